// gs_simt.cu -- fp32 CUDA-core kernels of the Gram-Space apply path.
//
// These kernels carry the small workloads (a handful of codewords, a few
// hundred queries: launch-latency bound) and the precise fp32 path that any
// shape can take (GS_PATH_SIMT).  The large-batch hot path is on tcgen05 in
// gs_tc.cu.
//
//  k_ps_small     fused project + similarity, 4 to 16 queries per block, r <= 32
//                 (Sec. 3.1 t = U^T x; Sec. 2.2 similarity; Eq. 2-3)
//  k_scores       similarity of Gram-loc queries (or of K-split partial sums of them), one warp per
//                 query, r <= 64 (Sec. 3.2, Eq. 2)
//  k_gemm         tiled fp32 GEMM with scale / cosine / bf16 epilogues; used for
//                 Y = X Q^T, S = Y R^T, V = P R (Sec. 2.2 / 3.3), Xhat = T Q
//                 (Sec. 3.1 / 3.3) and batched attention logits (Sec. 2.2)
//  k_row_finish   argmax / maxval / softmax over each score row
//  k_row_softmax  softmax over each attention row
//  k_rownorm      full-D query norms for cosine scores
//  k_group_argmax argmax / max of each score row within each group of a grouped codebook
//  k_bind16       block circular convolution / correlation (binding / unbinding), L % 16 == 0
//  k_bind8        the same for L % 8 == 0
//  k_bind_reg     the same for short blocks (L <= 32), one block per thread in registers
//  k_bind1        the same for any block length, one output per thread

#include <float.h>

#include <algorithm>

#include "gs_internal.h"

namespace gs {
namespace {

__device__ __forceinline__ float warp_sum(float v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_max(float v) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
// (value, index) argmax across a warp: larger value wins, lower index on ties.
__device__ __forceinline__ void warp_argmax(float& v, int& i) {
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, v, o);
        const int oi = __shfl_xor_sync(0xffffffffu, i, o);
        if (ov > v || (ov == v && oi < i)) {
            v = ov;
            i = oi;
        }
    }
}

// ----------------------------------------------------------------- scores of Gram-loc rows, r <= 64
constexpr int kCoefR = 64;
constexpr int kCoefWarps = 8;
constexpr int kRSmemFloats = 12 * 1024;  // codeword rows staged at a time: 48 KB

// p[0] + p[stride] + ... + p[(ks - 1) stride] in eight sums of every eighth term: their loads are in flight
// together, and the rounding grows with an eighth of the terms.
__device__ __forceinline__ float sum_parts(const float* __restrict__ p, long long stride, int ks) {
    float a[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) a[u] = u < ks ? p[u * stride] : 0.f;
    for (int z = 8; z < ks; z += 8) {
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (z + u < ks) a[u] += p[(z + u) * stride];
    }
    return ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
}

struct ScoreParams {
    const float* Y;       // N x r (ld ldy), or null: y_j = sum over z < ks (in a fixed order) of part[z][n][j]
    int ldy;
    const float* part;
    const float* xx;      // with part: ||x||^2 in ks parts (ks x N), or null
    int ks;
    const float* xnorm;   // with Y (optional): ||x_n||; otherwise ||y_n|| stands for it (Eq. 3)
    float* Yout;          // with part (optional): the Gram-loc rows
    int ldyo;
    long long N;
    int r;
    const float* R;
    int ldr, M;
    const float* cnorm;
    int mode;
    float scale;
    float* S;
    int lds;
    int* argmax;
    float* maxval;
    int chunk, pitch;     // codewords staged at a time, floats between their rows
};

// One warp per Gram-loc row, lane l scoring codewords l, l + 32, ...  R is staged in shared memory once
// per block (pitch: whole float4s, an odd number of them, so that a float4 from 32 consecutive rows
// falls in disjoint banks), the warp's row beside it: per codeword r / 4 conflict-free 16-byte reads and
// as many broadcasts.  Reading R's rows from global memory, a row per lane, took r loads of 32 lines
// each per codeword (8,000 rows x 16 codewords: 11.1 us, now 6.5; 1,024 x 40: 5.3, now 4.6).  A codebook past 48 KB goes through in chunks; softmax rows are then scored twice.
__global__ void __launch_bounds__(kCoefWarps * 32) k_scores(const ScoreParams p) {
    extern __shared__ float4 coef_sm[];
    float* Rs = reinterpret_cast<float*>(coef_sm);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float* ys = Rs + (size_t)p.chunk * p.pitch + warp * kCoefR;
    const int r4 = (p.r + 3) / 4;
    const bool whole = p.chunk >= p.M;  // one chunk: staged once, kept
    auto stage = [&](int i0) {
        const int n = min(p.chunk, p.M - i0);
        for (int e = threadIdx.x; e < n * 4 * r4; e += kCoefWarps * 32) {
            const int i = e / (4 * r4), j = e - i * 4 * r4;
            Rs[i * p.pitch + j] = j < p.r ? __ldg(p.R + (size_t)(i0 + i) * p.ldr + j) : 0.f;
        }
    };
    if (whole) {
        stage(0);
        __syncthreads();
    }
    const long long step = (long long)gridDim.x * kCoefWarps;
    const long long rounds = (p.N + step - 1) / step;
    for (long long it = 0; it < rounds; ++it) {
        const long long n = it * step + (long long)blockIdx.x * kCoefWarps + warp;
        const bool in = n < p.N;
        float ynorm = 0.f;
        __syncwarp();
        if (in) {
            float yy = 0.f;
            for (int j = lane; j < 4 * r4; j += 32) {
                float y = 0.f;
                if (j < p.r) {
                    if (p.part) {
                        y = sum_parts(p.part + n * p.r + j, p.N * p.r, p.ks);
                        if (p.Yout) p.Yout[(size_t)n * p.ldyo + j] = y;
                    } else {
                        y = __ldg(p.Y + (size_t)n * p.ldy + j);
                    }
                }
                ys[j] = y;
                yy = fmaf(y, y, yy);
            }
            if (p.mode == GS_SCORE_COSINE) {
                if (p.part) {
                    ynorm = sqrtf(sum_parts(p.xx + n, p.N, p.ks));
                } else {
                    ynorm = p.xnorm ? p.xnorm[n] : sqrtf(warp_sum(yy));
                }
            }
        }
        __syncwarp();
        const bool wanted = p.S || p.argmax || p.maxval;
        float bv = -FLT_MAX, m = -FLT_MAX, z = 0.f;
        int bi = 0x7fffffff;
        const bool soft = p.mode == GS_SCORE_SOFTMAX;
        const int sweeps = soft && p.S ? 2 : 1;
        float inv = 0.f;
        for (int sweep = 0; sweep < sweeps && wanted; ++sweep) {
            for (int i0 = 0; i0 < p.M; i0 += p.chunk) {
                if (!whole) {
                    __syncthreads();
                    stage(i0);
                    __syncthreads();
                }
                if (!in) continue;
                const int i1 = min(p.M, i0 + p.chunk);
                for (int i = i0 + lane; i < i1; i += 32) {
                    const float4* Ri = reinterpret_cast<const float4*>(Rs + (i - i0) * p.pitch);
                    const float4* yv = reinterpret_cast<const float4*>(ys);
                    float g = 0.f;
#pragma unroll 4
                    for (int q = 0; q < r4; ++q) {
                        const float4 a = yv[q], b = Ri[q];
                        g = fmaf(a.x, b.x, g);
                        g = fmaf(a.y, b.y, g);
                        g = fmaf(a.z, b.z, g);
                        g = fmaf(a.w, b.w, g);
                    }
                    g *= p.scale;
                    if (p.mode == GS_SCORE_COSINE) {
                        const float den = ynorm * p.cnorm[i];
                        g = den > 0.f ? g / den : 0.f;
                    }
                    if (sweep == 1) {
                        p.S[(size_t)n * p.lds + i] = __expf(g - m) * inv;
                        continue;
                    }
                    if (g > bv) {
                        bv = g;
                        bi = i;
                    }
                    if (soft) {
                        const float nm = fmaxf(m, g);
                        z = z * __expf(m - nm) + __expf(g - nm);
                        m = nm;
                    } else if (p.S) {
                        p.S[(size_t)n * p.lds + i] = g;
                    }
                }
            }
            if (sweep == 0 && soft && in) {  // the lanes' maxima and sums, merged
                const float mm = warp_max(m);
                inv = 1.f / warp_sum(z * __expf(m - mm));
                m = mm;
            }
        }
        if (!in || !wanted) continue;
        warp_argmax(bv, bi);
        if (bi == 0x7fffffff) bi = 0;
        if (lane == 0) {
            if (p.argmax) p.argmax[n] = bi;
            if (p.maxval) p.maxval[n] = soft ? inv : bv;  // the largest score's share is 1 / sum
        }
    }
}

// ----------------------------------------------------------------- fused project + score, r <= 32
// A block takes QB queries against the whole basis (RB >= r rows): chunks of 128 dimensions of both go
// through a cp.async ring, each of the eight warps takes 16 dimensions of a chunk for all
// QB x RB products (a lane QB / 4 x RB / 8 of them, 16-byte shared reads without conflicts), the warps'
// sums meet in shared memory, and the warps score the queries.  Bound by the loads' latency at the usual
// few hundred queries.  One warp per query read all of Q per query, 4 bytes a lane (2,048 queries of D =
// 1024, r = 30: 45 us, now 14.5; of D = 2560: 103, now 29); four queries' products in one warp's registers left
// few for loads in flight (19 and 57 us; at 512 queries, r = 10, it was the faster one, 5 us against 8).
constexpr int kSmallR = 32;
constexpr int kSmallM = 64;   // codewords kept in shared memory of their own
constexpr int kSmallKC = 128, kSmallPitch = kSmallKC + 4;
// ring depth: the few-query blocks have an SM each and are bound by latency alone
constexpr int small_stages(int qb) { return qb == 4 ? 8 : 4; }

__device__ __forceinline__ void cp_async_zfill16(float* dst, const float* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_zfill4(float* dst, const float* src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ float dot4(const float4& a, const float4& b) {
    return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, a.w * b.w)));
}

// BIG: more than kSmallM codewords (a template parameter: the usual small codebooks' kernel keeps its registers)
template <int QB, int RB, bool VEC, bool BIG>
__global__ void __launch_bounds__(256) k_ps_small(const float* __restrict__ X, long long N, int ldx, int D,
                                                  const float* __restrict__ Q, int r, const float* __restrict__ R,
                                                  int ldr, int M, const float* __restrict__ cnorm, int mode,
                                                  float scale, float* __restrict__ Y, int ldy, float* __restrict__ S,
                                                  int lds, int* __restrict__ argmax, float* __restrict__ maxval) {
    constexpr int NQ = QB / 4, NJ = RB / 8, kRows = QB + RB, kSmallStages = small_stages(QB);
    extern __shared__ float4 small_sm[];
    float* ring = reinterpret_cast<float*>(small_sm);  // kSmallStages x kRows rows: the queries, then Q
    __shared__ float ysm[QB][kSmallR], xsm[QB];
    __shared__ float Rs[BIG ? 1 : kSmallM][kSmallR + 1];  // the codewords, odd pitch: a row per lane
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long n0 = (long long)blockIdx.x * QB;
    const int nch = (D + kSmallKC - 1) / kSmallKC;
    auto fetch = [&](int c) {
        float* st = ring + (size_t)(c % kSmallStages) * kRows * kSmallPitch;
        constexpr int W = VEC ? 4 : 1, kPer = kSmallKC / W;
        for (int e = threadIdx.x; e < kRows * kPer; e += 256) {
            const int row = e / kPer, d = e % kPer * W, gd = c * kSmallKC + d;
            // rows past the end: any valid one, whose sums nobody reads; past D: zeros
            const float* src = row < QB ? X + (size_t)(n0 + row < N ? n0 + row : N - 1) * ldx
                                        : Q + (size_t)(row - QB < r ? row - QB : 0) * D;
            const int left = min(W, max(0, D - gd));
            float* dst = st + row * kSmallPitch + d;
            if (VEC)
                cp_async_zfill16(dst, src + (left ? gd : 0), 4 * left);
            else
                cp_async_zfill4(dst, src + (left ? gd : 0), 4 * left);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int c = 0; c < kSmallStages - 1; ++c) {
        if (c < nch) fetch(c);
        else asm volatile("cp.async.commit_group;" ::: "memory");
    }
    if (!BIG)  // in flight under the projection
        for (int e = threadIdx.x; e < M * RB; e += 256) {
            const int i = e / RB, j = e % RB;
            Rs[i][j] = j < r ? __ldg(R + (size_t)i * ldr + j) : 0.f;
        }
    const int jg = lane & 7, qg = lane >> 3;  // queries qg + 4 v, basis rows jg + 8 u
    float acc[NQ][NJ] = {}, xx[NQ] = {};
    for (int c = 0; c < nch; ++c) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kSmallStages - 2) : "memory");
        __syncthreads();  // chunk c is here for every thread, and chunk c - 1's stage has been read
        if (c + kSmallStages - 1 < nch) fetch(c + kSmallStages - 1);
        else asm volatile("cp.async.commit_group;" ::: "memory");
        const float* st = ring + (size_t)(c % kSmallStages) * kRows * kSmallPitch + 16 * warp;
        // a chunk's 16 terms are summed by themselves, by fours: chains of 4, 4 and D / 128 steps (one chain
        // of D / 8 lost up to twice as much; 28.5 against 28.0 us for 2,048 queries of D = 2560)
        float part[NQ][NJ] = {}, px[NQ] = {};
#pragma unroll
        for (int k = 0; k < 16; k += 4) {
            float4 x[NQ], q[NJ];
#pragma unroll
            for (int v = 0; v < NQ; ++v) x[v] = *reinterpret_cast<const float4*>(st + (qg + 4 * v) * kSmallPitch + k);
#pragma unroll
            for (int u = 0; u < NJ; ++u) q[u] = *reinterpret_cast<const float4*>(st + (QB + jg + 8 * u) * kSmallPitch + k);
#pragma unroll
            for (int v = 0; v < NQ; ++v) {
                px[v] += dot4(x[v], x[v]);
#pragma unroll
                for (int u = 0; u < NJ; ++u) part[v][u] += dot4(x[v], q[u]);
            }
        }
#pragma unroll
        for (int v = 0; v < NQ; ++v) {
            xx[v] += px[v];
#pragma unroll
            for (int u = 0; u < NJ; ++u) acc[v][u] += part[v][u];
        }
    }
    // the warps' sums, through the ring's memory: [warp][query][RB + 1], the last the squared norm
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    float* red = ring;
#pragma unroll
    for (int v = 0; v < NQ; ++v) {
        float* row = red + ((size_t)warp * QB + qg + 4 * v) * (RB + 1);
#pragma unroll
        for (int u = 0; u < NJ; ++u) row[jg + 8 * u] = acc[v][u];
        if (jg == 0) row[RB] = xx[v];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < QB * (RB + 1); e += 256) {
        const int qi = e / (RB + 1), j = e - qi * (RB + 1);
        const float t = sum_parts(red + qi * (RB + 1) + j, QB * (RB + 1), 8);
        if (j == RB) {
            xsm[qi] = t;
        } else {
            ysm[qi][j] = t;
            if (Y && j < r && n0 + qi < N) Y[(size_t)(n0 + qi) * ldy + j] = t;
        }
    }
    __syncthreads();
    if (BIG) {
        // the codebook goes through the ring's memory, as much of it at a time as fits (read in place, a row per lane
        // and r loads of 32 lines a codeword: 20,000 queries of D = 256, r = 20 against 700 codewords 269 us, 772
        // with the softmax and scores; 97 and 202 so)
        constexpr int NW = (QB + 7) / 8;  // queries of a warp
        constexpr int kCap = kSmallStages * kRows * kSmallPitch / (RB + 1) / 32 * 32;
        const int passes = mode != GS_SCORE_SOFTMAX ? 1 : S ? 3 : 2;
        float bv[NW], z[NW];
        int bi[NW];
#pragma unroll
        for (int v = 0; v < NW; ++v) bv[v] = -FLT_MAX, z[v] = 0.f, bi[v] = 0x7fffffff;
        for (int pass = 0; pass < passes; ++pass) {
            for (int i0 = 0; i0 < M; i0 += kCap) {
                const int nc = min(kCap, M - i0);
                if (pass == 0 || M > kCap) {
                    __syncthreads();  // every warp is through with the last chunk
                    for (int e = threadIdx.x; e < nc * RB; e += 256) {
                        const int i = e / RB, j = e % RB;
                        ring[i * (RB + 1) + j] = j < r ? __ldg(R + (size_t)(i0 + i) * ldr + j) : 0.f;
                    }
                    __syncthreads();
                }
#pragma unroll
                for (int v = 0; v < NW; ++v) {
                    const int qi = warp + 8 * v;
                    if (qi >= QB || n0 + qi >= N) continue;
                    const long long n = n0 + qi;
                    const float xnorm = sqrtf(xsm[qi]);
                    float y[RB];
#pragma unroll
                    for (int j = 0; j < RB; ++j) y[j] = j < r ? ysm[qi][j] : 0.f;
                    for (int c = lane; c < nc; c += 32) {
                        const int i = i0 + c;
                        float g = 0.f;
#pragma unroll
                        for (int j = 0; j < RB; ++j) g = fmaf(y[j], ring[c * (RB + 1) + j], g);
                        g *= scale;
                        if (mode == GS_SCORE_COSINE) {
                            const float den = xnorm * cnorm[i];
                            g = den > 0.f ? g / den : 0.f;
                        }
                        if (pass == 0) {
                            if (g > bv[v]) {
                                bv[v] = g;
                                bi[v] = i;
                            }
                            if (S && mode != GS_SCORE_SOFTMAX) S[(size_t)n * lds + i] = g;
                        } else if (pass == 1) {
                            z[v] += __expf(g - bv[v]);
                        } else {
                            S[(size_t)n * lds + i] = __expf(g - bv[v]) * z[v];
                        }
                    }
                }
            }
#pragma unroll
            for (int v = 0; v < NW; ++v) {
                if (pass == 0) warp_argmax(bv[v], bi[v]);
                if (pass == 1) z[v] = 1.f / warp_sum(z[v]);
            }
        }
#pragma unroll
        for (int v = 0; v < NW; ++v) {
            const int qi = warp + 8 * v;
            if (lane != 0 || qi >= QB || n0 + qi >= N) continue;
            if (argmax) argmax[n0 + qi] = bi[v] == 0x7fffffff ? 0 : bi[v];
            if (maxval) maxval[n0 + qi] = mode == GS_SCORE_SOFTMAX ? z[v] : bv[v];
        }
        return;
    }
    for (int qi = warp; qi < QB; qi += 8) {
        const long long n = n0 + qi;
        if (n >= N) break;
        float y[RB];
#pragma unroll
        for (int j = 0; j < RB; ++j) y[j] = j < r ? ysm[qi][j] : 0.f;
        const float x2 = xsm[qi];
        const float xnorm = sqrtf(x2);
        // scores: lane handles codewords i = lane, lane + 32, ...
        auto score = [&](int i) {
            float g = 0.f;
#pragma unroll
            for (int j = 0; j < RB; ++j) g = fmaf(y[j], Rs[i][j], g);
            g *= scale;
            if (mode == GS_SCORE_COSINE) {
                const float den = xnorm * cnorm[i];
                g = den > 0.f ? g / den : 0.f;
            }
            return g;
        };
        float bv = -FLT_MAX;
        int bi = 0x7fffffff;
        for (int i = lane; i < M; i += 32) {
            const float g = score(i);
            if (g > bv) {
                bv = g;
                bi = i;
            }
            if (S && mode != GS_SCORE_SOFTMAX) S[(size_t)n * lds + i] = g;
        }
        warp_argmax(bv, bi);
        if (bi == 0x7fffffff) bi = 0;
        float outmax = bv;
        if (mode == GS_SCORE_SOFTMAX) {
            float z = 0.f;
            for (int i = lane; i < M; i += 32) z += __expf(score(i) - bv);
            z = warp_sum(z);
            const float inv = 1.f / z;
            if (S)
                for (int i = lane; i < M; i += 32) S[(size_t)n * lds + i] = __expf(score(i) - bv) * inv;
            outmax = inv;
        }
        if (lane == 0) {
            if (argmax) argmax[n] = M > 0 ? bi : 0;
            if (maxval) maxval[n] = M > 0 ? outmax : 0.f;
        }
    }
}

// ----------------------------------------------------------------- tiled GEMM
// 256 threads, each MT x 4 outputs: tiles of 16 MT x 64 (MT = 8 reads 3 shared vectors per 32 FMAs, MT = 4
// two per 16; the smaller tile where the larger would leave SMs without work)
constexpr int kTN = 64, kTK = 16;
constexpr int kTM = 64;  // MT = 4

template <int T>
__device__ __forceinline__ float ld_elem(const void* p, long long i) {
    if (T == MAT_F32) return __ldg((const float*)p + i);
    return __bfloat162float(((const __nv_bfloat16*)p)[i]);
}

// Four consecutive elements i .. i + 3 of a row, those at or past `left` zero; vec: one 16-byte load
template <int T>
__device__ __forceinline__ void ld4(const void* p, long long i, int left, bool vec, float (&v)[4]) {
    if (T == MAT_F32 && vec && left >= 4) {
        const float4 x = __ldg(reinterpret_cast<const float4*>((const float*)p + i));
        v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
        return;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = u < left ? ld_elem<T>(p, i + u) : 0.f;
}

// One 64 x 64 output tile (rows m0.., columns n0..) of batch b, or of K chunk kz with ksplit;
// called by every thread of the block.  A thread loads four consecutive elements of each operand per
// K step (one 16-byte load where rows are aligned), the next step's while the current one is multiplied
// (two shared buffers, one barrier a step).  16,384 x 922 -> 10,000: 8,240 us with scalar loads and nothing in
// flight (37 TFLOP/s), 6,750 us here (45); 1,024 x 40 over K = 8192, summed and scored: 51, now 38.
template <int TA, int TB, int TC, bool BT, int MT>
__device__ __forceinline__ void gemm_tile(const GemmArgs& g, long long m0, int n0, int kz,
                                          float (&As)[2][kTK][16 * MT + 4], float (&Bs)[2][kTK][kTN + 4]) {
    const int tid = threadIdx.x;
    const int tx = tid % 16, ty = tid / 16;
    const bool split = g.ksplit > 1;
    const int b = split ? 0 : kz;
    const char* Ab = (const char*)g.A + (size_t)b * g.a_bstride * (TA == MAT_F32 ? 4 : 2);
    const char* Bb = (const char*)g.B + (size_t)b * g.b_bstride * (TB == MAT_F32 ? 4 : 2);
    int kend = g.k;
    if (BT && g.b_rowlen) {
        // rows n0..n0+63 of B are zero beyond their row length: stop at the max
        int mx = 0;
        for (int j = tid; j < kTN; j += 256)
            if (n0 + j < g.n) mx = max(mx, g.b_rowlen[n0 + j]);
        for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        __shared__ int smx[8];
        if ((tid & 31) == 0) smx[tid >> 5] = mx;
        __syncthreads();
        mx = 0;
        for (int w = 0; w < 8; ++w) mx = max(mx, smx[w]);
        kend = min(kend, mx);
    }
    int kbeg = 0;
    if (split) {  // this block's chunk of K (chunks are whole kTK steps)
        const int chunk = ((g.k + g.ksplit - 1) / g.ksplit + kTK - 1) / kTK * kTK;
        kbeg = kz * chunk;
        kend = min(kend, kbeg + chunk);
    }
    // A: row lr, k lk .. lk + 3 of the step; B the same (K-major), or k br, columns bc .. bc + 3
    const int lr = tid / 4, lk = tid % 4 * 4, br = tid / 16, bc = tid % 16 * 4;
    constexpr int AR = MT / 4;  // rows lr, lr + 64 of A
    long long arow[AR];
    bool a_in[AR];
#pragma unroll
    for (int h = 0; h < AR; ++h) {
        const long long gm = m0 + lr + 64 * h;
        a_in[h] = gm < g.m;
        arow[h] = (a_in[h] ? gm : g.m - 1) * g.lda;
    }
    const bool b_in = n0 + lr < g.n;
    const long long brow = BT ? (long long)(b_in ? n0 + lr : g.n - 1) * g.ldb : 0;
    // bf16 operands, which no 16-byte load takes here: consecutive threads on consecutive elements, k sk of rows sr +
    // 16 t (four of a row each: 64 x 64 x 1,100 x 128 53 us, 46 so)
    const int sr = tid / 16, sk = tid % 16;
    const int rows = (int)(g.m - m0 < 16 * MT ? g.m - m0 : 16 * MT), cols = min(kTN, g.n - n0);
    float av[AR][4], bv[4], xx[AR] = {};
    auto load = [&](int k0) {
        if (TA == MAT_F32) {
#pragma unroll
            for (int h = 0; h < AR; ++h) ld4<TA>(Ab, arow[h] + k0 + lk, a_in[h] ? kend - (k0 + lk) : 0, g.a_vec, av[h]);
        } else {
#pragma unroll
            for (int t = 0; t < 4 * AR; ++t)
                av[t / 4][t % 4] = sr + 16 * t < rows && k0 + sk < kend ? ld_elem<TA>(Ab, (m0 + sr + 16 * t) * g.lda + k0 + sk) : 0.f;
        }
        if (TB == MAT_BF16) {  // (n x k)
#pragma unroll
            for (int t = 0; t < 4; ++t)
                bv[t] = sr + 16 * t < cols && k0 + sk < kend ? ld_elem<TB>(Bb, (long long)(n0 + sr + 16 * t) * g.ldb + k0 + sk) : 0.f;
        } else if (BT)
            ld4<TB>(Bb, brow + k0 + lk, b_in ? kend - (k0 + lk) : 0, g.b_vec, bv);
        else
            ld4<TB>(Bb, (long long)(k0 + br) * g.ldb + n0 + bc, k0 + br < kend ? g.n - (n0 + bc) : 0, g.b_vec, bv);
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
#pragma unroll
            for (int h = 0; h < AR; ++h) {
                if (TA == MAT_F32) {
                    As[buf][lk + u][lr + 64 * h] = av[h][u];
                    xx[h] = fmaf(av[h][u], av[h][u], xx[h]);
                } else {
                    As[buf][sk][sr + 16 * (4 * h + u)] = av[h][u];
                }
            }
            if (TB == MAT_BF16) Bs[buf][sk][sr + 16 * u] = bv[u];
            else if (BT) Bs[buf][lk + u][lr] = bv[u];
        }
        if (!BT) *reinterpret_cast<float4*>(&Bs[buf][br][bc]) = make_float4(bv[0], bv[1], bv[2], bv[3]);
    };
    float acc[MT][4] = {};
    if (kbeg < kend) {
        load(kbeg);
        store(0);
    }
    __syncthreads();
    int buf = 0;
    for (int k0 = kbeg; k0 < kend; k0 += kTK, buf ^= 1) {
        const bool more = k0 + kTK < kend;
        if (more) load(k0 + kTK);
#pragma unroll
        for (int kk = 0; kk < kTK; ++kk) {
            float a[MT];
#pragma unroll
            for (int h = 0; h < AR; ++h)
                *reinterpret_cast<float4*>(a + 4 * h) = *reinterpret_cast<const float4*>(&As[buf][kk][ty * 4 + 64 * h]);
            const float4 b4 = *reinterpret_cast<const float4*>(&Bs[buf][kk][tx * 4]);
            const float bb[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], bb[j], acc[i][j]);
        }
        if (more) store(buf ^ 1);
        __syncthreads();
    }
    if (g.xx_part && n0 == 0) {  // this chunk's part of each row's squared norm
#pragma unroll
        for (int h = 0; h < AR; ++h) {
            float x = xx[h];
            x += __shfl_xor_sync(0xffffffffu, x, 1);
            x += __shfl_xor_sync(0xffffffffu, x, 2);
            if (lk == 0 && a_in[h]) g.xx_part[(size_t)kz * g.m + m0 + lr + 64 * h] = x;
        }
    }
    char* Cb = (char*)g.C + (size_t)b * g.c_bstride * (TC == MAT_F32 ? 4 : 2);
#pragma unroll
    for (int i = 0; i < MT; ++i) {
        const long long gi = m0 + ty * 4 + 64 * (i / 4) + i % 4;
        if (gi >= g.m) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int gn = n0 + tx * 4 + j;
            if (gn >= g.n) continue;
            float v = g.alpha * acc[i][j];
            if (g.rownorm) {
                const float den = g.rownorm[gi] * g.colnorm[gn];
                v = den > 0.f ? v / den : 0.f;
            }
            if (TC == MAT_F32) {
                if (g.kpart) g.kpart[((size_t)kz * g.m + gi) * g.n + gn] = v;
                else ((float*)Cb)[gi * g.ldc + gn] = v;
            } else {
                ((__nv_bfloat16*)Cb)[gi * g.ldc + gn] = __float2bfloat16_rn(v);
            }
        }
    }
}

template <int TA, int TB, int TC, bool BT, int MT>
__global__ void __launch_bounds__(256, MT == 8 ? 3 : 4) k_gemm(GemmArgs g) {
    __shared__ __align__(16) float As[2][kTK][16 * MT + 4];
    __shared__ __align__(16) float Bs[2][kTK][kTN + 4];
    gemm_tile<TA, TB, TC, BT, MT>(g, (long long)blockIdx.y * (16 * MT), blockIdx.x * kTN, blockIdx.z, As, Bs);
}

// The gated product (gate_xn2): each block takes a run of consecutive 64 x 64 tiles, n fastest, and
// computes only those whose 64 rows hold a selected row.  It looks at all its rows first (a run spans few
// row blocks), so with no such row the launch is one round of loads and a barrier (12 us before, with a
// barrier per tile: 16,384 x 922; 3.6 now).
template <int TA, int TB, int TC, bool BT>
__global__ void __launch_bounds__(256) k_gemm_gated(GemmArgs g, long long per) {
    __shared__ __align__(16) float As[2][kTK][kTM + 4];
    __shared__ __align__(16) float Bs[2][kTK][kTN + 4];
    const int tiles_n = (g.n + kTN - 1) / kTN;
    const long long tiles = (g.m + kTM - 1) / kTM * tiles_n;
    const long long t0 = (long long)blockIdx.x * per, t1 = t0 + per < tiles ? t0 + per : tiles;
    if (t0 >= t1) return;
    auto selected = [&](long long i) {
        const float xn2 = g.gate_xn2[i] + g.gate_xn2[g.gate_ld + i];
        return xn2 > 0.f && !(xn2 >= g.gate_lo && xn2 <= g.gate_hi);
    };
    const long long r0 = t0 / tiles_n * kTM, r1 = (t1 - 1) / tiles_n * kTM + kTM;
    bool mine = false;
    for (long long i = r0 + threadIdx.x; i < r1 && i < g.m; i += 256) mine |= selected(i);
    if (!__syncthreads_or(mine)) return;
    long long last_m0 = -1;
    bool any = false;
    for (long long t = t0; t < t1; ++t) {
        const long long m0 = t / tiles_n * kTM;
        if (m0 != last_m0) {
            mine = threadIdx.x < kTM && m0 + threadIdx.x < g.m && selected(m0 + threadIdx.x);
            any = __syncthreads_or(mine) != 0;
            last_m0 = m0;
        }
        if (any) gemm_tile<TA, TB, TC, BT, 4>(g, m0, (int)(t % tiles_n) * kTN, 0, As, Bs);
    }
}

// C[i][j] = sum over z (in a fixed order) of part[z][i][j]: the split-K partials of k_gemm
__global__ void k_ksum(const float* __restrict__ part, int ks, long long m, int n, float* __restrict__ C,
                       long long ldc) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= m * n) return;
    C[(idx / n) * ldc + idx % n] = sum_parts(part + idx, m * n, ks);
}

// ----------------------------------------------------------------- row kernels
__global__ void __launch_bounds__(256) k_row_finish(float* __restrict__ S, long long N, int M,
                                                     int lds, int softmax, int* __restrict__ argmax,
                                                     float* __restrict__ maxval) {
    const int lane = threadIdx.x & 31;
    const long long n = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (n >= N) return;
    float* s = S + (size_t)n * lds;
    float bv = -FLT_MAX;
    int bi = 0x7fffffff;
    for (int i = lane; i < M; i += 32) {
        const float g = s[i];
        if (g > bv) {
            bv = g;
            bi = i;
        }
    }
    warp_argmax(bv, bi);
    if (bi == 0x7fffffff) bi = 0;
    float outmax = bv;
    if (softmax) {
        float z = 0.f;
        for (int i = lane; i < M; i += 32) z += __expf(s[i] - bv);
        z = warp_sum(z);
        const float inv = 1.f / z;
        for (int i = lane; i < M; i += 32) s[i] = __expf(s[i] - bv) * inv;
        outmax = inv;
    }
    if (lane == 0) {
        if (argmax) argmax[n] = M > 0 ? bi : 0;
        if (maxval) maxval[n] = M > 0 ? outmax : 0.f;
    }
}

__global__ void __launch_bounds__(256) k_row_softmax(float* __restrict__ A, long long rows, int L,
                                                      long long ld) {
    const int lane = threadIdx.x & 31;
    const long long n = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (n >= rows) return;
    float* a = A + (size_t)n * ld;
    float mx = -FLT_MAX;
    for (int i = lane; i < L; i += 32) mx = fmaxf(mx, a[i]);
    mx = warp_max(mx);
    float z = 0.f;
    for (int i = lane; i < L; i += 32) z += __expf(a[i] - mx);
    z = warp_sum(z);
    const float inv = 1.f / z;
    for (int i = lane; i < L; i += 32) a[i] = __expf(a[i] - mx) * inv;
}

__global__ void __launch_bounds__(256) k_rownorm(const float* __restrict__ X, long long N, int ldx,
                                                  int D, float* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    const long long n = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (n >= N) return;
    const float* x = X + (size_t)n * ldx;
    float s = 0.f;
    for (int d = lane; d < D; d += 32) s = fmaf(x[d], x[d], s);
    s = warp_sum(s);
    if (lane == 0) out[n] = sqrtf(s);
}

// Column ranges of the groups of a grouped codebook, passed by value.
struct GroupOffsets {
    int G;
    int off[kMaxGroups + 1];
};

// one warp per score row: for each group, the max over its columns and the index (within
// the group) of its first occurrence
__global__ void __launch_bounds__(256) k_group_argmax(const float* __restrict__ S, long long N, int lds,
                                                       const GroupOffsets go, int* __restrict__ argmax,
                                                       float* __restrict__ maxval) {
    const int lane = threadIdx.x & 31;
    const long long n = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (n >= N) return;
    const float* s = S + (size_t)n * lds;
    for (int g = 0; g < go.G; ++g) {
        const int c0 = go.off[g], c1 = go.off[g + 1];
        float bv = -INFINITY;
        int bi = c1;
        for (int j = c0 + lane; j < c1; j += 32) {
            const float v = s[j];
            if (v > bv) {  // columns rise with j: the first of equal values stays
                bv = v;
                bi = j;
            }
        }
        warp_argmax(bv, bi);
        if (lane == 0) {
            if (argmax) argmax[(size_t)n * go.G + g] = bi - c0;
            if (maxval) maxval[(size_t)n * go.G + g] = bv;
        }
    }
}

// Binding (UNB = false: Z_k = sum_j X_j Y_(k-j mod L)) or unbinding (UNB = true:
// Z_k = sum_j X_j Y_(j-k mod L)) within blocks of L components.  A CTA takes one block of
// 256 / tpr rows (tpr = min(L / 8, 256) threads per row) and stages the rows' X and Y
// blocks in shared memory, Y index-reversed for unbinding (Y'_m = Y_(-m mod L) turns the
// correlation into a convolution).  A thread computes eight consecutive outputs
// k0..k0+7: per eight-wide step of j it reads X_j..X_(j+7) (the same words for the whole
// row: broadcast) and the sixteen Y' values (k0 - j - 8 .. k0 - j + 7) mod L -- two aligned
// chunks, since L, k0 and j are multiples of 8 -- and does 64 fma.  ldy = 0: one partner row.
template <bool UNB>
__global__ void __launch_bounds__(256) k_bind8(const float* __restrict__ X, long long N, int ldx,
                                                const float* __restrict__ Y, long long ldy, int L,
                                                float* __restrict__ Z, int ldz, int zvec) {
    extern __shared__ float4 bind_sm[];
    const int tpr = min(L >> 3, 256);
    const int rpc = 256 / tpr;
    const int tr = threadIdx.x / tpr, tk = threadIdx.x - tr * tpr;
    const long long n = (long long)blockIdx.x * rpc + tr;
    const int b0 = blockIdx.y * L;
    float* xs = reinterpret_cast<float*>(bind_sm) + (size_t)tr * 2 * L;
    float* ys = xs + L;
    if (tr < rpc && n < N) {
        const float* x = X + (size_t)n * ldx + b0;
        const float* y = Y + (size_t)n * ldy + b0;
        for (int j = tk; j < L; j += tpr) {
            xs[j] = x[j];
            ys[j] = y[UNB ? (j == 0 ? 0 : L - j) : j];
        }
    }
    __syncthreads();
    if (tr >= rpc || n >= N) return;
    for (int k0 = 8 * tk; k0 < L; k0 += 8 * tpr) {
        float z[8];
#pragma unroll
        for (int t = 0; t < 8; ++t) z[t] = 0.f;
        for (int j = 0; j < L; j += 8) {
            int a = k0 - j - 8;
            if (a < 0) a += L;
            const int c = a + 8 == L ? 0 : a + 8;
            float xv[8], w[16];
            *reinterpret_cast<float4*>(xv) = *reinterpret_cast<const float4*>(xs + j);
            *reinterpret_cast<float4*>(xv + 4) = *reinterpret_cast<const float4*>(xs + j + 4);
            *reinterpret_cast<float4*>(w) = *reinterpret_cast<const float4*>(ys + a);
            *reinterpret_cast<float4*>(w + 4) = *reinterpret_cast<const float4*>(ys + a + 4);
            *reinterpret_cast<float4*>(w + 8) = *reinterpret_cast<const float4*>(ys + c);
            *reinterpret_cast<float4*>(w + 12) = *reinterpret_cast<const float4*>(ys + c + 4);
#pragma unroll
            for (int u = 0; u < 8; ++u)
#pragma unroll
                for (int t = 0; t < 8; ++t) z[t] = fmaf(xv[u], w[8 + t - u], z[t]);
        }
        float* zo = Z + (size_t)n * ldz + b0 + k0;
        if (zvec) {
            reinterpret_cast<float4*>(zo)[0] = make_float4(z[0], z[1], z[2], z[3]);
            reinterpret_cast<float4*>(zo)[1] = make_float4(z[4], z[5], z[6], z[7]);
        } else {
#pragma unroll
            for (int t = 0; t < 8; ++t) zo[t] = z[t];
        }
    }
}

// The same with 16 x 16 register tiles (L % 16 == 0): a thread computes 16 consecutive
// outputs; per 16-wide step of j it reads X_j..X_(j+15) (broadcast within the row) and the
// 32 Y' values (k0 - j - 16 .. k0 - j + 15) mod L as two aligned 16-value segments, and does
// 256 fma.  Y' is stored with 4 words of padding after every 16 (segment i at word 20 i), so
// the segments of consecutive threads, 64 bytes apart unpadded, fall in disjoint banks.
template <bool UNB>
__global__ void __launch_bounds__(256) k_bind16(const float* __restrict__ X, long long N, int ldx,
                                                 const float* __restrict__ Y, long long ldy, int L,
                                                 float* __restrict__ Z, int ldz, int zvec) {
    extern __shared__ float4 bind_sm16[];
    const int tpr = min(L >> 4, 256);
    const int rpc = 256 / tpr;
    const int tr = threadIdx.x / tpr, tk = threadIdx.x - tr * tpr;
    const long long n = (long long)blockIdx.x * rpc + tr;
    const int b0 = blockIdx.y * L;
    const int Lp = L + (L >> 2);  // padded length of Y'
    float* xs = reinterpret_cast<float*>(bind_sm16) + (size_t)tr * (L + Lp);
    float* ys = xs + L;
    if (tr < rpc && n < N) {
        const float* x = X + (size_t)n * ldx + b0;
        const float* y = Y + (size_t)n * ldy + b0;
        for (int j = tk; j < L; j += tpr) {
            xs[j] = x[j];
            ys[j + (j >> 4) * 4] = y[UNB ? (j == 0 ? 0 : L - j) : j];
        }
    }
    __syncthreads();
    if (tr >= rpc || n >= N) return;
    for (int k0 = 16 * tk; k0 < L; k0 += 16 * tpr) {
        float z[16];
#pragma unroll
        for (int t = 0; t < 16; ++t) z[t] = 0.f;
        for (int j = 0; j < L; j += 16) {
            int a = k0 - j - 16;
            if (a < 0) a += L;
            const int c = a + 16 == L ? 0 : a + 16;
            float xv[16], w[32];
            const float* sa = ys + a + (a >> 2);
            const float* sc = ys + c + (c >> 2);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                *reinterpret_cast<float4*>(xv + 4 * q) = *reinterpret_cast<const float4*>(xs + j + 4 * q);
                *reinterpret_cast<float4*>(w + 4 * q) = *reinterpret_cast<const float4*>(sa + 4 * q);
                *reinterpret_cast<float4*>(w + 16 + 4 * q) = *reinterpret_cast<const float4*>(sc + 4 * q);
            }
#pragma unroll
            for (int u = 0; u < 16; ++u)
#pragma unroll
                for (int t = 0; t < 16; ++t) z[t] = fmaf(xv[u], w[16 + t - u], z[t]);
        }
        float* zo = Z + (size_t)n * ldz + b0 + k0;
        if (zvec) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                reinterpret_cast<float4*>(zo)[q] = make_float4(z[4 * q], z[4 * q + 1], z[4 * q + 2], z[4 * q + 3]);
        } else {
#pragma unroll
            for (int t = 0; t < 16; ++t) zo[t] = z[t];
        }
    }
}

// Short blocks (L <= 32, L % 4 == 0): one thread per block, its X and Y blocks in registers
// (float4 loads when every row start is 16-byte aligned), L sums of L products in j order;
// consecutive threads take consecutive blocks of a row, so a warp's loads and stores are
// contiguous.  The tiled kernels above would give each row's few outputs a thread group of
// their own and read rows 4 L bytes at a time.
template <int L, bool UNB>
__global__ void __launch_bounds__(256) k_bind_reg(const float* __restrict__ X, long long N, int nb, int ldx,
                                                   const float* __restrict__ Y, long long ldy,
                                                   float* __restrict__ Z, int ldz, int vec) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= N * nb) return;
    const long long n = e / nb;
    const int b = (int)(e - n * nb);
    const float* x = X + (size_t)n * ldx + (size_t)b * L;
    const float* y = Y + (size_t)n * ldy + (size_t)b * L;
    float* z = Z + (size_t)n * ldz + (size_t)b * L;
    float xv[L], yv[L], zv[L];
    if (vec) {
#pragma unroll
        for (int q = 0; q < L / 4; ++q) {
            const float4 a = __ldcs(reinterpret_cast<const float4*>(x) + q);
            const float4 c = __ldg(reinterpret_cast<const float4*>(y) + q);
            xv[4 * q] = a.x, xv[4 * q + 1] = a.y, xv[4 * q + 2] = a.z, xv[4 * q + 3] = a.w;
            yv[4 * q] = c.x, yv[4 * q + 1] = c.y, yv[4 * q + 2] = c.z, yv[4 * q + 3] = c.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < L; ++j) {
            xv[j] = x[j];
            yv[j] = y[j];
        }
    }
#pragma unroll
    for (int k = 0; k < L; ++k) {
        float acc = 0.f;
#pragma unroll
        for (int j = 0; j < L; ++j) acc = fmaf(xv[j], yv[UNB ? (j - k + L) % L : (k - j + L) % L], acc);
        zv[k] = acc;
    }
    if (vec) {
#pragma unroll
        for (int q = 0; q < L / 4; ++q)
            __stcs(reinterpret_cast<float4*>(z) + q, make_float4(zv[4 * q], zv[4 * q + 1], zv[4 * q + 2], zv[4 * q + 3]));
    } else {
#pragma unroll
        for (int k = 0; k < L; ++k) z[k] = zv[k];
    }
}

// Any block length: one thread per output, operands read through the cache.
template <bool UNB>
__global__ void __launch_bounds__(256) k_bind1(const float* __restrict__ X, long long N, int D, int ldx,
                                                const float* __restrict__ Y, long long ldy, int L,
                                                float* __restrict__ Z, int ldz) {
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= N * D) return;
    const long long n = e / D;
    const int d = (int)(e - n * D);
    const int b0 = d - d % L, k = d - b0;
    const float* x = X + (size_t)n * ldx + b0;
    const float* y = Y + (size_t)n * ldy + b0;
    float acc = 0.f;
    for (int j = 0; j < L; ++j) {
        int m = UNB ? j - k : k - j;
        if (m < 0) m += L;
        acc = fmaf(x[j], y[m], acc);
    }
    Z[(size_t)n * ldz + d] = acc;
}

inline unsigned rows_grid(long long n) { return (unsigned)((n + 7) / 8); }

}  // namespace

cudaError_t launch_ps_small(const float* X, long long N, int ldx, int D, const float* Q, int r,
                            const float* R, int ldr, int M, const float* cnorm, int mode, float scale,
                            float* Y, int ldy, float* S, int lds, int* argmax, float* maxval,
                            cudaStream_t s) {
    const bool vec = (uintptr_t)X % 16 == 0 && ldx % 4 == 0 && D % 4 == 0 && (uintptr_t)Q % 16 == 0;
    // queries per block: few while blocks are fewer than the SMs, more once they queue (each block
    // reads all of Q)
    const int qb = N <= 4 * 152 ? 4 : N <= 16 * 152 ? 8 : 16;
    const int rb = r <= 8 ? 8 : r <= 16 ? 16 : 32;
    const size_t smem = sizeof(float) * std::max((size_t)small_stages(qb) * (qb + rb) * kSmallPitch, (size_t)8 * qb * (rb + 1));
    const unsigned blocks = (unsigned)((N + qb - 1) / qb);
    static bool opted[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
#define GS_SMALL_CASE(QB, RB)                                                                          \
    if (!opted[dev])                                                                                   \
        for (auto fn : {k_ps_small<QB, RB, true, false>, k_ps_small<QB, RB, false, false>,             \
                        k_ps_small<QB, RB, true, true>, k_ps_small<QB, RB, false, true>}) {            \
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);     \
            if (e != cudaSuccess) return e;                                                            \
        }                                                                                              \
    if (qb == QB && rb == RB)                                                                          \
        kern = M <= kSmallM ? (vec ? k_ps_small<QB, RB, true, false> : k_ps_small<QB, RB, false, false>) \
                            : (vec ? k_ps_small<QB, RB, true, true> : k_ps_small<QB, RB, false, true>);
    auto kern = k_ps_small<4, 8, true, false>;
    GS_SMALL_CASE(4, 8)
    GS_SMALL_CASE(4, 16)
    GS_SMALL_CASE(4, 32)
    GS_SMALL_CASE(8, 8)
    GS_SMALL_CASE(8, 16)
    GS_SMALL_CASE(8, 32)
    GS_SMALL_CASE(16, 8)
    GS_SMALL_CASE(16, 16)
    GS_SMALL_CASE(16, 32)
#undef GS_SMALL_CASE
    opted[dev] = true;
    kern<<<blocks, 256, smem, s>>>(X, N, ldx, D, Q, r, R, ldr, M, cnorm, mode, scale, Y, ldy, S, lds, argmax, maxval);
    return cudaGetLastError();
}

static int scores_pitch(int r) { return 4 * (((r + 3) / 4) | 1); }
int scores_chunk(int r) { return (kRSmemFloats - kCoefWarps * kCoefR) / scores_pitch(r); }

cudaError_t launch_scores(const ScoreArgs& a, cudaStream_t s) {
    if (a.N <= 0) return cudaSuccess;
    if (a.r < 1 || a.r > kCoefR) return cudaErrorInvalidValue;
    ScoreParams p;
    p.Y = a.Y, p.ldy = a.ldy;
    p.part = a.part, p.xx = a.xx, p.ks = a.ks;
    p.xnorm = a.xnorm;
    p.Yout = a.Yout, p.ldyo = a.ldyo;
    p.N = a.N, p.r = a.r;
    p.R = a.R, p.ldr = a.ldr, p.M = a.M, p.cnorm = a.cnorm;
    p.mode = a.mode, p.scale = a.scale;
    p.S = a.S, p.lds = a.lds, p.argmax = a.argmax, p.maxval = a.maxval;
    p.pitch = scores_pitch(a.r);
    p.chunk = std::min(a.M, scores_chunk(a.r));
    const size_t smem = sizeof(float) * ((size_t)p.chunk * p.pitch + kCoefWarps * kCoefR);
    // a block stages R once, so at most about two blocks' worth of rounds per SM of a large batch
    const long long blocks = std::min<long long>((a.N + kCoefWarps - 1) / kCoefWarps, 152LL * 8);
    k_scores<<<(unsigned)blocks, kCoefWarps * 32, smem, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_ksum(const GemmArgs& g, int ks, cudaStream_t s) {
    const long long mn = g.m * g.n;
    k_ksum<<<(unsigned)((mn + 255) / 256), 256, 0, s>>>(g.kpart, ks, g.m, g.n, (float*)g.C, g.ldc);
    return cudaGetLastError();
}

cudaError_t launch_gemm_simt(const GemmArgs& g, cudaStream_t s) {
    return launch_gemm_simt_parts(g, s, true);
}

cudaError_t launch_gemm_simt_parts(const GemmArgs& args, cudaStream_t s, bool sum) {
    GemmArgs g = args;
    if (g.m <= 0 || g.n <= 0 || g.batch <= 0) return cudaSuccess;
    if (g.ksplit <= 1 && sum) g.kpart = nullptr;
    // 16-byte loads of four elements: rows (and batches) of fp32 operands on 16-byte boundaries
    g.a_vec = g.a_type == MAT_F32 && (uintptr_t)g.A % 16 == 0 && g.lda % 4 == 0 && g.a_bstride % 4 == 0;
    g.b_vec = g.b_type == MAT_F32 && (uintptr_t)g.B % 16 == 0 && g.ldb % 4 == 0 && g.b_bstride % 4 == 0;
    if (g.ksplit > 1 && (g.batch != 1 || g.c_type != MAT_F32 || !g.kpart)) return cudaErrorInvalidValue;
    if (g.gate_xn2) {
        if (g.batch != 1 || g.ksplit > 1 || g.a_type != MAT_F32 || g.b_type != MAT_F32 || g.c_type != MAT_F32 ||
            !g.b_trans)
            return cudaErrorInvalidValue;
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const long long tiles = (g.m + kTM - 1) / kTM * ((g.n + kTN - 1) / kTN);
        const long long grid = std::min<long long>(tiles, 4LL * std::max(sms, 1)), per = (tiles + grid - 1) / grid;
        k_gemm_gated<MAT_F32, MAT_F32, MAT_F32, true><<<(unsigned)((tiles + per - 1) / per), 256, 0, s>>>(g, per);
        return cudaGetLastError();
    }
    const long long z = g.ksplit > 1 ? g.ksplit : g.batch, tn = (g.n + kTN - 1) / kTN;
    // 128-row tiles: about two of them for every SM, and at most a quarter more rows of padding than 64-row ones (64
    // products of 64 x 1,100 x 128 took 62 us in half-empty ones, 44 so; 40 of 129 x 1,100 x 64 43.6 / 39.4; but 300 x
    // 9,001 x 63, a fifth more, 16.8 in 128-row tiles, 20.6 in 64-row ones)
    const long long t128 = (g.m + 127) / 128, t64 = (g.m + 63) / 64;
    const bool tall = t128 * tn * z >= 300 && 8 * t128 <= 5 * t64;
    const int tm = tall ? 128 : kTM;
    dim3 grid((unsigned)tn, (unsigned)((g.m + tm - 1) / tm), (unsigned)z);
    if (grid.y > 65535u) return cudaErrorInvalidConfiguration;
#define GS_GEMM_CASE(TA, TB, TC, BT)                                                        \
    if (g.a_type == TA && g.b_type == TB && g.c_type == TC && g.b_trans == BT) {            \
        if (tall) k_gemm<TA, TB, TC, BT, 8><<<grid, 256, 0, s>>>(g);                        \
        else k_gemm<TA, TB, TC, BT, 4><<<grid, 256, 0, s>>>(g);                             \
        if (g.ksplit > 1 && sum) return launch_ksum(g, g.ksplit, s);                        \
        return cudaGetLastError();                                                          \
    }
    GS_GEMM_CASE(MAT_F32, MAT_F32, MAT_F32, true)
    GS_GEMM_CASE(MAT_F32, MAT_F32, MAT_F32, false)
    GS_GEMM_CASE(MAT_F32, MAT_F32, MAT_BF16, false)
    GS_GEMM_CASE(MAT_BF16, MAT_F32, MAT_F32, false)
    GS_GEMM_CASE(MAT_BF16, MAT_BF16, MAT_F32, true)
#undef GS_GEMM_CASE
    return cudaErrorInvalidValue;
}

cudaError_t launch_rownorm(const float* X, long long N, int ldx, int D, float* out, cudaStream_t s) {
    if (N <= 0) return cudaSuccess;
    k_rownorm<<<rows_grid(N), 256, 0, s>>>(X, N, ldx, D, out);
    return cudaGetLastError();
}

cudaError_t launch_row_finish(float* S, long long N, int M, int lds, bool softmax, int* argmax,
                              float* maxval, cudaStream_t s) {
    if (N <= 0) return cudaSuccess;
    k_row_finish<<<rows_grid(N), 256, 0, s>>>(S, N, M, lds, softmax ? 1 : 0, argmax, maxval);
    return cudaGetLastError();
}

cudaError_t launch_group_argmax(const float* S, long long N, int lds, const int* off, int G, int* argmax,
                                float* maxval, cudaStream_t s) {
    if (N <= 0) return cudaSuccess;
    if (G < 1 || G > kMaxGroups) return cudaErrorInvalidValue;
    GroupOffsets go;
    go.G = G;
    for (int g = 0; g <= G; ++g) go.off[g] = off[g];
    k_group_argmax<<<rows_grid(N), 256, 0, s>>>(S, N, lds, go, argmax, maxval);
    return cudaGetLastError();
}

template <int L>
static cudaError_t launch_bind_reg(const float* X, long long N, int D, int ldx, const float* Y, long long ldy,
                                   bool unbind, float* Z, int ldz, cudaStream_t s) {
    const int nb = D / L;
    const int vec = ((uintptr_t)X % 16 == 0 && (uintptr_t)Y % 16 == 0 && (uintptr_t)Z % 16 == 0 && ldx % 4 == 0 &&
                     ldy % 4 == 0 && ldz % 4 == 0)
                        ? 1
                        : 0;
    const unsigned blocks = (unsigned)((N * nb + 255) / 256);
    if (unbind)
        k_bind_reg<L, true><<<blocks, 256, 0, s>>>(X, N, nb, ldx, Y, ldy, Z, ldz, vec);
    else
        k_bind_reg<L, false><<<blocks, 256, 0, s>>>(X, N, nb, ldx, Y, ldy, Z, ldz, vec);
    return cudaGetLastError();
}

cudaError_t launch_bind(const float* X, long long N, int D, int ldx, const float* Y, long long ldy, int L, bool unbind,
                        float* Z, int ldz, cudaStream_t s) {
    if (N <= 0) return cudaSuccess;
    switch (L) {
        case 4: return launch_bind_reg<4>(X, N, D, ldx, Y, ldy, unbind, Z, ldz, s);
        case 8: return launch_bind_reg<8>(X, N, D, ldx, Y, ldy, unbind, Z, ldz, s);
        case 12: return launch_bind_reg<12>(X, N, D, ldx, Y, ldy, unbind, Z, ldz, s);
        case 16: return launch_bind_reg<16>(X, N, D, ldx, Y, ldy, unbind, Z, ldz, s);
        case 20: return launch_bind_reg<20>(X, N, D, ldx, Y, ldy, unbind, Z, ldz, s);
        case 24: return launch_bind_reg<24>(X, N, D, ldx, Y, ldy, unbind, Z, ldz, s);
        case 28: return launch_bind_reg<28>(X, N, D, ldx, Y, ldy, unbind, Z, ldz, s);
        case 32: return launch_bind_reg<32>(X, N, D, ldx, Y, ldy, unbind, Z, ldz, s);
        default: break;
    }
    // the staged kernels hold a row's X and Y blocks in shared memory: opt in past 48 KB once
    static bool opted[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!opted[dev]) {
        for (auto fn : {k_bind16<true>, k_bind16<false>, k_bind8<true>, k_bind8<false>}) {
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
            if (e != cudaSuccess) return e;
        }
        opted[dev] = true;
    }
    const int zvec = ((uintptr_t)Z % 16 == 0 && ldz % 4 == 0) ? 1 : 0;
    if (L % 16 == 0 && L <= kMaxBindFastL && D / L <= 65535) {
        const int tpr = std::min(L / 16, 256);
        const int rpc = 256 / tpr;
        const size_t smem = (size_t)rpc * (2 * L + L / 4) * sizeof(float);
        const dim3 grid((unsigned)((N + rpc - 1) / rpc), (unsigned)(D / L));
        if (unbind)
            k_bind16<true><<<grid, 256, smem, s>>>(X, N, ldx, Y, ldy, L, Z, ldz, zvec);
        else
            k_bind16<false><<<grid, 256, smem, s>>>(X, N, ldx, Y, ldy, L, Z, ldz, zvec);
        return cudaGetLastError();
    }
    if (L % 8 == 0 && L <= kMaxBindFastL && D / L <= 65535) {
        const int tpr = std::min(L / 8, 256);
        const int rpc = 256 / tpr;
        const size_t smem = (size_t)rpc * 2 * L * sizeof(float);
        const dim3 grid((unsigned)((N + rpc - 1) / rpc), (unsigned)(D / L));
        if (unbind)
            k_bind8<true><<<grid, 256, smem, s>>>(X, N, ldx, Y, ldy, L, Z, ldz, zvec);
        else
            k_bind8<false><<<grid, 256, smem, s>>>(X, N, ldx, Y, ldy, L, Z, ldz, zvec);
        return cudaGetLastError();
    }
    const long long total = N * D;
    const unsigned blocks = (unsigned)((total + 255) / 256);
    if (unbind)
        k_bind1<true><<<blocks, 256, 0, s>>>(X, N, D, ldx, Y, ldy, L, Z, ldz);
    else
        k_bind1<false><<<blocks, 256, 0, s>>>(X, N, D, ldx, Y, ldy, L, Z, ldz);
    return cudaGetLastError();
}

cudaError_t launch_row_softmax(float* A, long long rows, int L, long long ld, cudaStream_t s) {
    if (rows <= 0) return cudaSuccess;
    k_row_softmax<<<rows_grid(rows), 256, 0, s>>>(A, rows, L, ld);
    return cudaGetLastError();
}

}  // namespace gs
