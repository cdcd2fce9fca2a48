// gs_build.cu -- basis construction (paper Sec. 3.1, Eq. 1; Sec. 3.3 "during
// initialization ... Gram-Schmidt orthogonalization of the codebook").
//
// Row-order Gram-Schmidt with two projection passes per row and a relative
// rank tolerance, in fp64 on the device.  Rows are taken in panels of
// kPanel.  For each panel:
//   1. the rows' norms ||c_i|| (once, before the panels);
//   2. twice (reorthogonalisation): H = V Q_old^T (fp64 dot products over
//      column slices, then a slice reduction that also accumulates R), and
//      V -= H Q_old -- a block projection against the basis built so far;
//   3. inside the panel: Cholesky QR, twice (two passes again), with the rank
//      decisions (||v|| > tol * ||c_i||) taken from the pivots; accepted rows are
//      appended to Q.  A panel whose decisions the pivots cannot settle is done
//      row by row instead, on a cluster of CTAs.
// In exact arithmetic this is the row-wise two-pass Gram-Schmidt of the
// paper's construction (projections onto orthonormal directions commute, and
// Cholesky QR of a panel is its Gram-Schmidt factorisation); the block passes
// against the old basis and the column slices are what make it data-parallel.
// Measured (GB300): M = 512, D = 4096: 7.25 ms (19.9 before the slices were cut to the
// number of SMs and the panels factored by Cholesky QR); M = 1,024, D = 10,000, rank
// 922: 38 ms (97).  The fp64 arithmetic of the block projections takes ~2.7 ms of the
// first, the rest is the chain of eight launches per panel.
// The only host synchronisation is the read of the final rank r.
//
// Afterwards fp32 copies of Q and R are made for the caller, plus the
// fp16 operand copies of the tensor-core kernels (unbiased dithered rounding
// of the fp64 basis, see dither_half).

#include <float.h>

#include <algorithm>
#include <cmath>
#include <memory>
#include <vector>

#include "gs_internal.h"
#include "gs_tc_ptx.cuh"

namespace gs {
namespace {

constexpr int kPanel = 16;      // rows per panel
constexpr int kMaxSlice = 96;   // columns per slice CTA (shared memory; 3 x 512 update outputs)

__device__ unsigned g_err_build = 0;

template <int NT>
__device__ double block_sum(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();  // protect sh from a previous use
    if (l == 0) sh[w] = v;
    __syncthreads();
    double t = 0.0;
    if (w == 0) {
        t = l < NT / 32 ? sh[l] : 0.0;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (l == 0) sh[32] = t;
    }
    __syncthreads();
    return sh[32];
}

// Row norms ||c_i|| and, with normalize, the rows' scales 1 / ||c_i|| (the norm is then that of the
// scaled row).  One CTA per row of C.
__global__ void __launch_bounds__(256) k_row_norms(const float* __restrict__ C, long long ldc, int D, int normalize,
                                                   double* __restrict__ cn, double* __restrict__ sc) {
    __shared__ double sh[33];
    const float* c = C + (size_t)blockIdx.x * ldc;
    double ss = 0.0;
    for (int d = threadIdx.x; d < D; d += 256) ss += (double)c[d] * (double)c[d];
    double nrm = sqrt(block_sum<256>(ss, sh)), scale = 1.0;
    if (normalize && nrm > 0.0) {
        scale = 1.0 / nrm;
        ss = 0.0;
        for (int d = threadIdx.x; d < D; d += 256) {
            const double x = (double)c[d] * scale;
            ss += x * x;
        }
        nrm = sqrt(block_sum<256>(ss, sh));
    }
    if (threadIdx.x == 0) {
        cn[blockIdx.x] = nrm;
        sc[blockIdx.x] = scale;
    }
}

// 2. Block projections.  The D columns are cut into slices of w, one CTA each (about one per SM: GB300
//    does ~2 fp64 FMAs per clock and SM, so a pass over the basis is bound by that pipe and wants every
//    SM busy for the same time; 64-column CTAs left 88 of 152 SMs idle at D = 4096: dots 64 us and update
//    77 us per panel and pass, now 36 us for dots alone, 68 us for an update and the next dots, 29 us for
//    the fp32 update with the Gram matrix).  A CTA keeps its slice of the panel in shared memory and streams the basis' slice
//    through two buffers (cp.async).  kind:
//      kDots1    V = C;           Hp = V Q^T                  (first pass' dots, over the slice)
//      kUpdDots  V = C - H Q;     Hp = V Q^T                  (first pass' update, second's dots)
//      kUpdGram  V -= H Q;        Gp = V V^T, V stored        (second update, and the panel's Gram matrix)
//    The second update runs in fp32: its coefficients are what the first pass left over, ~1e-16 of the
//    row, so that one fp32 rounding of each term is ~1e-23 of it.
//    Gp sums the slices of a cluster of kSliceCluster CTAs through distributed shared memory (fixed order).
enum { kDots1 = 0, kUpdDots = 1, kUpdGram = 2 };
constexpr int kSliceCluster = 8;
constexpr int kPairs = kPanel * (kPanel + 1) / 2;  // 136: the Gram matrix' lower triangle

// What a panel's factorisation hands from kernel to kernel.
struct PanelState {
    int slow;    // a rank decision needs the row-by-row kernel
    int nacc;    // accepted rows, in order
    int acc[kPanel];
    double G[kPanel][kPanel];  // V V^T
    double T[kPanel][kPanel];  // V' = T V (nacc rows)
};

__device__ __forceinline__ void cp_async8(double* dst, const double* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(ptx::smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// A double rounded towards zero to fp32 with integer instructions (conversions would share the fp64
// pipe); magnitudes below fp32's normal range become 0.  For |d| <= 1.
__device__ __forceinline__ float trunc_f32(double d) {
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const uint32_t mag = ((hi & 0x7fffffffu) << 3) | (lo >> 29);  // exponent still biased by 1023
    const uint32_t r = ((hi >> 20) & 0x7ffu) > 896u ? mag - (896u << 23) : 0u;
    return __uint_as_float(r | (hi & 0x80000000u));
}

struct SliceParams {
    const float* C;     // the panel's first row
    long long ldc;
    const double* sc;   // the panel rows' scales and norms
    const double* cn;
    double* V;          // kPanel x D
    const double* Qw;
    int D, w, bp, jc;   // jc: basis rows per chunk
    const int* r_start;
    const double* H;
    double* Hp;
    int ldh;
    double* Gp;         // per cluster: kPairs
};

// the sums over a cluster's CTAs of part[kPairs] (each CTA's own, in shared memory): CTA q adds the
// entries e = q mod kSliceCluster in CTA order and writes them to out
__device__ __forceinline__ void cluster_add_pairs(const double* part, double* out) {
    ptx::cluster_sync_all();
    const int rank = (int)ptx::cluster_ctarank();
    const int e = rank + kSliceCluster * (int)threadIdx.x;
    if (e < kPairs) {
        double v = 0.0;
        for (int c = 0; c < kSliceCluster; ++c) {
            double x;
            asm volatile("ld.shared::cluster.f64 %0, [%1];"
                         : "=d"(x)
                         : "r"(ptx::mapa_shared(ptx::smem_u32(part + e), (uint32_t)c))
                         : "memory");
            v += x;
        }
        out[e] = v;
    }
    ptx::cluster_sync_all();  // no CTA leaves while a peer may still read its part
}

// part[e] = sum over the slice of V_i V_j for the pairs e = (i, j <= i); Vs: kPanel rows of w, ld vl
__device__ __forceinline__ void gram_slice(const double* Vs, int vl, int w, double* part) {
    for (int e = threadIdx.x; e < kPairs; e += blockDim.x) {
        int i = 0;
        while ((i + 1) * (i + 2) / 2 <= e) ++i;
        const int j = e - i * (i + 1) / 2;
        double a = 0.0, b = 0.0;
        int c = 0;
        for (; c + 1 < w; c += 2) {
            a += Vs[i * vl + c] * Vs[j * vl + c];
            b += Vs[i * vl + c + 1] * Vs[j * vl + c + 1];
        }
        if (c < w) a += Vs[i * vl + c] * Vs[j * vl + c];
        part[e] = a + b;
    }
}

// 2^(+-e) with 2^e <= n < 2^(e+1) (1 for n = 0 or not finite): a row's scale as an exact factor
__device__ __forceinline__ double row_pow2(double n, int sign) {
    const int e = n > 0.0 && n <= DBL_MAX ? ilogb(n) : 0;
    return __hiloint2double((1023 + sign * e) << 20, 0);
}

// shared memory of k_panel_slice for slices of w columns and chunks of jc basis rows
constexpr size_t slice_smem(int w, int jc) {
    return sizeof(double) * ((size_t)(kPanel + 2 * jc) * (w | 1) + (2 * kPanel * jc > kPairs ? 2 * kPanel * jc : kPairs)) +
           sizeof(float) * ((size_t)jc * (w | 1) + (size_t)kPanel * jc);
}
constexpr int kSliceThreads = 512;  // at most
constexpr size_t kSliceSmemMax = slice_smem(kMaxSlice, kSliceThreads / kPanel * 2);
static_assert(kSliceSmemMax <= 227 * 1024, "a slice of the panel and its chunks of the basis fit a CTA's shared memory");

template <int KIND>
__global__ void __launch_bounds__(kSliceThreads) k_panel_slice(const SliceParams p) {
    extern __shared__ double sm[];
    const int tid = threadIdx.x, nt = blockDim.x;
    const int r0 = *p.r_start;
    const int c0 = blockIdx.x * p.w, w = max(0, min(p.w, p.D - c0));
    const int vl = p.w | 1;  // odd row pitches: lanes on consecutive rows hit different banks
    double* Vs = sm;
    double* Qs[2] = {Vs + kPanel * vl, Vs + kPanel * vl + p.jc * vl};
    double* Hs[2] = {Qs[1] + p.jc * vl, Qs[1] + p.jc * vl + kPanel * p.jc};  // updates only
    double* part = Hs[0];  // the Gram partials: after the last chunk of H
    float* Qf = reinterpret_cast<float*>(Hs[1] + kPanel * p.jc);  // kUpdGram: the current chunk in fp32
    float* Hf = Qf + p.jc * vl;
    const int nchunks = (r0 + p.jc - 1) / p.jc;

    auto fetch = [&](int ch, int b, bool with_h) {
        const int j0 = ch * p.jc, nj = min(p.jc, r0 - j0);
        for (int e = tid; e < nj * w; e += nt) {
            const int j = e / w, c = e - j * w;
            cp_async8(&Qs[b][j * vl + c], p.Qw + (size_t)(j0 + j) * p.D + c0 + c);
        }
        if (with_h)
            for (int e = tid; e < kPanel * nj; e += nt) {
                const int k = e / nj, j = e - k * nj;
                if (k < p.bp) cp_async8(&Hs[b][k * p.jc + j], p.H + (size_t)k * p.ldh + j0 + j);
            }
        cp_async_commit();
    };
    if (nchunks > 0) fetch(0, 0, KIND != kDots1);
    for (int e = tid; e < kPanel * w; e += nt) {
        const int k = e / w, c = e - k * w;
        double v = 0.0;
        if (k < p.bp)
            v = KIND == kUpdGram && r0 > 0 ? p.V[(size_t)k * p.D + c0 + c]
                                           : (double)p.C[(size_t)k * p.ldc + c0 + c] * p.sc[k];
        Vs[k * vl + c] = v;
    }
    if (KIND != kDots1) {
        // V -= H Q: thread outputs (k, c), at most three a thread (kPanel w <= 3 nt), summed over chunks
        constexpr int kOut = 3;
        double acc[kOut] = {};
        float accf[kOut] = {};
        int ko[kOut], co[kOut];
#pragma unroll
        for (int o = 0; o < kOut; ++o) {
            const int e = tid + o * nt;
            ko[o] = w > 0 && e < kPanel * w ? e / w : 0;
            co[o] = w > 0 && e < kPanel * w ? e % w : 0;
        }
        for (int ch = 0; ch < nchunks; ++ch) {
            const int b = ch & 1, nj = min(p.jc, r0 - ch * p.jc);
            if (ch + 1 < nchunks) {
                fetch(ch + 1, b ^ 1, true);
                cp_async_wait<1>();
            } else {
                cp_async_wait<0>();
            }
            __syncthreads();
            if (KIND == kUpdGram) {  // the chunk once into fp32, the coefficients relative to the row's norm
                for (int e = tid; e < nj * vl; e += nt) Qf[e] = trunc_f32(Qs[b][e]);
                for (int e = tid; e < kPanel * nj; e += nt) {
                    const int k = e / nj, j = e - k * nj;
                    Hf[k * p.jc + j] = k < p.bp ? (float)(Hs[b][k * p.jc + j] * row_pow2(p.cn[k], -1)) : 0.f;
                }
                __syncthreads();
            }
#pragma unroll
            for (int o = 0; o < kOut; ++o) {
                if (tid + o * nt >= kPanel * w) continue;
                if (KIND == kUpdGram) {
                    const float* h = &Hf[ko[o] * p.jc];
                    for (int j = 0; j < nj; ++j) accf[o] = fmaf(h[j], Qf[j * vl + co[o]], accf[o]);
                } else {
                    const double* h = &Hs[b][ko[o] * p.jc];
                    for (int j = 0; j < nj; ++j) acc[o] += h[j] * Qs[b][j * vl + co[o]];
                }
            }
            __syncthreads();
        }
        if (nchunks == 0) __syncthreads();
#pragma unroll
        for (int o = 0; o < kOut; ++o) {
            if (tid + o * nt >= kPanel * w || ko[o] >= p.bp) continue;
            double v = Vs[ko[o] * vl + co[o]];
            v -= KIND == kUpdGram ? (double)accf[o] * row_pow2(p.cn[ko[o]], 1) : acc[o];
            Vs[ko[o] * vl + co[o]] = v;
            p.V[(size_t)ko[o] * p.D + c0 + co[o]] = v;
        }
    }
    if (KIND == kUpdGram) {
        __syncthreads();
        gram_slice(Vs, vl, w, part);
        cluster_add_pairs(part, p.Gp + (size_t)(blockIdx.x / kSliceCluster) * kPairs);
        return;
    }
    // Hp = V Q^T over the slice: thread (k = tid % 16, basis rows j and j + jc / 2 of a chunk)
    if (KIND == kUpdDots) {
        __syncthreads();
        if (nchunks > 0) fetch(0, 0, false);
    }
    const int k = tid % kPanel, jl = tid / kPanel, jh = p.jc / 2;
    for (int ch = 0; ch < nchunks; ++ch) {
        const int b = ch & 1, j0 = ch * p.jc, nj = min(p.jc, r0 - j0);
        if (ch + 1 < nchunks) {
            fetch(ch + 1, b ^ 1, false);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        if (jl < nj) {
            const double* v = &Vs[k * vl];
            const double* q0 = &Qs[b][jl * vl];
            const double* q1 = &Qs[b][min(jl + jh, nj - 1) * vl];
            double a0 = 0.0, a1 = 0.0;
            if (jl + jh < nj) {
                for (int c = 0; c < w; ++c) {
                    const double x = v[c];
                    a0 += x * q0[c];
                    a1 += x * q1[c];
                }
            } else {
                for (int c = 0; c < w; ++c) a0 += v[c] * q0[c];
            }
            double* out = p.Hp + ((size_t)blockIdx.x * kPanel + k) * p.ldh + j0;
            out[jl] = a0;
            if (jl + jh < nj) out[jl + jh] = a1;
        }
        __syncthreads();
    }
}

// H[k][j] = sum over slices; R64[p0+k][j] += H[k][j].  16 consecutive outputs a block, 16 threads each
// (fp64 adds take the fp64 FMA's time here, and the loads their latency: four threads an output took
// 17 us at 152 slices), their parts added in a fixed order.
__global__ void __launch_bounds__(256) k_panel_reduce(const double* __restrict__ Hp, int nslices, int bp,
                                                      const int* __restrict__ r_start, int ldh, double* __restrict__ H,
                                                      double* __restrict__ R64, int ldr) {
    __shared__ double sh[16][17];
    const int r0 = *r_start;
    const int oi = threadIdx.x & 15, q = threadIdx.x >> 4;
    const long long o = (long long)blockIdx.x * 16 + oi;
    const bool in = o < (long long)bp * r0;
    const int k = in ? (int)(o / r0) : 0, j = in ? (int)(o % r0) : 0;
    double s = 0.0;
    if (in) {
        const double* src = Hp + (size_t)k * ldh + j;
#pragma unroll 8
        for (int t = q; t < nslices; t += 16) s += src[(size_t)t * kPanel * ldh];
    }
    sh[q][oi] = s;
    __syncthreads();
    if (in && q == 0) {
        double v = 0.0;
#pragma unroll
        for (int t = 0; t < 16; ++t) v += sh[t][oi];
        H[(size_t)k * ldh + j] = v;
        R64[(size_t)k * ldr + j] += v;
    }
}

// 3. Inside the panel: Cholesky QR, twice.  G = V V^T (summed over the slices) = L L^T, V' = T V with T ~
//    L^-1 has rows orthonormal up to the rounding of T and G times the panel's condition squared; a
//    second round on V' brings that to eps: V'' = T2 V', and the panel's rows of R are V V''^T =
//    G T^T T2^T.  Each round is one pass over the slices with every CTA doing the 16 x 16 factorisation
//    itself, against three cluster-wide sums per row (k_panel_gs2: 326 us a panel at D = 4096, of which
//    ~65 us were arithmetic).
//    T need not be exact, V' = T V only has to be taken in fp64 with the T that is used: the first
//    round's factorisation runs in fp32, one warp, a row per lane (rows scaled by powers of two), where
//    every pivot stays above 1e-3 of its row and certain of its rank decision; otherwise in fp64.  The
//    second round's Gram matrix is then I + E with |E| ~ 1e-7, whose Cholesky factor I + X and T2 come
//    from their series (X = lower(E - X X^T) iterated, T2 = I - X + X^2 - X^3: errors below |E|^4) in four
//    16 x 16 products; otherwise by the fp64 factorisation.  (fp64 runs at 2 FMAs per clock and SM here,
//    16 dependent steps of it cost ~20 us: the two rounds took 57 us a panel with both in fp64, 39 now.)
//    Row k is accepted exactly as the row-by-row kernel would: its norm against what came before it,
//    sqrt(pivot), > tau ||c_k||.  A panel with a pivot that is closer to the tolerance than its own noise
//    (see chol_factor), or within 1e-6 of it, is left to k_panel_gs2.
//
// The factorisation in one CTA (all threads): A (the Gram matrix; the fp64 form overwrites it), T: rows of
// the transform for the accepted rows (T[k] over the panel's rows).
struct Chol {
    double A[kPanel][kPanel + 1], T[kPanel][kPanel + 1], L[kPanel][kPanel], diag[kPanel], nv[kPanel], rs;
    double W[kPanel][kPanel + 1];
    float Af[kPanel][kPanel + 1];
    int acc[kPanel], nacc, slow, take, quick;
};

__device__ __forceinline__ void chol_load(Chol& c, const double* Gp, int ncl) {
    for (int e = threadIdx.x; e < kPairs; e += blockDim.x) {
        double v = 0.0;
        for (int t = 0; t < ncl; ++t) v += Gp[(size_t)t * kPairs + e];
        int i = 0;
        while ((i + 1) * (i + 2) / 2 <= e) ++i;
        const int j = e - i * (i + 1) / 2;
        c.A[i][j] = v;
        c.A[j][i] = v;
        if (i == j) {
            c.diag[i] = v;
            c.nv[i] = sqrt(fmax(v, 0.0));
        }
    }
    for (int e = threadIdx.x; e < kPanel * kPanel; e += blockDim.x) {
        c.T[e / kPanel][e % kPanel] = e / kPanel == e % kPanel ? 1.0 : 0.0;
        c.L[e / kPanel][e % kPanel] = 0.0;
    }
    if (threadIdx.x == 0) c.nacc = c.slow = 0;
    __syncthreads();
}

// gerr: the first round's Gram matrix and its factorisation are off by at most gerr ||v_i|| ||v_j|| an entry, so
// row k's pivot is by gerr (sum_j |t_j| ||v_j||)^2, t the combination of the panel's rows that it is the
// squared norm of (a panel whose taken rows lie close to each other has large t: the noise can exceed the
// tolerance although 1e-14 ||v_k||^2 does not)
__device__ __forceinline__ void chol_factor(Chol& c, int n, bool first, const double* cn, double tau, int room,
                                            double gerr) {
    for (int k = 0; k < n; ++k) {
        double amp = 0.0;
        if (first && threadIdx.x < 32) {
            const int j = threadIdx.x & (kPanel - 1);
            amp = fabs(c.T[k][j]) * c.nv[j];
#pragma unroll
            for (int o = kPanel / 2; o > 0; o >>= 1) amp += __shfl_xor_sync(0xffffffffu, amp, o);
        }
        if (threadIdx.x == 0) {
            const double piv = c.A[k][k];
            int take = 1;
            if (first) {
                const double lim = tau * cn[k], lim2 = lim * lim, v2 = c.diag[k];
                if (c.nacc >= room) {
                    take = 0;  // the basis is full: every further row is dependent
                } else if (!(v2 > lim2 * (1.0 - 1e-6))) {
                    take = 0;  // what the basis so far leaves of the row is below the tolerance already
                    if (v2 != v2) c.slow = 1;
                } else {
                    take = piv > lim2;
                    if (!(fabs(piv - lim2) >= fmax(gerr * amp * amp, 1e-6 * lim2))) c.slow = 1;
                }
            }
            c.take = take;
            if (take) {
                c.rs = rsqrt(piv);
                c.acc[c.nacc] = k;
            }
        }
        __syncthreads();
        if (c.take) {
            const int a = c.nacc;
            const double rs = c.rs;
            for (int e = threadIdx.x; e < kPanel; e += blockDim.x) {
                if (e >= k) c.L[e][a] = c.A[e][k] * rs;
                else c.T[k][e] *= rs;
                if (e == k) c.T[k][k] *= rs;
            }
            __syncthreads();
            for (int e = threadIdx.x; e < 2 * kPanel * kPanel; e += blockDim.x) {
                const int i = (e / kPanel) % kPanel, j = e % kPanel;
                if (i <= k) continue;
                if (e < kPanel * kPanel) {
                    if (j > k) c.A[i][j] -= c.L[i][a] * c.L[j][a];
                } else if (j <= k) {
                    c.T[i][j] -= c.L[i][a] * c.T[k][j];
                }
            }
            if (threadIdx.x == 0) ++c.nacc;
        }
        __syncthreads();
    }
}

// 2^-e for a squared norm in [4^e, 4^(e+1)) (1 when it is not a positive finite number)
__device__ __forceinline__ double row_unscale(double n2) {
    if (!(n2 > 0.0) || !(n2 <= DBL_MAX)) return 1.0;
    const int e = (((__double2hiint(n2) >> 20) & 0x7ff) - 1023) >> 1;
    return __hiloint2double((1023 - e) << 20, 0);
}

// The first round's factorisation in fp32 on warp 0 (all threads call it): sets T, acc, nacc and quick when
// every decision is certain.
__device__ __forceinline__ void chol_quick(Chol& c, int n, const double* cn, double tau, int room) {
    for (int e = threadIdx.x; e < kPanel * kPanel; e += blockDim.x) {
        const int i = e / kPanel, j = e % kPanel;
        c.Af[i][j] = (float)(c.A[i][j] * row_unscale(c.diag[i]) * row_unscale(c.diag[j]));
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x, i = lane & 15;
        float a[kPanel], t[kPanel];
#pragma unroll
        for (int j = 0; j < kPanel; ++j) {
            a[j] = c.Af[i][j];
            t[j] = i == j ? 1.f : 0.f;
        }
        const float d = c.Af[i][i];
        // rows below the tolerance already are dependent; the others' tolerance in the scaled units
        bool out = true;
        float lim = 0.f;
        bool sure = true;
        if (i < n) {
            const double l = tau * cn[i], l2 = l * l, v2 = c.diag[i], u = row_unscale(v2);
            out = !(v2 > l2 * (1.0 - 1e-6));
            lim = (float)(l2 * u * u);
            sure = v2 == v2 && v2 <= DBL_MAX && (out || (d >= 1.f && d < 4.1f));
        }
        bool ok = __all_sync(0xffffffffu, sure);
        int na = 0;
        unsigned taken = 0;
#pragma unroll
        for (int k = 0; k < kPanel; ++k) {
            const bool skip = __shfl_sync(0xffffffffu, (int)out, k) != 0;
            const float piv = __shfl_sync(0xffffffffu, a[k], k), dk = __shfl_sync(0xffffffffu, d, k),
                        lk = __shfl_sync(0xffffffffu, lim, k);
            if (k >= n || skip || na >= room) continue;  // (warp-uniform)
            ok = ok && piv > 1e-3f * dk && piv > 1.01f * lk;
            const float rs = rsqrtf(piv), l = a[k] * rs;
#pragma unroll
            for (int j = 0; j < kPanel; ++j) {
                if (j > k) {
                    const float lj = __shfl_sync(0xffffffffu, l, j);
                    if (i > k) a[j] = fmaf(-l, lj, a[j]);
                } else {
                    const float tj = __shfl_sync(0xffffffffu, t[j], k) * rs;
                    if (i > k) t[j] = fmaf(-l, tj, t[j]);
                    if (i == k) t[j] = tj;
                }
            }
            if (lane == 0) c.acc[na] = k;
            taken |= 1u << k;
            ++na;
        }
        // T's rounding reaches V' V'^T times (sum_j |t_j| ||v_j||)^2, and a pivot 18 x 2^-24 of that square: below
        // 0.4 % of a taken one, which the 1 % from its tolerance covers
        float amp = 0.f;
#pragma unroll
        for (int j = 0; j < kPanel; ++j) amp += fabsf(t[j]) * 2.f;
        ok = ok && __all_sync(0xffffffffu, !((taken >> i) & 1u) || amp < 60.f);
        if (ok && lane < kPanel) {
#pragma unroll
            for (int j = 0; j < kPanel; ++j) c.T[i][j] = (double)t[j] * row_unscale(c.diag[j]);
        }
        if (lane == 0) {
            c.quick = ok;
            if (ok) c.nacc = na;
        }
    }
    __syncthreads();
}

// The second round's transform from the series, when the Gram matrix is that close to I: T[0..n).  Entry
// (i, j <= i) of each 16 x 16 product in one thread, ordered so that a warp's sums have about one length.
__device__ __forceinline__ bool chol_series(Chol& c, int n) {
    bool far = false;
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
        const int i = e / n, j = e % n;
        far |= !(fabs(c.A[i][j] - (i == j ? 1.0 : 0.0)) < 4e-6);
    }
    if (__syncthreads_or(far)) return false;
    // entries by column (sum length j + 1) and by diagonal (sum length i - j + 1)
    int ci = -1, cj = 0, di = -1, dj = 0;
    if (threadIdx.x < kPairs) {
        int e = threadIdx.x, len = kPanel;
        while (e >= len) e -= len--;
        cj = kPanel - len, ci = cj + e;
        di = kPanel - len + e, dj = e;
    }
    const bool con = ci >= 0 && ci < n, don = di >= 0 && di < n;
    const double eij = con ? (ci == cj ? 0.5 * (c.A[ci][cj] - 1.0) : c.A[ci][cj]) : 0.0;
    if (con) c.L[ci][cj] = eij;
    __syncthreads();
    for (int it = 0; it < 2; ++it) {  // X = lower(E - X X^T), the diagonal halved
        double s = 0.0;
        if (con)
            for (int m = 0; m <= cj; ++m) s += c.L[ci][m] * c.L[cj][m];
        __syncthreads();
        if (con) c.L[ci][cj] = eij - (ci == cj ? 0.5 * s : s);
        __syncthreads();
    }
    if (don) c.T[di][dj] = (di == dj ? 1.0 : 0.0) - c.L[di][dj];
    __syncthreads();
    for (int it = 0; it < 2; ++it) {  // T = I - X T
        double s = 0.0;
        if (don)
            for (int m = dj; m <= di; ++m) s += c.L[di][m] * c.T[m][dj];
        __syncthreads();
        if (don) c.T[di][dj] = (di == dj ? 1.0 : 0.0) - s;
        __syncthreads();
    }
    if (threadIdx.x == 0) c.nacc = n;
    if (threadIdx.x < n) c.acc[threadIdx.x] = threadIdx.x;
    __syncthreads();
    return true;
}

struct CholParams {
    double* V;
    double* Qw;
    int D, w, bp, ncl;
    const double* Gp;   // this round's Gram partials
    double* Gp2;        // the next round's (round 1)
    const double* cn;   // the panel rows' norms
    double tau, gerr;   // rank tolerance; bound of the first Gram matrix' relative error (see chol_factor)
    double* R64;        // the panel's first row
    int ldr, rmax;
    const int* r_start;
    int* r_next;
    PanelState* st;
};

// ROUND 1: V' = L^-1 V in place (rows 0 .. nacc), its Gram partials, and the panel's state.
// ROUND 2: the same on V', written to the basis; R's new columns; the rank for the next panel.
template <int ROUND>
__global__ void __launch_bounds__(512) k_panel_chol(const CholParams p) {
    extern __shared__ double sm[];
    __shared__ Chol c;
    __shared__ double part[kPairs];
    const int tid = threadIdx.x, nt = blockDim.x;
    const int r0 = *p.r_start;
    const int c0 = blockIdx.x * p.w, w = max(0, min(p.w, p.D - c0));
    const int vl = p.w | 1;
    double* Vs = sm;
    if (ROUND == 2 && p.st->slow) return;  // k_panel_gs2 does this panel
    const int n = ROUND == 1 ? p.bp : p.st->nacc;
    for (int e = tid; e < n * w; e += nt) Vs[(e / w) * vl + e % w] = p.V[(size_t)(e / w) * p.D + c0 + e % w];
    chol_load(c, p.Gp, p.ncl);
    if (ROUND == 1) {
        if (blockIdx.x == 0)
            for (int e = tid; e < kPanel * kPanel; e += nt) p.st->G[e / kPanel][e % kPanel] = c.A[e / kPanel][e % kPanel];
        chol_quick(c, n, p.cn, p.tau, p.rmax - r0);
        if (!c.quick) {
            chol_factor(c, n, true, p.cn, p.tau, p.rmax - r0, p.gerr);
            // V' = T V multiplies G's rounding by (sum_j |T_kj| ||v_j||)^2: beyond 1e8 the second round would
            // not bring it back to eps
            if (tid < p.bp && !c.slow) {
                double amp = 0.0;
                for (int j = 0; j <= tid; ++j) amp += fabs(c.T[tid][j]) * c.nv[j];
                bool taken = false;
                for (int a = 0; a < c.nacc; ++a) taken |= c.acc[a] == tid;
                if (taken && !(amp < 1e4)) c.slow = 1;
            }
            __syncthreads();
        }
    } else if (!chol_series(c, n)) {
        chol_factor(c, n, false, p.cn, p.tau, p.rmax - r0, 0.0);
    }
    const bool slow = ROUND == 1 && c.slow != 0;
    if (ROUND == 1 && blockIdx.x == 0) {
        if (tid == 0) {
            p.st->slow = slow;
            p.st->nacc = c.nacc;
        }
        for (int e = tid; e < kPanel; e += nt) p.st->acc[e] = c.acc[e];
        for (int e = tid; e < c.nacc * kPanel; e += nt) {
            const int a = e / kPanel, j = e % kPanel;
            p.st->T[a][j] = j <= c.acc[a] ? c.T[c.acc[a]][j] : 0.0;
        }
    }
    if (slow) return;  // the same data and so the same answer in every CTA of the grid
    const int na = c.nacc;
    for (int e = tid; e < na * w; e += nt) {
        const int a = e / w, cc = e - a * w, k = c.acc[a];
        double v = 0.0;
        for (int j = 0; j <= k; ++j) v += c.T[k][j] * Vs[j * vl + cc];
        if (ROUND == 1)
            p.V[(size_t)a * p.D + c0 + cc] = v;  // this CTA's columns, already read
        else
            p.Qw[(size_t)(r0 + a) * p.D + c0 + cc] = v;
    }
    if (ROUND == 1) {
        __syncthreads();  // every value of Vs has been used: the Gram matrix of the new rows, read back
        for (int e = tid; e < kPanel * w; e += nt) {
            const int a = e / w, cc = e - a * w;
            Vs[a * vl + cc] = a < na ? p.V[(size_t)a * p.D + c0 + cc] : 0.0;
        }
        __syncthreads();
        gram_slice(Vs, vl, w, part);
        cluster_add_pairs(part, p.Gp2 + (size_t)(blockIdx.x / kSliceCluster) * kPairs);
    } else if (blockIdx.x == 0) {
        // R's new columns, V V''^T = (G T^T) T2^T; entry (k, a) is zero where row k comes before accepted row a
        for (int e = tid; e < p.bp * na; e += nt) {
            const int k = e / na, a = e - k * na;
            double v = 0.0;
            for (int j = 0; j <= p.st->acc[a]; ++j) v += p.st->G[k][j] * p.st->T[a][j];
            c.W[k][a] = v;
        }
        __syncthreads();
        for (int e = tid; e < p.bp * na; e += nt) {
            const int k = e / na, a = e - k * na;
            if (p.st->acc[a] > k) continue;
            double v = 0.0;
            for (int b = 0; b <= a; ++b) v += c.W[k][b] * c.T[a][b];
            p.R64[(size_t)k * p.ldr + r0 + a] = v;
        }
        if (tid == 0) *p.r_next = r0 + na;
    }
}

// 3b. The row-by-row form, for the panels that k_panel_chol leaves (PanelState.slow):
//    Gram-Schmidt with two passes inside the panel, rank decision, normalisation and append, on a
//    cluster of kMgsCtas CTAs: CTA c owns columns [c S, (c + 1) S) of every vector (S = ceil(D /
//    kMgsCtas)), so the fp64 arithmetic of a row is spread over kMgsCtas SMs (GB300's fp64 rate
//    per SM is low: one CTA doing this took 1.5 ms per 16-row panel of 10,000-wide rows).  Each
//    pass takes the projections of v on all of the panel's new directions at once (classical
//    Gram-Schmidt, twice: the same factorisation as the row-by-row passes in exact arithmetic, and
//    as stable with the second pass), so a row needs three sums over the whole row: the two passes'
//    projections and the norm.  A sum is reduced in each CTA (a 16-lane butterfly, then across the
//    warps), and each CTA's partials are stored into every CTA's shared memory with st.async, whose
//    bytes complete on the receiver's mbarrier for that buffer (no release fence on the sending
//    side; a cluster barrier per sum cost ~11 us); every CTA adds the partials in CTA order, so all
//    hold the same values, take the same rank decisions and run the same sums.  Partial sums
//    alternate between two buffers: a CTA posts sum n + 2 only after it has every partial of sum
//    n + 1, which each CTA posts after reading sum n, so a buffer is never overwritten while read.
//    Every wait is bounded (on expiry: GS_DEV_ERR_TIMEOUT, and the kernel runs on to its end).
constexpr int kMgsCtas = 8;
constexpr int kMgsThreads = 256;
static_assert(kPanel == 16, "the sums' butterfly gives lane l entry l & 15");

__global__ void __launch_bounds__(kMgsThreads) k_panel_gs2(double* __restrict__ V, double* __restrict__ Qw, int D,
                                                          int bp, int p0, double tau, const double* __restrict__ cn,
                                                          double* __restrict__ R64, int ldr,
                                                          const int* __restrict__ r_start, int* __restrict__ r_next,
                                                          int rmax, const PanelState* __restrict__ st) {
    using namespace ptx;
    if (!st->slow) return;  // k_panel_chol has done this panel (the same flag in every CTA)
    __shared__ double part[2][kMgsCtas][kPanel];  // per sum: every CTA's partials (stored by that CTA)
    __shared__ double red[kMgsThreads / 32][kPanel];
    __shared__ uint64_t pbar[2];                  // one barrier per partial buffer: 1 arrival + the bytes
    __shared__ double total[kPanel];              // the last sum, added once for the whole CTA
    const uint32_t rank = cluster_ctarank();
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int S = (D + kMgsCtas - 1) / kMgsCtas;
    const int c0 = (int)rank * S, c1 = min(D, c0 + S);
    const int r0 = *r_start;
    int r = r0, nsum = 0;
    bool ok = true;  // false once a wait has run out (the results are then flagged as an error)
    if (tid == 0) {
        mbar_init(&pbar[0], 1);
        mbar_init(&pbar[1], 1);
        fence_barrier_init();
    }
    cluster_sync_all();  // every CTA's barriers exist before anyone stores into its memory

    // the sum over the cluster of acc[0..kPanel) (this thread's part): reduced in the CTA, stored into
    // every CTA, added in CTA order; the result is identical in every thread of every CTA
    auto cluster_sum = [&](double (&acc)[kPanel], double (&out)[kPanel]) {
        // warp: a butterfly over the lane bits 3..0 leaves lane l with the sum of entry l & 15 over
        // its half-warp (after the step with lane bit b a lane keeps the entries whose index has bit
        // b equal to its own), then the two half-warps are added: 16 shuffles instead of 80
#pragma unroll
        for (int wb = kPanel / 2; wb >= 1; wb >>= 1) {
            const bool up = (lane & wb) != 0;
#pragma unroll
            for (int j = 0; j < wb; ++j) {
                const double send = up ? acc[j] : acc[j + wb];
                const double keep = up ? acc[j + wb] : acc[j];
                acc[j] = keep + __shfl_xor_sync(0xffffffffu, send, wb);
            }
        }
        acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 16);
        __syncthreads();  // red and the last sum's buffer have been read by every thread of this CTA
        if (lane < kPanel) red[w][lane] = acc[0];
        __syncthreads();
        const int slot = nsum & 1;
        const uint32_t parity = (uint32_t)(nsum >> 1) & 1u;
        if (tid == 0) mbar_arrive_expect_tx(&pbar[slot], (uint32_t)(kMgsCtas * kPanel * sizeof(double)));
        if (tid < kPanel * kMgsCtas) {
            const int j = tid % kPanel, dest = tid / kPanel;
            double v = 0.0;
            for (int ww = 0; ww < kMgsThreads / 32; ++ww) v += red[ww][j];
            st_async_f64(mapa_shared(smem_u32(&part[slot][rank][j]), (uint32_t)dest), v,
                         mapa_shared(smem_u32(&pbar[slot]), (uint32_t)dest));
        }
        // sixteen threads wait for every CTA's partials and add them (fp64 adds run at a low rate
        // on GB300: every thread adding all 128 had cost ~9 us a sum)
        if (tid < kPanel) {
            if (ok) {
                const unsigned long long t0 = globaltimer();
                for (uint32_t it = 0; !mbar_try_wait_cluster(&pbar[slot], parity); ++it)
                    if ((it & 255u) == 255u && globaltimer() - t0 > kWaitLimitNs) {
                        atomicOr(&g_err_build, GS_DEV_ERR_TIMEOUT);
                        ok = false;
                        break;
                    }
            }
            double v = 0.0;
            for (int c = 0; c < kMgsCtas; ++c) v += part[slot][c][tid];
            total[tid] = v;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kPanel; ++j) out[j] = total[j];
        ++nsum;
    };

    for (int k = 0; k < bp; ++k) {
        double* v = V + (size_t)k * D;
        double* Rrow = R64 + (size_t)(p0 + k) * ldr;
        const int nj = r - r0;  // the panel's new directions so far
        for (int pass = 0; pass < 2; ++pass) {
            double acc[kPanel], h[kPanel];
#pragma unroll
            for (int j = 0; j < kPanel; ++j) acc[j] = 0.0;
            for (int d = c0 + tid; d < c1; d += kMgsThreads) {
                const double x = v[d];
#pragma unroll
                for (int j = 0; j < kPanel; ++j)
                    if (j < nj) acc[j] += Qw[(size_t)(r0 + j) * D + d] * x;
            }
            cluster_sum(acc, h);
            for (int d = c0 + tid; d < c1; d += kMgsThreads) {
                double x = v[d];
#pragma unroll
                for (int j = 0; j < kPanel; ++j)
                    if (j < nj) x -= h[j] * Qw[(size_t)(r0 + j) * D + d];
                v[d] = x;
            }
            if (rank == 0 && tid < nj) {
                double hv = 0.0;  // h[tid] without a dynamic index (which would move h to local memory)
#pragma unroll
                for (int j = 0; j < kPanel; ++j)
                    if (j == tid) hv = h[j];
                Rrow[r0 + tid] += hv;
            }
        }
        double acc[kPanel], nn[kPanel];
#pragma unroll
        for (int j = 0; j < kPanel; ++j) acc[j] = 0.0;
        for (int d = c0 + tid; d < c1; d += kMgsThreads) acc[0] += v[d] * v[d];
        cluster_sum(acc, nn);
        const double nu = sqrt(nn[0]);
        if (nu > tau * cn[p0 + k] && r < rmax) {
            double* q = Qw + (size_t)r * D;
            for (int d = c0 + tid; d < c1; d += kMgsThreads) q[d] = v[d] / nu;
            if (rank == 0 && tid == 0) Rrow[r] = nu;
            ++r;
        }
    }
    if (rank == 0 && tid == 0) *r_next = r;
    cluster_sync_all();  // no CTA leaves while a peer may still store into its memory
}

// ----------------------------------------------------------------- finalisation
__global__ void k_cast_rows(const double* __restrict__ src, long long lds, float* __restrict__ dst,
                            long long ldd, int rows, int cols) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)rows * cols) return;
    const int i = (int)(idx / cols), j = (int)(idx % cols);
    dst[(size_t)i * ldd + j] = (float)src[(size_t)i * lds + j];
}

// rlen[i] = 1 + last nonzero column of R_i among the first r; chunk max per 32 rows
__global__ void k_rlen(const double* __restrict__ R64, int ldr, int M, int r, int* __restrict__ rlen) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M) return;
    int last = 0;
    for (int j = 0; j < r; ++j)
        if (R64[(size_t)i * ldr + j] != 0.0) last = j + 1;
    rlen[i] = last;
}

__global__ void k_rlen_chunk(const int* __restrict__ rlen, int M, int* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c * 32 >= M) return;
    int m = 0;
    for (int i = c * 32; i < min(M, c * 32 + 32); ++i) m = max(m, rlen[i]);
    out[c] = m;
}

// Counter-based 32-bit mixer (the "lowbias32" integer hash).
__device__ __forceinline__ uint32_t mix32(uint32_t x) {
    x ^= x >> 16;
    x *= 0x7feb352du;
    x ^= x >> 15;
    x *= 0x846ca68bu;
    x ^= x >> 16;
    return x;
}

// Unbiased dithered (stochastic) rounding of a basis entry to fp16: round to
// the fp16 neighbour below or above in magnitude with probability given by the
// remainder, using a fixed hash of the element index.  The expected value is
// the input, and the rounding errors of different elements are independent
// even where the basis has few distinct magnitudes (the first basis vector of
// a bipolar codebook is +-1/sqrt(D) everywhere), so in X Q^T they average out
// over D instead of adding up coherently.  |q| <= 1, so no overflow.
__device__ __forceinline__ __half dither_half(double qd, unsigned long long index) {
    const float f = (float)qd;
    const __half lo = __float2half_rz(f);
    const float lof = __half2float(lo);
    if (lof == f) return lo;
    const __half hi = __ushort_as_half((unsigned short)(__half_as_ushort(lo) + 1));
    const float hif = __half2float(hi);
    const float frac = (f - lof) / (hif - lof);
    const uint32_t hsh = mix32((uint32_t)index ^ mix32((uint32_t)(index >> 32) + 0x9e3779b9u));
    const float u = (float)(hsh >> 8) * (1.0f / 16777216.0f);
    return u < frac ? hi : lo;
}

// Q16[j][d] (r x ldq) and Q16t[d][j] (D x ldt) from Qw (fp64, r x D); zero padding.
__global__ void k_q16(const double* __restrict__ Qw, int r, int D, __half* __restrict__ Q16, int ldq,
                      __half* __restrict__ Q16t, int ldt) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)r * ldq) return;
    const int j = (int)(idx / ldq), d = (int)(idx % ldq);
    __half hv = __float2half(0.0f);
    if (d < D) hv = dither_half(Qw[(size_t)j * D + d], (unsigned long long)j * D + d);
    Q16[idx] = hv;
    if (Q16t && d < D) Q16t[(size_t)d * ldt + j] = hv;
}

// dst[d][j] (cols x ldt fp16) = dithered rounding of src[j][d] (rows x cols fp32, ld lds), through
// 32 x 32 tiles in shared memory (coalesced reads and writes); the transposed operand of a
// reconstruction from fp32 rows that are not the basis itself (the basis bound with a partner).
__global__ void k_f16t_dither(const float* __restrict__ src, int rows, int cols, long long lds,
                              __half* __restrict__ dst, long long ldt) {
    __shared__ float tile[32][33];
    const int j0 = blockIdx.y * 32, d0 = blockIdx.x * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;  // 256 threads: 8 rows per step
    for (int k = ty; k < 32; k += 8) {
        const int j = j0 + k, d = d0 + tx;
        tile[k][tx] = (j < rows && d < cols) ? src[(size_t)j * lds + d] : 0.f;
    }
    __syncthreads();
    for (int k = ty; k < 32; k += 8) {
        const int d = d0 + k, j = j0 + tx;
        if (d < cols && j < rows)
            dst[(size_t)d * ldt + j] = dither_half((double)tile[tx][k], (unsigned long long)j * cols + d);
    }
}

__global__ void k_zero_half(__half* p, long long n) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = __float2half(0.0f);
}

inline unsigned grid1(long long n, int b) { return (unsigned)((n + b - 1) / b); }

// fp32 rows (ld lds) -> fp64 rows (ld ldd)
__global__ void k_widen_rows(const float* __restrict__ src, long long lds, double* __restrict__ dst,
                             long long ldd, int rows, int cols) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)rows * cols) return;
    const int i = (int)(idx / cols), j = (int)(idx % cols);
    dst[(size_t)i * ldd + j] = (double)src[(size_t)i * lds + j];
}

// ||R_i|| in fp64, one thread per row (C = R Q with orthonormal Q, so this is ||c_i||)
__global__ void k_row_norms64(const double* __restrict__ R64, int ldr, int M, int r, double* __restrict__ cn) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M) return;
    double ss = 0.0;
    for (int j = 0; j < r; ++j) ss += R64[(size_t)i * ldr + j] * R64[(size_t)i * ldr + j];
    cn[i] = sqrt(ss);
}

struct DevBuf {
    void* p = nullptr;
    ~DevBuf() { if (p) cudaFree(p); }
};

}  // namespace

unsigned take_device_error_build() {
    unsigned v = 0, z = 0;
    cudaMemcpyFromSymbol(&v, g_err_build, sizeof(v));
    if (v) cudaMemcpyToSymbol(g_err_build, &z, sizeof(z));
    return v;
}

#define GS_CK(x)                                                     \
    do {                                                             \
        cudaError_t e_ = (x);                                        \
        if (e_ != cudaSuccess) {                                     \
            return e_ == cudaErrorMemoryAllocation ? GS_ERR_NOMEM : GS_ERR_CUDA; \
        }                                                            \
    } while (0)

gs_status finalize_basis(const double* Qw, const double* R64, int ldr, const double* cn, int M, int D, int r,
                         cudaStream_t s, gs_basis* h);

// The fp64 factorisation C = R Q of M rows of C (Q: r x D orthonormal rows, R: M x r lower
// echelon, ldr = min(M, D); cn: the rows' norms), kept on the device.
struct Factor {
    double* Qw = nullptr;
    double* R64 = nullptr;
    double* cn = nullptr;
    int r = 0, ldr = 1;
    Factor() = default;
    Factor(const Factor&) = delete;
    Factor& operator=(const Factor&) = delete;
    ~Factor() {
        cudaFree(Qw);
        cudaFree(R64);
        cudaFree(cn);
    }
};

gs_status factor_rows(const float* C, int M, int D, int ldc, double tau, bool normalize, cudaStream_t s,
                      Factor& f) {
    const int rmax = std::min(M, D);
    const int ldr = rmax;                       // R64 leading dimension
    const int ldh = std::max(1, ((M + 15) / 16) * 16);  // >= any r0
    const int npanels = (M + kPanel - 1) / kPanel;
    // column slices: one per SM, at most kMaxSlice columns each; whole clusters of CTAs
    int dev = 0, sms = 0;
    GS_CK(cudaGetDevice(&dev));
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    sms = std::max(sms, kSliceCluster) / kSliceCluster * kSliceCluster;
    const int w = std::max(8, std::min(kMaxSlice, (D + sms - 1) / sms));
    const int nslices = ((D + w - 1) / w + kSliceCluster - 1) / kSliceCluster * kSliceCluster;
    const int ncl = nslices / kSliceCluster;
    // threads: the update's kPanel w outputs in as few full rounds as fit (at most three of 512)
    const int rounds = (kPanel * w + kSliceThreads - 1) / kSliceThreads;
    int threads = ((kPanel * w + rounds - 1) / rounds + 31) / 32 * 32;
    if (threads < 320) threads = kSliceThreads;  // short rows: few outputs, so longer chunks of the basis instead
    const int jc = threads / kPanel * 2;        // basis rows per chunk: two dot products a thread
    const int vl = w | 1;
    const size_t smem = slice_smem(w, jc);
    const size_t smem_chol = sizeof(double) * (size_t)kPanel * vl;
    // longest chains of sums behind an entry of a Gram matrix (w / 2 terms in a slice, the cluster's CTAs, the
    // clusters) and behind a pivot (kPanel steps), a unit roundoff each, and twice that for the second order
    const double gerr = 0x1p-52 * (w / 2 + kSliceCluster + ncl + kPanel + 4);
    // the limit belongs to the function on the device: one that covers every D, since another thread may be
    // building from rows of another length at the same time
    for (auto fn : {k_panel_slice<kDots1>, k_panel_slice<kUpdDots>, k_panel_slice<kUpdGram>})
        GS_CK(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSliceSmemMax));

    // the factors, and one workspace for everything else
    GS_CK(cudaMalloc(&f.Qw, sizeof(double) * (size_t)rmax * D));
    GS_CK(cudaMalloc(&f.R64, sizeof(double) * (size_t)M * ldr));
    GS_CK(cudaMalloc(&f.cn, sizeof(double) * (size_t)M));
    const size_t nV = (size_t)kPanel * D, nH = (size_t)kPanel * ldh, nHp = (size_t)nslices * kPanel * ldh,
                 nG = (size_t)ncl * kPairs, nst = (sizeof(PanelState) + 7) / 8;
    DevBuf ws;
    GS_CK(cudaMalloc(&ws.p, sizeof(double) * (nV + nH + nHp + 2 * nG + (size_t)M + nst) +
                                sizeof(int) * (size_t)(npanels + 1)));
    double* Qw = f.Qw;
    double* R64 = f.R64;
    double* cn = f.cn;
    double* V = (double*)ws.p;
    double* H = V + nV;
    double* Hp = H + nH;
    double* G1 = Hp + nHp;
    double* G2 = G1 + nG;
    double* sc = G2 + nG;
    PanelState* st = (PanelState*)(sc + M);
    int* r_at = (int*)(sc + M + nst);  // r_at[p]: the rank at the start of panel p
    GS_CK(cudaMemsetAsync(R64, 0, sizeof(double) * (size_t)M * ldr, s));
    GS_CK(cudaMemsetAsync(r_at, 0, sizeof(int), s));
    k_row_norms<<<M, 256, 0, s>>>(C, ldc, D, normalize ? 1 : 0, cn, sc);

    auto clustered = [&](int ctas, int cluster, int nthreads, size_t sm_bytes, cudaLaunchAttribute* at) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)ctas);
        cfg.blockDim = dim3((unsigned)nthreads);
        cfg.dynamicSmemBytes = sm_bytes;
        cfg.stream = s;
        at->id = cudaLaunchAttributeClusterDimension;
        at->val.clusterDim.x = (unsigned)cluster;
        at->val.clusterDim.y = 1;
        at->val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        return cfg;
    };
    for (int pn = 0; pn < npanels; ++pn) {
        const int p0 = pn * kPanel, bp = std::min(kPanel, M - p0);
        SliceParams sp;
        sp.C = C + (size_t)p0 * ldc, sp.ldc = ldc;
        sp.sc = sc + p0, sp.cn = cn + p0;
        sp.V = V, sp.Qw = Qw;
        sp.D = D, sp.w = w, sp.bp = bp, sp.jc = jc;
        sp.r_start = r_at + pn;
        sp.H = H, sp.Hp = Hp, sp.ldh = ldh;
        sp.Gp = G1;
        if (p0 > 0) {
            const unsigned rgrid = grid1((long long)bp * std::min(p0, rmax), 16);
            double* Rp = R64 + (size_t)p0 * ldr;
            k_panel_slice<kDots1><<<nslices, threads, smem, s>>>(sp);
            k_panel_reduce<<<rgrid, 256, 0, s>>>(Hp, nslices, bp, sp.r_start, ldh, H, Rp, ldr);
            k_panel_slice<kUpdDots><<<nslices, threads, smem, s>>>(sp);
            k_panel_reduce<<<rgrid, 256, 0, s>>>(Hp, nslices, bp, sp.r_start, ldh, H, Rp, ldr);
        }
        cudaLaunchAttribute at[1];
        cudaLaunchConfig_t cfg = clustered(nslices, kSliceCluster, threads, smem, at);
        GS_CK(cudaLaunchKernelEx(&cfg, k_panel_slice<kUpdGram>, (const SliceParams)sp));
        CholParams cp;
        cp.V = V, cp.Qw = Qw;
        cp.D = D, cp.w = w, cp.bp = bp, cp.ncl = ncl;
        cp.Gp = G1, cp.Gp2 = G2;
        cp.cn = cn + p0, cp.tau = tau, cp.gerr = gerr;
        cp.R64 = R64 + (size_t)p0 * ldr, cp.ldr = ldr, cp.rmax = rmax;
        cp.r_start = r_at + pn, cp.r_next = r_at + pn + 1;
        cp.st = st;
        cfg = clustered(nslices, kSliceCluster, 512, smem_chol, at);
        GS_CK(cudaLaunchKernelEx(&cfg, k_panel_chol<1>, (const CholParams)cp));
        cp.Gp = G2;
        k_panel_chol<2><<<nslices, 512, smem_chol, s>>>(cp);
        cfg = clustered(kMgsCtas, kMgsCtas, kMgsThreads, 0, at);
        GS_CK(cudaLaunchKernelEx(&cfg, k_panel_gs2, V, Qw, D, bp, p0, tau, (const double*)cn, R64, ldr,
                                 (const int*)(r_at + pn), r_at + pn + 1, rmax, (const PanelState*)st));
    }
    const int* r_dev = r_at + npanels;
    GS_CK(cudaGetLastError());
    int r = 0;
    GS_CK(cudaMemcpyAsync(&r, r_dev, sizeof(int), cudaMemcpyDeviceToHost, s));
    GS_CK(cudaStreamSynchronize(s));
    // a bounded wait of the panel kernel that ran out leaves the factorisation unusable
    if (take_device_error_build() & GS_DEV_ERR_TIMEOUT) return GS_ERR_TIMEOUT;
    f.r = r;
    f.ldr = ldr;
    return GS_OK;
}

gs_status build_basis(const float* C, int M, int D, int ldc, double tau, bool normalize,
                      cudaStream_t s, gs_basis* h) {
    Factor f;
    gs_status st = factor_rows(C, M, D, ldc, tau, normalize, s, f);
    if (st != GS_OK) return st;
    return finalize_basis(f.Qw, f.R64, f.ldr, f.cn, M, D, f.r, s, h);
}

// Sec. 3.1, D < M: the entries are split into subsets, each gets its own orthonormal basis,
// and the reconstructions are concatenated.  Group g (rows [off[g], off[g+1]) of C) is
// factored alone; the handle holds the stacked Q = [Q_0; Q_1; ...] (r = sum of r_g rows) and
// the block-diagonal R whose row i of group g holds R_g's row in columns [s_g, s_g + r_g),
// s_g = r_0 + ... + r_(g-1).  C = R Q holds row by row, so every call on the handle works
// unchanged (Q's rows are orthonormal within a group, not across groups).
gs_status build_basis_grouped(const float* C, int M, int D, int ldc, const int* off, int G, double tau,
                              bool normalize, cudaStream_t s, gs_basis* h) {
    std::vector<std::unique_ptr<Factor>> fs;
    int rt = 0;
    for (int g = 0; g < G; ++g) {
        fs.emplace_back(new Factor());
        gs_status st = factor_rows(C + (size_t)off[g] * ldc, off[g + 1] - off[g], D, ldc, tau, normalize, s,
                                   *fs.back());
        if (st != GS_OK) return st;
        rt += fs.back()->r;
    }
    const int ldr = std::max(rt, 1);
    DevBuf bQ, bR, bcn;
    GS_CK(cudaMalloc(&bQ.p, sizeof(double) * (size_t)ldr * D));
    GS_CK(cudaMalloc(&bR.p, sizeof(double) * (size_t)M * ldr));
    GS_CK(cudaMalloc(&bcn.p, sizeof(double) * (size_t)M));
    double* Q = (double*)bQ.p;
    double* R = (double*)bR.p;
    double* cn = (double*)bcn.p;
    GS_CK(cudaMemsetAsync(R, 0, sizeof(double) * (size_t)M * ldr, s));
    h->grp_rows.assign(off, off + G + 1);
    h->grp_coeffs.assign(1, 0);
    int sg = 0;
    for (int g = 0; g < G; ++g) {
        const Factor& f = *fs[g];
        const int mg = off[g + 1] - off[g];
        if (f.r > 0) {
            GS_CK(cudaMemcpyAsync(Q + (size_t)sg * D, f.Qw, sizeof(double) * (size_t)f.r * D,
                                  cudaMemcpyDeviceToDevice, s));
            GS_CK(cudaMemcpy2DAsync(R + (size_t)off[g] * ldr + sg, sizeof(double) * ldr, f.R64,
                                    sizeof(double) * f.ldr, sizeof(double) * f.r, mg, cudaMemcpyDeviceToDevice,
                                    s));
        }
        GS_CK(cudaMemcpyAsync(cn + off[g], f.cn, sizeof(double) * mg, cudaMemcpyDeviceToDevice, s));
        sg += f.r;
        h->grp_coeffs.push_back(sg);
    }
    return finalize_basis(Q, R, ldr, cn, M, D, rt, s, h);
}

// Everything a handle holds besides the fp64 factorisation: fp32 Q, R and norms for the
// caller, R's echelon lengths, the fp16 operand copies (dithered) and the chunk scratch.
gs_status finalize_basis(const double* Qw, const double* R64, int ldr, const double* cn, int M, int D, int r,
                         cudaStream_t s, gs_basis* h) {
    h->M = M;
    h->D = D;
    h->r = r;
    h->ldr = std::max(r, 1);

    // user-visible fp32 results
    GS_CK(cudaMalloc(&h->Q, sizeof(float) * (size_t)std::max(r, 1) * D));
    GS_CK(cudaMalloc(&h->R, sizeof(float) * (size_t)M * h->ldr));
    GS_CK(cudaMalloc(&h->cnorm, sizeof(float) * (size_t)M));
    GS_CK(cudaMalloc(&h->rlen, sizeof(int) * (size_t)M));
    GS_CK(cudaMalloc(&h->rlen_chunk, sizeof(int) * (size_t)((M + 31) / 32)));
    GS_CK(cudaMemsetAsync(h->R, 0, sizeof(float) * (size_t)M * h->ldr, s));
    if (r > 0) {
        k_cast_rows<<<grid1((long long)r * D, 256), 256, 0, s>>>(Qw, D, h->Q, D, r, D);
        k_cast_rows<<<grid1((long long)M * r, 256), 256, 0, s>>>(R64, ldr, h->R, h->ldr, M, r);
    }
    k_cast_rows<<<grid1(M, 256), 256, 0, s>>>(cn, 1, h->cnorm, 1, M, 1);
    k_rlen<<<grid1(M, 128), 128, 0, s>>>(R64, ldr, M, r, h->rlen);
    k_rlen_chunk<<<grid1((M + 31) / 32, 128), 128, 0, s>>>(h->rlen, M, h->rlen_chunk);

    // tensor-core operand copies (fp16, dithered)
    if (r > 0) {
        h->ldq16 = (D + 7) / 8 * 8;
        h->ldr16 = (r + 7) / 8 * 8;
        GS_CK(cudaMalloc(&h->Q16, sizeof(__half) * (size_t)r * h->ldq16));
        GS_CK(cudaMalloc(&h->Q16t, sizeof(__half) * (size_t)D * h->ldr16));
        if (h->ldr16 != r)
            k_zero_half<<<grid1((long long)D * h->ldr16, 256), 256, 0, s>>>(h->Q16t, (long long)D * h->ldr16);
        k_q16<<<grid1((long long)r * h->ldq16, 256), 256, 0, s>>>(Qw, r, D, h->Q16, h->ldq16, h->Q16t,
                                                                  h->ldr16);
    }

    // scratch for the chunked multi-kernel paths: rows x (r + M + 1) floats
    const long long per_row = (long long)r + M + 1;
    long long rows = std::max(256LL, (64LL << 20) / per_row);
    rows = std::min(rows, 65536LL);
    h->chunk_rows = rows;
    h->scratch_floats = rows * per_row;
    GS_CK(cudaMalloc(&h->scratch, sizeof(float) * (size_t)h->scratch_floats));
    GS_CK(cudaGetLastError());
    GS_CK(cudaStreamSynchronize(s));
    return GS_OK;
}

cudaError_t launch_f16t_dither(const float* src, int rows, int cols, long long lds, void* dst, long long ldt,
                               cudaStream_t s) {
    if (rows <= 0 || cols <= 0) return cudaSuccess;
    const dim3 grid((unsigned)((cols + 31) / 32), (unsigned)((rows + 31) / 32));
    if (grid.y > 65535u) return cudaErrorInvalidConfiguration;
    k_f16t_dither<<<grid, 256, 0, s>>>(src, rows, cols, lds, static_cast<__half*>(dst), ldt);
    return cudaGetLastError();
}

}  // namespace gs

namespace gs {

gs_status import_basis(const float* Q, int ldq, const float* R, int ldr_in, const float* cnorm, int M, int D,
                       int r, cudaStream_t s, gs_basis* h) {
    const int ldr = std::max(r, 1);
    DevBuf bQw, bR64, bcn;
    GS_CK(cudaMalloc(&bQw.p, sizeof(double) * (size_t)std::max(r, 1) * D));
    GS_CK(cudaMalloc(&bR64.p, sizeof(double) * (size_t)M * ldr));
    GS_CK(cudaMalloc(&bcn.p, sizeof(double) * (size_t)M));
    double* Qw = (double*)bQw.p;
    double* R64 = (double*)bR64.p;
    double* cn = (double*)bcn.p;
    GS_CK(cudaMemsetAsync(R64, 0, sizeof(double) * (size_t)M * ldr, s));
    if (r > 0) {
        k_widen_rows<<<grid1((long long)r * D, 256), 256, 0, s>>>(Q, ldq, Qw, D, r, D);
        k_widen_rows<<<grid1((long long)M * r, 256), 256, 0, s>>>(R, ldr_in, R64, ldr, M, r);
    }
    if (cnorm)
        k_widen_rows<<<grid1(M, 256), 256, 0, s>>>(cnorm, 1, cn, 1, M, 1);
    else
        k_row_norms64<<<grid1(M, 128), 128, 0, s>>>(R64, ldr, M, r, cn);
    GS_CK(cudaGetLastError());
    return finalize_basis(Qw, R64, ldr, cn, M, D, r, s, h);
}

}  // namespace gs
