// gs_gemm_x3.cu -- fp32-accurate GEMM on the tensor cores for large fp32 products that no 16-bit
// operand copy may serve: operands of any alignment and leading dimension, bf16 or fp32 A, short
// rows.
//
//     C = alpha * A op(B)          (optionally divided by rownorm[i] * colnorm[j])
//
//   A  m x K row-major, fp32 or bf16; B  fp32, n x K (b_trans) or K x n; C  fp32 or bf16; batched.
//
// Every fp32 operand is the sum of three bf16 numbers, x = h + m + l: h = bf16(x), m = bf16(x - h),
// l = bf16(x - h - m), each difference exact in fp32, 3 x 8 significant bits.  m and l are kept as 2^8 m and
// 2^16 l, no larger than x: bf16 ends at 2^-133, and without the factors every operand below 2^-110 lost
// bits of l, then of m (at 1e-37, 5e-4 of a row; now 6e-8 down to fp32's subnormals).  Six of the nine
// products (hh, hm, mh, mm, hl, lh) are taken on the tensor core; the three left out are below 2^-24 of each
// term.  The tensor core's fp32 accumulation loses a bounded amount at every step, which grows with the
// number of steps rather than with its square root, so (1) hh has an accumulator of its own, as have the
// products of each of the two scales, hm + mh and mm + hl + lh (their sums are ~2^-8 and 2^-16 of hh's, and so
// are their losses), and (2) hh's accumulator is emptied every kChunk K-blocks (128 terms)
// into fp32 registers (round to nearest).  Relative error against 64 bits, 16,384 x 922 -> 10,000:
// 9e-8, the CUDA-core GEMM's 5.4e-7; at 300 terms 9e-8 and 3.1e-7.  (Chunks of 256 terms: 1.3e-7 at the
// same speed, but 4.9e-7 against 4.1e-7 where all terms of a sum have one sign; of 512: 2.4e-7.)
// Outputs of a thread that holds one that is not finite (an operand that is not, or beyond 2^120, where
// the factors overflow) are computed again as plain fp32 dot products, so infinities and NaN come out as the
// CUDA-core GEMM has them.
//
// Measured (GB300, reconstruction of 16,384 rows, r = 922, D = 10,000, rows of 922 floats): 8,240 us on
// the CUDA cores (36.7 TFLOP/s), 1,800 us here (168 TFLOP/s; 1,734 without the factors and their third
// accumulator; multiplying both differences on the way, rather than what the second is taken from, 1,900).
// What bounds it: the converters' loads
// (long scoreboard is the top stall, the tensor pipe 40 % active).  Shared memory would be next: per
// K-block of 32 a 128 x 128 tile writes 48 KB of operand planes and its 12 MMAs read 96 KB of them,
// 1125 clk at 128 B/clk against 768 clk of MMA.  Tried: one group of eleven converter warps (3,670 to
// 4,000 us: every load's latency exposed, and code long enough to miss the instruction cache), one pair
// of k per lane with four-byte stores (1,785 us), loading A's next K-block before the hand-over
// (2,000 us: the hand-over's arrive waits for it), B's parts kept in memory and loaded by TMA (1,650 us, for
// 6 more bytes an entry of the basis).  Timing copies of that form say that no single part holds it: 4 to
// 17 % less time without A's loads, without the split's arithmetic, without stores, or with a third of the
// MMAs; the converters issue at 0.33 instructions a clock and sub-partition, two warps each.
// Sixteen converter warps, their registers taken from the other roles, ran no faster (1,877 against 1,860
// us; 20,000 x 131 -> 777 98 against 104).
//
// No workspace (but a K split's partial products, in the caller's) and no pass over the operands
// beforehand: rows that start anywhere are read with plain loads (no TMA), so nothing is allocated and
// calls on different streams share nothing.
//
// Warp roles (544 threads): 0 TMEM allocator + MMA issuer, 1-8 epilogue (two per TMEM lane quadrant,
// 64 columns each), 9-16 converters in two groups taking alternate K-blocks.  Every wait is bounded
// (see gs_tc_ptx.cuh).

#include <algorithm>
#include <cmath>

#include "gs_internal.h"
#include "gs_tc_ptx.cuh"

namespace gs {
namespace {

using namespace ptx;

__device__ unsigned g_err_x3 = 0;

constexpr int kBM = 128, kBN = 128, kBK = 32;
constexpr int kEpi0 = 1, kEpiWarps = 8;
constexpr int kCvt0 = kEpi0 + kEpiWarps, kCvtGroups = 2, kCvtGroupWarps = 4;
constexpr int kCvtWarps = kCvtGroups * kCvtGroupWarps;
constexpr int kThreads = (kCvt0 + kCvtWarps) * 32;  // 544: at most five warps a sub-partition, 96 registers each
constexpr int kPlane = 128 * 64 * 2;                // 16 KB: one bf16 plane of 128 rows, two K-blocks wide
constexpr int kPairBytes = 6 * kPlane;              // A h, m, l then B h, m, l of two K-blocks
constexpr int kStages = 4;                          // K-blocks: stage s is half s & 1 of pair s >> 1
constexpr int kChunk = 4;                           // K-blocks of hh summed on the tensor core at a time
constexpr int kSlots = 4;                           // tasks of one warp, per operand: 16 tasks over four warps
constexpr int kTmemCols = 512;                      // hh: 2 x 128, then hm + mh and mm + hl + lh: 128 each
constexpr uint32_t kColMid = 256, kColLow = 384;
constexpr float kPartScale = 256.f;                 // m and l are kept as 2^8 m and 2^16 l

struct X3Params {
    const void* A;
    const float* B;
    void* C;
    long long lda, ldb, ldc, a_bs, b_bs, c_bs;
    long long m, tiles_m, tiles;
    int n, k, nt, tiles_n, nkb;
    int k_last;          // K of the last batch plane (a K split's planes are chunks of one product)
    long long last;      // that plane
    int c_bf16, c_vec;
    float alpha;
    const float* rownorm;
    const float* colnorm;
    const int* b_rowlen;  // as in GemmArgs: B's row j is zero from there on
};

struct Ctl {
    uint64_t full[kStages], empty[kStages];
    uint64_t a_full[2], a_empty[2], x_empty;
    uint64_t mma_done;
    uint32_t tmem_base;
    int abort_flag;
};

// a converter group's position: its K-block, and where the tile's operands start
struct Step {
    int kb;
    const char* A;   // first row of A (in its batch plane), first row or column of B
    const char* B;
    int rows, cols;  // valid rows of A and columns of C in the tile
    int k;           // K of the tile's plane
};

template <int TA>
__device__ __forceinline__ float lda1(const void* p, long long i) {
    return TA == MAT_F32 ? __ldg((const float*)p + i) : __bfloat162float(((const __nv_bfloat16*)p)[i]);
}

// Eight consecutive elements (4 pairs) of a row.  VEC: log2 of the elements that one load may take
// (the row's start is aligned to them: 2, 1 or 0).  The slow form, for a K-block that K ends in, loads
// element by element, clamped to the row's last, and zeroes what lies past it.
template <int T, int VEC>
__device__ __forceinline__ void ld8(const char* p, float2 (&v)[4]) {
    if (T == MAT_F32) {
        if (VEC == 2) {
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float4 x = __ldg(reinterpret_cast<const float4*>(p) + u);
                v[2 * u] = make_float2(x.x, x.y);
                v[2 * u + 1] = make_float2(x.z, x.w);
            }
        } else if (VEC == 1) {
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = __ldg(reinterpret_cast<const float2*>(p) + u);
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                v[u] = make_float2(__ldg(reinterpret_cast<const float*>(p) + 2 * u),
                                   __ldg(reinterpret_cast<const float*>(p) + 2 * u + 1));
        }
    } else {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            uint32_t w;
            if (VEC >= 1) {
                w = __ldg(reinterpret_cast<const unsigned*>(p) + u);
            } else {
                const uint32_t w0 = __ldg(reinterpret_cast<const unsigned short*>(p) + 2 * u);
                const uint32_t w1 = __ldg(reinterpret_cast<const unsigned short*>(p) + 2 * u + 1);
                w = w0 | (w1 << 16);
            }
            v[u] = make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
        }
    }
}
template <int T>
__device__ __forceinline__ void ld8_end(const char* row, int k, int K, float2 (&v)[4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int k0 = k + 2 * u;
        v[u].x = lda1<T>(row, min(k0, K - 1));
        v[u].y = lda1<T>(row, min(k0 + 1, K - 1));
        if (k0 >= K) v[u].x = 0.f;
        if (k0 + 1 >= K) v[u].y = 0.f;
    }
}

// (a, b) minus the two bf16 values packed in w, exact here
__device__ __forceinline__ float2 sub_bf16x2(float2 a, uint32_t w) {
    float2 r;
    asm("{\n\t.reg .b64 x, y, z;\n\t"
        "mov.b64 x, {%2, %3};\n\t"
        "mov.b64 y, {%4, %5};\n\t"
        "sub.rn.f32x2 z, x, y;\n\t"
        "mov.b64 {%0, %1}, z;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(__uint_as_float(w << 16)), "f"(__uint_as_float(w & 0xffff0000u)));
    return r;
}

__device__ __forceinline__ float2 scale_part(float2 a) {
    float2 r;
    asm("{\n\t.reg .b64 x, y, z;\n\t"
        "mov.b64 x, {%2, %3};\n\t"
        "mov.b64 y, {%4, %4};\n\t"
        "mul.rn.f32x2 z, x, y;\n\t"
        "mov.b64 {%0, %1}, z;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(kPartScale));
    return r;
}

// a minus kPartScale times the two bf16 values packed in w, exact here
__device__ __forceinline__ float2 sub_scaled_bf16x2(float2 a, uint32_t w) {
    float2 r;
    asm("{\n\t.reg .b64 x, y, z, s;\n\t"
        "mov.b64 x, {%2, %3};\n\t"
        "mov.b64 y, {%4, %5};\n\t"
        "mov.b64 s, {%6, %6};\n\t"
        "fma.rn.f32x2 z, y, s, x;\n\t"
        "mov.b64 {%0, %1}, z;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(__uint_as_float(w << 16)), "f"(__uint_as_float(w & 0xffff0000u)), "f"(-kPartScale));
    return r;
}

// two elements into their three bf16 parts h, 2^8 m and 2^16 l, packed
__device__ __forceinline__ void split3(float2 x, uint32_t& h, uint32_t& m, uint32_t& l) {
    h = pack_bf16(x.x, x.y);
    x = scale_part(sub_bf16x2(x, h));
    m = pack_bf16(x.x, x.y);
    x = sub_scaled_bf16x2(scale_part(x), m);
    l = pack_bf16(x.x, x.y);
}

template <int TA, bool BT, int VEC>
__global__ void __maxnreg__(96) k_gemm_x3(const __grid_constant__ X3Params p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* base = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    Ctl& c = *reinterpret_cast<Ctl*>(base + (size_t)(kStages / 2) * kPairBytes);
    volatile int* abort_flag = &c.abort_flag;
    unsigned* err = &g_err_x3;
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;  // warp-uniform
    const int ntiles = p.tiles > blockIdx.x ? (int)((p.tiles - 1 - blockIdx.x) / gridDim.x + 1) : 0;
    constexpr int ta_size = TA == MAT_F32 ? 4 : 2;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&c.full[s], kCvtGroupWarps);
            mbar_init(&c.empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&c.a_full[b], 1);
            mbar_init(&c.a_empty[b], kEpiWarps);
        }
        mbar_init(&c.x_empty, kEpiWarps);
        mbar_init(&c.mma_done, 1);
        c.abort_flag = 0;
        fence_barrier_init();
    }
    if (warp == 0) {
        tmem_alloc(&c.tmem_base, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = c.tmem_base;
    // tile of this CTA: batch plane, row block, column tile (columns fastest: A rows shared in L2)
    auto tile_of = [&](int lt, long long& b, long long& tm, int& tn) {
        const long long tg = blockIdx.x + (long long)lt * gridDim.x;
        tn = (int)(tg % p.tiles_n);
        const long long q = tg / p.tiles_n;
        tm = q % p.tiles_m;
        b = q / p.tiles_m;
    };

    if (warp == 0) {
        // ------------------------------------------------------------- MMA issue
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16_f32(p.nt);
            RingPos rs;
            int chunk = 0;  // chunks of hh issued so far: accumulator chunk & 1
            bool ok = true;
            for (int lt = 0; lt < ntiles && ok; ++lt) {
                const uint32_t mid = tmem + kColMid, low = tmem + kColLow;
                if (!mbar_wait_1t(&c.x_empty, ((uint32_t)lt & 1u) ^ 1u, abort_flag, err)) break;
                tc_fence_after();
                for (int kb = 0; kb < p.nkb; ++kb, rs.next(kStages)) {
                    const bool first = kb % kChunk == 0;
                    const int ab = chunk & 1;
                    if (first && !mbar_wait_1t(&c.a_empty[ab], ((uint32_t)(chunk >> 1) & 1u) ^ 1u, abort_flag, err)) {
                        ok = false;
                        break;
                    }
                    if (!mbar_wait_1t(&c.full[rs.idx], rs.phase, abort_flag, err)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t at = tmem + (uint32_t)(ab * 128);
                    const uint32_t s0 = smem_u32(base + (size_t)(rs.idx >> 1) * kPairBytes) + 64u * (uint32_t)(rs.idx & 1);
                    const uint64_t ah = sdesc_sw128(s0), am = sdesc_sw128(s0 + kPlane), al = sdesc_sw128(s0 + 2 * kPlane);
                    const uint64_t bh = sdesc_sw128(s0 + 3 * kPlane), bm = sdesc_sw128(s0 + 4 * kPlane),
                                   bl = sdesc_sw128(s0 + 5 * kPlane);
#pragma unroll
                    for (int k = 0; k < kBK / 16; ++k) {
                        const uint64_t o = (uint64_t)(2 * k);
                        mma_f16_ss(low, ah + o, bl + o, idesc, (kb | k) != 0 ? 1u : 0u);
                        mma_f16_ss(low, al + o, bh + o, idesc, 1u);
                        mma_f16_ss(low, am + o, bm + o, idesc, 1u);
                        mma_f16_ss(mid, ah + o, bm + o, idesc, (kb | k) != 0 ? 1u : 0u);
                        mma_f16_ss(mid, am + o, bh + o, idesc, 1u);
                        mma_f16_ss(at, ah + o, bh + o, idesc, (!first || k != 0) ? 1u : 0u);
                    }
                    mma_commit(&c.empty[rs.idx]);
                    if (kb % kChunk == kChunk - 1 || kb == p.nkb - 1) {
                        mma_commit(&c.a_full[ab]);  // and, with a tile's last chunk, its small products
                        ++chunk;
                    }
                }
            }
            mma_commit(&c.mma_done);
            mbar_drain(&c.mma_done, 0, err);
        }
    } else if (warp >= kCvt0) {
        // ------------------------------------------------------------- converters
        // The two groups take alternate K-blocks, so that one group's loads are in flight while the
        // other converts; a group loads its next K-block only after it has handed this one on (the
        // hand-over's arrive is a release, which waits for the thread's own outstanding loads).
        // A K-block of each operand is 16 tasks of 8 values a lane, four tasks a warp: eight rows of
        // it, a lane eight consecutive k (one address, one 16-byte store per plane; rows are dealt to
        // the lanes so that eight consecutive lanes' stores fall in disjoint banks), or, for a B stored
        // K x n, eight k of 32 columns (a lane one column).  Rows, columns and k past the end are
        // clamped to the last valid one, whose products either land in outputs that are never stored
        // or, past K, are zeroed on A's side.
        const int g = (warp - kCvt0) / kCvtGroupWarps, cw = (warp - kCvt0) % kCvtGroupWarps;
        const int rl = (lane >> 3) + (lane & 4), ch = lane & 3;  // a lane's row of eight, its chunk of 8 k
        float2 va[kSlots][4], vb[kSlots][4];
        Step st{};
        int lt = 0;
        auto set_tile = [&]() {
            long long b, tm;
            int tn;
            tile_of(lt, b, tm, tn);
            const long long m0 = tm * kBM;
            const int n0 = tn * p.nt;
            st.A = (const char*)p.A + (size_t)(b * p.a_bs + m0 * p.lda) * ta_size;
            st.B = (const char*)(p.B + b * p.b_bs + (BT ? (long long)n0 * p.ldb : n0));
            st.rows = (int)(p.m - m0 < kBM ? p.m - m0 : kBM);
            st.cols = p.n - n0 < p.nt ? p.n - n0 : p.nt;
            st.k = b == p.last ? p.k_last : p.k;
        };
        // to K-block `kb` of tile lt, or into the tiles after it; false past the CTA's last tile
        auto seek = [&]() {
            bool moved = false;
            while (st.kb >= p.nkb) {
                st.kb -= p.nkb;
                if (++lt >= ntiles) return false;
                moved = true;
            }
            if (moved) set_tile();
            return true;
        };
        auto row_a = [&](int i) {
            const int row = min(8 * (cw + kCvtGroupWarps * i) + rl, st.rows - 1);
            return st.A + (size_t)((uint32_t)row * (uint32_t)p.lda) * ta_size;
        };
        auto row_b = [&](int i) {
            const int row = min(8 * (cw + kCvtGroupWarps * i) + rl, st.cols - 1);
            return st.B + (size_t)((uint32_t)row * (uint32_t)p.ldb) * 4;
        };
        auto load = [&]() {
            const int k0 = st.kb * kBK, kc = k0 + 8 * cw;  // kc: this warp's eight k of a B stored K x n
            if (k0 + kBK <= st.k) {
#pragma unroll
                for (int i = 0; i < kSlots; ++i) ld8<TA, VEC>(row_a(i) + (k0 + 8 * ch) * ta_size, va[i]);
#pragma unroll
                for (int i = 0; i < kSlots; ++i) {
                    if (BT) {
                        ld8<MAT_F32, VEC>(row_b(i) + (k0 + 8 * ch) * 4, vb[i]);
                        continue;
                    }
                    // slot i: columns 32 i ..
                    const char* src = st.B + 4 * (size_t)((uint32_t)kc * (uint32_t)p.ldb + (uint32_t)min(32 * i + lane, st.cols - 1));
                    const size_t step = 4 * (size_t)p.ldb;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        vb[i][u].x = __ldg(reinterpret_cast<const float*>(src));
                        src += step;
                        vb[i][u].y = __ldg(reinterpret_cast<const float*>(src));
                        src += step;
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < kSlots; ++i) ld8_end<TA>(row_a(i), k0 + 8 * ch, st.k, va[i]);
#pragma unroll
                for (int i = 0; i < kSlots; ++i) {
                    if (BT) {
                        ld8_end<MAT_F32>(row_b(i), k0 + 8 * ch, st.k, vb[i]);
                        continue;
                    }
                    const float* f = reinterpret_cast<const float*>(st.B) + min(32 * i + lane, st.cols - 1);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        vb[i][u].x = __ldg(f + (size_t)min(kc + 2 * u, st.k - 1) * p.ldb);
                        vb[i][u].y = __ldg(f + (size_t)min(kc + 2 * u + 1, st.k - 1) * p.ldb);
                    }
                }
            }
        };
        // four pairs into three planes: 16 bytes of row `row`, chunk `c` of its eight
        auto put = [&](const float2 (&v)[4], uint8_t* dst, int row, int c) {
            uint32_t h[4], m[4], l[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) split3(v[u], h[u], m[u], l[u]);
            uint8_t* d = dst + row * 128 + ((c ^ (row & 7)) << 4);
            *reinterpret_cast<uint4*>(d) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(d + kPlane) = make_uint4(m[0], m[1], m[2], m[3]);
            *reinterpret_cast<uint4*>(d + 2 * kPlane) = make_uint4(l[0], l[1], l[2], l[3]);
        };
        auto store = [&](uint8_t* pair, int hf) {
#pragma unroll
            for (int i = 0; i < kSlots; ++i) put(va[i], pair, 8 * (cw + kCvtGroupWarps * i) + rl, 4 * hf + ch);
#pragma unroll
            for (int i = 0; i < kSlots; ++i) {
                if (BT)
                    put(vb[i], pair + 3 * kPlane, 8 * (cw + kCvtGroupWarps * i) + rl, 4 * hf + ch);
                else
                    put(vb[i], pair + 3 * kPlane, 32 * i + lane, 4 * hf + cw);
            }
        };
        bool more = ntiles > 0;
        if (more) {
            set_tile();
            st.kb = g;
            more = seek();
        }
        RingPos rs;
        if (g) rs.next(kStages);
        while (more) {
            load();
            if (!mbar_wait_warp_inline(&c.empty[rs.idx], rs.phase ^ 1u, abort_flag, err)) break;
            uint8_t* pair = base + (size_t)(rs.idx >> 1) * kPairBytes;
            store(pair, rs.idx & 1);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&c.full[rs.idx]);
            st.kb += kCvtGroups;
            more = seek();
            for (int j = 0; j < kCvtGroups; ++j) rs.next(kStages);
        }
    } else {
        // ------------------------------------------------------------- epilogue
        const int quad = warp & 3, half = (warp - kEpi0) >> 2;  // lane quadrant, 64 columns
        int chunk = 0;
        bool ok = true;
        for (int lt = 0; lt < ntiles && ok; ++lt) {
            float acc[4][16];  // [32 columns x 2][16-lane half x 2] in the 16x256b pattern
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int j = 0; j < 16; ++j) acc[q][j] = 0.f;
            const uint32_t tb = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(64 * half);
            auto add = [&](uint32_t col) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (64 * half + 32 * (q >> 1) >= p.nt) continue;
                    float t[16];
                    tmem_ld16x256b_x4(tb + ((uint32_t)(16 * (q & 1)) << 16) + col + (uint32_t)(32 * (q >> 1)), t);
#pragma unroll
                    for (int j = 0; j < 16; ++j) acc[q][j] += t[j];
                }
                tc_fence_before();
                __syncwarp();
            };
            for (int kb = 0; kb < p.nkb; kb += kChunk, ++chunk) {
                const int ab = chunk & 1;
                if (!mbar_wait_warp_inline(&c.a_full[ab], (uint32_t)(chunk >> 1) & 1u, abort_flag, err)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                add((uint32_t)(ab * 128));
                if (lane == 0) mbar_arrive(&c.a_empty[ab]);
            }
            if (!ok) break;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (64 * half + 32 * (q >> 1) >= p.nt) continue;
                const uint32_t tq = tb + ((uint32_t)(16 * (q & 1)) << 16) + (uint32_t)(32 * (q >> 1));
                float t[16];
                tmem_ld16x256b_x4(tq + kColLow, t);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    float u[8];
                    tmem_ld16x256b_x2(tq + kColMid + 16u * e, u);
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[q][8 * e + j] = fmaf(fmaf(t[8 * e + j], 1.f / kPartScale, u[j]), 1.f / kPartScale, acc[q][8 * e + j]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&c.x_empty);

            long long b, tm;
            int tn;
            tile_of(lt, b, tm, tn);
            bool bad = false;  // one of this thread's outputs is not finite
            auto finish = [&](float g, long long row, int col) {
                g *= p.alpha;
                if (p.rownorm) {
                    const float d = p.rownorm[row] * p.colnorm[col];
                    g = d > 0.f ? g / d : 0.f;
                }
                return g;
            };
#pragma unroll
            for (int q = 0; q < 4; ++q) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    int ln = lane;
                    asm volatile("" : "+r"(ln));  // the 64 sums leave no registers for kept addresses
                    const long long row = tm * kBM + quad * 32 + 16 * (q & 1) + (ln >> 2) + 8 * h;
                    const int cl0 = 64 * half + 32 * (q >> 1) + 2 * (ln & 3);
                    if (row >= p.m) continue;
                    const size_t off0 = (size_t)(b * p.c_bs + row * p.ldc + tn * p.nt + cl0);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int col = tn * p.nt + cl0 + 8 * j;
                        if (cl0 + 8 * j >= p.nt || col >= p.n) continue;
                        const bool two = col + 1 < p.n;
                        float g0 = acc[q][4 * j + 2 * h], g1 = acc[q][4 * j + 2 * h + 1];
                        bad |= !isfinite(g0) || (two && !isfinite(g1));
                        g0 = finish(g0, row, col);
                        if (two) g1 = finish(g1, row, col + 1);
                        const size_t off = off0 + 8 * j;
                        if (p.c_bf16) {
                            __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(p.C) + off;
                            if (p.c_vec && two) {
                                *reinterpret_cast<uint32_t*>(dst) = pack_bf16(g0, g1);
                            } else {
                                dst[0] = __float2bfloat16_rn(g0);
                                if (two) dst[1] = __float2bfloat16_rn(g1);
                            }
                        } else {
                            float* dst = reinterpret_cast<float*>(p.C) + off;
                            if (p.c_vec && two) {
                                __stcs(reinterpret_cast<float2*>(dst), make_float2(g0, g1));
                            } else {
                                dst[0] = g0;
                                if (two) dst[1] = g1;
                            }
                        }
                    }
                }
            }
            if (bad) {  // this thread's outputs again, as plain fp32 dot products in K order
                const char* Ab = (const char*)p.A + (size_t)(b * p.a_bs) * ta_size;
                const float* Bb = p.B + b * p.b_bs;
                const int kend = b == p.last ? p.k_last : p.k;
#pragma unroll 1
                for (int e = 0; e < 64; ++e) {
                    const int cl = 64 * half + 32 * (e >> 5) + 8 * ((e >> 3) & 3) + 2 * (lane & 3) + (e & 1);
                    const int col = tn * p.nt + cl;
                    const long long row = tm * kBM + quad * 32 + 16 * ((e >> 2) & 1) + (lane >> 2) + 8 * ((e >> 1) & 1);
                    if (cl >= p.nt || col >= p.n || row >= p.m) continue;
                    float g = 0.f;
                    // where B's rows end: the CUDA-core GEMM multiplies no zeros past the longest of 64 (an
                    // infinity or a NaN of A's row that lies there does not reach these columns)
                    int end = kend;
                    if (p.b_rowlen) {
                        end = 0;
                        for (int j = col & ~63; j < min(p.n, (col & ~63) + 64); ++j) end = max(end, p.b_rowlen[j]);
                        end = min(end, kend);
                    }
#pragma unroll 4
                    for (int k = 0; k < end; ++k)
                        g = fmaf(lda1<TA>(Ab, row * p.lda + k),
                                 __ldg(Bb + (BT ? (long long)col * p.ldb + k : (long long)k * p.ldb + col)), g);
                    g = finish(g, row, col);
                    const size_t off = (size_t)(b * p.c_bs + row * p.ldc + col);
                    if (p.c_bf16)
                        reinterpret_cast<__nv_bfloat16*>(p.C)[off] = __float2bfloat16_rn(g);
                    else
                        reinterpret_cast<float*>(p.C)[off] = g;
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

}  // namespace

unsigned take_device_error_x3() {
    unsigned v = 0, z = 0;
    cudaMemcpyFromSymbol(&v, g_err_x3, sizeof(v));
    if (v) cudaMemcpyToSymbol(g_err_x3, &z, sizeof(z));
    return v;
}

static cudaError_t launch_gemm_x3(const GemmArgs& g, int k_last, int sms, int device, cudaStream_t s) {
    X3Params p;
    p.A = g.A;
    p.B = (const float*)g.B;
    p.C = g.C;
    p.lda = g.lda, p.ldb = g.ldb, p.ldc = g.ldc;
    p.a_bs = g.a_bstride, p.b_bs = g.b_bstride, p.c_bs = g.c_bstride;
    p.m = g.m, p.n = g.n, p.k = g.k;
    p.k_last = k_last, p.last = g.batch - 1;
    p.tiles_n = (g.n + kBN - 1) / kBN;
    p.nt = ((g.n + p.tiles_n - 1) / p.tiles_n + 15) / 16 * 16;
    p.tiles_m = (g.m + kBM - 1) / kBM;
    p.tiles = p.tiles_m * p.tiles_n * g.batch;
    p.nkb = (g.k + kBK - 1) / kBK;
    // log2 of the elements that one load of a row of A (and of B, when its rows run along K) may take:
    // every row's start is aligned to them
    auto align = [](const void* ptr, int esize, long long ld, long long bs) {
        const unsigned long long a = (uintptr_t)ptr / esize | (unsigned long long)ld | (unsigned long long)bs;
        return a % 4 == 0 ? 2 : a % 2 == 0 ? 1 : 0;
    };
    int vec = align(g.A, g.a_type == MAT_F32 ? 4 : 2, g.lda, g.a_bstride);
    if (g.b_trans) vec = std::min(vec, align(g.B, 4, g.ldb, g.b_bstride));
    if (g.a_type == MAT_BF16) vec = std::min(vec, 1);
    p.c_bf16 = g.c_type == MAT_BF16;
    p.c_vec = (uintptr_t)g.C % (p.c_bf16 ? 4 : 8) == 0 && g.ldc % 2 == 0 && g.c_bstride % 2 == 0;
    p.alpha = g.alpha;
    p.rownorm = g.rownorm;
    p.colnorm = g.colnorm;
    p.b_rowlen = g.b_rowlen;
    const size_t smem = 1024 + (size_t)(kStages / 2) * kPairBytes + sizeof(Ctl);
    const int grid = (int)std::min<long long>(sms, p.tiles);
#define GS_X3_CASE(TA, BT, VEC)                                                                     \
    if (g.a_type == TA && g.b_trans == BT && vec == VEC) {                                          \
        static bool set[64];                                                                        \
        if (device < 0 || device >= 64) return cudaErrorInvalidDevice;                              \
        if (!set[device]) {                                                                         \
            cudaError_t e = cudaFuncSetAttribute(k_gemm_x3<TA, BT, VEC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); \
            if (e != cudaSuccess) return e;                                                         \
            set[device] = true;                                                                     \
        }                                                                                           \
        k_gemm_x3<TA, BT, VEC><<<grid, kThreads, smem, s>>>(p);                                     \
        return cudaGetLastError();                                                                  \
    }
    GS_X3_CASE(MAT_F32, true, 0)
    GS_X3_CASE(MAT_F32, true, 1)
    GS_X3_CASE(MAT_F32, true, 2)
    GS_X3_CASE(MAT_F32, false, 0)
    GS_X3_CASE(MAT_F32, false, 1)
    GS_X3_CASE(MAT_F32, false, 2)
    GS_X3_CASE(MAT_BF16, false, 0)
    GS_X3_CASE(MAT_BF16, false, 1)
#undef GS_X3_CASE
    return cudaErrorInvalidValue;
}

// K chunks for the product on the tensor cores; 0: it stays on the CUDA cores.
static int x3_ksplit(const GemmArgs& g, bool simt, int device) {
    const bool takes = !simt && g.b_type == MAT_F32 && (g.a_type == MAT_F32 || !g.b_trans) && !g.gate_xn2 && g.k >= 1 &&
                       g.k <= 32768 && g.lda <= 1 << 22 &&
                       (g.b_trans ? g.ldb <= 1 << 22 : (double)g.ldb * g.k < 1e9) && g.m > 0 && g.n > 0 && g.batch > 0;
    // times of both kernels, fitted to measured ones: a wave of tiles takes ~0.9 us per K-block and ~6 us
    // around it (512 x 3001 x 257: 21 us against 36 on the CUDA cores; 3000 x 1000 x 300: 32 / 56; 20,000 x
    // 777 x 131: 95 / 128; 1,300 x 13,823 x 130: 84 / 154); the CUDA-core GEMM runs at 28 to 45 TFLOP/s
    // where it is full, and unsplit takes at least 0.42 us a step of 16 and 0.4 more for each of an SM's 64 x 64
    // tiles (700 x 922 x 922, two on some SMs: 84 us; 100 x 922 x 922, one: 50)
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    double simt_us = 2e-6 * g.m * g.n * g.k * g.batch / 30.0;
    if (g.ksplit <= 1) {
        const double t64 = (double)((g.m + 63) / 64) * ((g.n + 63) / 64) * g.batch;
        simt_us = std::max(simt_us, g.k / 16 * (0.42 + 0.4 * std::ceil(t64 / std::max(sms, 1))));
    }
    if (!takes || simt_us <= 15.0 || !tc_available(device)) return 0;
    const double tiles = (double)((g.m + kBM - 1) / kBM) * ((g.n + kBN - 1) / kBN) * g.batch;
    const int nkb = (g.k + kBK - 1) / kBK;
    // few tiles over a deep K: chunks of at least eight K-blocks to partial products in the caller's
    // workspace, and their sum.  Whole scoring calls: 2,000 x 8192, r = M = 512: 239 -> 150 us; 1,000 x
    // 4096, 512: 138 -> 74; 300 x 8192, 1,000: 250 -> 102; 500 x 16,384, 256: 125 -> 60
    const bool may = g.kpart && g.batch == 1 && g.c_type == MAT_F32 && !g.rownorm && !g.colnorm && g.alpha == 1.f;
    const long long most = may ? std::min<long long>(g.kpart_floats / (g.m * g.n), std::min(32, nkb / 8)) : 1;
    int best = 0;
    double best_us = simt_us;
    for (int ks = 1; ks <= std::max(1LL, most); ++ks) {
        const double us = 8.0 + std::ceil(tiles * ks / std::max(sms, 1)) * (0.9 * ((nkb + ks - 1) / ks) + 6.0) +
                          (ks > 1 ? 4.0 + 4e-6 * g.m * g.n * (ks + 1) / 3.0 : 0.0);
        if (us < best_us) best = ks, best_us = us;
    }
    return best;
}

bool gemm_fp32_on_tensor(const GemmArgs& g, bool simt, int device) { return x3_ksplit(g, simt, device) > 0; }

cudaError_t launch_gemm_fp32(const GemmArgs& g, bool simt, int device, cudaStream_t s) {
    const int ks = x3_ksplit(g, simt, device);
    if (ks == 0) return launch_gemm_simt(g, s);
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (ks == 1) return launch_gemm_x3(g, g.k, std::max(sms, 1), device, s);
    GemmArgs q = g;  // the chunks as batch planes, the last one shorter
    const int nkb = (g.k + kBK - 1) / kBK, each = (nkb + ks - 1) / ks;
    q.k = each * kBK;
    q.batch = (nkb + each - 1) / each;
    q.a_bstride = q.k;
    q.b_bstride = g.b_trans ? q.k : (long long)q.k * g.ldb;
    q.C = g.kpart;
    q.ldc = g.n;
    q.c_bstride = g.m * g.n;
    cudaError_t e = launch_gemm_x3(q, g.k - (q.batch - 1) * q.k, std::max(sms, 1), device, s);
    return e != cudaSuccess ? e : launch_ksum(g, q.batch, s);
}

}  // namespace gs
