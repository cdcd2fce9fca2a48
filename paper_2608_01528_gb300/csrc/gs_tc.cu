// gs_tc.cu -- tcgen05 (5th-generation tensor core) kernels for sm_103a.
//
// k_ps_tc: fused project + similarity for large query batches (paper Sec. 3.1
// t = U^T x, Sec. 2.2 scaled dot-product similarity, Sec. 3.2 Eq. 2-3), for
// bases with r <= 256 and codebooks with M <= 256.
//
//   GEMM1  Y = X Q^T   tcgen05.mma kind::f16, M = 128 queries, N = r,
//                      fp32 accumulator in TMEM columns [0, 256).
//                      A = X: fp32 tiles streamed from HBM by TMA into a staging
//                      ring (several 32 KB tiles in flight per SM), rounded to
//                      fp16 (RN) by converter warps into the 128-byte-swizzled
//                      K-major layout the MMA reads.
//                      B = Q: the basis' fixed fp16 copy (dithered rounding, see
//                      gs_build.cu), fetched per K-block by TMA (L2-resident).
//   GEMM2  S = Y R^T   tcgen05.mma kind::f16 with bf16 operands split in two,
//                      Y = Yh + Yl and R = Rh + Rl, S = Yh Rh + Yl Rh + Yh Rl
//                      (relative error ~2^-16, fp32's exponent range), fp32
//                      accumulator in TMEM columns [256, 512).  The epilogue
//                      splits Y in place in TMEM (each 16-column fp32 chunk
//                      becomes 8 columns of packed Yh and 8 of packed Yl), and
//                      the MMA reads that A operand straight from TMEM.  S runs
//                      in halves of up to 128 codewords; one B-ring slot holds
//                      one K-block of both Rh and Rl of a half, so each slot is
//                      consumed on its own and the next one loads meanwhile.
//                      Gram-Schmidt leaves R lower echelon (codeword i has no
//                      component past the basis vectors built before it), so a
//                      half stops at the K-block holding its last nonzero.
//                      A single fp16/tf32 rounding would not do here: the
//                      dominant terms of S are single products Y_i R_ii.
//   epilogue           scale / cosine (full-D ||x|| accumulated by the
//                      converters from the fp32 input) / online softmax, argmax
//                      (lowest index on ties), maxval, optional Y and S stores.
//
// Why the X tiles go through TMA rather than through registers: a thread that
// signals "A stage full" with an mbarrier arrive (a release) cannot complete
// that arrive while its own prefetched global loads are still in flight, so a
// register-prefetch loader serialises on one memory round trip per K-block.
// With TMA the bytes in flight are the hardware's, and the converters' release
// only orders shared-memory traffic.
//
// Work split: one persistent CTA per SM; each CTA takes a contiguous, balanced
// range of rows and cuts it into tiles of at most 128 rows, so every CTA moves
// the same number of bytes.  Warp roles (480 threads):
//   warps 0-3    epilogue: warp w owns TMEM lanes 32w..32w+31 (rows of the tile)
//   warp  4      TMA producer of the X tiles
//   warp  5      TMEM allocator and MMA issuer (one elected lane)
//   warp  6      TMA producer of the B operand tiles (Q per K-block, then Rh / Rl)
//   warps 7-14   converters (fp32 -> fp16, row norms, range check), two groups of
//                four warps taking alternate K-blocks so two blocks convert at once; with a
//                K split they share the tile's tail with the epilogue (split_tail)
// Every wait on an mbarrier is bounded (wall-clock limit): on expiry the CTA
// records GS_DEV_ERR_TIMEOUT, raises a CTA-wide abort flag so the other roles
// leave their loops, waits (bounded) for its own TMA copies and MMAs to land,
// frees TMEM and returns.

#include <float.h>

#include <algorithm>
#include <vector>

#include "gs_internal.h"
#include "gs_tc_ptx.cuh"

namespace gs {
namespace {

using namespace ptx;

__device__ unsigned g_err_tc = 0;

constexpr int kBM = 128;             // queries per tile (MMA M)
constexpr int kBK = 64;              // K elements per block (fp16 A row = 128 B, fp32 staging row = 256 B)
constexpr int kEpiWarps = 4;
constexpr int kXWarp = 4;
constexpr int kMmaWarp = 5;
constexpr int kBWarp = 6;
constexpr int kCvt0 = 7;
constexpr int kCvtGroups = 2;        // converter groups take alternate K-blocks
constexpr int kCvtGroupWarps = 4;
constexpr int kCvtWarps = kCvtGroups * kCvtGroupWarps;
constexpr int kThreads = (kCvt0 + kCvtWarps) * 32;  // 480
constexpr int kCvtThreads = kCvtGroupWarps * 32;     // 128 per group
constexpr int kCvtRowStep = kCvtThreads / 16;        // 8 rows per sweep of the 16 float4 columns
constexpr int kCvtRows = kBM / kCvtRowStep;          // 16 rows per converter thread
constexpr int kAStageBytes = kBM * kBK * 2;          // 16 KB fp16 operand tile
constexpr int kBStageBytes = 256 * kBK * 2;          // 32 KB: up to 256 rows of one B operand K-block
constexpr int kMaxSX = 6, kMaxSA = 2, kMaxSB = 4;
constexpr int kTmemCols = 512;
constexpr int kMaxKR = 4;            // K-blocks of 64 in r <= 256
constexpr int kSCol = 256;           // first TMEM column of the score accumulator
constexpr int kMaxKS = 8;            // CTAs that may share a tile's K range
constexpr int kSendLd = 36;          // SPLIT: floats between the rows of a sending warp's 32 x 32 scratch
constexpr int kTailRoles = 1 + kCvtGroups;            // SPLIT: warps of a lane quadrant that share its columns
constexpr int kTailWarps = kEpiWarps * kTailRoles;    // SPLIT: warps that share the rows to be scored
static_assert(kCvtGroupWarps == 4, "every converter group has a warp in each lane quadrant");

// ----------------------------------------------------------------- work split
struct TileRange {
    long long row0;
    int nrows;
};

// Balanced contiguous row range of CTA c, cut into tiles of at most 128 rows.
struct CtaRows {
    long long rb;
    long long rows;
    int ntiles;
    int tsize;
    __host__ __device__ CtaRows(long long N, int G, int c) {
        const long long base = N / G, rem = N % G;
        rows = base + (c < rem ? 1 : 0);
        rb = (long long)c * base + (c < rem ? c : rem);
        ntiles = (int)((rows + kBM - 1) / kBM);
        tsize = ntiles ? (int)((rows + ntiles - 1) / ntiles) : 0;
    }
    __host__ __device__ TileRange tile(int t) const {
        TileRange tr;
        tr.row0 = rb + (long long)t * tsize;
        const long long left = rb + rows - tr.row0;
        tr.nrows = (int)(left < tsize ? left : tsize);
        return tr;
    }
};

struct PsParams {
    long long N;
    int D, r, npad, M, mpad, nkb;
    int nh, half_rows, nkr_h[2];  // GEMM2: halves of codewords, K-blocks of R each half needs
    int ks;                 // SPLIT: CTAs of a cluster that share a tile's K range
    int xch_ld;             // SPLIT: floats between exchanged Y rows (npad + 4)
    int send_off;           // SPLIT: the senders' scratch, behind the exchanged rows and the rows to be scored, then ||x||
    int s_ld;               // SPLIT: floats between the rows to be scored (mpad + 4)
    int bs_off;             // bytes from the X staging to the B ring
    int sx, sa, sb;         // ring depths: fp32 X staging, fp16 A, B operand tiles
    int box_rows;           // rows of each X TMA box (>= every tile's rows)
    int xstage;             // bytes between X staging tiles (box_rows x 256, 1 KB aligned)
    float xn2_lo, xn2_hi;   // rows with ||x||^2 outside [lo, hi] (and > 0) are redone scaled
    const float* cnorm;     // M
    int mode;
    float scale;
    float* Y;
    int ldy;
    float* S;
    int lds;
    int s_vec;              // S rows are 16-byte aligned
    int* argmax;
    float* maxval;
};

struct Ctl {
    uint64_t x_full[kMaxSX], x_empty[kMaxSX];
    uint64_t a_full[kMaxSA], a_empty[kMaxSA];
    uint64_t b_full[kMaxSB], b_empty[kMaxSB];
    uint64_t y_full, s_full, s_empty, gemm2_done;
    uint64_t ysplit[kMaxKR];  // Y columns [64 k, 64 k + 64) split in TMEM (GEMM2 K-block k may start)
    uint64_t xn_full[2], xn_empty[2];
    uint64_t dec_full[2];     // redo decision of regular tile t published in slot t % 2
    uint64_t peer_ready, xch_full;  // SPLIT: every CTA's GEMM1 is done; the peers' parts of my rows are here
    uint64_t sent_full, rows_full, tail_done;  // SPLIT: other owners' lanes are sent; S is in shared memory; scored
    uint64_t mma_done;
    float xn[2][kBM];  // ||x||^2 per row, both converter groups add into it
    int8_t rsc[2][kBM];      // per-row exponent s of the redo's scale 2^s, for the tile in that slot
    int redo[2][kMaxKS];     // per epilogue warp (SPLIT: per deciding warp of the cluster): some row needs the redo
    uint32_t tmem_base;
    int abort_flag;
};

// Exact power of two 2^k (|k| <= 126).
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((127 + k) << 23); }

// The exponent s that brings a row of squared norm xn2 to 2^14 <= ||x|| 2^s < 2^15: every
// element then lies below 2^15 (inside fp16's range) and the row's mass far above fp16's
// subnormals.  s lies in [-49, 89] for any finite positive fp32 xn2; rows whose squared norm is
// not a finite positive number keep s = 0.
__device__ __forceinline__ int row_scale_exp(float xn2) {
    if (!(xn2 > 0.f) || !(xn2 <= FLT_MAX)) return 0;
    return 14 - (ilogbf(xn2) >> 1);  // ilogbf(xn2) >> 1 = floor(log2 ||x||)
}

// one fp16 rounding of x is accurate when every element is inside fp16's range
// (||x|| <= 2^15) and the row's mass is far above its subnormals (||x|| >= 2^-8
// sqrt(D): the subnormals' absolute errors, at most 2^-25 each, then add at most
// 2^-19 ||x|| to the error of <x, q_j>); any other nonzero row has its tile redone
// with an exact power-of-two scale (a norm that is not a number keeps scale 1)
__device__ __forceinline__ bool out_of_range(float xn2, const PsParams& p) {
    return xn2 > 0.f && !(xn2 >= p.xn2_lo && xn2 <= p.xn2_hi);
}

// w (16 or 32) columns of Y at TMEM address ty, split in place: a chunk of 16 fp32 columns -> 8 columns of
// packed bf16(Y) + 8 columns of packed bf16(Y - bf16(Y)).
__device__ __forceinline__ void split_y(uint32_t ty, int w, const float (&y)[32]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h * 16 >= w) break;
        uint32_t hl[16];  // 8 columns of packed hi, then 8 of packed lo
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float a = y[16 * h + 2 * j], b = y[16 * h + 2 * j + 1];
            const float ah = __bfloat162float(__float2bfloat16_rn(a));
            const float bh = __bfloat162float(__float2bfloat16_rn(b));
            hl[j] = pack_bf16(ah, bh);
            hl[8 + j] = pack_bf16(a - ah, b - bh);
        }
        tmem_st16(ty + (uint32_t)(16 * h), hl);
    }
}

// Largest value over the warp's lanes (no NaN among them).
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Processing order of a CTA's tiles: regular tile t, and once tile t + 1 has been handed on, the
// redo of tile t when its epilogue asked for one (the decision is published in slot t % 2, so it
// is always known by then and nobody waits on it in the common case).  body(t, redo, q) runs one
// tile; q counts processed tiles (the per-tile barrier phases and the norm buffers follow it).
// wait(bar, parity) is the role's bounded wait.  Returns false when a wait or the body gave up.
template <class Wait, class Body>
__device__ __forceinline__ bool walk_tiles(const CtaRows& cr, Ctl& c, Wait wait, Body body) {
    int q = 0;
    for (int t = 0; t <= cr.ntiles; ++t) {
        if (t < cr.ntiles && !body(t, false, q++)) return false;
        if (t >= 1) {
            const int d = t - 1, slot = d & 1;
            if (!wait(&c.dec_full[slot], (uint32_t)(d >> 1) & 1u)) return false;
            const volatile int* rd = c.redo[slot];
            bool again = false;
#pragma unroll
            for (int w = 0; w < kMaxKS; ++w) again |= rd[w] != 0;
            if (again && !body(d, true, q++)) return false;
        }
    }
    return true;
}

// SPLIT: for batches with fewer 128-row tiles than half the SMs, a cluster of ks CTAs takes one tile:
// each runs GEMM1 over its part of D, then sends its partial Y (and ||x||^2) of the rows that peer q
// owns (rows [q 128 / ks, (q + 1) 128 / ks)) into q's shared memory; q adds the parts in a fixed order
// and goes on alone with its rows (GEMM2 over all 128 TMEM lanes, of which its own are read).  Without
// it a 4,096-query batch ran on 32 of 152 SMs, each streaming its X tile and all of Q: 150 us at D =
// 8192, r = M = 256 (softmax, scores out) against 46.5 us on 36 clusters of 4 (92 and 44 us for raw
// argmax): 23.5 until GEMM1's last K-block, 1.7 until every CTA is there, 4.1 for the exchange, 3.2 for the
// split, 2.3 for GEMM2, 2.5 for scores and rows, the rest launch and exit.  Splitting the rows instead would
// have every SM stream all of Q (4 MB each, 620 MB of L2 reads).  The exchange reuses the X staging and A
// stages, after every CTA of the cluster has finished GEMM1 (peer_ready).
// FULL = false: raw scores with only argmax / maxval out (the large-batch lookup); true: every
// mode and output.  A template parameter, so the lookup kernel carries none of the other paths.
template <bool FULL, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 1)
    k_ps_tc(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_q,
            const __grid_constant__ CUtensorMap tmap_rh, const __grid_constant__ CUtensorMap tmap_rl,
            const PsParams p) {
    extern __shared__ uint8_t smem_raw[];
    // 1024-byte aligned operand area (SW128 atoms), control block after it
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* base = smem_raw + (((raw + 1023u) & ~1023u) - raw);
    uint8_t* Xs = base;
    uint8_t* As = Xs + (size_t)p.sx * p.xstage;
    uint8_t* Bs = Xs + p.bs_off;
    Ctl& c = *reinterpret_cast<Ctl*>(Bs + (size_t)p.sb * kBStageBytes);
    volatile int* abort_flag = &c.abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ks = SPLIT ? p.ks : 1;
    const int rank = SPLIT ? (int)cluster_ctarank() : 0;
    const CtaRows cr(p.N, gridDim.x / ks, blockIdx.x / ks);
    const int kb0 = SPLIT ? p.nkb * rank / ks : 0, kb1 = SPLIT ? p.nkb * (rank + 1) / ks : p.nkb;
    constexpr int kRoles = SPLIT ? kTailRoles : 1;
    const int own_rows = kBM / ks;                                    // rows this CTA carries on with
    const int own_warps = SPLIT ? std::max(1, kEpiWarps / ks) : kEpiWarps;  // epilogue warps that hold them

    if (threadIdx.x == 0) {
        for (int s = 0; s < p.sx; ++s) {
            mbar_init(&c.x_full[s], 1);
            mbar_init(&c.x_empty[s], kCvtGroupWarps);
        }
        for (int s = 0; s < p.sa; ++s) {
            mbar_init(&c.a_full[s], kCvtGroupWarps);
            mbar_init(&c.a_empty[s], 1);
        }
        for (int s = 0; s < p.sb; ++s) {
            mbar_init(&c.b_full[s], 1);
            mbar_init(&c.b_empty[s], 1);
        }
        mbar_init(&c.y_full, 1);
        for (int k = 0; k < kMaxKR; ++k) mbar_init(&c.ysplit[k], own_warps * kRoles);
        mbar_init(&c.s_full, 1);
        mbar_init(&c.s_empty, own_warps * kRoles);
        mbar_init(&c.gemm2_done, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&c.xn_full[b], kCvtWarps);
            mbar_init(&c.xn_empty[b], kEpiWarps);
            mbar_init(&c.dec_full[b], SPLIT ? ks * own_warps * kRoles : kEpiWarps);
            for (int w = 0; w < kMaxKS; ++w) c.redo[b][w] = 0;
        }
        if (SPLIT) {
            mbar_init(&c.peer_ready, ks);
            mbar_init(&c.xch_full, (ks - 1) * own_warps);
            mbar_init(&c.sent_full, own_warps);
            mbar_init(&c.rows_full, own_warps * kRoles);
            mbar_init(&c.tail_done, kTailWarps);
        }
        mbar_init(&c.mma_done, 1);
        c.abort_flag = 0;
        for (int j = 0; j < 2 * kBM; ++j) (&c.xn[0][0])[j] = 0.f;
        fence_barrier_init();
    }
    if (warp == kMmaWarp) {
        tmem_alloc(&c.tmem_base, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    if (SPLIT) cluster_sync_all();  // every CTA's barriers exist before a peer signals them
    tc_fence_after();
    const uint32_t tmem = c.tmem_base;
    auto wait_1t = [&](uint64_t* bar, uint32_t par) { return mbar_wait_1t(bar, par, abort_flag, &g_err_tc); };
    auto wait_warp = [&](uint64_t* bar, uint32_t par) { return mbar_wait_warp(bar, par, abort_flag, &g_err_tc); };
    // a tile's redo decision: from this CTA's epilogue, or (SPLIT) from every CTA of the cluster
    auto dec_1t = [&](uint64_t* bar, uint32_t par) {
        return SPLIT ? mbar_wait_cluster(bar, par, abort_flag, &g_err_tc) : wait_1t(bar, par);
    };
    auto dec_warp = [&](uint64_t* bar, uint32_t par) {
        return SPLIT ? __all_sync(0xffffffffu, mbar_wait_cluster(bar, par, abort_flag, &g_err_tc)) != 0
                     : wait_warp(bar, par);
    };

    // SPLIT: what follows GEMM1 of a tile, on the epilogue's and the converters' twelve warps.  Three warps
    // (`role`) share a lane quadrant: the first sends the rows that peers own, then all three add the
    // peers' parts of this CTA's own rows and split them for GEMM2, column chunks in turn.  S goes through shared memory, from
    // which every warp (`wi`) scores whole rows: the own rows are 32 TMEM lanes at ks = 4, so that one
    // scheduler's warps did all the arithmetic (9.7 us for 32 rows of 256 scores with the softmax against 1.9),
    // and the rows left 16 bytes at a time.
    auto split_tail = [&](int role, int qd, int wi, int t, bool redo, int q) {
        const uint32_t pt = (uint32_t)q & 1u;
        const int b = q & 1;
        const int i = qd * 32 + lane;  // row within the tile = TMEM lane
        const uint32_t ty = tmem + ((uint32_t)(qd * 32) << 16), ts = ty + kSCol;
        const TileRange tr = cr.tile(t);
        const int owner = i / own_rows;  // the CTA that carries on with this row
        const bool mine = owner == rank;
        float* fin = reinterpret_cast<float*>(Xs + p.send_off) + kBM * kSendLd;  // ||x|| per row
        float* rows = reinterpret_cast<float*>(Xs);  // S of the own rows, once their parts are read
        if (!wait_warp(&c.y_full, pt)) return false;
        tc_fence_after();
        float xn2 = 0.f;
        if (role == 0) {
            if (!wait_warp(&c.xn_full[b], (uint32_t)(q >> 1) & 1u)) return false;
            xn2 = c.xn[b][i];
            c.xn[b][i] = 0.f;
            __syncwarp();
            if (lane == 0) mbar_arrive(&c.xn_empty[b]);
            // the peers may write over this CTA's X and A stages, and it over theirs
            if (qd == 0 && lane < ks) mbar_arrive_cluster(mapa_shared(smem_u32(&c.peer_ready), (uint32_t)lane));
        }
        if (!__all_sync(0xffffffffu, mbar_wait_cluster(&c.peer_ready, pt, abort_flag, &g_err_tc))) return false;
        const unsigned own_lanes = __ballot_sync(0xffffffffu, mine);
        if (role == 0 && own_lanes != 0xffffffffu) {
            // 32 columns at a time through this warp's scratch, so that a store takes 128 contiguous bytes of
            // each of four rows: 4.1 us for 96 rows of 256 columns, 24 bytes/ns, which is what the SM-to-SM
            // network carries (5.9 with a row per lane, 5.1 with 64 bytes of a row from three warps)
            float* tile = reinterpret_cast<float*>(Xs + p.send_off) + qd * 32 * kSendLd;
            const int u0 = lane >> 3, c4 = (lane & 7) * 4;  // rows u0 + 4 u of the warp, four columns
            uint32_t half_dst[2];  // rows u0 of the warp's two halves (which have an owner each at ks = 8)
            bool half_out[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int ri = qd * 32 + 16 * h, own = ri / own_rows, from = rank < own ? rank : rank - 1;
                half_out[h] = own != rank;
                half_dst[h] = mapa_shared(smem_u32(Xs) + 4u * (uint32_t)((from * own_rows + ri % own_rows + u0) * p.xch_ld + c4),
                                          (uint32_t)own);
            }
            const float* sent_from = tile + u0 * kSendLd + c4;
            for (int jc = 0; jc < p.npad; jc += 32) {
                const int w = p.npad - jc >= 32 ? 32 : 16;
                for (int e = 0; e < w; e += 16) {
                    float y[16];
                    tmem_ld16(ty + (uint32_t)(jc + e), y);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        *reinterpret_cast<float4*>(tile + lane * kSendLd + e + 4 * j) =
                            make_float4(y[4 * j], y[4 * j + 1], y[4 * j + 2], y[4 * j + 3]);
                }
                __syncwarp();
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const float4 f = *reinterpret_cast<const float4*>(sent_from + 4 * u * kSendLd);
                    if (half_out[u >> 2] && c4 < w)
                        st_cluster_f32x4(half_dst[u >> 2] + 4u * (uint32_t)(4 * (u & 3) * p.xch_ld + jc), f.x, f.y, f.z,
                                         f.w);
                }
                __syncwarp();
            }
            const int src = rank < owner ? rank : rank - 1;
            if (!mine)
                st_cluster_f32x4(mapa_shared(smem_u32(Xs) + 4u * (uint32_t)((src * own_rows + i % own_rows) * p.xch_ld + p.npad),
                                             (uint32_t)owner),
                                 xn2, 0.f, 0.f, 0.f);
            __syncwarp();
            // one arrival per group of rows of one owner (a release: the lanes' stores come before it)
            if (!mine && lane % std::min(32, own_rows) == 0)
                mbar_arrive_cluster(mapa_shared(smem_u32(&c.xch_full), (uint32_t)owner));
        }
        if (own_lanes != 0u) {
            if (own_rows < 32) {  // the split overwrites the other owners' lanes too, which role 0 sends
                tc_fence_before();
                if (role == 0 && lane == 0) mbar_arrive(&c.sent_full);
                if (!wait_warp(&c.sent_full, pt)) return false;
                tc_fence_after();
            }
            if (!__all_sync(0xffffffffu, mbar_wait_cluster(&c.xch_full, pt, abort_flag, &g_err_tc))) return false;
            // this row's parts from the peers, in CTA order
            const float* parts = reinterpret_cast<const float*>(Xs) + (size_t)(i % own_rows) * p.xch_ld;
            // a redone tile ran on x 2^s: Y and ||x|| come back multiplied by 2^s
            const float unscale = redo ? pow2f(-c.rsc[t & 1][i]) : 1.f;
            if (role == 0) {
                if (mine) {
                    for (int u = 0; u < ks - 1; ++u) xn2 += parts[(size_t)u * own_rows * p.xch_ld + p.npad];
                    fin[i] = sqrtf(xn2) * unscale;
                }
                if (!redo) {  // the redo's data, to every CTA of the cluster (this one among them)
                    const int slot = t & 1;
                    const uint32_t e = (uint32_t)(uint8_t)(int8_t)row_scale_exp(xn2);
                    const unsigned any = __ballot_sync(0xffffffffu, mine && out_of_range(xn2, p));
                    const uint32_t a_rsc = smem_u32(&c.rsc[slot][i]);
                    const uint32_t a_redo = smem_u32(&c.redo[slot][own_warps > 1 ? qd : rank]);
                    for (int d = 0; d < ks; ++d)
                        if (mine) st_cluster_u8(mapa_shared(a_rsc, (uint32_t)d), e);
                    if (lane < ks) st_cluster_u32(mapa_shared(a_redo, (uint32_t)lane), any != 0u);
                }
            }
            for (int jc = 0; jc < p.npad; jc += 32) {
                if ((jc >> 5) % kRoles == role) {
                    const int w = p.npad - jc >= 32 ? 32 : 16;
                    float y[32];
                    if (w == 32)
                        tmem_ld32(ty + (uint32_t)jc, y);
                    else
                        tmem_ld16(ty + (uint32_t)jc, y);
                    if (mine) {
                        for (int u = 0; u < ks - 1; ++u) {
                            const float4* src = reinterpret_cast<const float4*>(parts + (size_t)u * own_rows * p.xch_ld + jc);
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                if (4 * j >= w) break;
                                const float4 f = src[j];
                                y[4 * j] += f.x;
                                y[4 * j + 1] += f.y;
                                y[4 * j + 2] += f.z;
                                y[4 * j + 3] += f.w;
                            }
                        }
                    }
                    if (redo) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) y[j] *= unscale;
                    }
                    if (FULL && p.Y && mine && i < tr.nrows) {
                        float* dst = p.Y + (size_t)(tr.row0 + i) * p.ldy + jc;
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            if (j < w && jc + j < p.r) dst[j] = y[j];
                    }
                    split_y(ty + (uint32_t)jc, w, y);
                }
                if (((jc + 32) & 63) == 0 || jc + 32 >= p.npad) {  // this role's part of K-block jc / 64 is split
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&c.ysplit[jc >> 6]);
                }
            }
            // the parts are read and the redo's data sent
            if (!redo && lane < ks) mbar_arrive_cluster(mapa_shared(smem_u32(&c.dec_full[t & 1]), (uint32_t)lane));
            if (!wait_warp(&c.s_full, pt)) return false;
            tc_fence_after();
            for (int ic = 16 * role; ic < p.mpad; ic += 16 * kRoles) {
                float sv[16];
                tmem_ld16(ts + (uint32_t)ic, sv);
                if (p.nkr_h[ic >= p.half_rows ? 1 : 0] == 0) {  // a half with no nonzero R: S = 0
#pragma unroll
                    for (int j = 0; j < 16; ++j) sv[j] = 0.f;
                }
                if (mine) {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        *reinterpret_cast<float4*>(rows + (i % own_rows) * p.s_ld + ic + 4 * j) =
                            make_float4(sv[4 * j], sv[4 * j + 1], sv[4 * j + 2], sv[4 * j + 3]);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&c.s_empty);
                mbar_arrive(&c.rows_full);
            }
        }
        if (!wait_warp(&c.rows_full, pt)) return false;
        const bool softmax = FULL && p.mode == GS_SCORE_SOFTMAX;
        for (int il = wi; il < own_rows && rank * own_rows + il < tr.nrows; il += kTailWarps) {
            const long long row = tr.row0 + rank * own_rows + il;
            float v[8];  // columns 4 lane + j and 128 + 4 lane + j
            float best = -FLT_MAX;
            int besti = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int col = 128 * h + 4 * lane;
                const float4 f = col < p.mpad ? *reinterpret_cast<const float4*>(rows + il * p.s_ld + col)
                                              : make_float4(0.f, 0.f, 0.f, 0.f);
                v[4 * h] = f.x;
                v[4 * h + 1] = f.y;
                v[4 * h + 2] = f.z;
                v[4 * h + 3] = f.w;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float& x = v[4 * h + j];
                    x *= p.scale;
                    if (FULL && p.mode == GS_SCORE_COSINE) {
                        const float den = col + j < p.M ? fin[rank * own_rows + il] * p.cnorm[col + j] : 0.f;
                        x = den > 0.f ? x / den : 0.f;
                    }
                    if (col + j >= p.M) x = -INFINITY;  // columns past M never win and add nothing
                    if (x > best) {
                        best = x;
                        besti = col + j;
                    }
                }
            }
            const float top = warp_max(best);
            // the first of equal scores, and entry 0 where none is above the type's lowest value
            const int idx = top > -FLT_MAX ? (int)__reduce_min_sync(0xffffffffu, best == top ? (unsigned)besti : 0x7fffffffu) : 0;
            float outmax = top;
            if (softmax) {
                float sum = 0.f;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    v[j] = __expf(v[j] - top);
                    sum += v[j];
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                const float inv = 1.f / sum;
                outmax = __expf(top - top) * inv;
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] *= inv;
            }
            if (FULL && p.S) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int col = 128 * h + 4 * lane;
                    float* dst = p.S + (size_t)row * p.lds + col;
                    if (p.s_vec && col + 4 <= p.M) {
                        *reinterpret_cast<float4*>(dst) = make_float4(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (col + j < p.M) dst[j] = v[4 * h + j];
                    }
                }
            }
            if (lane == 0 && p.argmax) p.argmax[row] = idx;
            if (lane == 0 && p.maxval) p.maxval[row] = outmax;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&c.tail_done);
        return true;
    };

    if (warp == kXWarp) {
        // ------------------------------------------------------------- X tiles via TMA
        if (lane == 0) {
            const uint64_t pol = l2_policy_evict_first();
            const uint32_t bytes = (uint32_t)p.box_rows * kBK * 4;
            int it = 0;
            RingPos xs;
            walk_tiles(cr, c, dec_1t, [&](int t, bool redo, int q) {
                const TileRange tr = cr.tile(t);
                if (SPLIT && redo) {  // the exchanged rows and the scores lay where X lands again
                    if (!wait_1t(&c.tail_done, (uint32_t)(q - 1) & 1u)) return false;
                    fence_proxy_async();
                }
                for (int kb = kb0; kb < kb1; ++kb, ++it, xs.next(p.sx)) {
                    if (!wait_1t(&c.x_empty[xs.idx], xs.phase ^ 1u)) return false;
                    mbar_arrive_expect_tx(&c.x_full[xs.idx], bytes);
                    tma_load_2d(Xs + (size_t)xs.idx * p.xstage, &tmap_x, &c.x_full[xs.idx], kb * kBK, (int)tr.row0,
                                pol);
                }
                return true;
            });
            // every copy this thread started lands before the CTA can exit
            for (int j = std::max(0, it - p.sx); j < it; ++j) mbar_drain(&c.x_full[j % p.sx], (uint32_t)(j / p.sx) & 1u, &g_err_tc);
        }
    } else if (warp == kBWarp) {
        // ------------------------------------------------------------- B operand tiles via TMA:
        // per tile, nkb Q tiles (GEMM1), then per half of the codewords its K-blocks of
        // Rh and Rl, both in one slot (GEMM2)
        if (lane == 0) {
            const uint64_t pol = l2_policy_evict_last();
            const uint32_t qbytes = (uint32_t)p.npad * kBK * 2, rbytes = 2u * (uint32_t)p.half_rows * kBK * 2;
            const uint32_t rl_off = (uint32_t)p.half_rows * kBK * 2;  // Rl after Rh in the slot
            const int nkb = kb1 - kb0, per_tile = nkb + p.nkr_h[0] + p.nkr_h[1];
            int it = 0;
            RingPos bs;
            walk_tiles(cr, c, dec_1t, [&](int, bool, int) {
                for (int k = 0; k < per_tile; ++k, ++it, bs.next(p.sb)) {
                    const int s = bs.idx;
                    if (!wait_1t(&c.b_empty[s], bs.phase ^ 1u)) return false;
                    uint8_t* dst = Bs + (size_t)s * kBStageBytes;
                    if (k < nkb) {
                        mbar_arrive_expect_tx(&c.b_full[s], qbytes);
                        tma_load_2d(dst, &tmap_q, &c.b_full[s], (kb0 + k) * kBK, 0, pol);
                    } else {
                        const int j = k - nkb;
                        const int h = j < p.nkr_h[0] ? 0 : 1;
                        const int kr = h ? j - p.nkr_h[0] : j;
                        mbar_arrive_expect_tx(&c.b_full[s], rbytes);
                        tma_load_2d(dst, &tmap_rh, &c.b_full[s], kr * kBK, h * p.half_rows, pol);
                        tma_load_2d(dst + rl_off, &tmap_rl, &c.b_full[s], kr * kBK, h * p.half_rows, pol);
                    }
                }
                return true;
            });
            for (int j = std::max(0, it - p.sb); j < it; ++j) mbar_drain(&c.b_full[j % p.sb], (uint32_t)(j / p.sb) & 1u, &g_err_tc);
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------- MMA issue
        if (lane == 0) {
            const uint32_t idesc1 = idesc_f16_f32(p.npad);
            const uint32_t idesc2 = idesc_bf16_f32(p.half_rows);
            const uint32_t y_tmem = tmem, s_tmem = tmem + kSCol;
            RingPos ra, rb;
            walk_tiles(cr, c, dec_1t, [&](int, bool, int q) {
                const uint32_t pt = (uint32_t)q & 1u;
                // GEMM1: Y = X Q^T into columns [0, npad)
                for (int kb = kb0; kb < kb1; ++kb, ra.next(p.sa), rb.next(p.sb)) {
                    const int sa = ra.idx, sb = rb.idx;
                    if (!wait_1t(&c.a_full[sa], ra.phase) || !wait_1t(&c.b_full[sb], rb.phase)) return false;
                    tc_fence_after();
                    const uint64_t ad = sdesc_sw128(smem_u32(As + (size_t)sa * kAStageBytes));
                    const uint64_t bd = sdesc_sw128(smem_u32(Bs + (size_t)sb * kBStageBytes));
#pragma unroll
                    for (int k = 0; k < kBK / 16; ++k)
                        mma_f16_ss(y_tmem, ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), idesc1,
                                   (kb != kb0 || k != 0) ? 1u : 0u);
                    mma_commit(&c.a_empty[sa]);
                    mma_commit(&c.b_empty[sb]);
                }
                mma_commit(&c.y_full);
                // GEMM2: S = Yh Rh + Yl Rh + Yh Rl into columns [256, 256 + mpad), once the
                // epilogue has split Y in place and released the previous tile's S
                if (!wait_1t(&c.s_empty, pt ^ 1u)) return false;
                int nsplit = 0;  // K-blocks of Y known to be split; the epilogue signals each one
                for (int h = 0; h < p.nh; ++h) {
                    const uint32_t s_half = s_tmem + (uint32_t)(h * p.half_rows);
                    for (int kr = 0; kr < p.nkr_h[h]; ++kr, rb.next(p.sb)) {
                        for (; nsplit <= kr; ++nsplit)
                            if (!wait_1t(&c.ysplit[nsplit], pt)) return false;
                        const int sr = rb.idx;
                        if (!wait_1t(&c.b_full[sr], rb.phase)) return false;
                        tc_fence_after();
                        const uint32_t rs = smem_u32(Bs + (size_t)sr * kBStageBytes);
                        const uint64_t rh = sdesc_sw128(rs);
                        const uint64_t rl = sdesc_sw128(rs + (uint32_t)p.half_rows * kBK * 2);
#pragma unroll
                        for (int k = 0; k < kBK / 16; ++k) {
                            // r columns [64 kr + 16 k, +16) were split into TMEM columns
                            // [16 kk, 16 kk + 8) (Yh) and [16 kk + 8, 16 kk + 16) (Yl), kk = 4 kr + k
                            const int kk = 4 * kr + k;
                            if (16 * kk >= p.npad) break;  // past r: no split columns there
                            const uint32_t a_hi = y_tmem + (uint32_t)(16 * kk);
                            const uint32_t a_lo = a_hi + 8;
                            mma_bf16_ts(s_half, a_hi, rh + (uint64_t)(2 * k), idesc2, (kr | k) != 0 ? 1u : 0u);
                            mma_bf16_ts(s_half, a_lo, rh + (uint64_t)(2 * k), idesc2, 1u);
                            mma_bf16_ts(s_half, a_hi, rl + (uint64_t)(2 * k), idesc2, 1u);
                        }
                        mma_commit(&c.b_empty[sr]);
                    }
                }
                // K-blocks of Y that no codeword uses (R may end before r): the epilogue may still be reading
                // them, and with a K split the peers' parts of them, where the scores go once S is there
                for (; nsplit < (p.npad + kBK - 1) / kBK; ++nsplit)
                    if (!wait_1t(&c.ysplit[nsplit], pt)) return false;
                mma_commit(&c.s_full);
                // the next tile's GEMM1 overwrites the columns GEMM2 reads: wait for it to finish
                mma_commit(&c.gemm2_done);
                if (!wait_1t(&c.gemm2_done, pt)) return false;
                tc_fence_after();
                return true;
            });
            // all MMAs issued by this thread complete before TMEM is released
            mma_commit(&c.mma_done);
            mbar_drain(&c.mma_done, 0, &g_err_tc);
        }
    } else if (warp >= kCvt0) {
        // ------------------------------------------------------------- converters
        const int g = (warp - kCvt0) / kCvtGroupWarps;           // group: K-blocks with it % 2 == g
        const int l = threadIdx.x - (kCvt0 + g * kCvtGroupWarps) * 32;  // 0..127 within the group
        const int c4 = l & 15;                   // float4 column of the 64-wide K-block
        const int rbase = l >> 4;                // rows rbase + 8u, u < 16
        float nrm[kCvtRows];
#pragma unroll
        for (int u = 0; u < kCvtRows; ++u) nrm[u] = 0.f;
        float amax = 0.f;
        int it = 0;
        RingPos rx, ra;  // every K-block advances both rings; this group takes those with it % 2 == g
        walk_tiles(cr, c, dec_warp, [&](int t, bool redo, int q) {
            const TileRange tr = cr.tile(t);
            const int b = q & 1;
            const int8_t* rs = c.rsc[t & 1];  // the rows' scale exponents (redo only)
            for (int kb = kb0; kb < kb1; ++kb, ++it, rx.next(p.sx), ra.next(p.sa)) {
                if ((it & 1) != g) continue;
                const int sx = rx.idx, sa = ra.idx;
                if (!wait_warp(&c.x_full[sx], rx.phase) || !wait_warp(&c.a_empty[sa], ra.phase ^ 1u)) return false;
                const uint8_t* Xt = Xs + (size_t)sx * p.xstage;
                uint8_t* At = As + (size_t)sa * kAStageBytes;
#pragma unroll
                for (int u = 0; u < kCvtRows; ++u) {
                    const int row = rbase + kCvtRowStep * u;
                    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (row < tr.nrows) x = *reinterpret_cast<const float4*>(Xt + row * (kBK * 4) + c4 * 16);
                    if (redo) {  // exact power-of-two scale: the fp16 rounding below loses nothing to range
                        const float sc = pow2f(rs[row]);
                        x.x *= sc;
                        x.y *= sc;
                        x.z *= sc;
                        x.w *= sc;
                        amax = fmaxf(amax, fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))));
                    }
                    nrm[u] = fmaf(x.x, x.x, fmaf(x.y, x.y, fmaf(x.z, x.z, fmaf(x.w, x.w, nrm[u]))));
                    const __half2 h0 = __floats2half2_rn(x.x, x.y);
                    const __half2 h1 = __floats2half2_rn(x.z, x.w);
                    uint2 pk;
                    pk.x = *reinterpret_cast<const uint32_t*>(&h0);
                    pk.y = *reinterpret_cast<const uint32_t*>(&h1);
                    const int chunk = (c4 >> 1) ^ (row & 7);
                    *reinterpret_cast<uint2*>(At + row * 128 + chunk * 16 + (c4 & 1) * 8) = pk;
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&c.a_full[sa]);
                    mbar_arrive(&c.x_empty[sx]);
                }
            }
            // tile finished: this group's part of ||x||^2 of each row is added into shared memory
#pragma unroll
            for (int u = 0; u < kCvtRows; ++u) {
                float v = nrm[u];
                v += __shfl_xor_sync(0xffffffffu, v, 8);
                v += __shfl_xor_sync(0xffffffffu, v, 4);
                v += __shfl_xor_sync(0xffffffffu, v, 2);
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                nrm[u] = v;
            }
            if (!wait_warp(&c.xn_empty[b], ((uint32_t)(q >> 1) & 1u) ^ 1u)) return false;
            if ((lane & 15) == 0) {
#pragma unroll
                for (int u = 0; u < kCvtRows; ++u) atomicAdd(&c.xn[b][rbase + kCvtRowStep * u], nrm[u]);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&c.xn_full[b]);
#pragma unroll
            for (int u = 0; u < kCvtRows; ++u) nrm[u] = 0.f;
            return SPLIT ? split_tail(1 + g, warp & 3, kEpiWarps + warp - kCvt0, t, redo, q) : true;
        });
        // only a redone row can still leave fp16's range (a norm that is not a finite fp32 number)
        if (amax > 65504.f) atomicOr(&g_err_tc, GS_DEV_ERR_RANGE);
    } else {
        // ------------------------------------------------------------- epilogue (warps 0-3)
        const int i = threadIdx.x;  // row within the tile = TMEM lane
        const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
        const uint32_t ty = tmem + lane_base, ts = tmem + lane_base + kSCol;
        walk_tiles(cr, c, dec_warp, [&](int t, bool redo, int q) {
            if (SPLIT) return split_tail(0, warp, warp, t, redo, q);
            const uint32_t pt = (uint32_t)q & 1u;
            const int b = q & 1;
            if (!wait_warp(&c.y_full, pt)) return false;
            tc_fence_after();
            const TileRange tr = cr.tile(t);
            const long long row = tr.row0 + i;
            const bool valid = i < tr.nrows;
            // a redone tile ran on x 2^s: Y and ||x|| come back multiplied by 2^s
            const float unscale = redo ? pow2f(-c.rsc[t & 1][i]) : 1.f;
            // split Y in place: chunk of 16 fp32 columns -> 8 columns bf16(Y) + 8 columns
            // bf16(Y - bf16(Y)), read 32 columns per TMEM load wait.  Each finished K-block
            // of 64 columns is signalled on its own, so GEMM2 starts on it while the rest
            // of Y is still being split.
            for (int jc = 0; jc < p.npad; jc += 32) {
                const int w = p.npad - jc >= 32 ? 32 : 16;
                float y[32];
                if (w == 32)
                    tmem_ld32(ty + (uint32_t)jc, y);
                else
                    tmem_ld16(ty + (uint32_t)jc, y);
                if (redo) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) y[j] *= unscale;
                }
                if (FULL && p.Y && valid) {
                    float* dst = p.Y + (size_t)row * p.ldy + jc;
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (j < w && jc + j < p.r) dst[j] = y[j];
                }
                split_y(ty + (uint32_t)jc, w, y);
                if (((jc + 32) & 63) == 0 || jc + 32 >= p.npad) {  // K-block jc / 64 is split
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&c.ysplit[jc >> 6]);
                }
            }
            if (!wait_warp(&c.xn_full[b], (uint32_t)(q >> 1) & 1u)) return false;
            const float xn2 = c.xn[b][i];
            c.xn[b][i] = 0.f;  // ready for the tile after next (both groups add into it)
            __syncwarp();
            if (lane == 0) mbar_arrive(&c.xn_empty[b]);
            const float xnorm = sqrtf(xn2) * unscale;
            if (!redo) {
                const int slot = t & 1;
                c.rsc[slot][i] = (int8_t)row_scale_exp(xn2);
                const unsigned any = __ballot_sync(0xffffffffu, out_of_range(xn2, p));
                if (lane == 0) c.redo[slot][warp] = any != 0u;
                __syncwarp();
                if (lane == 0) mbar_arrive(&c.dec_full[slot]);
            }
            if (!wait_warp(&c.s_full, pt)) return false;
            tc_fence_after();
            // scores ci .. ci + 15 of this thread's row
            auto scores = [&](int ic, float (&sv)[16]) {
                tmem_ld16(ts + (uint32_t)ic, sv);
                if (p.nkr_h[ic >= p.half_rows ? 1 : 0] == 0) {  // a half with no nonzero R: S = 0
#pragma unroll
                    for (int j = 0; j < 16; ++j) sv[j] = 0.f;
                }
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    sv[j] *= p.scale;
                    if (FULL && p.mode == GS_SCORE_COSINE) {
                        const float den = ic + j < p.M ? xnorm * p.cnorm[ic + j] : 0.f;
                        sv[j] = den > 0.f ? sv[j] / den : 0.f;
                    }
                }
            };
            auto store = [&](int ic, const float (&sv)[16]) {
                float* dst = p.S + (size_t)row * p.lds + ic;
                if (p.s_vec && ic + 16 <= p.M) {
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        reinterpret_cast<float4*>(dst)[u] = make_float4(sv[4 * u], sv[4 * u + 1], sv[4 * u + 2], sv[4 * u + 3]);
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (ic + j < p.M) dst[j] = sv[j];
                }
            };
            float best = -FLT_MAX, run_max = -FLT_MAX, run_sum = 0.f;
            int besti = 0;
            for (int ic = 0; ic < p.mpad; ic += 16) {
                float sv[16];
                scores(ic, sv);
                if (ic + 16 > p.M) {  // columns past M never win and add nothing
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (ic + j >= p.M) sv[j] = -INFINITY;
                }
                // the chunk's first largest score by a tree, left before right (one compare after the other
                // took 4.6 against 2.5 us a tile of 256 scores, 11.2 against 5.8 with the softmax); a NaN never wins
                float tv[16];
                int ti[8];
#pragma unroll
                for (int j = 0; j < 16; ++j) tv[j] = fmaxf(sv[j], -FLT_MAX);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const bool g = tv[2 * j + 1] > tv[2 * j];
                    ti[j] = g ? 2 * j + 1 : 2 * j;
                    tv[j] = g ? tv[2 * j + 1] : tv[2 * j];
                }
#pragma unroll
                for (int n = 4; n > 0; n >>= 1) {
#pragma unroll
                    for (int j = 0; j < n; ++j) {
                        const bool g = tv[2 * j + 1] > tv[2 * j];
                        ti[j] = g ? ti[2 * j + 1] : ti[2 * j];
                        tv[j] = g ? tv[2 * j + 1] : tv[2 * j];
                    }
                }
                if (tv[0] > best) {
                    best = tv[0];
                    besti = ic + ti[0];
                }
                if (FULL && p.mode == GS_SCORE_SOFTMAX) {
                    // online, sixteen at a time: one rescaling exponential per chunk, one per score
                    const float nm = best;
                    float e[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) e[j] = __expf(sv[j] - nm);
#pragma unroll
                    for (int n = 8; n > 0; n >>= 1) {
#pragma unroll
                        for (int j = 0; j < n; ++j) e[j] += e[j + n];
                    }
                    run_sum = run_sum * __expf(run_max - nm) + e[0];
                    run_max = nm;
                }
                if (FULL && p.S && valid && p.mode != GS_SCORE_SOFTMAX) store(ic, sv);
            }
            float outmax = best;
            if (FULL && p.mode == GS_SCORE_SOFTMAX) {
                const float inv = 1.f / run_sum;
                outmax = __expf(best - run_max) * inv;
                // the scores once more from TMEM (they were written unnormalised and read back before:
                // three passes of one 4-byte access per lane and row)
                for (int ic = 0; p.S && ic < p.mpad; ic += 16) {
                    float sv[16];
                    scores(ic, sv);
#pragma unroll
                    for (int j = 0; j < 16; ++j) sv[j] = __expf(sv[j] - run_max) * inv;
                    if (valid) store(ic, sv);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&c.s_empty);
            if (!valid) return true;
            if (p.argmax) p.argmax[row] = besti;
            if (p.maxval) p.maxval[row] = outmax;
            return true;
        });
    }

    tc_fence_before();
    __syncthreads();
    if (SPLIT) cluster_sync_all();  // no CTA leaves while a peer may still write to it or signal it
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// ----------------------------------------------------------------- host side
// R (M x r fp32) -> Rh = bf16(R), Rl = bf16(R - Rh) (mpad x npad) and the same
// split of R^T (npad x mpad), all zero padded.
__global__ void k_split_r(const float* __restrict__ R, int M, int r, int ldr, __nv_bfloat16* __restrict__ Rh,
                          __nv_bfloat16* __restrict__ Rl, __nv_bfloat16* __restrict__ Rth,
                          __nv_bfloat16* __restrict__ Rtl, int mpad, int npad) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)mpad * npad) return;
    const int i = (int)(idx / npad), j = (int)(idx % npad);
    const float v = (i < M && j < r) ? R[(size_t)i * ldr + j] : 0.f;
    const __nv_bfloat16 hv = __float2bfloat16_rn(v);
    const __nv_bfloat16 lv = __float2bfloat16_rn(v - __bfloat162float(hv));
    Rh[idx] = hv;
    Rl[idx] = lv;
    Rth[(size_t)j * mpad + i] = hv;
    Rtl[(size_t)j * mpad + i] = lv;
}

// Q (r x D fp32, ld = D) -> Qh = bf16(Q), Ql = bf16(Q - Qh), both r x ldq, zero padded.
__global__ void k_split_q(const float* __restrict__ Q, int r, int D, int ldq, __nv_bfloat16* __restrict__ Qh,
                          __nv_bfloat16* __restrict__ Ql) {
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long long)r * ldq) return;
    const int j = (int)(idx / ldq), d = (int)(idx % ldq);
    const float v = d < D ? Q[(size_t)j * D + d] : 0.f;
    const __nv_bfloat16 hv = __float2bfloat16_rn(v);
    Qh[idx] = hv;
    Ql[idx] = __float2bfloat16_rn(v - __bfloat162float(hv));
}

int num_sms(int dev) {
    int n = 0;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

struct Rings {
    int sx, sa, sb;
};

constexpr size_t kSmemCap = 227 * 1024;

// bytes between fp32 X staging tiles of `box_rows` rows (SW128 operand areas follow: 1 KB aligned)
int ps_xstage(int box_rows) { return (box_rows * kBK * 4 + 1023) / 1024 * 1024; }

// xch: bytes of the exchanged rows, the senders' scratch and the norms (0: no K split), which share the X
// staging's and A stages' place
size_t ps_bs_off(Rings g, int xstage, size_t xch) {
    return std::max((size_t)g.sx * xstage + (size_t)g.sa * kAStageBytes, (xch + 1023) / 1024 * 1024);
}
size_t ps_smem_bytes(Rings g, int xstage, size_t xch) {
    return 1024 + ps_bs_off(g, xstage, xch) + (size_t)g.sb * kBStageBytes + sizeof(Ctl);
}

// Ring depths for X boxes of `box_rows` rows: the deepest X ring that fits, then the
// deepest B ring.  The X depth must be even.  The two converter groups take alternate
// K-blocks, so with an even depth every X stage belongs to one group, which waits on its
// phases in order.  With an odd depth a stage alternates between the groups: one group
// can reach the stage two phases on while the other group's load into it is still in
// flight (TMA loads may land out of order), and the parity test would then pass on the
// stage's older, completed phase and hand over stale data.
Rings ps_rings(int box_rows, size_t xch) {
    const int xs = ps_xstage(box_rows);
    for (int sx = kMaxSX; sx >= 2; sx -= 2)
        for (int sb = kMaxSB; sb >= 2; --sb) {
            Rings g{sx, kMaxSA, sb};
            if (ps_smem_bytes(g, xs, xch) <= kSmemCap) return g;
        }
    return Rings{2, kMaxSA, 2};
}

// launch configuration of a K-split launch: `ctas` CTAs in clusters of ks
cudaLaunchConfig_t ps_cluster_config(int ctas, int ks, size_t smem, cudaStream_t s, cudaLaunchAttribute* at) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)ks;
    at->val.clusterDim.y = 1;
    at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

}  // namespace

namespace {
// Self-test of the bounded waits: one thread waits, through the same mbar_wait the
// tensor-core kernels use, on an mbarrier that nothing ever arrives on.  The wait gives up
// after its limit, records GS_DEV_ERR_TIMEOUT in this file's device word and returns.
__global__ void k_wait_selftest() {
    __shared__ uint64_t bar;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        abort_flag = 0;
        fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) mbar_wait(&bar, 0u, &abort_flag, &g_err_tc);  // phase 0 never completes
}
}  // namespace

cudaError_t launch_wait_selftest(cudaStream_t s) {
    k_wait_selftest<<<1, 32, 0, s>>>();
    return cudaGetLastError();
}

unsigned take_device_error_tc() {
    unsigned v = 0, z = 0;
    cudaMemcpyFromSymbol(&v, g_err_tc, sizeof(v));
    if (v) cudaMemcpyToSymbol(g_err_tc, &z, sizeof(z));
    return v;
}

bool tc_available(int device) {
    int major = 0, minor = 0;
    cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device);
    cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, device);
    return major == 10 && minor == 3 && encode_fn() != nullptr;
}

gs_status tc_prepare(gs_basis* h) {
    if (h->r < 1) return GS_OK;
    const int npad = (h->r + 15) / 16 * 16;
    const int mpad = (h->M + 15) / 16 * 16;
    const size_t n = (size_t)mpad * npad;
    // bf16 hi / lo splits of R (mpad x npad) and of R^T (npad x mpad)
    for (void** ptr : {&h->tc_Rh, &h->tc_Rl, &h->tc_Rth, &h->tc_Rtl})
        if (cudaMalloc(ptr, sizeof(__nv_bfloat16) * n) != cudaSuccess) return GS_ERR_NOMEM;
    k_split_r<<<(unsigned)((n + 255) / 256), 256>>>(h->R, h->M, h->r, h->ldr, (__nv_bfloat16*)h->tc_Rh,
                                                    (__nv_bfloat16*)h->tc_Rl, (__nv_bfloat16*)h->tc_Rth,
                                                    (__nv_bfloat16*)h->tc_Rtl, mpad, npad);
    // bf16 hi / lo split of Q (r x ldq16, zero padded)
    const size_t nq = (size_t)h->r * h->ldq16;
    for (void** ptr : {&h->tc_Qh, &h->tc_Ql})
        if (cudaMalloc(ptr, sizeof(__nv_bfloat16) * nq) != cudaSuccess) return GS_ERR_NOMEM;
    k_split_q<<<(unsigned)((nq + 255) / 256), 256>>>(h->Q, h->r, h->D, h->ldq16, (__nv_bfloat16*)h->tc_Qh,
                                                     (__nv_bfloat16*)h->tc_Ql);
    if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return GS_ERR_CUDA;
    h->tc_npad = npad;
    h->tc_mpad = mpad;
    h->has_split = true;
    // R's echelon structure on the host, for the GEMMs' K trimming
    h->rlen_host.assign((size_t)h->M, 0);
    if (cudaMemcpy(h->rlen_host.data(), h->rlen, sizeof(int) * (size_t)h->M, cudaMemcpyDeviceToHost) != cudaSuccess)
        return GS_ERR_CUDA;
    h->kzero_host.assign((size_t)h->M, 0);
    h->kM_host.assign((size_t)h->r, h->M);
    h->pivot_host.assign((size_t)h->r, h->M);
    for (int j = 0, i = 0; j < h->r; ++j) {  // first row reaching column j (nondecreasing in j)
        while (i < h->M && h->rlen_host[(size_t)i] <= j) ++i;
        h->pivot_host[(size_t)j] = i;
    }
    // the fused kernel keeps Y (r <= 256 columns) and S (M <= 256 columns) in TMEM
    if (h->r > 256 || h->M > 256) return GS_OK;
    // GEMM2 halves: up to 128 codewords each; K-blocks per half from the last nonzero of R
    h->tc_half_rows = mpad > 128 ? 128 : mpad;
    h->tc_nh = (mpad + h->tc_half_rows - 1) / h->tc_half_rows;
    {
        std::vector<int> rl((size_t)h->M);
        if (cudaMemcpy(rl.data(), h->rlen, sizeof(int) * (size_t)h->M, cudaMemcpyDeviceToHost) != cudaSuccess)
            return GS_ERR_CUDA;
        for (int hh = 0; hh < 2; ++hh) {
            int last = 0;
            for (int i = hh * h->tc_half_rows; hh < h->tc_nh && i < std::min(h->M, (hh + 1) * h->tc_half_rows); ++i)
                last = std::max(last, rl[(size_t)i]);
            h->tc_nkr_half[hh] = (last + kBK - 1) / kBK;
        }
    }
    if (!make_tmap_2d(&h->tmap_q16, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, h->Q16, h->r, h->D, h->ldq16, kBK, npad,
                      CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_tmap_2d(&h->tmap_rh, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, h->tc_Rh, mpad, npad, npad, kBK,
                      h->tc_half_rows, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_tmap_2d(&h->tmap_rl, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, h->tc_Rl, mpad, npad, npad, kBK,
                      h->tc_half_rows, CU_TENSOR_MAP_SWIZZLE_128B))
        return GS_ERR_CUDA;
    // the fused kernel needs all of its threads resident in one CTA; otherwise the
    // basis simply has no fused tensor-core similarity path
    bool fits = true;
    for (auto fn : {k_ps_tc<false, false>, k_ps_tc<true, false>, k_ps_tc<false, true>, k_ps_tc<true, true>}) {
        cudaFuncAttributes fa;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemCap) != cudaSuccess ||
            cudaFuncGetAttributes(&fa, fn) != cudaSuccess)
            return GS_ERR_CUDA;
        fits = fits && fa.maxThreadsPerBlock >= kThreads;
    }
    h->has_tmap_q16 = fits;
    // clusters of 2, 4 and 8 CTAs that the GPU holds at once (GPCs need not hold whole numbers of them)
    for (int i = 0; i < 3; ++i) {
        cudaLaunchAttribute at[1];
        cudaLaunchConfig_t cfg = ps_cluster_config(2 << i, 2 << i, kSmemCap, 0, at);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k_ps_tc<true, true>, &cfg) != cudaSuccess) return GS_ERR_CUDA;
        h->ps_clusters[i] = n;
    }
    return GS_OK;
}

cudaError_t launch_ps_tc(const gs_basis* h, const float* X, long long N, int ldx, int mode, float scale, float* Y,
                         int ldy, float* S, int lds, int* argmax, float* maxval, cudaStream_t s) {
    if (!h->has_tmap_q16) return cudaErrorNotSupported;
    const long long tiles = (N + kBM - 1) / kBM;
    // Fewer tiles than half the SMs: clusters of ks CTAs share each tile's K range, as many clusters as
    // the GPU holds (their rows even out).  A K-block takes a CTA ~0.65 us, the exchange and what only the
    // row's owner does after it ~15 us at r = M = 256, so the K-blocks saved have to be worth 20 us.
    // Measured at r = M = 256, 4,096 queries: D = 4096: 33 us (50 without), 8192: 44 (92), 16,384: 65;
    // D = 2048 is left alone.
    const int nkb = (h->D + kBK - 1) / kBK;
    int ks = 1, clusters = 0;
    for (int i = 0; i < 3; ++i)
        if (tiles <= h->ps_clusters[i] && 0.65 * (nkb - nkb / (2 << i)) > 20.0)
            ks = 2 << i, clusters = h->ps_clusters[i];
    const int grid = (int)(ks > 1 ? std::min<long long>(clusters, N) : std::min<long long>(num_sms(h->device), tiles));
    // the X box must cover the largest tile of any CTA (CTAs differ by one row)
    int box_rows = 1;
    for (int cta : {0, grid - 1}) box_rows = std::max(box_rows, CtaRows(N, grid, cta).tsize);
    CUtensorMap tmx;
    if (!make_tmap_2d(&tmx, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, X, N, h->D, ldx, kBK, box_rows,
                      CU_TENSOR_MAP_SWIZZLE_NONE))
        return cudaErrorInvalidValue;
    const int xch_ld = h->tc_npad + 4;  // 16 bytes of shift per row: the row-per-thread accesses spread over the banks
    const int s_ld = h->tc_mpad + 4;
    const size_t send_off = sizeof(float) * (size_t)(kBM / ks) * std::max((ks - 1) * xch_ld, s_ld);
    const size_t xch = ks > 1 ? send_off + sizeof(float) * (kBM * kSendLd + kBM) : 0;
    const Rings g = ps_rings(box_rows, xch);
    if (g.sx % kCvtGroups != 0 || g.sa % kCvtGroups != 0) return cudaErrorInvalidConfiguration;
    PsParams p;
    p.N = N;
    p.D = h->D;
    p.r = h->r;
    p.npad = h->tc_npad;
    p.M = h->M;
    p.mpad = h->tc_mpad;
    p.nkb = nkb;
    p.nh = h->tc_nh;
    p.half_rows = h->tc_half_rows;
    p.nkr_h[0] = h->tc_nkr_half[0];
    p.nkr_h[1] = h->tc_nkr_half[1];
    p.sx = g.sx;
    p.sa = g.sa;
    p.sb = g.sb;
    p.box_rows = box_rows;
    p.xstage = ps_xstage(box_rows);
    p.ks = ks;
    p.xch_ld = xch_ld;
    p.send_off = (int)send_off;
    p.s_ld = s_ld;
    p.bs_off = (int)ps_bs_off(g, p.xstage, xch);
    p.s_vec = (uintptr_t)S % 16 == 0 && lds % 4 == 0;
    // one fp16 rounding of a row is accurate for 2^-8 sqrt(D) <= ||x|| <= 2^15; other rows are redone
    p.xn2_lo = (float)h->D * 0x1p-16f;
    p.xn2_hi = 0x1p30f;
    p.cnorm = h->cnorm;
    p.mode = mode;
    p.scale = scale;
    p.Y = Y;
    p.ldy = ldy;
    p.S = S;
    p.lds = lds;
    p.argmax = argmax;
    p.maxval = maxval;
    const bool full = mode != GS_SCORE_RAW || Y || S;
    const size_t smem = ps_smem_bytes(g, p.xstage, xch);
    if (smem > kSmemCap) return cudaErrorInvalidConfiguration;
    if (ks == 1) {
        if (full)
            k_ps_tc<true, false><<<grid, kThreads, smem, s>>>(tmx, h->tmap_q16, h->tmap_rh, h->tmap_rl, p);
        else
            k_ps_tc<false, false><<<grid, kThreads, smem, s>>>(tmx, h->tmap_q16, h->tmap_rh, h->tmap_rl, p);
        return cudaGetLastError();
    }
    cudaLaunchAttribute at[1];
    cudaLaunchConfig_t cfg = ps_cluster_config(grid * ks, ks, smem, s, at);
    return cudaLaunchKernelEx(&cfg, full ? k_ps_tc<true, true> : k_ps_tc<false, true>, tmx, h->tmap_q16, h->tmap_rh,
                              h->tmap_rl, p);
}

}  // namespace gs
