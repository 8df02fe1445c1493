// FP64-equivalent matrix product (precision pattern OO_PREC_FP64EQ) for the
// matrix-product function block (Sec. 3.2.2): C = A B for FP64 row-major
// A (m x k) and B (k x n), computed on the BF16 tensor cores by an
// Ozaki-type error-free splitting (Ozaki, Ogita, Oishi, Rump 2012):
//
//   a_il = 2^ea_i * sum_{p=1..s} d^A_p(i,l) 2^(-beta p) + r   (|r| < 2^(ea_i - beta s))
//   b_lj = 2^eb_j * sum_{q=1..s} d^B_q(l,j) 2^(-beta q) + r'
//
// Each digit d is a signed integer with |d| <= 2^beta - 1, read directly
// as a beta-bit group of the entry's fixed-point mantissa relative to its
// row (A) or column (B) scale 2^e (no floating-point arithmetic in the
// split).  Digits are exact in BF16 (beta <= 8), their products exact in
// FP32, and with K-blocks of kb terms, kb (2^beta - 1)^2 < 2^24, every
// product's K-block sum D_pq = sum_l d^A_p d^B_q accumulates exactly in the
// FP32 accumulators of tensor memory, whatever order the hardware adds in.
//
//   C_ij = 2^(ea_i + eb_j) sum_{p + q <= L} 2^(-beta (p + q)) D_pq(i, j)
//
// The terms are summed in float-float (about 48 bits) in tensor memory,
// smallest level first, then widened to FP64 and scaled.  Dropping the
// levels p + q > L and the split remainders costs at most about
// (L + 2) 2^(-beta (L - 1)) 2^(ea_i + eb_j) k per element; L is the
// smallest level for which 4 (L + 2) 2^(-beta (L - 1)) <= 2^-42, i.e. at
// most ~2.3e-13 of sum_l |a_il| |b_lj| when the entries of a row (column)
// are of comparable size.
//
//   K-block kb: the fewest blocks of at most 1024 terms, multiples of 64,
//   all about as long;  beta = 8 (kb <= 256) or 7;
//   beta 8: L = 7 (21 products); beta 7: L = 8 (28 products).
//
// Kernel: persistent, one CTA per SM over 128 x 128 output tiles.  The
// products are grouped in units that share the A slice: (p, q1) and
// (p, q2) become one M = 128, N = 256 MMA whose B operand is the two B
// slices' tiles stacked (a product without a partner runs alone at
// N = 128).  A unit of work is one such group over one K-block (K-blocks
// outermost, so one K-block's slices serve all groups while in L2): warp 0
// streams its A_p and B_q tiles (TMA, 128-byte swizzle) through a 4-stage
// ring, warp 1 issues tcgen05.mma (K = 16) into one of two 256-column FP32
// accumulators in tensor memory (double-buffered), and eight epilogue warps
// (two per tensor-memory lane quarter, one per 64-column half) add each
// finished accumulator, scaled by 2^(-beta (p + q)), into a float-float
// running sum held in registers; after the tile's last unit they write
// FP64 C.  Sharing A_p raises the MMA work per staged byte by a third.
// Every mbarrier wait is bounded.
// A row of A or column of B holding a NaN or an infinity gives NaN in every
// entry of C it meets (tc.cuh, kNonFiniteExp); other entries are unaffected.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "ff.cuh"
#include "oo_internal.h"
#include "eq_digits.cuh"
#include "tc.cuh"

namespace oo {

namespace {

using namespace tc;
using eq::eff_exp;
using eq::fixed_frac;

constexpr int kBM = 128, kBN = 128, kBK = 64, kStages = 4;
constexpr int kThreads = 320;              // producer, MMA issuer, 8 epilogue warps
constexpr int kEpiWarps = 8;
constexpr uint32_t kTile = kBM * kBK * 2;  // 16 KB, A and B tiles alike
constexpr uint32_t kStageBytes = 3 * kTile;  // A_p, B_q1, B_q2
constexpr int kGroupM = 8;
constexpr int kMaxUnits = 24;
constexpr uint32_t kIdescPair = idesc_bf16(kBM, 2 * kBN);
constexpr uint32_t kIdescOne = idesc_bf16(kBM, kBN);

using EqShape = eq::Shape;
// the scheme the library uses for inner dimension k
EqShape eq_used_shape(int k) { return eq::shape(eq_scheme_for(k), k); }

struct EqMaps {
    CUtensorMap a, b;  // all slices stacked: slice p at rows [p m, (p + 1) m)
};

struct EqArgs {
    int m, n, ksteps, kb_steps, nkb, nunits;
    int m_tiles, n_tiles;
    double *C;
    long long ldc;
    const int *ea, *eb;
    unsigned *err;
    unsigned char up[kMaxUnits], uq[kMaxUnits], unq[kMaxUnits];  // 0-based slices p, q .. q + nq - 1
    float us[kMaxUnits];                                         // 2^(-beta (p + q)), 1-based p and first q
    float uq_step;                                               // 2^-beta
};

__device__ __forceinline__ void eq_tile(const EqArgs &a, int t, int &m0, int &n0) {
    const int per_group = kGroupM * a.n_tiles;
    const int g = t / per_group, r = t % per_group;
    const int rows = min(kGroupM, a.m_tiles - g * kGroupM);
    m0 = (g * kGroupM + r % rows) * kBM;
    n0 = (r / rows) * kBN;
}

// Single CTAs (OO_OPT_GEMM_PAIR = 0): what the CTA-pair kernel's bits are
// compared with, so its roles and its store stay plain.
__global__ void __launch_bounds__(kThreads, 1) gemm_fp64eq_kernel(const __grid_constant__ EqMaps maps,
                                                                 const __grid_constant__ EqArgs a) {
    extern __shared__ __align__(1024) unsigned char esm_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(esm_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint64_t *bars = reinterpret_cast<uint64_t *>(sm + kStages * kStageBytes);
    uint64_t *full = bars, *empty = bars + kStages;
    uint64_t *tfull = bars + 2 * kStages, *tempty = bars + 2 * kStages + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * kStages + 4);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tiles = a.m_tiles * a.n_tiles;
    const int units = a.nunits * a.nkb;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            bar_init(su32(&full[s]), 1);
            bar_init(su32(&empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            bar_init(su32(&tfull[b]), 1);
            bar_init(su32(&tempty[b]), kEpiWarps);  // one arrival per epilogue warp
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        tmem_alloc(su32(tmem_slot), 512);
        fence_before();
    }
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;

    int loaded = 0;      // producer: stages issued
    int units_mma = 0;   // MMA issuer: units whose accumulation was issued
    if (warp == 0 && lane == 0) {
        // ---------------------------------------------------- TMA producer
        int it = 0;
        bool ok = true;
        for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
            int m0, n0;
            eq_tile(a, t, m0, n0);
            for (int u = 0; ok && u < units; ++u) {
                const int kbi = u / a.nunits, pr = u % a.nunits;  // K-block outer: its slices stay in L2
                const bool pair = a.unq[pr] == 2;
                const int rowA = a.up[pr] * a.m + m0, rowB1 = a.uq[pr] * a.n + n0;
                const int rowB2 = pair ? rowB1 + a.n : 0;
                const int ks1 = min(a.ksteps, (kbi + 1) * a.kb_steps);
                for (int ks = kbi * a.kb_steps; ks < ks1; ++ks, ++it) {
                    const int s = it % kStages;
                    const uint32_t use = it / kStages;
                    if (use > 0 && !bar_wait(su32(&empty[s]), (use - 1) & 1, abort_flag, a.err, 1u)) {
                        ok = false;
                        break;
                    }
                    unsigned char *st = sm + (size_t)s * kStageBytes;
                    const uint32_t fb = su32(&full[s]);
                    bar_expect_tx(fb, pair ? 3 * kTile : 2 * kTile);
                    tma_2d(su32(st), &maps.a, ks * kBK, rowA, fb);
                    tma_2d(su32(st + kTile), &maps.b, ks * kBK, rowB1, fb);
                    if (pair) tma_2d(su32(st + 2 * kTile), &maps.b, ks * kBK, rowB2, fb);
                    ++loaded;
                }
            }
        }
    } else if (warp == 1 && lane == 0) {
        // ---------------------------------------------------- MMA issuer
        int it = 0, gu = 0;
        bool ok = true;
        for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
            for (int u = 0; ok && u < units; ++u, ++gu) {
                const int b = gu & 1;
                const uint32_t buse = gu >> 1;
                if (buse > 0 && !bar_wait(su32(&tempty[b]), (buse - 1) & 1, abort_flag, a.err, 2u)) {
                    ok = false;
                    break;
                }
                fence_after();
                const uint32_t d = tmem + (uint32_t)(b * 2 * kBN);
                const int kbi = u / a.nunits, pr = u % a.nunits;  // K-block outer: its slices stay in L2
                const bool pair = a.unq[pr] == 2;
                const int ks0 = kbi * a.kb_steps, ks1 = min(a.ksteps, (kbi + 1) * a.kb_steps);
                for (int ks = ks0; ks < ks1; ++ks, ++it) {
                    const int s = it % kStages;
                    if (!bar_wait(su32(&full[s]), (it / kStages) & 1, abort_flag, a.err, 2u)) {
                        ok = false;
                        break;
                    }
                    fence_after();
                    const uint32_t sa = su32(sm + (size_t)s * kStageBytes), sb = sa + kTile;
#pragma unroll
                    for (int kk = 0; kk < kBK / 16; ++kk) {
                        const uint32_t off = kk * 32;  // 16 BF16 along K inside the 128-byte row
                        const uint32_t acc = (ks == ks0 && kk == 0) ? 0u : 1u;
                        if (pair)  // B_q1 and B_q2 tiles stacked: one N = 256 operand
                            mma_bf16<kIdescPair>(d, sdesc_sw128(sa + off), sdesc_sw128(sb + off), acc);
                        else
                            mma_bf16<kIdescOne>(d, sdesc_sw128(sa + off), sdesc_sw128(sb + off), acc);
                    }
                    mma_commit(su32(&empty[s]));
                }
                if (!ok) break;
                mma_commit(su32(&tfull[b]));  // this unit's accumulator is complete
                ++units_mma;
            }
        }
    } else if (warp >= 2) {
        // ---------------------------------------------------- epilogue
        const int q = warp & 3;              // TMEM lane quarter this warp may access
        const int h = (warp - 2) >> 2;       // 64-column half of the tile
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        float Sh[64], Sl[64];                // running float-float sum of this row's 64 columns
        int gu = 0;
        bool ok = true;
        for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
            int m0, n0;
            eq_tile(a, t, m0, n0);
#pragma unroll
            for (int j = 0; j < 64; ++j) Sh[j] = Sl[j] = 0.0f;
            for (int u = 0; u < units; ++u, ++gu) {
                const int b = gu & 1;
                if (!bar_wait(su32(&tfull[b]), (gu >> 1) & 1, abort_flag, a.err, 4u)) {
                    ok = false;
                    break;
                }
                fence_after();
                const int pr = u % a.nunits;
                const bool pair = a.unq[pr] == 2;
                const float f1 = a.us[pr], f2 = f1 * a.uq_step;
                const uint32_t acc = tmem + (uint32_t)(b * 2 * kBN) + lane_off + (uint32_t)(h * 64);
#pragma unroll
                for (int c = 0; c < 64; c += 8) {
                    uint32_t v[8], w[8];
                    OO_TMEM_LD8(acc + c, v);
                    if (pair) OO_TMEM_LD8(acc + kBN + c, w);
                    tmem_wait_ld();
                    if (pair)
                        eq::add_two8(Sh + c, Sl + c, w, f2, v, f1);  // powers of two: exact scales
                    else
                        eq::add_one8(Sh + c, Sl + c, v, f1);
                }
                fence_before();
                __syncwarp();
                if (lane == 0) bar_arrive(su32(&tempty[b]));
                if (u == units - 1) {
                    // column scales: lane l holds columns l and l + 32 of this
                    // half (coalesced) and hands them out by shuffle
                    const int row = m0 + q * 32 + lane;
                    const int c0 = n0 + h * 64;
                    const int e0 = c0 + lane < a.n ? a.eb[c0 + lane] : 0;
                    const int e1 = c0 + 32 + lane < a.n ? a.eb[c0 + 32 + lane] : 0;
                    const bool row_ok = row < a.m;
                    const int sa = row_ok ? a.ea[row] : 0;
                    double *crow = a.C + (long long)row * a.ldc + c0;
#pragma unroll
                    for (int j = 0; j < 64; ++j) {
                        const int sb = __shfl_sync(0xffffffffu, j < 32 ? e0 : e1, j & 31);
                        if (row_ok && c0 + j < a.n)
                        {
                            double v;
                            if (!eq::scaled_value(Sh[j], Sl[j], sa + sb, v)) v = eq::general_value(Sh[j], Sl[j], sa + sb);
                            crow[j] = v;
                        }
                    }
                }
            }
        }
    }
    // drain on abort: wait (bounded) for issued MMAs and copies before TMEM
    // is released and the CTA exits
    if (*abort_flag) {
        if (warp == 1 && lane == 0 && units_mma > 0)
            bar_drain(su32(&tfull[(units_mma - 1) & 1]), ((units_mma - 1) >> 1) & 1);
        if (warp == 0 && lane == 0)
            for (int it = (loaded > kStages ? loaded - kStages : 0); it < loaded; ++it)
                bar_drain(su32(&full[it % kStages]), (it / kStages) & 1);
    }
    fence_before();
    __syncthreads();
    if (warp == 1) {
        fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// ------------------------------------------------------------ CTA pairs
// The same products on CTA pairs (cta_group::2, M = 256): a tile is 256 rows
// x TN = 128 columns, CTA r of the pair holding rows m0 + 128 r .. +127 of the
// tile and its own accumulators and running sums.  A two-product unit
// (p, q1) + (p, q2) is one M = 256, N = 256 MMA whose B operand is B_q1's
// tile in rank 0's shared memory and B_q2's in rank 1's, so an SM stages
// 32 KB (A_p and one B slice tile) per K step where a single CTA stages
// 48 KB for the same MMA work; a one-product unit is an N = 128 MMA, each
// CTA holding 64 of the tile's columns of B_q.  Rank 0 issues the MMAs;
// the commits arrive on both CTAs' barriers; both epilogues report to rank
// 0 that their accumulator buffer is free.  The D_pq of a K-block are exact
// whatever the instruction shape, and the epilogue adds the units in the
// same order, so the result is the single-CTA kernel's bit for bit.
// The producer and the MMA issuer run as whole warps (tc.cuh): with one lane
// running each loop, the issuer's own instructions took 611 clocks a K step,
// and 1050 while the epilogue ran, for 512 clocks of MMA; n = 4096 took 2.92
// ms in this kernel, 2.29 ms so (3.13 -> 2.56 ms with the splits).
// The epilogue: C is stored through shared memory (eq::store_columns) and a
// running sum costs 8 operations a product, the power-of-two scale folded
// into them.  With a row of C per lane and the conversion unrolled over the
// columns the store took 122,000 clocks a tile, in which the tensor cores did
// two units of the next tile and then waited: n = 4096 2.50 -> 2.18 ms, n =
// 2048 444 -> 356 us, 1024 118 -> 105 us with the splits.  A unit's epilogue takes
// about as long as a K-block of 1024 terms' MMAs, so K-blocks are balanced
// (eq::shape): 1000 x 777 x 1300 in blocks of 1024 + 320 159 us, 704 + 640
// 144 us with both (wide tiles).  What binds now at n = 4096 is the tensor rate, 0.91 of
// 1.96 PFLOP/s over the products' 3.85 PFLOP with the splits, under the power limit.
// Narrow tiles, TN = 64: a unit is up to four slices of B against one of A,
// beside each other in the same 256 accumulator columns, so that A_p's 16 KB
// still come with up to 16 KB of B for 512 clocks of MMA a K step, and half
// the columns need half the time: 1000 x 777 x 1300 is 28 wide tiles on 76
// CTA pairs, 144 us with the splits, and 52 narrow ones, 92 us (90 with two
// products added at once); 1024^3 105 -> 72 us.  (64-column tiles of two-product
// units would stage 24 KB for 256 clocks of MMA, more than the 65 bytes a clock
// that one SM gets from L2.)
constexpr int kStagesPair = 6;
constexpr uint32_t kStageBytesPair = 2 * kTile;  // A_p and this CTA's B tile

struct EqPairMaps {
    CUtensorMap a, b, bh;  // B slices in boxes of a tile's columns and of half as many
};

template <int TN>
__device__ __forceinline__ void eq_tile_pair(const EqArgs &a, int t, int &m0, int &n0) {
    const int per_group = (kGroupM / 2) * a.n_tiles;
    const int g = t / per_group, r = t % per_group;
    const int rows = min(kGroupM / 2, a.m_tiles - g * (kGroupM / 2));
    m0 = (g * (kGroupM / 2) + r % rows) * 2 * kBM;
    n0 = (r / rows) * TN;
}

// a.m_tiles counts 256-row slabs here
template <int TN>
__global__ void __launch_bounds__(kThreads, 1) gemm_fp64eq_pair_kernel(const __grid_constant__ EqPairMaps maps,
                                                                      const __grid_constant__ EqArgs a) {
    extern __shared__ __align__(1024) unsigned char esm_raw[];
    unsigned char *sm = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(esm_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    unsigned char *out = sm + kStagesPair * kStageBytesPair;  // the epilogue warps' store staging
    uint64_t *bars = reinterpret_cast<uint64_t *>(out + kEpiWarps * eq::kOutBytes);
    uint64_t *full = bars, *empty = bars + kStagesPair;
    uint64_t *tfull = bars + 2 * kStagesPair, *tempty = tfull + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(tempty + 2);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);

    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const bool leader = rank == 0;
    const int cid = (int)(blockIdx.x >> 1), ncl = (int)(gridDim.x >> 1);
    const int tiles = a.m_tiles * a.n_tiles;
    const int units = a.nunits * a.nkb;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStagesPair; ++s) {
            bar_init(su32(&full[s]), 1);   // rank 0's: its expect-tx arrival + both CTAs' bytes
            bar_init(su32(&empty[s]), 1);  // the MMA commit
        }
        for (int b = 0; b < 2; ++b) {
            bar_init(su32(&tfull[b]), 1);
            bar_init(su32(&tempty[b]), 2 * kEpiWarps);  // rank 0's: every epilogue warp of both CTAs
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        tmem_alloc_pair(su32(tmem_slot), 512);
        fence_before();
    }
    __syncthreads();
    cluster_sync_all();  // both CTAs' barriers and TMEM exist before either uses the other's
    fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    wait_previous();

    int loaded = 0, units_mma = 0;
    if (warp == 0) {
        // ---------------------------------------------------- TMA producer (both CTAs, whole warp)
        const uint32_t el = elect_one();
        const uint32_t sm0 = su32(sm), empty0 = su32(empty);
        const uint32_t full_here = su32(full), full0 = map_to_rank(full_here, 0);
        int s = 0;
        uint32_t phase = 1;  // the ring's first use needs no wait
        bool ok = true;
        for (int t = cid; ok && t < tiles; t += ncl) {
            int m0, n0;
            eq_tile_pair<TN>(a, t, m0, n0);
            for (int kbi = 0; ok && kbi < a.nkb; ++kbi)  // K-block outer: its slices stay in L2
                for (int pr = 0; ok && pr < a.nunits; ++pr) {
                    const int rowA = a.up[pr] * a.m + m0 + (int)rank * kBM;
                    // this CTA's B rows: half tiles c .. c + nq - 1 of the unit's 2 nq, in one
                    // or two boxes (nq = 3: a whole tile and half of the middle one)
                    const int nq = a.unq[pr], c = (int)rank * nq;
                    const int rowB = (a.uq[pr] + (c >> 1)) * a.n + n0 + (c & 1) * (TN / 2);
                    const bool half1 = nq == 1 || (c & 1) != 0;
                    const CUtensorMap *mb = half1 ? &maps.bh : &maps.b;
                    const int rowB2 = (a.uq[pr] + (c >> 1) + 1) * a.n + n0;  // nq > 2
                    const CUtensorMap *mb2 = nq == 3 && !half1 ? &maps.bh : &maps.b;
                    const uint32_t off2 = kTile + (half1 ? TN / 2 : TN) * kBK * 2;
                    const uint32_t tx = 2 * kTile + nq * TN * kBK * 2;
                    const int ks1 = min(a.ksteps, (kbi + 1) * a.kb_steps);
                    for (int ks = kbi * a.kb_steps; ks < ks1; ++ks) {
                        if (loaded >= kStagesPair && !warp_wait<true>(empty0 + s * 8, phase, abort_flag, a.err, 1u)) {
                            ok = false;
                            break;
                        }
                        const uint32_t st = sm0 + s * kStageBytesPair, fb = full0 + s * 8;
                        if (leader) bar_expect_tx_if(el, full_here + s * 8, tx);
                        tma_2d_pair_if(el, st, &maps.a, ks * kBK, rowA, fb);
                        tma_2d_pair_if(el, st + kTile, mb, ks * kBK, rowB, fb);
                        if (TN < kBN && nq > 2) tma_2d_pair_if(el, st + off2, mb2, ks * kBK, rowB2, fb);
                        ++loaded;
                        if (++s == kStagesPair) {
                            s = 0;
                            phase ^= 1;
                        }
                    }
                }
        }
    } else if (warp == 1 && leader) {
        // ---------------------------------------------------- MMA issuer (rank 0, whole warp)
        const uint32_t el = elect_one();
        const uint64_t da0 = sdesc_sw128(su32(sm)), db0 = sdesc_sw128(su32(sm) + kTile);
        const uint32_t full0 = su32(full), empty0 = su32(empty), tfull0 = su32(tfull), tempty0 = su32(tempty);
        int s = 0, gu = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int t = cid; ok && t < tiles; t += ncl) {
            for (int kbi = 0; ok && kbi < a.nkb; ++kbi)
                for (int pr = 0; ok && pr < a.nunits; ++pr, ++gu) {
                    const int b = gu & 1;
                    if (gu > 1 &&
                        !warp_wait<true>(tempty0 + b * 8, ((gu >> 1) - 1) & 1, abort_flag, a.err, 2u)) {
                        ok = false;
                        break;
                    }
                    fence_after();
                    const uint32_t d = tmem + (uint32_t)(b * 2 * kBN);
                    const uint32_t idesc = idesc_bf16(2 * kBM, a.unq[pr] * TN);
                    const int steps = min(a.ksteps, (kbi + 1) * a.kb_steps) - kbi * a.kb_steps;
                    uint32_t acc = 0;
                    for (int ks = 0; ks < steps; ++ks) {
                        if (!warp_wait<true>(full0 + s * 8, phase, abort_flag, a.err, 2u)) {
                            ok = false;
                            break;
                        }
                        fence_after();
                        const uint64_t da = da0 + (uint64_t)(s * (int)(kStageBytesPair >> 4)),
                                       db = db0 + (uint64_t)(s * (int)(kStageBytesPair >> 4));
#pragma unroll
                        for (int kk = 0; kk < kBK / 16; ++kk) {  // 32 bytes of each row per MMA
                            mma_bf16_pair_if(el, d, da + kk * 2, db + kk * 2, idesc, acc);
                            acc = 1;
                        }
                        mma_commit_pair_if(el, empty0 + s * 8, 3);  // stage s free in both CTAs
                        if (++s == kStagesPair) {
                            s = 0;
                            phase ^= 1;
                        }
                    }
                    if (!ok) break;
                    mma_commit_pair_if(el, tfull0 + b * 8, 3);  // this unit's accumulators complete in both CTAs
                    ++units_mma;
                }
        }
    } else if (warp >= 2) {
        // ---------------------------------------------------- epilogue (both CTAs)
        const int q = warp & 3;
        const int h = (warp - 2) >> 2;
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        constexpr int NC = TN / 2;  // columns of a warp
        float Sh[NC], Sl[NC];
        int gu = 0;
        bool ok = true;
        for (int t = cid; ok && t < tiles; t += ncl) {
            int m0, n0;
            eq_tile_pair<TN>(a, t, m0, n0);
            m0 += (int)rank * kBM;
#pragma unroll
            for (int j = 0; j < NC; ++j) Sh[j] = Sl[j] = 0.0f;
            for (int u = 0; u < units; ++u, ++gu) {
                const int b = gu & 1;
                if (!bar_wait_cluster(su32(&tfull[b]), (gu >> 1) & 1, abort_flag, a.err, 4u)) {
                    ok = false;
                    break;
                }
                fence_after();
                const int pr = u % a.nunits;
                const int nq = a.unq[pr];
                const float f1 = a.us[pr], f2 = f1 * a.uq_step;  // powers of two: exact scales
                const float f3 = f2 * a.uq_step, f4 = f3 * a.uq_step;
                const uint32_t acc = tmem + (uint32_t)(b * 2 * kBN) + lane_off + (uint32_t)(h * NC);
#pragma unroll
                for (int c = 0; c < NC; c += 8) {
                    uint32_t v[8], w[8], x[8], y[8];
                    OO_TMEM_LD8(acc + c, v);
                    if (nq > 1) OO_TMEM_LD8(acc + TN + c, w);
                    if (TN < kBN && nq > 2) OO_TMEM_LD8(acc + 2 * TN + c, x);
                    if (TN < kBN && nq > 3) OO_TMEM_LD8(acc + 3 * TN + c, y);
                    tmem_wait_ld();
                    if (TN < kBN && nq > 3)  // smallest first
                        eq::add_two8(Sh + c, Sl + c, y, f4, x, f3);
                    else if (TN < kBN && nq > 2)
                        eq::add_one8(Sh + c, Sl + c, x, f3);
                    if (nq > 1)
                        eq::add_two8(Sh + c, Sl + c, w, f2, v, f1);
                    else
                        eq::add_one8(Sh + c, Sl + c, v, f1);
                }
                fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (leader)
                        bar_arrive(su32(&tempty[b]));
                    else
                        bar_arrive_remote(map_to_rank(su32(&tempty[b]), 0));
                }
            }
            const int row0 = m0 + q * 32, c0 = n0 + h * NC, ncols = min(NC, a.n - c0);
            if (ok && row0 < a.m && ncols > 0) {
                // scales: lane l holds row row0 + l's and columns c0 + l's (and c0 + 32 + l's)
                const int ea = row0 + lane < a.m ? a.ea[row0 + lane] : 0;
                int eb[NC / 32];
#pragma unroll
                for (int i = 0; i < NC / 32; ++i) eb[i] = 32 * i + lane < ncols ? a.eb[c0 + 32 * i + lane] : 0;
                eq::store_columns(Sh, Sl, out + (warp - 2) * eq::kOutBytes, a.C, a.ldc, row0, c0,
                                  min(32, a.m - row0), ncols, ea, eb);
            }
        }
    }
    // drain on abort (bounded): rank 0 waits for its issued MMAs and for the
    // copies counted on its barriers; rank 1 for the commits that free its
    // stages (its copies complete on rank 0's barriers)
    if (*abort_flag) {
        if (warp == 1 && lane == 0 && leader && units_mma > 0)
            bar_drain(su32(&tfull[(units_mma - 1) & 1]), ((units_mma - 1) >> 1) & 1);
        if (warp == 0 && lane == 0)
            for (int it = (loaded > kStagesPair ? loaded - kStagesPair : 0); it < loaded; ++it)
                bar_drain(su32(leader ? &full[it % kStagesPair] : &empty[it % kStagesPair]),
                          (it / kStagesPair) & 1);
    }
    fence_before();
    __syncthreads();
    cluster_sync_all();  // neither CTA leaves while the other may still signal it or read its TMEM
    if (warp == 1) {
        fence_after();
        tmem_dealloc_pair(tmem, 512);
    }
}

// ------------------------------------------------------------ splitting
// A (m x k, lda) -> ea and slices As[p] (m x kp each, p < s); one warp per row
__device__ __forceinline__ void split_rows(const double *A, long long lda, int m, int k, int kp, int beta, int s,
                                           int *ea, __nv_bfloat16 *As, int block) {
    const int row = block * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= m) return;
    const int lane = threadIdx.x & 31;
    const double *src = A + (long long)row * lda;
    int mx = 0;
#pragma unroll 4
    for (int l = lane; l < k; l += 32) mx = max(mx, eff_exp(src[l]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) ea[row] = mx == 0 ? 0 : mx - 1022;
    const size_t plane = (size_t)m * kp;
    __nv_bfloat162 *dst = reinterpret_cast<__nv_bfloat162 *>(As + (size_t)row * kp);
    for (int l2 = lane; l2 < kp / 2; l2 += 32) {
        const int l = 2 * l2;
        unsigned n0 = 0, n1 = 0;
        const unsigned long long X0 = (mx != 0 && l < k) ? fixed_frac(src[l], mx, n0) : 0ull;
        const unsigned long long X1 = (mx != 0 && l + 1 < k) ? fixed_frac(src[l + 1], mx, n1) : 0ull;
        for (int p = 0; p < s; ++p)
            reinterpret_cast<unsigned *>(dst)[p * (plane / 2) + l2] = eq::digit_pair(X0, n0, X1, n1, beta, p);
    }
}

// Same split, one 256-thread CTA per row and 16-byte loads (lda even, A
// 16-byte aligned): the row's second read hits L1, and each thread keeps
// eight loads in flight in the exponent pass.
__device__ __forceinline__ void split_row_v2(const double *A, long long lda, int m, int k, int kp, int beta, int s,
                                             int *ea, __nv_bfloat16 *As, int row) {
    const double2 *src = reinterpret_cast<const double2 *>(A + (long long)row * lda);
    const int k2 = k >> 1;
    int mx = 0;
#pragma unroll 8
    for (int l2 = threadIdx.x; l2 < k2; l2 += 256) {
        const double2 v = src[l2];
        mx = max(mx, max(eff_exp(v.x), eff_exp(v.y)));
    }
    if ((k & 1) && threadIdx.x == 0) mx = max(mx, eff_exp(A[(long long)row * lda + k - 1]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    __shared__ int red[8];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    mx = red[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) mx = max(mx, red[w]);
    if (threadIdx.x == 0) ea[row] = mx == 0 ? 0 : mx - 1022;
    const size_t plane2 = (size_t)m * kp / 2;
    __nv_bfloat162 *dst = reinterpret_cast<__nv_bfloat162 *>(As + (size_t)row * kp);
#pragma unroll 2
    for (int l2 = threadIdx.x; l2 < kp / 2; l2 += 256) {
        const int l = 2 * l2;
        double2 v = make_double2(0.0, 0.0);
        if (l + 1 < k) {
            v = src[l2];
        } else if (l < k) {
            v.x = A[(long long)row * lda + l];
        }
        unsigned n0 = 0, n1 = 0;
        const unsigned long long X0 = mx != 0 ? fixed_frac(v.x, mx, n0) : 0ull;
        const unsigned long long X1 = mx != 0 ? fixed_frac(v.y, mx, n1) : 0ull;
        for (int p = 0; p < s; ++p)
            reinterpret_cast<unsigned *>(dst)[p * plane2 + l2] = eq::digit_pair(X0, n0, X1, n1, beta, p);
    }
}

// The split of A and, before it in the grid, the largest effective exponents
// of B's columns (mxo, zero on entry; blocks of 32 columns x rows_per rows),
// which the split of B waits for: one launch, so that the column blocks'
// latency hides behind the rows' traffic.
template <bool V2>
__global__ void __launch_bounds__(256) eq_split_rows_kernel(const double *A, long long lda, int m, int k, int kp,
                                                          int beta, int s, int *ea, __nv_bfloat16 *As,
                                                          const double *B, long long ldb, int n, int rows_per,
                                                          int col_blocks, int max_blocks, int *mxo) {
    if ((int)blockIdx.x >= max_blocks) {
        if (V2)
            split_row_v2(A, lda, m, k, kp, beta, s, ea, As, blockIdx.x - max_blocks);
        else
            split_rows(A, lda, m, k, kp, beta, s, ea, As, blockIdx.x - max_blocks);
        return;
    }
    const int col = (int)(blockIdx.x % col_blocks) * 32 + (threadIdx.x & 31);
    const int r0 = (int)(blockIdx.x / col_blocks) * rows_per, r1 = min(k, r0 + rows_per);
    int mx = 0;
    if (col < n) {
#pragma unroll 8
        for (int l = r0 + (threadIdx.x >> 5); l < r1; l += 8) mx = max(mx, eff_exp(B[(long long)l * ldb + col]));
    }
    __shared__ int red[256];
    red[threadIdx.x] = mx;
    __syncthreads();
    if (threadIdx.x < 32 && col < n) {
#pragma unroll
        for (int w = 1; w < 8; ++w) mx = max(mx, red[w * 32 + threadIdx.x]);
        if (mx > 0) atomicMax(mxo + col, mx);
    }
}

// B tile of 64 (k) x 64 (columns) -> transposed slices Bs[q] (n x kp each) and
// the columns' scale exponents eb; mxo holds the column maxima (exponent
// fields); 256 threads
__global__ void eq_split_cols_t_kernel(const double *B, long long ldb, int k, int n, int kp, int beta, int s,
                                       const int *mxo, int *eb, __nv_bfloat16 *Bs) {
    __shared__ double t[64][65];
    next_may_start();
    const int c0 = blockIdx.x * 64, l0 = blockIdx.y * 64;
    const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
    if (l0 == 0 && ty == 0 && c0 + tx < n) eb[c0 + tx] = mxo[c0 + tx] == 0 ? 0 : mxo[c0 + tx] - 1022;
#pragma unroll
    for (int yy = ty; yy < 64; yy += 4) {
        const int l = l0 + yy, c = c0 + tx;
        t[yy][tx] = (l < k && c < n) ? B[(long long)l * ldb + c] : 0.0;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const size_t plane = (size_t)n * kp;
    for (int cc = w * 8; cc < w * 8 + 8; ++cc) {
        const int c = c0 + cc;
        if (c >= n) break;
        const int mx = mxo[c];
        unsigned n0 = 0, n1 = 0;
        const unsigned long long X0 = mx != 0 ? fixed_frac(t[2 * lane][cc], mx, n0) : 0ull;
        const unsigned long long X1 = mx != 0 ? fixed_frac(t[2 * lane + 1][cc], mx, n1) : 0ull;
        __nv_bfloat162 *dst = reinterpret_cast<__nv_bfloat162 *>(Bs + (size_t)c * kp + l0) + lane;
        for (int p = 0; p < s; ++p)
            reinterpret_cast<unsigned *>(dst)[p * (plane / 2)] = eq::digit_pair(X0, n0, X1, n1, beta, p);
    }
}

size_t smem_eq() { return 1024 + (size_t)kStages * kStageBytes + 256; }
constexpr size_t kSmemEqPair = 1024 + (size_t)kStagesPair * kStageBytesPair + kEpiWarps * eq::kOutBytes + 256;
static_assert(kSmemEqPair <= 232448, "pair kernel exceeds the shared memory of a CTA");

// 2-CTA clusters of the pair kernel that fit on the device at once (cached)
template <int TN>
int eq_pair_clusters() {
    int dev = 0;
    OO_CUDA_TRY(cudaGetDevice(&dev));
    static std::atomic<int> max_clusters[64];
    int ncl = dev < 64 ? max_clusters[dev].load() : 0;
    if (ncl > 0) return ncl;
    static std::atomic<uint64_t> attr{0};
    set_smem_limit_once((const void *)gemm_fp64eq_pair_kernel<TN>, kSmemEqPair, attr);
    int sms = 148;
    OO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(sms / 2 * 2));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemEqPair;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    OO_CUDA_TRY(cudaOccupancyMaxActiveClusters(&ncl, (const void *)gemm_fp64eq_pair_kernel<TN>, &cfg));
    OO_REQUIRE(ncl >= 1, OO_ECUDA, "no 2-CTA cluster of the FP64-equivalent kernel fits on this device");
    if (dev < 64) max_clusters[dev].store(ncl);
    return ncl;
}

struct EqLayout {
    size_t err, ea, eb, mxo, as, bs, total;
};
EqLayout eq_layout(int m, int n, int k) {
    const EqShape e = eq_used_shape(k);
    const size_t kp = (size_t)(k + kBK - 1) / kBK * kBK;
    auto up = [](size_t x) { return (x + 255) / 256 * 256; };
    EqLayout L{};
    L.err = 0;
    L.mxo = 256;
    L.ea = L.mxo + up((size_t)n * 4);
    L.eb = L.ea + up((size_t)m * 4);
    L.as = L.eb + up((size_t)n * 4);
    L.bs = L.as + up((size_t)e.slices * m * kp * 2);
    L.total = L.bs + up((size_t)e.slices * n * kp * 2);
    return L;
}

}  // namespace

// ------------------------------------------- level schemes' digit split
// The split of products with k <= 512, in batches and single calls (eight
// BF16 digits of 16 bytes leave a thread at once; digit width and count are
// constants, so a digit is a shift, a mask, a subtraction and half a
// permute).  Bound by HBM in batches (8 bytes read and 2 S written an entry)
// and by latency for one product.  4096 products, m, n, k log-uniform in [16,
// 512]: rows 625 us and columns 1030 us with a warp per row or 64 columns per
// block, 4-byte stores and every entry of B read twice; 520 and 795 us so.  One
// 256 x 256 x 256 product: 34 us in four launches and two clears, 11 us in one.
namespace {

template <int BETA, int S>
struct LevelSplit {
    // digits of eight consecutive entries relative to 2^(mx - 1022) -> dst, one
    // 16-byte store per slice
    static __device__ __forceinline__ void eight(const double (&v)[8], int mx, __nv_bfloat16 *dst, size_t plane) {
        unsigned long long X[8];
        unsigned sign[4];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            unsigned n = 0;
            X[i] = mx != 0 ? fixed_frac(v[i], mx, n) : 0ull;
            if (mx == 0) n = 0;
            if (i & 1)
                sign[i >> 1] |= n << 31;
            else
                sign[i >> 1] = n << 15;
        }
#pragma unroll
        for (int p = 0; p < S; ++p) {
            unsigned w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                // d < 2^8 is exact as 2^23 + d - 2^23, its BF16 bits the float's top half
                auto digit = [&](unsigned long long x) {
                    const unsigned d = (unsigned)(x >> (64 - BETA * (p + 1))) & ((1u << BETA) - 1u);
                    return __float_as_uint(__fsub_rn(__uint_as_float(0x4b000000u | d), 8388608.0f));
                };
                w[i] = __byte_perm(digit(X[2 * i]), digit(X[2 * i + 1]), 0x7632) | sign[i];
            }
            *reinterpret_cast<uint4 *>(dst + p * plane) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }

    // rows [r0, r0 + 32) of A: eight lanes a row, eight entries a lane
    static __device__ __forceinline__ void rows(const eq::GSplit &G, int r0) {
        const int lane = threadIdx.x & 31, sub = lane & 7;
        const int row = r0 + (threadIdx.x >> 5) * 4 + (lane >> 3);
        const bool in = row < G.m;
        const double *src = G.A + (long long)(in ? row : 0) * G.lda;
        const int k = in ? G.k : 0;
        const bool vec = (((uintptr_t)G.A | (uintptr_t)(G.lda * 8)) & 15u) == 0;
        auto load = [&](int l, double (&v)[8]) {
            if (vec && l + 8 <= k) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const double2 x = reinterpret_cast<const double2 *>(src + l)[i];
                    v[2 * i] = x.x;
                    v[2 * i + 1] = x.y;
                }
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = l + i < k ? src[l + i] : 0.0;
            }
        };
        int mx = 0;
        double v[8];
        for (int l = 8 * sub; l < G.kp; l += 64) {
            load(l, v);
#pragma unroll
            for (int i = 0; i < 8; ++i) mx = max(mx, eff_exp(v[i]));
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (!in) return;
        if (sub == 0) G.ea[row] = mx == 0 ? 0 : mx - 1022;
        __nv_bfloat16 *dst = G.As + (size_t)row * G.pitch;
        for (int l = 8 * sub; l < G.kp; l += 64) {
            if (G.kp > 64) load(l, v);  // from L1; one chunk is still in registers
            eight(v, mx, dst + l, (size_t)G.m * G.pitch);
        }
    }

    // columns [c0, c0 + C) of B through shared memory, read once: t holds C
    // columns of kp + 1 doubles (an odd pitch, so a row's stores fall in
    // different banks), red 256 ints.  Every thread of the block calls it.
    template <int C>
    static __device__ __forceinline__ void cols(const eq::GSplit &G, int c0, double *t, int *red) {
        constexpr int R = 256 / C;  // rows read at a time
        const int tx = threadIdx.x % C, ty = threadIdx.x / C, col = c0 + tx, pitch = G.kp + 1;
        int mx = 0;
#pragma unroll 8
        for (int l = ty; l < G.kp; l += R) {
            const double x = l < G.k && col < G.n ? G.B[(long long)l * G.ldb + col] : 0.0;
            mx = max(mx, eff_exp(x));
            t[tx * pitch + l] = x;
        }
        red[threadIdx.x] = mx;
        __syncthreads();
        if (ty == 0) {
#pragma unroll 8
            for (int y = 1; y < R; ++y) mx = max(mx, red[y * C + tx]);
            red[tx] = mx;
            if (col < G.n) G.eb[col] = mx == 0 ? 0 : mx - 1022;
        }
        __syncthreads();
        const int sub = threadIdx.x & 7, chunks = G.kp / 64;
        for (int u = threadIdx.x >> 3; u < C * chunks; u += 32) {
            const int c = u % C, l = (u / C) * 64 + 8 * sub;
            if (c0 + c >= G.n) continue;
            double v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = t[c * pitch + l + i];
            eight(v, red[c], G.Bs + (size_t)(c0 + c) * G.pitch + l, (size_t)G.n * G.pitch);
        }
    }
};

// columns per job and its shared memory: small enough for a full SM of blocks
template <int BETA>
struct LevelCols;
template <>
struct LevelCols<7> {  // k <= 128
    static constexpr int C = 16, kMax = 128;
};
template <>
struct LevelCols<6> {  // k <= 512
    static constexpr int C = 8, kMax = 512;
};
template <int BETA>
constexpr size_t level_cols_smem(int kp) {
    return (size_t)LevelCols<BETA>::C * (kp + 1) * 8;
}

// jobs (first row), then jobs (first column) of one kind per launch
template <int BETA, int S>
__global__ void __launch_bounds__(256) eq_level_rows_kernel(const eq::GSplit *gs, const int4 *jobs) {
    const int4 jb = jobs[blockIdx.x];
    const eq::GSplit G = gs[jb.y];
    LevelSplit<BETA, S>::rows(G, jb.z);
}
template <int BETA, int S>
__global__ void __launch_bounds__(256) eq_level_cols_kernel(const eq::GSplit *gs, const int4 *jobs) {
    extern __shared__ __align__(16) double lv_t[];
    __shared__ int red[256];
    const int4 jb = jobs[blockIdx.x];
    const eq::GSplit G = gs[jb.y];
    LevelSplit<BETA, S>::template cols<LevelCols<BETA>::C>(G, jb.z, lv_t, red);
}
// one product: the first row_blocks blocks take rows, the others columns
template <int BETA, int S>
__global__ void __launch_bounds__(256) eq_level_split_kernel(const __grid_constant__ eq::GSplit G, int row_blocks,
                                                            unsigned *err) {
    extern __shared__ __align__(16) double lv_t[];
    __shared__ int red[256];
    next_may_start();
    if (blockIdx.x == 0 && threadIdx.x == 0) *err = 0;  // of the product kernel that follows
    if ((int)blockIdx.x < row_blocks)
        LevelSplit<BETA, S>::rows(G, blockIdx.x * 32);
    else
        LevelSplit<BETA, S>::template cols<LevelCols<BETA>::C>(G, (blockIdx.x - row_blocks) * LevelCols<BETA>::C,
                                                               lv_t, red);
}

template <int BETA, int S>
void launch_level_split(const eq::GSplit &G, unsigned *err, cudaStream_t s) {
    constexpr int C = LevelCols<BETA>::C;
    const int row_blocks = (G.m + 31) / 32, col_blocks = (G.n + C - 1) / C;
    eq_level_split_kernel<BETA, S><<<row_blocks + col_blocks, 256, level_cols_smem<BETA>(G.kp), s>>>(G, row_blocks,
                                                                                                   err);
    OO_CUDA_TRY(cudaGetLastError());
}

// The grouped split of pair-scheme products (k > 512): eight rows of A a
// block, then 64 columns of B a block (eq_digits.cuh).
__global__ void __launch_bounds__(256) eq_group_split_rows_kernel(const eq::GSplit *gs, const int4 *jobs) {
    const int4 jb = jobs[blockIdx.x];
    eq::split_rows_job(gs[jb.y], jb.z);
}
__global__ void __launch_bounds__(256) eq_group_split_cols_kernel(const eq::GSplit *gs, const int4 *jobs) {
    __shared__ double t[64][65];
    __shared__ int red[4][64];
    const int4 jb = jobs[blockIdx.x];
    eq::split_cols_job(gs[jb.y], jb.z, t, red);
}

// the pair scheme's units and scales, up to `most` slices of B a unit
void set_units(EqArgs &a, const EqShape &e, int most) {
    const std::vector<eq::PairUnit> U = eq::pair_units(e, most);
    OO_REQUIRE((int)U.size() <= kMaxUnits, OO_EINVAL, "too many product groups");
    a.nunits = (int)U.size();
    a.uq_step = std::ldexp(1.0f, -e.beta);
    for (size_t i = 0; i < U.size(); ++i) {
        a.up[i] = (unsigned char)U[i].p;
        a.uq[i] = (unsigned char)U[i].q;
        a.unq[i] = (unsigned char)U[i].nq;
        a.us[i] = std::ldexp(1.0f, -e.beta * (U[i].p + U[i].q + 2));
    }
}

template <int TN>
void launch_pair(EqArgs &a, const EqShape &e, __nv_bfloat16 *As, __nv_bfloat16 *Bs, int kp, int clusters,
                 cudaStream_t s) {
    set_units(a, e, 2 * kBN / TN);
    EqPairMaps pm;
    map_bf16(&pm.a, As, (long long)e.slices * a.m, kp, kBM);
    map_bf16(&pm.b, Bs, (long long)e.slices * a.n, kp, TN);
    map_bf16(&pm.bh, Bs, (long long)e.slices * a.n, kp, TN / 2);
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1] = programmatic();
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(2 * clusters));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemEqPair;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    OO_CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_fp64eq_pair_kernel<TN>, (const EqPairMaps)pm, (const EqArgs)a));
}

}  // namespace

void eq_group_split_jobs(int scheme, int problem, int m, int n, std::vector<int4> (&jobs)[6]) {
    const bool pairs = scheme == eq::kSchemePairs;
    const int base = pairs ? 0 : (scheme == eq::kSchemeLevel7 ? 2 : 4);
    const int rows = pairs ? 8 : 32;
    const int cols = pairs ? 64 : (scheme == eq::kSchemeLevel7 ? LevelCols<7>::C : LevelCols<6>::C);
    for (int r = 0; r < m; r += rows) jobs[base].push_back(make_int4(0, problem, r, 0));
    for (int c = 0; c < n; c += cols) jobs[base + 1].push_back(make_int4(1, problem, c, 0));
}

void launch_eq_group_split(const eq::GSplit *gs, const int4 *jobs, const int (&count)[6], cudaStream_t s) {
    for (int x = 0; x < 6; jobs += count[x++]) {
        if (count[x] == 0) continue;
        switch (x) {
            case 0: eq_group_split_rows_kernel<<<count[x], 256, 0, s>>>(gs, jobs); break;
            case 1: eq_group_split_cols_kernel<<<count[x], 256, 0, s>>>(gs, jobs); break;
            case 2: eq_level_rows_kernel<7, 7><<<count[x], 256, 0, s>>>(gs, jobs); break;
            case 3:
                eq_level_cols_kernel<7, 7><<<count[x], 256, level_cols_smem<7>(LevelCols<7>::kMax), s>>>(gs, jobs);
                break;
            case 4: eq_level_rows_kernel<6, 8><<<count[x], 256, 0, s>>>(gs, jobs); break;
            case 5:
                eq_level_cols_kernel<6, 8><<<count[x], 256, level_cols_smem<6>(LevelCols<6>::kMax), s>>>(gs, jobs);
                break;
        }
        OO_CUDA_TRY(cudaGetLastError());
    }
}

size_t gemm_fp64eq_scratch_bytes(int m, int n, int k) { return eq_layout(m, n, k).total; }

int gemm_fp64eq_products(int k) { return eq_used_shape(k).nprod; }

void gemm_fp64eq_shape(int k, int *beta, int *levels, int *k_block) {
    const EqShape e = eq_used_shape(k);
    if (beta) *beta = e.beta;
    if (levels) *levels = e.levels;
    if (k_block) *k_block = e.kb;
}

void launch_gemm_fp64eq(int m, int n, int k, const double *A, long long lda, const double *B, long long ldb,
                        double *C, long long ldc, void *scratch, cudaStream_t s, int width, bool pair) {
    OO_REQUIRE(m >= 1 && n >= 1 && k >= 1, OO_EINVAL, "m, n, k must be >= 1");
    OO_REQUIRE(lda >= k && ldb >= n && ldc >= n, OO_EINVAL, "leading dimensions too small");
    const EqShape e = eq_used_shape(k);
    OO_REQUIRE((long long)e.slices * m < (1ll << 31) && (long long)e.slices * n < (1ll << 31), OO_EINVAL,
               "matrix too large for the FP64-equivalent mode");
    const int kp = (k + kBK - 1) / kBK * kBK;
    const EqLayout L = eq_layout(m, n, k);
    char *p = static_cast<char *>(scratch);
    unsigned *err = reinterpret_cast<unsigned *>(p + L.err);
    int *ea = reinterpret_cast<int *>(p + L.ea), *eb = reinterpret_cast<int *>(p + L.eb);
    int *mxo = reinterpret_cast<int *>(p + L.mxo);
    auto *As = reinterpret_cast<__nv_bfloat16 *>(p + L.as);
    auto *Bs = reinterpret_cast<__nv_bfloat16 *>(p + L.bs);
    int dev = 0, sms = 148;
    OO_CUDA_TRY(cudaGetDevice(&dev));
    OO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (e.scheme != eq::kSchemePairs) {
        // level schemes: split and tiled kernel as in batches
        const eq::GSplit G{A, B, lda, ldb, kp, m, n, k, kp, e.beta, e.slices, As, Bs, ea, eb};
        if (e.scheme == eq::kSchemeLevel7)
            launch_level_split<7, 7>(G, err, s);
        else
            launch_level_split<6, 8>(G, err, s);
        launch_gemm_eq_tiles(m, n, k, As, Bs, ea, eb, C, ldc, width, err, sms, s);
        return;
    }
    OO_CUDA_TRY(cudaMemsetAsync(err, 0, L.ea - L.err, s));  // the error word and the column maxima
    {
        constexpr int kRowsPer = 128;  // 16 loads a thread, in two batches
        const int col_blocks = (n + 31) / 32, max_blocks = col_blocks * ((k + kRowsPer - 1) / kRowsPer);
        const bool v2 = lda % 2 == 0 && ((uintptr_t)A & 15u) == 0;
        const long long blocks = (long long)max_blocks + (v2 ? m : (m + 7) / 8);
        OO_REQUIRE(blocks < (1ll << 31), OO_EINVAL, "matrix too large");
        (v2 ? eq_split_rows_kernel<true> : eq_split_rows_kernel<false>)<<<(unsigned)blocks, 256, 0, s>>>(
            A, lda, m, k, kp, e.beta, e.slices, ea, As, B, ldb, n, kRowsPer, col_blocks, max_blocks, mxo);
        OO_CUDA_TRY(cudaGetLastError());
    }
    {
        dim3 grid((n + 63) / 64, kp / 64);
        OO_REQUIRE(grid.y <= 65535, OO_EINVAL, "k too large");
        eq_split_cols_t_kernel<<<grid, 256, 0, s>>>(B, ldb, k, n, kp, e.beta, e.slices, mxo, eb, Bs);
        OO_CUDA_TRY(cudaGetLastError());
    }
    EqArgs ga{};
    ga.m = m;
    ga.n = n;
    ga.ksteps = kp / kBK;
    ga.kb_steps = e.kb / kBK;
    ga.nkb = e.nkb;
    ga.m_tiles = (m + kBM - 1) / kBM;
    ga.n_tiles = (n + kBN - 1) / kBN;
    ga.C = C;
    ga.ldc = ldc;
    ga.ea = ea;
    ga.eb = eb;
    ga.err = err;
    if (pair) {
        const int slabs = (m + 2 * kBM - 1) / (2 * kBM), n128 = (n + kBN - 1) / kBN, n64 = (n + 63) / 64;
        ga.m_tiles = slabs;
        const long long t128 = (long long)slabs * n128, t64 = (long long)slabs * n64;
        OO_REQUIRE(t64 < (1ll << 31), OO_EINVAL, "too many tiles");
        const int ncl = std::min(eq_pair_clusters<128>(), eq_pair_clusters<64>());
        // A narrow tile costs 0.57 of a wide one (a K step of all products 4,314 against
        // 7,656 clocks by staged bytes and MMA rate): narrow where that makes the waves
        // shorter.  1000 x 777 x 1300: 52 of 76 pairs for 28, 92 us for 144; 300 x 4000 x
        // 1000 would take two waves for one, and 2048^3 four for two, 2.28 times a wave.
        const long long w128 = (t128 + ncl - 1) / ncl, w64 = (t64 + ncl - 1) / ncl;
        if (57 * w64 < 100 * w128) {
            ga.n_tiles = n64;
            launch_pair<64>(ga, e, As, Bs, kp, (int)std::min<long long>(t64, ncl), s);
        } else {
            ga.n_tiles = n128;
            launch_pair<128>(ga, e, As, Bs, kp, (int)std::min<long long>(t128, ncl), s);
        }
        return;
    }
    EqMaps maps;
    map_bf16(&maps.a, As, (long long)e.slices * m, kp, kBM);
    map_bf16(&maps.b, Bs, (long long)e.slices * n, kp, kBN);
    set_units(ga, e, 2);
    static std::atomic<uint64_t> attr{0};
    set_smem_limit_once((const void *)gemm_fp64eq_kernel, smem_eq(), attr);
    const long long tiles = (long long)ga.m_tiles * ga.n_tiles;
    OO_REQUIRE(tiles < (1ll << 31), OO_EINVAL, "too many tiles");
    const int grid = (int)std::min<long long>(tiles, sms);
    OO_REQUIRE(grid >= 1, OO_EINVAL, "empty product");
    gemm_fp64eq_kernel<<<grid, kThreads, smem_eq(), s>>>(maps, ga);
    OO_CUDA_TRY(cudaGetLastError());
}

unsigned *gemm_fp64eq_error_word(void *scratch) { return static_cast<unsigned *>(scratch); }

unsigned gemm_fp64eq_check_error(void *scratch, cudaStream_t s) {
    unsigned *err = static_cast<unsigned *>(scratch);
    unsigned e = 0;
    OO_CUDA_TRY(cudaMemcpyAsync(&e, err, 4, cudaMemcpyDeviceToHost, s));
    OO_CUDA_TRY(cudaStreamSynchronize(s));
    if (e) OO_CUDA_TRY(cudaMemsetAsync(err, 0, 4, s));
    return e;
}

}  // namespace oo
