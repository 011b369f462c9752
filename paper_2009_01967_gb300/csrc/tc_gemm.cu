// Tensor-core (tcgen05) path of the Gamma-only linewidths: the per-mode
// contractions T = E Y_mu^T-form and phi = T E^T (paper Eq. projection_plus at
// q = 0) on 5th-generation tensor cores with a 16-bit hi+lo split.
//
// Every operand x is carried as two FP16 planes, hi = fp16(x), lo = fp16(x - hi),
// and a product is formed from three MMAs, A_hi B_hi + A_hi B_lo + A_lo B_hi,
// accumulated in FP32 in tensor memory; the dropped lo*lo term and the rounding of
// lo leave about 22 significant bits per product (two BF16 pieces left 16, and the
// error of gamma from that, 1e-5 for the smallest cells, grows when each triple of
// modes is projected once instead of three times).  FP16's narrow range is met by
// powers of two (Scales): each atom by how strongly Phi3 holds it, each mode's
// eigenvector by its largest component, the rows of Y_mu of one atom by their largest
// element as built, T by the norms of its two factors; the epilogues take them out
// exactly.
//
// Several modes go through each launch (a batch of MB modes, so that small
// systems still fill the GPU): the Y and T planes of the batch are stacked
// (plane b at rows b * rows .. ), GEMM1 takes the mode from blockIdx.z and
// GEMM2 from its tile record.
//
// Kernel shape (one 128 x 128 output tile per CTA, 128 threads; 512 for the triples'
// weights, four warps per 32 rows, since nothing overlaps an epilogue here: with 128
// threads it took 35 of that product's 50 ms for twelve cells of 324 to 1500 modes):
//   warp 0 lane 0   TMA producer: 4 tiled loads per K block of 64 (A hi/lo,
//                   B hi/lo; 128-byte swizzle), 3-stage ring of mbarriers
//   warp 1          allocates 512 TMEM columns (four accumulators); lane 0 issues the MMAs
//                   (M = 128, N = 128, K = 16, kind::f16, FP16 in, FP32 out)
//                   and commits each stage back to the producer
//   warps 0-3       epilogue: tcgen05.ld of their 32 accumulator lanes
// Every mbarrier wait is bounded; on expiry the CTA records the failure in a
// device flag, lets its copies and MMAs drain (bounded again), frees its TMEM
// and returns, and the host reports KALD_E_TIMEOUT.

#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

#include "kald_internal.h"
#include "tc_common.cuh"
#include "wdiff.cuh"

namespace kald {
namespace {

constexpr int kBM = 128, kBN = 128, kBK = 64;      // tile; 64 FP16 = one 128-byte swizzle row
constexpr int kStages = 3;
constexpr int kMaxBatch = 64;                      // modes per launch
// Tensor-core accumulation truncates: a long chain of MMAs into one accumulator
// (2592 / 16 x 3 for the 864-atom cell) drifts towards zero by about 1e-5 relative.
// The hi hi products go round-robin into three accumulators and the two small
// products into a fourth, whose own truncations are 2^-8 of that (all 512 TMEM
// columns); the epilogue adds the four in FP32.  A third of the K steps then
// truncate a full-size sum: all three products over four accumulators did so three
// quarters as often as there are steps.
constexpr int kAcc = 4;
constexpr int kTileBytes = kBM * kBK * 2;          // 16 KB per operand plane per stage
constexpr int kStageBytes = 4 * kTileBytes;        // A hi, A lo, B hi, B lo

enum : int { EPI_SPLIT = 0, EPI_GAMMA = 1, EPI_GSYM = 2 };
constexpr uint32_t kIdesc = tc::idesc_f16(kBN);

using namespace tc;

struct EpiGamma {
    const double *omega;      // [nb] rad/ps (0 = masked)
    const double *occ;        // [nb]
    int mu0;                  // first mode of the batch
    int a_rows;               // rows of one T plane (stacked per mode of the batch)
    double sig2inv, cut;      // delta-shape parameter (delta_param), window half width
    int shape;                // energy-delta shape
    double *partial;          // [n_tiles] per-tile sums of this batch
    unsigned long long *allowed;
    const int2 *tiles;        // (tm | b << 16, tn): band tile (tm, tn) of mode mu0 + b
    int symmetric;            // phi symmetric: upper-triangle tiles, symmetrised weights
    double *rowp, *colp;      // EPI_GSYM: [n_tiles][128] sums for the modes of a tile's rows and columns
};
struct EpiSplit {
    __half *hi, *lo;   // [batch][rows][ld] output planes
    int ld;
    int b_rows;               // rows of one Y / T plane (stacked per mode of the batch)
    int tm0;                  // first row tile
    int mu0;                  // first mode of the batch
    const int *yk;            // [batch][N / 3] exponents of the rows of Y (ybuild_rows_kernel)
};

// Powers of two that bring the operands into FP16's range.  With k the exponents of
// the atoms (atom_scale_kernel), E^(m, b) = 2^k_b E(m, b) and
// Y^_mu(c, b) = 2^(-k_b - k_c) Y_mu(c, b), whose contractions over b and c are those
// of E and Y:
//   E^(m, .) = 2^e_m E', |E'| <= 1 and |E'|_2 <= 2^h_m, stored x 2^kEBits;
//   Y^_mu(c, .) = 2^y_mu,k Y', |Y'| <= 1 (the largest element of the rows of c's atom
//   k), stored x 2^kYBits; y_mu = max over k;
//   T^ = E^ Y^_mu = 2^(e_m + y_mu) T', |T'| <= 2^(h_m + hR) (Cauchy-Schwarz: the rows
//   of Y_mu have at most 4^hR entries), stored x 2^(kTBits - h_m - hR).
// FP16's step is 2^-24, so an element keeps the 16 bits of two BF16 pieces down to
// 2^-23 of the largest one of its row of E or rows of Y_mu, and to some 2^-16 of a
// usual one of T.  The scales therefore follow what is measured: Y_mu per mode, since
// the strong couplings inside a molecule cancel for the modes that move it as a whole,
// and the atoms, since a mode may extend over parts whose Phi3 differs by orders of
// magnitude.  With one exponent for the whole Phi3 the modes of the weaker part lost
// 3e-4 of gamma where its Phi3 is 2^-16 of the stronger part's, 4e-3 at 2^-20 and 0.3
// at 2^-24; 4e-7 now, as in a uniform cell, and 2e-6 for modes mixed of the two parts
// at 2^-24 (216 modes).  What this takes: 256 atoms 2.88 -> 3.05 ms (3.14 with Y_mu
// built in FP32 first and scaled by its mode's largest element in a second pass).
constexpr int kEBits = 15, kYBits = 15, kTBits = 15;
struct Scales {
    const int *e, *h;         // [nb] e_m, h_m
    const int *ymax;          // [nb] y_mu (far below any exponent: no element)
    int hR;
    __device__ __forceinline__ int y(int mu) const {
        const int x = __ldg(ymax + mu);
        return x < -1000000 ? 0 : x;
    }
    // what takes an accumulator of the second contraction to phi, for row m of mode mu
    // and for column n
    __device__ __forceinline__ float row(int m, int mu) const {
        return ldexpf(1.0f, __ldg(e + m) + __ldg(h + m) + y(mu) + hR - kTBits - kEBits);
    }
    __device__ __forceinline__ float col(int n) const { return ldexpf(1.0f, __ldg(e + n)); }
};

// Columns [c, c + 32) of the accumulators, added in a fixed order.
__device__ __forceinline__ void tmem_ld_sum(uint32_t taddr, float v[32]) {
    tmem_ld32(taddr, v);
#pragma unroll
    for (int a = 1; a < kAcc; ++a) {
        float u[32];
        tmem_ld32(taddr + (uint32_t)(a * kBN), u);
#pragma unroll
        for (int x = 0; x < 32; ++x) v[x] += u[x];
    }
}

// Columns [c, c + 16) of the accumulators, added in the same order.
__device__ __forceinline__ void tmem_ld_sum16(uint32_t taddr, float v[16]) {
    tmem_ld16(taddr, v);
#pragma unroll
    for (int a = 1; a < kAcc; ++a) {
        float u[16];
        tmem_ld16(taddr + (uint32_t)(a * kBN), u);
#pragma unroll
        for (int x = 0; x < 16; ++x) v[x] += u[x];
    }
}

// Sums over the 32 lanes of 16 values each: lane l returns value l / 2 (both
// lanes of a pair the same), added pairwise in a fixed order.
__device__ __forceinline__ float lane_sums16(float (&v)[16]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 8; h > 0; h >>= 1) {
        const bool up = lane & (2 * h);
#pragma unroll
        for (int x = 0; x < h; ++x) {
            const float keep = up ? v[x + h] : v[x], send = up ? v[x] : v[x + h];
            v[x] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * h);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// The projections of mode a with the unordered pair {b, c} of two other positions:
// sum of the weights of (a; b, c) and (a; c, b) (of one of them for b = c) and
// their window hits, the energy differences formed as EPI_GAMMA forms them -- b the
// row and c the column, exchanged as well where both lie in one tile (`same`).
__device__ __forceinline__ float pair_terms(F2 wa, F2 wb, F2 wc, F2 nb_, F2 nc_, bool equal, bool same, float cut,
                                            int shape, float s2i, int &cnt) {
    const F2 dif = f2_add(wa, f2_neg(wb));
    const float dp = f2_diff(f2_add(wa, wb), wc), dm = f2_diff(dif, wc);
    const float dn = f2_diff(nb_, nc_), sn = 1.0f + nb_.h + nc_.h;
    const bool hp = fabsf(dp) < cut, hm = fabsf(dm) < cut;
    float g = 0.0f;
    if (hp) g += dn * delta_shape(dp, shape, s2i);
    if (hm) g += 0.5f * sn * delta_shape(dm, shape, s2i);
    cnt += hp || hm;
    if (equal) return g;
    const float dp2 = same ? f2_diff(f2_add(wa, wc), wb) : f2_diff(dif, f2_neg(wc));
    const float dm2 = same ? f2_diff(f2_add(wa, f2_neg(wc)), wb) : dm;
    const bool hp2 = fabsf(dp2) < cut, hm2 = fabsf(dm2) < cut;
    if (hp2) g -= dn * delta_shape(dp2, shape, s2i);
    if (hm2) g += 0.5f * sn * delta_shape(dm2, shape, s2i);
    cnt += hp2 || hm2;
    return g;
}

// C[m][n] = sum_k A[m][k] B[n][k]; A, B as FP16 hi/lo planes behind four
// tensor maps (box 64 x 128, 128-byte swizzle).  Grid: one CTA per tile.
constexpr int gemm_threads(int epi) { return epi == EPI_GSYM ? 512 : 128; }
template <int EPI>
__global__ void __launch_bounds__(gemm_threads(EPI), 1)
tc_gemm_kernel(const __grid_constant__ CUtensorMap mAh, const __grid_constant__ CUtensorMap mAl,
               const __grid_constant__ CUtensorMap mBh, const __grid_constant__ CUtensorMap mBl,
               int M, int N, int K, Scales sc, EpiSplit es, EpiGamma eg, int *err, uint32_t wait_limit) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // 1024-byte alignment for the swizzled tiles
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full[kStages], empty[kStages], done;
    __shared__ uint32_t tmem_base_sm;
    __shared__ int fail_sm;
    __shared__ float wn_sm[kBN], wl_sm[kBN], nn_sm[kBN], nl_sm[kBN];
    __shared__ __align__(16) float cf_sm[kBN];
    __shared__ double red[gemm_threads(EPI) / 32];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int tm, tn, bz;                              // tile and mode of the batch
    if (EPI != EPI_SPLIT) {
        const int2 t = eg.tiles[blockIdx.x];
        tm = t.x & 0xffff; bz = t.x >> 16; tn = t.y;
    } else {
        tm = es.tm0 + blockIdx.y; tn = blockIdx.x; bz = blockIdx.z;
    }
    // row coordinates of the A and B tiles: T (GEMM2's A) and Y (GEMM1's B)
    // are stacked per mode of the batch
    const int a_row = tm * kBM + (EPI != EPI_SPLIT ? bz * eg.a_rows : 0);
    const int b_row = tn * kBN + (EPI == EPI_SPLIT ? bz * es.b_rows : 0);
    const int nkb = (K + kBK - 1) / kBK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        mbar_init(&done, 1);
        fail_sm = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_base_sm)), "r"(kAcc * kBN) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_sm;

    int issued = 0;      // stages handed to TMA by the producer (drain bookkeeping)
    if (warp == 0 && lane == 0) {
        // ---- producer
        for (int kb = 0; kb < nkb; ++kb) {
            const int s = kb % kStages;
            if (kb >= kStages && !mbar_wait(&empty[s], ((kb / kStages) - 1) & 1, wait_limit)) { fail_sm = 1; break; }
            unsigned char *st = base + (size_t)s * kStageBytes;
            mbar_expect_tx(&full[s], kStageBytes);
            tma_load_2d(st, &mAh, &full[s], kb * kBK, a_row);
            tma_load_2d(st + kTileBytes, &mAl, &full[s], kb * kBK, a_row);
            tma_load_2d(st + 2 * kTileBytes, &mBh, &full[s], kb * kBK, b_row);
            tma_load_2d(st + 3 * kTileBytes, &mBl, &full[s], kb * kBK, b_row);
            ++issued;
        }
    } else if (warp == 1 && lane == 0) {
        // ---- MMA issuer
        for (int kb = 0; kb < nkb; ++kb) {
            const int s = kb % kStages;
            if (!mbar_wait(&full[s], (kb / kStages) & 1, wait_limit) || *(volatile int *)&fail_sm) { fail_sm = 1; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            unsigned char *st = base + (size_t)s * kStageBytes;
            const uint64_t ah = smem_desc(st), al = smem_desc(st + kTileBytes);
            const uint64_t bh = smem_desc(st + 2 * kTileBytes), bl = smem_desc(st + 3 * kTileBytes);
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k) {
                const uint64_t dk = (uint64_t)((k * 32) >> 4);     // 16 FP16 = 32 B along K
                const int step = kb * (kBK / 16) + k;
                const uint32_t dacc = tmem + (uint32_t)((step % (kAcc - 1)) * kBN), dlo = tmem + (kAcc - 1) * kBN;
                mma_bf16(dacc, ah + dk, bh + dk, kIdesc, step >= kAcc - 1 ? 1u : 0u);
                mma_bf16(dlo, ah + dk, bl + dk, kIdesc, step > 0 ? 1u : 0u);
                mma_bf16(dlo, al + dk, bh + dk, kIdesc, 1u);
            }
            mma_commit(&empty[s]);               // stage free once these MMAs finish
        }
        mma_commit(&done);                       // accumulator complete
    } else if (EPI == EPI_SPLIT && warp >= 2) {
        // what takes T's columns to the mode's y
        const int y = sc.y(es.mu0 + bz);
        for (int x = threadIdx.x - 64; x < kBN; x += 64) {
            const int c = tn * kBN + x;
            cf_sm[x] = c < N ? ldexpf(1.0f, __ldg(es.yk + (size_t)bz * (N / 3) + c / 3) - y) : 0.0f;
        }
    }
    __syncwarp();
    const int row = (warp & 3) * 32 + lane;      // accumulator lane = tile row
    const int m = tm * kBM + row;
    const int hm = EPI == EPI_SPLIT && m < M ? __ldg(sc.h + m) : 0;
    // ---- epilogue: wait for the accumulator (bounded)
    bool ok = mbar_wait(&done, 0, wait_limit);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!ok || *(volatile int *)&fail_sm) {
        ok = false;
        if (threadIdx.x == 0) atomicOr(err, 1);
    }
    const int quad = warp & 3;                   // the 32 lanes a warp may read
    const uint32_t taddr = tmem + ((uint32_t)(quad * 32) << 16);
    if (EPI == EPI_SPLIT) {
        // whole tile: rows and columns past M, N hold exact zeros (their A rows
        // / B rows are zero padding) and the planes are allocated to the padded
        // size (ld a multiple of 128).  The lanes of a warp hold consecutive
        // rows, so each lane pair writes two whole 64-byte row segments per
        // chunk with 32-byte stores (st_rowpair_v8).
        __syncthreads();                         // (cf_sm)
        const bool okw = __all_sync(0xffffffffu, ok);
        const float tsc = ldexpf(1.0f, kTBits - hm - sc.hR - kEBits - kYBits);
        const size_t orow = (size_t)bz * es.b_rows + m;
        char *ph = reinterpret_cast<char *>(es.hi + orow * es.ld + tn * kBN);
        char *pl = reinterpret_cast<char *>(es.lo + orow * es.ld + tn * kBN);
        const size_t rs = sizeof(__half) * (size_t)es.ld;
#pragma unroll 1
        for (int c0 = 0; c0 < kBN; c0 += 32) {
            float v[32];
            tmem_ld_sum(taddr + c0, v);
            if (!okw) continue;
            uint32_t hw[16], lw[16];
#pragma unroll
            for (int x = 0; x < 16; ++x) {
                const float2 s = __fmul2_rn(*reinterpret_cast<const float2 *>(cf_sm + c0 + 2 * x), make_float2(tsc, tsc));
                const float2 u = __fmul2_rn(make_float2(v[2 * x], v[2 * x + 1]), s);
                const __half2 h = __floats2half2_rn(u.x, u.y);
                const __half2 l = __floats2half2_rn(u.x - __low2float(h), u.y - __high2float(h));
                hw[x] = *reinterpret_cast<const uint32_t *>(&h);
                lw[x] = *reinterpret_cast<const uint32_t *>(&l);
            }
            st_rowpair_v8(ph + 2 * c0, rs, hw, lane & 1);
            st_rowpair_v8(pl + 2 * c0, rs, lw, lane & 1);
        }
    } else if (EPI == EPI_GSYM) {
        // Phi3 symmetric under every permutation: mode mu of the batch, rows m >= mu
        // and columns n >= m stand for all orders of {mu, m, n}.  The three modes'
        // sums share |phi|^2 / (w_mu w_m w_n) and the three energy differences
        //   s3 = mu + m - n,  s2 = mu - m + n,  s1 = -(mu - m - n);
        // mode m's go to rowp, mode n's to colp (FP64 across tiles).  With every
        // frequency above two windows, differences inside the window are exact but
        // for their last rounding, so that one set serves the three positions;
        // below that each position forms its own (pair_terms).
        constexpr int kCols = kBN / 4;                   // columns of a warp
        __shared__ float cs_sm[4][kBN], rs_sm[4][kBM];
        const int tc = threadIdx.x & (kBN - 1), nc = tn * kBN + tc;
        const F2 wcol = nc < N ? f2_of(eg.omega[nc]) : F2{0.f, 0.f};
        if (threadIdx.x < kBN) {
            const F2 ncol = nc < N ? f2_of(eg.occ[nc]) : F2{0.f, 0.f};
            wn_sm[tc] = wcol.h; wl_sm[tc] = wcol.l;
            nn_sm[tc] = ncol.h; nl_sm[tc] = ncol.l;
            cf_sm[tc] = nc < N ? sc.col(nc) : 0.0f;
        }
        const float cut = (float)eg.cut, s2i = (float)eg.sig2inv;
        const int mu = eg.mu0 + bz;
        const float rf = m < M ? sc.row(m, mu) : 0.0f;
        const F2 wmu = f2_of(eg.omega[mu]), nmu = f2_of(eg.occ[mu]);
        const F2 w1p = m < M ? f2_of(eg.omega[m]) : F2{0.f, 0.f};
        const F2 n1p = m < M ? f2_of(eg.occ[m]) : F2{0.f, 0.f};
        const float w1 = w1p.h, n1 = n1p.h, two = 2.01f * cut;
        const bool fast = __syncthreads_and((!(w1 > 0.0f) || w1 >= two) && (!(wcol.h > 0.0f) || wcol.h >= two)) &&
                          wmu.h >= two;                // (the columns are in shared memory, too)
        const F2 wsum = f2_add(wmu, w1p), wdif = f2_add(wmu, f2_neg(w1p));
        const float dmu = f2_diff(nmu, n1p);
        const bool live = w1 > 0.0f && m >= mu;
        const int tmu = mu / kBM;
        float acc1 = 0.0f, acc2 = 0.0f;
        int cnt = 0;
        const int cq = warp >> 2;
#pragma unroll 1
        for (int c0 = cq * kCols; c0 < (cq + 1) * kCols; c0 += 16) {
            float v[16];
            tmem_ld_sum16(taddr + c0, v);
            bool any = false;
#pragma unroll
            for (int x = 0; x < 16; ++x) {
                const float f = v[x] * rf * cf_sm[c0 + x];
                v[x] = 0.0f;
                const F2 w2p{wn_sm[c0 + x], wl_sm[c0 + x]};
                const float w2 = w2p.h;
                const int n = tn * kBN + c0 + x;
                const float s3 = f2_diff(wsum, w2p), s1 = f2_diff(wdif, w2p), s2 = f2_diff(wdif, f2_neg(w2p));
                if (!live || n < m || !(w2 > 0.0f)) continue;
                const F2 n2p{nn_sm[c0 + x], nl_sm[c0 + x]};
                const float n2 = n2p.h;
                float g1, g2, g3;
                if (fast) {
                    const bool h3 = fabsf(s3) < cut, h1 = fabsf(s1) < cut, h2 = fabsf(s2) < cut;
                    if (!(h3 || h1 || h2)) continue;
                    const float G3 = h3 ? delta_shape(s3, eg.shape, s2i) : 0.0f;
                    const float G1 = h1 ? delta_shape(s1, eg.shape, s2i) : 0.0f;
                    const float G2 = h2 ? delta_shape(s2, eg.shape, s2i) : 0.0f;
                    g1 = f2_diff(n1p, n2p) * (G3 - G2) + (m == n ? 0.5f : 1.0f) * (1.0f + n1 + n2) * G1;
                    g2 = f2_diff(nmu, n2p) * (G3 - G1) + (1.0f + nmu.h + n2) * G2;
                    g3 = dmu * (G2 - G1) + (m == mu ? 0.5f : 1.0f) * (1.0f + nmu.h + n1) * G3;
                    const int h31 = h3 || h1, h21 = h2 || h1, h32 = h3 || h2;
                    cnt += h31 + (m < n ? h21 : 0);                      // (mu; m, n)
                    if (m > mu) cnt += h32 + h21;                        // (m; mu, n)
                    if (m < n) cnt += h32 + (m > mu ? h31 : 0);          // (n; mu, m)
                } else {
                    int h = 0;
                    g1 = pair_terms(wmu, w1p, w2p, n1p, n2p, m == n, tm == tn, cut, eg.shape, s2i, h);
                    g2 = g3 = 0.0f;
                    if (m > mu) g2 = pair_terms(w1p, wmu, w2p, nmu, n2p, false, tmu == tn, cut, eg.shape, s2i, h);
                    if (m < n) g3 = pair_terms(w2p, wmu, w1p, nmu, n1p, m == mu, tmu == tm, cut, eg.shape, s2i, h);
                    if (!h) continue;
                    cnt += h;
                }
                any = true;
                const float c = f * f / (w1 * w2);
                acc1 += c * g1;
                if (m > mu) acc2 += c * g2;
                if (m < n) v[x] = c * g3;
            }
            if (__any_sync(0xffffffffu, any)) {
                const float s = lane_sums16(v);
                if (!(lane & 1)) cs_sm[quad][c0 + (lane >> 1)] = s;
            } else if (lane < 16) {
                cs_sm[quad][c0 + lane] = 0.0f;
            }
        }
        double accd = (double)acc1;
        unsigned long long cn = (unsigned long long)cnt;
        for (int o = 16; o > 0; o >>= 1) {
            accd += __shfl_xor_sync(0xffffffffu, accd, o);
            cn += __shfl_xor_sync(0xffffffffu, cn, o);
        }
        if (lane == 0) red[warp] = accd;
        if (lane == 0 && cn && ok) atomicAdd(eg.allowed, cn);
        rs_sm[cq][row] = acc2;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
            eg.partial[blockIdx.x] = ok ? s : 0.0;
        }
        // the other modes' sums, with their own frequency in place of mu's below the line
        const double iw = 1.0 / (double)wmu.h;
        const size_t o = (size_t)blockIdx.x * kBM;
        auto sum4 = [&](const float (&v)[4][kBM], int x) {
            return ((double)v[0][x] + (double)v[1][x]) + ((double)v[2][x] + (double)v[3][x]);
        };
        if (warp < 4) eg.rowp[o + row] = ok ? sum4(rs_sm, row) * ((double)w1 * iw) : 0.0;
        else if (warp < 8) eg.colp[o + tc] = ok ? sum4(cs_sm, tc) * ((double)wcol.h * iw) : 0.0;
    } else {
        // delta weights in FP32 (window test first; the FP64 unit is slow),
        // the energy and occupation differences from FP32 pairs (wdiff.cuh)
        for (int x = threadIdx.x; x < kBN; x += blockDim.x) {
            const int n = tn * kBN + x;
            const F2 wv = n < N ? f2_of(eg.omega[n]) : F2{0.f, 0.f};
            const F2 nv = n < N ? f2_of(eg.occ[n]) : F2{0.f, 0.f};
            wn_sm[x] = wv.h; wl_sm[x] = wv.l;
            nn_sm[x] = nv.h; nl_sm[x] = nv.l;
            cf_sm[x] = n < N ? sc.col(n) : 0.0f;
        }
        __syncthreads();
        const float cut = (float)eg.cut, s2i = (float)eg.sig2inv;
        const F2 wmu = f2_of(eg.omega[eg.mu0 + bz]);
        const float rf = m < M ? sc.row(m, eg.mu0 + bz) : 0.0f;
        const F2 w1p = m < M ? f2_of(eg.omega[m]) : F2{0.f, 0.f};
        const F2 n1p = m < M ? f2_of(eg.occ[m]) : F2{0.f, 0.f};
        const float w1 = w1p.h, n1 = n1p.h;
        const F2 wsum = f2_add(wmu, w1p), wdif = f2_add(wmu, f2_neg(w1p));
        const bool upper = eg.symmetric && (tn > tm);
        float acc = 0.0f;
        unsigned long long cnt = 0;
#pragma unroll 1
        for (int c0 = 0; c0 < kBN; c0 += 32) {
            float v[32];
            tmem_ld_sum(taddr + c0, v);
            if (!(w1 > 0.0f)) continue;
#pragma unroll 4
            for (int x = 0; x < 32; ++x) {
                const F2 w2p{wn_sm[c0 + x], wl_sm[c0 + x]};
                const float w2 = w2p.h;
                // w + w' - w'', w - w' - w'' and (symmetric half) w + w'' - w'
                const float dp = f2_diff(wsum, w2p), dm = f2_diff(wdif, w2p), dp2 = f2_diff(wdif, f2_neg(w2p));
                const bool hp = fabsf(dp) < cut, hm = fabsf(dm) < cut;
                const bool hp2 = upper && fabsf(dp2) < cut;
                if (!(w2 > 0.0f) || !(hp || hm || hp2)) continue;
                const F2 n2p{nn_sm[c0 + x], nl_sm[c0 + x]};
                const float n2 = n2p.h;
                const float dn = f2_diff(n1p, n2p);
                float g = 0.0f;
                if (hp) g += dn * delta_shape(dp, eg.shape, s2i);
                if (hm) g += (upper ? 1.0f : 0.5f) * (1.0f + n1 + n2) * delta_shape(dm, eg.shape, s2i);
                if (hp2) g -= dn * delta_shape(dp2, eg.shape, s2i);
                const float f = v[x] * rf * cf_sm[c0 + x];
                acc += f * f * g / (w1 * w2);
                cnt += (unsigned long long)(hp || hm) + (unsigned long long)(upper && (hp2 || hm));
            }
        }
        double accd = (double)acc;
        for (int o = 16; o > 0; o >>= 1) {
            accd += __shfl_xor_sync(0xffffffffu, accd, o);
            cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        }
        if (lane == 0) red[warp] = accd;
        if (lane == 0 && cnt && ok) atomicAdd(eg.allowed, cnt);
        __syncthreads();
        if (threadIdx.x == 0) eg.partial[blockIdx.x] = ok ? red[0] + red[1] + red[2] + red[3] : 0.0;
    }
    // ---- teardown: let in-flight TMA/MMA work finish before freeing TMEM
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if ((*(volatile int *)&fail_sm || !ok) && threadIdx.x == 0) {
        // drain: the latest load of each stage completes its transaction, and
        // every MMA the issuer committed has finished (bounded, full limit)
        for (int s = 0; s < kStages; ++s) {
            int last = -1;
            for (int kb = s; kb < issued; kb += kStages) last = kb;
            if (last >= 0) mbar_wait(&full[s], (last / kStages) & 1);
        }
        mbar_wait(&done, 0);
    }
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kAcc * kBN)
                     : "memory");
    }
}

// What the tiles leave for the modes of their rows and columns (EPI_GSYM), added in a
// fixed order: part[c][m] the sums from the tiles of modes kSumModes c .., tile by tile,
// for mode m; then gacc[m] over the c.  (One kernel per batch of modes that added to
// gacc took 13 us each: a 256-atom cell 3.42 ms, 3.15 so.)
constexpr int kSumModes = 8;
__global__ void __launch_bounds__(kBM)
gsym_part_kernel(int nb, const int *__restrict__ tile_start, const int2 *__restrict__ tiles,
                 const double *__restrict__ rowp, const double *__restrict__ colp, double *__restrict__ part) {
    const int t = blockIdx.x, x = threadIdx.x, mu0 = blockIdx.y * kSumModes, m = t * kBM + x;
    const int y1 = tile_start[min(nb, mu0 + kSumModes)];
    double s = 0.0;
#pragma unroll 4
    for (int y = tile_start[mu0]; y < y1; ++y) {
        const int2 r = __ldg(tiles + y);
        if ((r.x & 0xffff) == t) s += rowp[(size_t)y * kBM + x];
        if (r.y == t) s += colp[(size_t)y * kBM + x];
    }
    if (m < nb) part[(size_t)blockIdx.y * nb + m] = s;
}
__global__ void gsym_sums_kernel(int nb, int n_part, const double *__restrict__ part, double *__restrict__ gacc) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= nb) return;
    double s = 0.0;
#pragma unroll 8
    for (int c = 0; c < n_part; ++c) s += part[(size_t)c * nb + m];
    gacc[m] = s;
}

// Bits of the largest |Phi3| (FP32) of the blocks of each atom, in s.  A warp per (j, k)
// group, a lane per block.
__global__ void __launch_bounds__(256)
atom_strength_kernel(int n_groups, const int *__restrict__ group_start, const int *__restrict__ group_jk,
                     const int *__restrict__ blk_i, const float2 *__restrict__ fc3, unsigned *s) {
    const int g = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (g >= n_groups) return;                         // whole warps
    auto put = [&](int atom, unsigned v) {
        if (v > __ldcg(s + atom)) atomicMax(s + atom, v);
    };
    unsigned top = 0;
    for (int b = group_start[g] + lane; b < group_start[g + 1]; b += 32) {
        float m = 0.0f;
#pragma unroll
        for (int x = 0; x < 27; ++x) m = fmaxf(m, fabsf(__ldg(fc3 + (size_t)27 * b + x).x));
        put(__ldg(blk_i + b), __float_as_uint(m));
        top = max(top, __float_as_uint(m));
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane < 2) put(group_jk[2 * g + lane], top);
}
// Exponents of the atoms: a third of how far their Phi3 is below the largest one, so
// that Phi3 2^(-k_i - k_j - k_k) is of one size throughout.  One CTA.
__global__ void __launch_bounds__(256)
atom_scale_kernel(int n_at, const unsigned *__restrict__ s, int *__restrict__ k) {
    __shared__ unsigned top;
    if (threadIdx.x == 0) top = 0;
    __syncthreads();
    unsigned m = 0;
    for (int a = threadIdx.x; a < n_at; a += blockDim.x) m = max(m, s[a]);
    atomicMax(&top, m);
    __syncthreads();
    int x0;
    frexpf(__uint_as_float(top), &x0);
    for (int a = threadIdx.x; a < n_at; a += blockDim.x) {
        int x = -256;                                  // (no Phi3 at all: the least)
        if (s[a]) frexpf(__uint_as_float(s[a]), &x);
        k[a] = max(-30, min(0, (x - x0 - 1) / 3));
    }
}
// Exponents of each mode: |E^(m, .)| <= 2^e[m], its norm <= 2^(e[m] + h[m]).
__global__ void __launch_bounds__(128)
mode_scale_kernel(int nb, const double2 *__restrict__ eig, const int *__restrict__ k, int *__restrict__ e,
                  int *__restrict__ h) {
    __shared__ float red[2][4];
    float v = 0.0f, n2 = 0.0f;
    for (int c = threadIdx.x; c < nb; c += blockDim.x) {
        const float x = fabsf(ldexpf((float)eig[(size_t)blockIdx.x * nb + c].x, __ldg(k + c / 3)));
        v = fmaxf(v, x);
        n2 = fmaf(x, x, n2);
    }
    for (int o = 16; o > 0; o >>= 1) {
        v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        n2 += __shfl_xor_sync(0xffffffffu, n2, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = v;
        red[1][threadIdx.x >> 5] = n2;
    }
    __syncthreads();
    if (threadIdx.x) return;
    int x, y;
    frexpf(fmaxf(fmaxf(red[0][0], red[0][1]), fmaxf(red[0][2], red[0][3])), &x);
    frexpf(1.001f * sqrtf(red[1][0] + red[1][1] + red[1][2] + red[1][3]), &y);
    e[blockIdx.x] = x;
    h[blockIdx.x] = max(0, y - x);
}
// hi/lo FP16 planes of the scaled eigenvectors (padding stays zero from the caller's
// memset).
__global__ void split_kernel(int nb, const double2 *__restrict__ eig, const int *__restrict__ k,
                             const int *__restrict__ e, int ld, __half *__restrict__ hi, __half *__restrict__ lo) {
    const size_t n = (size_t)nb * nb;
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < n; x += (size_t)gridDim.x * blockDim.x) {
        const size_t r = x / nb, c = x % nb;
        const float v = (float)ldexp(eig[x].x, kEBits - __ldg(e + r) + __ldg(k + c / 3));
        const __half h = __float2half_rn(v);
        hi[r * ld + c] = h;
        lo[r * ld + c] = __float2half_rn(v - __half2float(h));
    }
}

// FP32 pairs (hi, lo) of the scaled Phi3 blocks, 27 per block.
__global__ void fc3_pair_kernel(size_t n, const double *__restrict__ src, float2 *__restrict__ out) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < n; x += (size_t)gridDim.x * blockDim.x) {
        const F2 v = f2_of(src[x]);
        out[x] = make_float2(v.h, v.l);
    }
}
// FP32 pairs of the eigenvectors with the modes contiguous: Et[d][mu], row
// length ldm (32 x 32 tiles through shared memory).
__global__ void __launch_bounds__(256)
eig_pair_kernel(int nb, const double2 *__restrict__ eig, int ldm, float2 *__restrict__ Et) {
    __shared__ float2 tile[32][33];
    const int d0 = blockIdx.x * 32, m0 = blockIdx.y * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int r = ty; r < 32; r += 8)
        if (m0 + r < nb && d0 + tx < nb) {
            const F2 v = f2_of(eig[(size_t)(m0 + r) * nb + d0 + tx].x);
            tile[r][tx] = make_float2(v.h, v.l);
        }
    __syncthreads();
    for (int r = ty; r < 32; r += 8)
        if (d0 + r < nb && m0 + tx < nb) Et[(size_t)(d0 + r) * ldm + m0 + tx] = tile[tx][r];
}

// acc += a b for FP32 pairs: the product to about 2^-46 of itself (FMA
// residual plus the cross terms), the sum by Knuth's two-sum.
__device__ __forceinline__ void pair_fma(F2 &acc, float2 a, float2 b) {
    const float p = __fmul_rn(a.x, b.x);
    float e = __fmaf_rn(a.x, b.x, -p);
    e = __fmaf_rn(a.x, b.y, e);
    e = __fmaf_rn(a.y, b.x, e);
    const float s = __fadd_rn(acc.h, p);
    const float v = __fsub_rn(s, acc.h);
    const float r = __fadd_rn(__fsub_rn(acc.h, __fsub_rn(s, v)), __fsub_rn(p, v));
    acc.h = s;
    acc.l = __fadd_rn(acc.l, __fadd_rn(r, e));
}

// The rows c = 3 k .. 3 k + 2 of Y^_mu(c, b) of modes mu0 .. mu0 + nm - 1, scaled, in
// their FP16 hi/lo planes (plane stride plane_elems); CTA = (k, MT modes).  Sums of FP32
// pairs (about 46 bits), rounded once to FP32 and, when the rows' largest element is
// known (its exponent goes to yk[mode][k], the mode's to ymax), split.  The other
// elements of the planes are zero and stay so.
//
// Bound: FP32 issue (a batch of 34 modes of 768 branches 74 us, of 22 modes 34 us; 65
// and 33 without the largest elements, which a CTA of any groups can do).  As plain FP64
// sums (one thread per output and mode, 2
// FP64 FMA per clock and SM) this build took 173 us per launch of 18 modes of a 768-mode
// cell, three times both GEMMs together; a pair FMA is 12 FP32 operations
// against the 64 that one FP64 FMA costs here.  A thread takes MT modes
// of one output, so a block's values are read once for all of them and the
// modes of an eigenvector component are contiguous.  The groups of k come longest
// first: the k_start[k].y longest -- the atoms paired with themselves hold
// one block per neighbour where the others hold two or three -- take a warp
// each, three lanes per output, or the whole CTA; the warps take the others from a
// counter.
constexpr int kYAll = 24;
constexpr int kNoRow = -100000;                        // exponent of rows without an element
template <int MT>
__global__ void __launch_bounds__(256, 6)
ybuild_rows_kernel(const int2 *__restrict__ k_start, const int4 *__restrict__ k_grp, const int *__restrict__ blk_i,
                   const float2 *__restrict__ fc3, const float2 *__restrict__ Et, int ldm, int mu0, int nm,
                   const int *__restrict__ kx, int ld, size_t plane_elems, int n_val, __half *__restrict__ hi,
                   __half *__restrict__ lo, int *__restrict__ yk, int *ymax) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *val = reinterpret_cast<float *>(smem_raw);            // [MT][n_val]
    __shared__ unsigned top_sm[8][MT];
    __shared__ float2 part_sm[8][MT][9];
    __shared__ int next;
    const int k = blockIdx.x, m0 = blockIdx.y * MT, n_m = min(MT, nm - m0);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int2 ks = k_start[k];
    const int n_g = k_start[k + 1].x - ks.x, n_w = ks.y + (9 * (n_g - ks.y) + 31) / 32;
    const int kk = __ldg(kx + k);
    if (threadIdx.x == 0) next = 0;
    __syncthreads();
    unsigned top[MT];
#pragma unroll
    for (int m = 0; m < MT; ++m) top[m] = 0;
    // sum of the blocks b0, b0 + step .. b1 - 1 of a group for output bg
    auto blocks = [&](F2(&acc)[MT], int b0, int b1, int step, int bg) {
#pragma unroll
        for (int m = 0; m < MT; ++m) acc[m] = F2{0.f, 0.f};
#pragma unroll 2
        for (int bl = b0; bl < b1; bl += step) {
            const float2 *e = Et + (size_t)(3 * __ldg(blk_i + bl)) * ldm + mu0 + m0;
            const float2 *f = fc3 + (size_t)27 * bl + bg;
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float2 v = __ldg(f + 9 * a);
#pragma unroll
                for (int m = 0; m < MT; ++m) pair_fma(acc[m], v, __ldg(e + (size_t)a * ldm + m));
            }
        }
    };
    // the three lanes of an output (lane / 9), in order, to lanes 0 .. 8
    auto lanes3 = [&](F2(&acc)[MT]) {
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            F2 p[2];
#pragma unroll
            for (int z = 0; z < 2; ++z) {
                p[z].h = __shfl_down_sync(0xffffffffu, acc[m].h, 9 * (z + 1));
                p[z].l = __shfl_down_sync(0xffffffffu, acc[m].l, 9 * (z + 1));
            }
            acc[m] = f2_add(f2_add(acc[m], p[0]), p[1]);
        }
    };
    auto put = [&](const F2 &s, int m, int e, int sh) {
        const float v = ldexpf(__fadd_rn(s.h, s.l), -sh);
        val[m * n_val + e] = v;
        top[m] = max(top[m], __float_as_uint(fabsf(v)));
    };
    F2 acc[MT];
    // groups of more than kYAll blocks by all warps, three lanes per output each
    for (int gi = 0; gi < ks.y; ++gi) {
        const int4 g = __ldg(k_grp + ks.x + gi);       // (first block, end, j)
        if (g.y - g.x <= kYAll) continue;              // uniform
        const int sh = kk + __ldg(kx + g.z);
        blocks(acc, lane < 27 ? g.x + 3 * warp + lane / 9 : g.y, g.y, 24, lane % 9);
        lanes3(acc);
        __syncthreads();                               // (part_sm has been read)
        if (lane < 9)
#pragma unroll
            for (int m = 0; m < MT; ++m) part_sm[warp][m][lane] = make_float2(acc[m].h, acc[m].l);
        __syncthreads();
        if (threadIdx.x < 9) {
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                F2 s{part_sm[0][m][threadIdx.x].x, part_sm[0][m][threadIdx.x].y};
                for (int w = 1; w < 8; ++w) s = f2_add(s, F2{part_sm[w][m][threadIdx.x].x, part_sm[w][m][threadIdx.x].y});
                put(s, m, 9 * gi + threadIdx.x, sh);
            }
        }
    }
    for (;;) {
        int w = 0;
        if (lane == 0) w = atomicAdd(&next, 1);
        w = __shfl_sync(0xffffffffu, w, 0);
        if (w >= n_w) break;
        const bool lng = w < ks.y;                     // uniform over the warp
        const int t = lng ? 0 : (w - ks.y) * 32 + lane;
        const int gi = lng ? w : ks.y + t / 9, bg = lng ? lane % 9 : t % 9;
        const bool act = gi < n_g && (!lng || lane < 27);
        const int4 g = act ? __ldg(k_grp + ks.x + gi) : make_int4(0, 0, 0, 0);
        if (lng && __shfl_sync(0xffffffffu, g.y - g.x, 0) > kYAll) continue;       // (done above)
        const int sh = kk + __ldg(kx + g.z);
        blocks(acc, g.x + (lng ? lane / 9 : 0), g.y, lng ? 3 : 1, bg);
        if (lng) lanes3(acc);
        if (act && !(lng && lane >= 9))
#pragma unroll
            for (int m = 0; m < MT; ++m) put(acc[m], m, 9 * gi + bg, sh);
    }
#pragma unroll
    for (int m = 0; m < MT; ++m) {
        const unsigned t1 = __reduce_max_sync(0xffffffffu, top[m]);
        if (lane == 0) top_sm[threadIdx.x >> 5][m] = t1;
    }
    __syncthreads();
    int ex[MT];
#pragma unroll
    for (int m = 0; m < MT; ++m) {
        unsigned t1 = 0;
        for (int w = 0; w < 8; ++w) t1 = max(t1, top_sm[w][m]);
        frexpf(__uint_as_float(t1), &ex[m]);
        if (threadIdx.x == 0 && m < n_m) {
            yk[(size_t)(m0 + m) * gridDim.x + k] = t1 ? ex[m] : kNoRow;
            if (t1) atomicMax(ymax + mu0 + m0 + m, ex[m]);
        }
    }
    for (int x = threadIdx.x; x < 9 * n_g; x += 256) {
        const int bg = x % 9;
        const size_t off = (size_t)(3 * k + bg % 3) * ld + 3 * __ldg(k_grp + ks.x + x / 9).z + bg / 3;
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            if (m >= n_m) break;
            const float s = ldexpf(val[m * n_val + x], kYBits - ex[m]);
            const __half h = __float2half_rn(s);
            const size_t o = (size_t)(m0 + m) * plane_elems + off;
            hi[o] = h;
            lo[o] = __float2half_rn(s - __half2float(h));
        }
    }
}
// Shared memory of the Y build for mt modes and at most n_val entries of a k.
size_t ybuild_smem(int mt, int n_val) { return sizeof(float) * mt * (size_t)n_val; }

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// Tensor map of an FP16 plane [rows][ld] (ld a multiple of 64), box 64 x 128.
bool make_map(CUtensorMap *map, const __half *ptr, int rows, int ld) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)ld, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)kBM};
    const cuuint32_t estr[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half *>(ptr), dims, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

constexpr size_t kSmemBytes = kStages * kStageBytes + 1024;

}  // namespace

int tc_tile(void) { return kBM; }

// Modes per launch: enough tiles of the first contraction for about two CTAs per SM,
// at most 32; twice as many, at most 64, where each triple is projected once (a mode
// has half of those tiles, and a sixth as many of the second contraction's: 768 modes
// 3.9 -> 3.3 ms).
int tc_gamma_batch(int nb, int sms, int sym3) {
    const int nt = (nb + kBM - 1) / kBM;
    const int want = (2 * std::max(sms, 1) + nt * nt - 1) / (nt * nt);
    return std::max(1, std::min({sym3 ? 2 * want : want, sym3 ? kMaxBatch : 32, nb}));
}

// Largest modes per launch the autotuner may choose (twice the default, at most 32
// or 64).
int tc_gamma_batch_max(int nb, int sms, int sym3) {
    return std::max(1, std::min({2 * tc_gamma_batch(nb, sms, sym3), sym3 ? kMaxBatch : 32, nb}));
}

// Modes per row of the transposed eigenvector pairs (the Y build reads up to
// three modes past the last one).
static int tc_ldm(int nb) { return (nb + 3 + 31) / 32 * 32; }

// Row (or column) sums of the tiles, and the parts of the modes' sums (EPI_GSYM).
static size_t tc_gsym_bytes(size_t n_tiles) { return ws_round(sizeof(double) * kBM * std::max<size_t>(n_tiles, 1)); }
static int tc_gsym_parts(int nb) { return (nb + kSumModes - 1) / kSumModes; }

// e, h and ymax of the modes, the strengths and the exponents of the atoms, those of the
// rows of Y of a batch.
static size_t tc_scale_ints(int nb, int mb_max) { return 3 * (size_t)nb + (2 + (size_t)mb_max) * ((nb + 2) / 3); }

size_t tc_gamma_scratch_bytes(int nb, int mb_max, size_t n_fc3, int sym3, size_t n_tiles) {
    const int ld = (nb + kBN - 1) / kBN * kBN;     // whole 128-column tiles per row
    const int rows = (nb + kBM - 1) / kBM * kBM;
    const size_t plane = ws_round(sizeof(__half) * (size_t)rows * ld);
    // E hi/lo, then Y hi, Y lo, T hi, T lo of every mode of a batch (the largest batch)
    // then the FP32 pairs of Phi3 and of the eigenvectors and the scales, then (Phi3 symmetric under
    // every permutation) the tiles' sums and the modes' sums
    return (2 + 4 * (size_t)mb_max) * plane + ws_round(sizeof(float2) * 27 * std::max<size_t>(n_fc3, 1)) +
           ws_round(sizeof(float2) * (size_t)nb * tc_ldm(nb)) + ws_round(sizeof(int) * tc_scale_ints(nb, mb_max)) +
           (sym3 ? 2 * tc_gsym_bytes(n_tiles) + ws_round(sizeof(double) * (size_t)nb * (1 + tc_gsym_parts(nb))) : 0);
}

// The tensor-core pipeline for one Gamma-only system (Y build, T = E Y^T-form,
// phi tiles of the delta band with the weight epilogue), gp.mb modes per
// launch (0: tc_gamma_batch), modes below mode_limit only (tuning runs).
cudaError_t launch_gamma_only_tc(const GammaPlan &gp, const GammaDev &d, const LwParams &p, void *scratch,
                                 const std::vector<int2> &tiles, const std::vector<int> &tile_start,
                                 int2 *tiles_dev, int symmetric, double *partial_tc, int *err, int sms,
                                 cudaStream_t st, int mode_limit, const double **gacc_out) {
    const int nb = p.nb;
    const int ld = (nb + kBN - 1) / kBN * kBN;     // whole 128-column tiles per row
    const int rows = (nb + kBM - 1) / kBM * kBM;
    const int mb = std::min(gp.mb > 0 ? gp.mb : tc_gamma_batch(nb, sms, gp.sym3), gp.mb_max);
    const size_t plane = ws_round(sizeof(__half) * (size_t)rows * ld);
    const size_t stack = (size_t)mb * plane;        // one operand plane for every mode of a batch
    char *b = static_cast<char *>(scratch);
    __half *Eh = reinterpret_cast<__half *>(b);
    __half *El = reinterpret_cast<__half *>(b + plane);
    auto S = [&](int i) { return reinterpret_cast<__half *>(b + 2 * plane + i * stack); };
    __half *Yh = S(0), *Yl = S(1), *Th = S(2), *Tl = S(3);
    cudaError_t e = cudaMemsetAsync(b, 0, 2 * plane + 2 * stack, st);       // E and Y
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(err, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
    const int ldm = tc_ldm(nb);
    char *pairs = b + (2 + 4 * (size_t)gp.mb_max) * plane;
    float2 *fc3p = reinterpret_cast<float2 *>(pairs);
    float2 *Et = reinterpret_cast<float2 *>(pairs + ws_round(sizeof(float2) * 27 * std::max<size_t>(gp.n_fc3, 1)));
    char *sums = reinterpret_cast<char *>(Et) + ws_round(sizeof(float2) * (size_t)nb * ldm);
    char *gsums = sums + ws_round(sizeof(int) * tc_scale_ints(nb, gp.mb_max));
    double *rowp = nullptr, *colp = nullptr, *gacc = nullptr;
    // tile_start follows the tiles (same allocation)
    int *ts = reinterpret_cast<int *>(tiles_dev + std::max<size_t>(tiles.size(), 1));
    e = cudaMemcpyAsync(ts, tile_start.data(), sizeof(int) * (nb + 1), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    if (gp.sym3) {
        rowp = reinterpret_cast<double *>(gsums);
        colp = reinterpret_cast<double *>(gsums + tc_gsym_bytes(tiles.size()));
        gacc = reinterpret_cast<double *>(gsums + 2 * tc_gsym_bytes(tiles.size()));
    }
    if (gacc_out) *gacc_out = gacc;
    const size_t nf = 27 * gp.n_fc3;
    if (nf) fc3_pair_kernel<<<counted((unsigned)std::min<size_t>((nf + 255) / 256, 4096)), 256, 0, st>>>(nf, d.fc3, fc3p);
    eig_pair_kernel<<<counted(dim3((nb + 31) / 32, (nb + 31) / 32)), 256, 0, st>>>(
        nb, reinterpret_cast<const double2 *>(d.eig), ldm, Et);
    const int n_at = nb / 3;
    int *em = reinterpret_cast<int *>(sums), *hm = em + nb, *ymax = hm + nb, *kx = ymax + nb;
    unsigned *strength = reinterpret_cast<unsigned *>(kx + n_at);
    int *yk = reinterpret_cast<int *>(strength + n_at);
    e = cudaMemsetAsync(ymax, 0x80, sizeof(int) * (size_t)nb, st);          // (no element yet)
    if (e == cudaSuccess) e = cudaMemsetAsync(strength, 0, sizeof(int) * (size_t)n_at, st);
    if (e != cudaSuccess) return e;
    if (gp.n_groups)
        atom_strength_kernel<<<counted((gp.n_groups + 7) / 8), 256, 0, st>>>(gp.n_groups, d.group_start, d.group_jk,
                                                                            d.blk_i, fc3p, strength);
    atom_scale_kernel<<<counted(1), 256, 0, st>>>(n_at, strength, kx);
    mode_scale_kernel<<<counted(nb), 128, 0, st>>>(nb, reinterpret_cast<const double2 *>(d.eig), kx, em, hm);
    int hR = 0;
    while ((1LL << (2 * hR)) < gp.row_entries) ++hR;
    const Scales sc{em, hm, ymax, hR};
    const int n_val = 3 * gp.row_entries;          // entries of the three rows of one k
    split_kernel<<<counted(4096), 256, 0, st>>>(nb, reinterpret_cast<const double2 *>(d.eig), kx, em, ld, Eh, El);
    // the planes of one stack are contiguous: plane_elems = plane / 2 elements apart
    const size_t plane_elems = plane / sizeof(__half);
    const int stack_rows = (int)((size_t)mb * plane_elems / ld);
    CUtensorMap mEh, mEl, mYh, mYl, mTh, mTl;
    if (plane_elems % ld != 0 || !make_map(&mEh, Eh, rows, ld) || !make_map(&mEl, El, rows, ld) ||
        !make_map(&mYh, Yh, stack_rows, ld) || !make_map(&mYl, Yl, stack_rows, ld) ||
        !make_map(&mTh, Th, stack_rows, ld) || !make_map(&mTl, Tl, stack_rows, ld))
        return cudaErrorInvalidValue;
    const int prow = (int)(plane_elems / ld);      // rows from one plane to the next (>= rows)
    auto k1 = tc_gemm_kernel<EPI_SPLIT>;
    auto k2 = gp.sym3 ? tc_gemm_kernel<EPI_GSYM> : tc_gemm_kernel<EPI_GAMMA>;
    e = cudaFuncSetAttribute(k1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    if (e != cudaSuccess) return e;
    // tile records carry the mode's place in its batch: (tm | b << 16, tn)
    std::vector<int2> enc(std::max<size_t>(tiles.size(), 1), make_int2(0, 0));
    for (int mu = 0; mu < nb; ++mu)
        for (int t = tile_start[mu]; t < tile_start[mu + 1]; ++t)
            enc[t] = make_int2(tiles[t].x | ((mu % mb) << 16), tiles[t].y);
    // (a copy from pageable memory returns once the host buffer is staged)
    e = cudaMemcpyAsync(tiles_dev, enc.data(), sizeof(int2) * enc.size(), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    const int nt = rows / kBM;
    const double sig2inv = delta_param(p.shape, p.sigma_w);
    const int mu_end = std::min(nb, mode_limit);
    for (int mu0 = 0; mu0 < mu_end; mu0 += mb) {
        const int nm = std::min(mb, nb - mu0);
        const int t0 = tile_start[mu0], t1 = tile_start[mu0 + nm];
        if (t1 == t0) continue;                     // no delta-band tile (masked modes)
        auto ybuild = [&](auto kern, int mt) {
            const size_t smem = ybuild_smem(mt, n_val);
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e == cudaSuccess)
                kern<<<counted(dim3(n_at, (nm + mt - 1) / mt)), 256, smem, st>>>(d.k_start, d.k_grp, d.blk_i, fc3p, Et, ldm,
                                                                               mu0, nm, kx, ld, plane_elems, n_val, Yh,
                                                                               Yl, yk, ymax);
        };
        // modes per CTA: 4, or 3 where that leaves fewer of them unused, and fewer where
        // their entries do not fit
        int mt = nm < 3 ? nm : (nm + 2) / 3 * 3 < (nm + 3) / 4 * 4 ? 3 : 4;
        while (mt > 1 && ybuild_smem(mt, n_val) > (size_t)96 << 10) --mt;
        if (mt == 1) ybuild(ybuild_rows_kernel<1>, 1);
        else if (mt == 2) ybuild(ybuild_rows_kernel<2>, 2);
        else if (mt == 3) ybuild(ybuild_rows_kernel<3>, 3);
        else ybuild(ybuild_rows_kernel<4>, 4);
        if (e != cudaSuccess) return e;
        // (with sym3 the tiles of a mode start at its own row tile)
        const int tm0 = gp.sym3 ? mu0 / kBM : 0;
        EpiSplit es{Th, Tl, ld, prow, tm0, mu0, yk};
        EpiGamma eg{};
        ProfMark p1(p.prof, KALD_PROF_TC_GEMM1, st);
        k1<<<counted(dim3(nt, nt - tm0, nm)), 128, kSmemBytes, st>>>(mEh, mEl, mYh, mYl, nb, nb, ld, sc, es, eg, err,
                                                               p.wait_limit);
        p1.end();
        EpiGamma eg2{d.omega, d.occ, mu0, prow, sig2inv, p.cut_w, p.shape, partial_tc + t0, d.allowed,
                     tiles_dev + t0, symmetric, rowp ? rowp + (size_t)t0 * kBM : nullptr,
                     colp ? colp + (size_t)t0 * kBM : nullptr};
        EpiSplit es0{nullptr, nullptr, 0, 0, 0, 0, nullptr};
        ProfMark p2(p.prof, KALD_PROF_TC_GEMM2, st);
        k2<<<counted(t1 - t0), gp.sym3 ? gemm_threads(EPI_GSYM) : 128, kSmemBytes, st>>>(mTh, mTl, mEh, mEl, nb, nb, ld, sc, es0, eg2, err, p.wait_limit);
        p2.end();
    }
    if (gp.sym3 && gacc_out) {
        double *part = gacc + nb;
        gsym_part_kernel<<<counted(dim3(nt, tc_gsym_parts(nb))), kBM, 0, st>>>(nb, ts, tiles_dev, rowp, colp, part);
        gsym_sums_kernel<<<counted((nb + 63) / 64), 64, 0, st>>>(nb, tc_gsym_parts(nb), part, gacc);
    }
    return cudaGetLastError();
}

}  // namespace kald
