// Three-phonon linewidths on the GPU (paper, section "Boltzman Transport
// Equation": Eq. projection_plus, gamma_operators, phase_space,
// delta_deconstructed, and Gamma^0).
//
// For every momentum-conserving triplet (q s, q' s', q'' s''), q'' = q + q',
//   phi(s, s', s'') = sum_{b c} eps'_b(s') Y_s(b, c) conj(eps''_c(s''))
//   Y_s(b, c) = sum_{blocks (i; j Rj; k Rk) -> (b, c)} sum_a Phi3~_{a b c}
//                 eps_{ia}(q s) chi(q', Rj) conj(chi(q'', Rk))
// with Phi3~ = Phi3 / sqrt(mi mj mk), eps = eta (mass scaling lives in Phi3~)
// and chi(q, R) = exp(-i q.R).  The first (home) index is contracted on the
// sparse blocks, the two others are dense complex contractions:
//   T'(s', c) = sum_b eps'(b, s') Y(b, c),   phi(s', s'') = sum_c T'(s', c) conj(eps''(c, s'')).
// The epilogue applies both processes to the one projection (the - process of
// (q, -q') has the same |phi|^2 up to gauge):
//   acc_s += |phi|^2 / (w' w'') [ (n' - n'') G(w + w' - w'') + 1/2 (1 + n' + n'') G(w - w' - w'') ]
// where G(d) = exp(-d^2 / 2 sigma^2) for |d| < n_sigma sigma; the constant
// hbar pi / (8 N_k) (eV/A^2 amu -> ps^-2)^3 / (sqrt(2 pi) sigma w) is applied
// per mode at the end in FP64.
//
// Work: a persistent grid pulls items -- (q, chunk of q'), or one orbit of
// momentum triples (OrbitPlan) -- from a device counter (atomicAdd only; nothing
// waits).  Each item writes its own FP64 partial sums, which a second kernel adds
// in a fixed order, so results do not depend on the schedule.

#include <algorithm>
#include <array>
#include <type_traits>
#include <vector>

#include "kald_internal.h"
#include "wdiff.cuh"

namespace kald {
namespace {

template <typename R> struct C2;
template <> struct C2<float> { using T = float2; };
template <> struct C2<double> { using T = double2; };

template <typename T2> __device__ __forceinline__ T2 mk(double x, double y);
template <> __device__ __forceinline__ float2 mk<float2>(double x, double y) {
    return make_float2((float)x, (float)y);
}
template <> __device__ __forceinline__ double2 mk<double2>(double x, double y) {
    return make_double2(x, y);
}

constexpr int kThreads = 512;          // most threads of a CTA
constexpr int kTR = 6;                 // register tile: kTR rows (s') ...
constexpr int kTC = 3;                 // ... by kTC columns (complex)

// ---------------------------------------------------------------- prep kernels
__global__ void mode_prep_kernel(int n, const double *__restrict__ nu, double omega_min_w,
                                 double T, int classical, double *__restrict__ omega,
                                 double *__restrict__ occ) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n) return;
    const double w = kTwoPi * nu[x];
    const bool ok = isfinite(w) && (w > omega_min_w);
    double n_b = 0.0;
    if (ok) {
        const double xx = kHbarEvPs * w / (kKbEvK * T);
        n_b = classical ? 1.0 / xx : 1.0 / expm1(fmin(xx, 700.0));
    }
    omega[x] = ok ? w : 0.0;
    occ[x] = n_b;
}

// FP32 pairs (hi, lo) of omega and n for the compensated epilogue differences.
__global__ void wn_pair_kernel(int n, const double *__restrict__ omega, const double *__restrict__ occ,
                               float4 *__restrict__ out) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= n) return;
    const F2 w = f2_of(omega[x]), o = f2_of(occ[x]);
    out[x] = make_float4(w.h, w.l, o.h, o.l);
}

template <typename R2>
__global__ void chi_kernel(int nq, int n_rep, const double *__restrict__ qcart,
                           const double *__restrict__ rep, R2 *__restrict__ chi) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= nq * n_rep) return;
    const int q = x / n_rep, r = x % n_rep;
    double s, c;
    sincos(qcart[3 * q] * rep[3 * r] + qcart[3 * q + 1] * rep[3 * r + 1] +
               qcart[3 * q + 2] * rep[3 * r + 2], &s, &c);
    chi[x] = mk<R2>(c, -s);                    // exp(-i q.R)
}

// epsT[q][b][s] = eta[q][s][b] in the working precision
template <typename R2>
__global__ void eps_transpose_kernel(int nq, int nb, const double2 *__restrict__ eig,
                                     R2 *__restrict__ epsT) {
    const size_t n = (size_t)nq * nb * nb;
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < n;
         x += (size_t)gridDim.x * blockDim.x) {
        const size_t q = x / ((size_t)nb * nb);
        const int r = (int)(x % ((size_t)nb * nb));
        const int b = r / nb, s = r % nb;
        const double2 v = eig[(q * nb + s) * nb + b];
        epsT[x] = mk<R2>(v.x, v.y);
    }
}

// -------------------------------------------------------------- main kernel
template <typename R2>
__device__ __forceinline__ void cfma(R2 &acc, const R2 a, const R2 b) {   // acc += a b
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.y = fma(a.y, b.x, acc.y);
}
template <typename R2>
__device__ __forceinline__ R2 cmul(const R2 a, const R2 b) {
    R2 r;
    r.x = a.x * b.x - a.y * b.y;
    r.y = a.x * b.y + a.y * b.x;
    return r;
}

// Phase sums of one q-point, [nq][slots][27] per class: the blocks of each
// (j, k, i) whose phase depends on q' alone (class 0: Rk = 0, chi(q', Rj)), on
// q'' alone (class 1: Rj = 0, conj chi(q'', Rk)) or on q alone (class 2:
// Rj = Rk, conj chi(q, R)); see LwTerms.  One thread per value, sums in FP64.
template <typename R>
__global__ void lw_tables_kernel(int nq, int n_rep, LwTerms t, const int4 *__restrict__ blkinfo,
                                 const R *__restrict__ fc3, const typename C2<R>::T *__restrict__ chi) {
    using R2 = typename C2<R>::T;
    for (int cls = 0; cls < 3; ++cls) {
        const size_t per = (size_t)t.n_slot[cls] * 27, n = per * nq;
        R2 *out = static_cast<R2 *>(t.tab[cls]);
        for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < n; x += (size_t)gridDim.x * blockDim.x) {
            const size_t q = x / per, e = x - q * per;
            const int slot = t.slot0[cls] + (int)(e / 27), v = (int)(e % 27);
            double re = 0.0, im = 0.0;
            for (int y = t.slot_start[slot]; y < t.slot_start[slot + 1]; ++y) {
                const int b = t.slot_blk[y];
                const int4 bi = __ldg(blkinfo + b);
                const R2 z = chi[q * n_rep + (cls == 1 ? bi.z : bi.y)];
                const double f = (double)fc3[(size_t)28 * b + v];
                re += f * (double)z.x;
                im += cls == 0 ? f * (double)z.y : -f * (double)z.y;
            }
            out[x] = mk<R2>(re, im);
        }
    }
}

// One thread per mode, CTA = (row, group set apart).
template <typename R>
__global__ void __launch_bounds__(kMaxNbSmall)
lw_same_kernel(int nb, LwTerms t, const int2 *__restrict__ rows, const typename C2<R>::T *__restrict__ epsT_all) {
    using R2 = typename C2<R>::T;
    const int c = blockIdx.y, q = rows ? rows[blockIdx.x].x : blockIdx.x, s = threadIdx.x;
    if (s >= nb) return;
    const R2 *eps = epsT_all + (size_t)q * nb * nb + s;
    const R2 *tab = static_cast<const R2 *>(t.tab[2]) + (size_t)q * t.n_slot[2] * 27;
    R2 acc[9];
#pragma unroll
    for (int e = 0; e < 9; ++e) acc[e] = mk<R2>(0.0, 0.0);
    for (int y = t.cterm_start[c]; y < t.cterm_start[c + 1]; ++y) {
        const int2 tm = __ldg(t.cterm + y);                    // (i, slot)
#pragma unroll
        for (int al = 0; al < 3; ++al) {
            const R2 u = eps[(size_t)(3 * tm.x + al) * nb];
#pragma unroll
            for (int e = 0; e < 9; ++e) cfma(acc[e], u, tab[(size_t)27 * tm.y + 9 * al + e]);
        }
    }
    R2 *yc = static_cast<R2 *>(t.yc) + ((size_t)q * t.n_cg + c) * 9 * nb + s;
#pragma unroll
    for (int e = 0; e < 9; ++e) yc[(size_t)e * nb] = acc[e];
}

// out [n_pairs][per]: the n_sblk mode blocks' position sums of a pair added in order.
__global__ void lw_block_sums_kernel(size_t n, int per, int n_sblk, const double *__restrict__ out3,
                                     double *__restrict__ out) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < n; x += (size_t)gridDim.x * blockDim.x) {
        const size_t pair = x / per, e = x - pair * per;
        double v = 0.0;
        for (int b = 0; b < n_sblk; ++b) v += out3[(pair * n_sblk + b) * per + e];
        out[x] = v;
    }
}

// Shared memory of a CTA of sb modes and nthr threads (R2 = complex of the
// working precision; P = nb rounded up to a multiple of kTR, Q = P + 1):
//   Y    [sb][P][Q]  Y(b, c) at b*P + c, then T'^T(c, s') at c*Q + s' (odd
//                    pitch: the transposed store walks distinct banks)
//   EpT, EppT [P][P] eps(q')^T and conj(eps(q''))^T (only when they fit: oper)
//   es   [sb][P]     eps(q, s) columns
//   wp, np_, wpp, npp [P]     omega and n of q' / q'' (R; the hi parts for FP32)
//   wpl, npl, wppl, nppl [P]  lo parts of the FP32 pairs (wdiff.cuh)
//   red  [3][nb] double  the item's sums per mode (of each position of an orbit)
//   psum [nthr], prow [nthr][6], pcol [nthr][3] double  sums of the listed tiles
//                    (rows and columns: orbits only)
//   tiles [nthr] int the (mode, tile) pairs the delta windows reach
template <typename R>
__host__ __device__ inline size_t lw_smem_bytes(int nb, int sb, int nthr, bool oper, bool orbit) {
    const size_t P = (size_t)((nb + kTR - 1) / kTR) * kTR;
    size_t b = 2 * sizeof(R) * (sb * P * (P + 1) + (oper ? 2 * P * P : 0) + sb * P);
    b += sizeof(R) * 8 * P;
    b = (b + 15) & ~size_t(15);
    b += sizeof(double) * (3 * (size_t)nb + (size_t)nthr * (orbit ? 10 : 1));
    b += sizeof(int) * (size_t)nthr;
    return b + 32;
}

// Bound: FMA issue (FP64: 2 per clock and SM).  Y_s(b, c) is summed from the
// tables of LwTerms, one thread per (mode, atom pair); both contractions run in
// 6 x 3 register tiles, sb modes side by side so that small cells fill the CTA;
// GEMM2 only on the tiles that a window reaches.  ORBIT: one projection per
// orbit of momentum triples, three weights per element, the sums of all three
// positions into out3.  Eight atoms (24 branches), 4^3 mesh, FP64: 74 ms with
// every block phased for every mode, one mode per CTA and one q-point of each
// pair {q, -q}; 3.3 ms now.
template <typename R, bool OPER_SMEM, bool ORBIT>
__global__ void __launch_bounds__(kThreads, 1)
lw_main_kernel(LwParams p, LwDev d, LwTerms t, int SB, const R *__restrict__ fc3,
               const typename C2<R>::T *__restrict__ epsT_all, const typename C2<R>::T *__restrict__ chi_all) {
    using R2 = typename C2<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nb = p.nb, nthr = blockDim.x;
    const int P = ((nb + kTR - 1) / kTR) * kTR;
    const int Q = P + 1, na = nb / 3, nap = P / 3;
    const int tcols = P / kTC;                       // column tiles
    const int n_tiles = (P / kTR) * tcols;
    const size_t ysz = (size_t)P * Q;
    R2 *Y = reinterpret_cast<R2 *>(smem_raw);
    R2 *EpT = Y + SB * ysz;
    R2 *EppT = OPER_SMEM ? EpT + (size_t)P * P : EpT;
    R2 *es = OPER_SMEM ? EppT + (size_t)P * P : EpT;
    R *wp = reinterpret_cast<R *>(es + SB * P);
    R *np_ = wp + P;
    R *wpp = np_ + P;
    R *npp = wpp + P;
    R *wpl = npp + P;
    R *npl = wpl + P;
    R *wppl = npl + P;
    R *nppl = wppl + P;
    constexpr bool kPair = std::is_same<R, float>::value;
    double *red = reinterpret_cast<double *>((reinterpret_cast<uintptr_t>(nppl + P) + 15) & ~uintptr_t(15));
    double *psum = red + 3 * nb;
    double *prow = psum + nthr, *pcol = prow + 6 * (size_t)(ORBIT ? nthr : 0);
    int *tiles = reinterpret_cast<int *>(pcol + 3 * (size_t)(ORBIT ? nthr : 0));
    __shared__ int item_sm, n_act_sm, warp_cnt[kThreads / 32];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = nthr >> 5;
    const R sig2inv = (R)delta_param(p.shape, p.sigma_w);   // the delta shape's parameter
    const R cut = (R)p.cut_w;
    // an orbit's count is formed member by member where a window's edge is near
    // (the members' sums round differently): closer than the rounding of FP32
    // pairs or FP64
    const R edge = cut * (kPair ? (R)1e-4 : (R)1e-9) + (kPair ? (R)1e-5 : (R)1e-12);
    // items: (pair or q chunk, block of modes), n_sblk blocks of s_per modes each
    const int n_items = (ORBIT ? t.n_pairs : p.nqc * p.n_chunks) * t.n_sblk;
    unsigned long long allowed = 0;

    for (;;) {
        if (tid == 0) item_sm = atomicAdd(d.queue, 1);
        __syncthreads();
        const int item_all = item_sm;
        __syncthreads();
        if (item_all >= n_items) break;
        const int item = item_all / t.n_sblk, sblk = item_all - item * t.n_sblk;
        const int sbeg = sblk * t.s_per, send = min(nb, sbeg + t.s_per);
        int q, qp0, qp1, mult;
        if (ORBIT) {
            const int2 pr = t.pairs[item];
            q = pr.x; qp0 = pr.y; qp1 = pr.y + 1;
            mult = t.orbit[item];
        } else {
            const int2 qm = d.qsel[item / p.n_chunks];
            q = qm.x;
            mult = qm.y;                             // an item of q stands for -q as well when it takes q's linewidths
            qp0 = (item % p.n_chunks) * p.qp_chunk;
            qp1 = min(p.nq, qp0 + p.qp_chunk);
        }
        unsigned long long hits = 0;
        for (int x = tid; x < 3 * nb; x += nthr) red[x] = 0.0;

        for (int qp = qp0; qp < qp1; ++qp) {
            // q'' = q + q' on the mesh
            const int *kq = d.qfrac + 3 * q, *kp = d.qfrac + 3 * qp;
            const int k0 = (kq[0] + kp[0]) % p.mesh[0];
            const int k1 = (kq[1] + kp[1]) % p.mesh[1];
            const int k2 = (kq[2] + kp[2]) % p.mesh[2];
            const int qpp = (k0 * p.mesh[1] + k1) * p.mesh[2] + k2;
            __syncthreads();
            for (int x = tid; x < P; x += nthr) {
                const bool in = x < nb;
                if constexpr (kPair) {
                    const float4 a = in ? d.wn32[(size_t)qp * nb + x] : make_float4(0.f, 0.f, 0.f, 0.f);
                    const float4 b = in ? d.wn32[(size_t)qpp * nb + x] : make_float4(0.f, 0.f, 0.f, 0.f);
                    wp[x] = a.x; wpl[x] = a.y; np_[x] = a.z; npl[x] = a.w;
                    wpp[x] = b.x; wppl[x] = b.y; npp[x] = b.z; nppl[x] = b.w;
                } else {
                    wp[x] = in ? (R)d.omega[(size_t)qp * nb + x] : (R)0;
                    np_[x] = in ? (R)d.occ[(size_t)qp * nb + x] : (R)0;
                    wpp[x] = in ? (R)d.omega[(size_t)qpp * nb + x] : (R)0;
                    npp[x] = in ? (R)d.occ[(size_t)qpp * nb + x] : (R)0;
                }
            }
            if (OPER_SMEM) {
                const R2 *src1 = epsT_all + (size_t)qp * nb * nb;
                const R2 *src2 = epsT_all + (size_t)qpp * nb * nb;
                for (int x = tid; x < P * P; x += nthr) {
                    const int b = x / P, s = x % P;
                    const bool in = (b < nb) && (s < nb);
                    R2 v1 = in ? src1[b * nb + s] : mk<R2>(0.0, 0.0);
                    R2 v2 = in ? src2[b * nb + s] : mk<R2>(0.0, 0.0);
                    v2.y = -v2.y;
                    EpT[x] = v1;
                    EppT[x] = v2;
                }
            }
            // the tables' rows of this pair
            const R2 *tab[3];
#pragma unroll
            for (int c = 0; c < 3; ++c)
                tab[c] = static_cast<const R2 *>(t.tab[c]) + (size_t)(c == 0 ? qp : c == 1 ? qpp : q) * t.n_slot[c] * 27;

            for (int s0 = sbeg; s0 < send; s0 += SB) {
                const int ns = min(SB, send - s0);
                __syncthreads();
                for (int x = tid; x < ns * P; x += nthr) {
                    const int m = x / P, b = x - m * P;
                    es[m * P + b] = b < nb ? epsT_all[((size_t)q * nb + b) * nb + s0 + m] : mk<R2>(0.0, 0.0);
                }
                __syncthreads();
                // ---- Y_s(3j.., 3k..): one thread per (atom pair, mode), modes fastest;
                // padding atoms and pairs without blocks are zero
                for (int x = tid; x < nap * nap * ns; x += nthr) {
                    const int jk = x / ns, m = x - jk * ns, j = jk / nap, k = jk - j * nap;
                    R2 acc9[9];
#pragma unroll
                    for (int e = 0; e < 9; ++e) acc9[e] = mk<R2>(0.0, 0.0);
                    const int g = (j < na && k < na) ? __ldg(t.group + j * na + k) : -1;
                    if (g >= 0) {
                        const int c2 = __ldg(t.group_c + g);
                        if (c2 >= 0) {
                            const R2 *yc = static_cast<const R2 *>(t.yc) + ((size_t)q * t.n_cg + c2) * 9 * nb + s0 + m;
#pragma unroll
                            for (int e = 0; e < 9; ++e) acc9[e] = yc[(size_t)e * nb];
                        }
                        const R2 *em = es + m * P;
                        for (int y = t.term_start[g]; y < t.term_start[g + 1]; ++y) {
                            const int4 tm = __ldg(t.term + y);               // (i, class, slot or block)
                            const R2 *e3 = em + 3 * tm.x;
                            if (tm.y < 3) {
                                const R2 *w = (tm.y == 0 ? tab[0] : tm.y == 1 ? tab[1] : tab[2]) + (size_t)27 * tm.z;
#pragma unroll
                                for (int a = 0; a < 3; ++a) {
                                    const R2 ev = e3[a];
#pragma unroll
                                    for (int e = 0; e < 9; ++e) cfma(acc9[e], ev, w[9 * a + e]);
                                }
                            } else {
                                const int4 bi = __ldg(d.blkinfo + tm.z);
                                const R2 u = chi_all[(size_t)qp * p.n_rep + bi.y], v = chi_all[(size_t)qpp * p.n_rep + bi.z];
                                R2 ph;                                       // chi(q', Rj) conj(chi(q'', Rk))
                                ph.x = u.x * v.x + u.y * v.y;
                                ph.y = u.y * v.x - u.x * v.y;
                                const R *f = fc3 + (size_t)28 * tm.z;
#pragma unroll
                                for (int a = 0; a < 3; ++a) {
                                    const R2 ev = cmul(e3[a], ph);
#pragma unroll
                                    for (int e = 0; e < 9; ++e) {
                                        const R fv = __ldg(f + 9 * a + e);
                                        acc9[e].x = fma(fv, ev.x, acc9[e].x);
                                        acc9[e].y = fma(fv, ev.y, acc9[e].y);
                                    }
                                }
                            }
                        }
                    }
                    R2 *Ym = Y + m * ysz + (size_t)(3 * j) * P + 3 * k;
#pragma unroll
                    for (int e = 0; e < 9; ++e) Ym[(e / 3) * P + e % 3] = acc9[e];
                }
                __syncthreads();

                // ---- GEMM1: T'(s', c) = sum_b epsT'(b, s') Y(b, c), dense.
                // A warp holds one row tile (broadcast A) over its column tiles.
                const int m1 = tid / n_tiles, tile1 = tid - m1 * n_tiles;
                const int ti = tile1 / tcols, tj = tile1 % tcols;
                const bool active = m1 < ns;
                int r0 = ti * kTR, c0 = tj * kTC;
                R2 acc[kTR][kTC];
                if (active) {
                    const R2 *Ym = Y + m1 * ysz;
#pragma unroll
                    for (int r = 0; r < kTR; ++r)
#pragma unroll
                        for (int c = 0; c < kTC; ++c) acc[r][c] = mk<R2>(0.0, 0.0);
                    for (int b = 0; b < nb; ++b) {
                        R2 av[kTR], bv[kTC];
                        const R2 *arow = OPER_SMEM ? EpT + (size_t)b * P
                                                   : epsT_all + ((size_t)qp * nb + b) * nb;
#pragma unroll
                        for (int r = 0; r < kTR; ++r)
                            av[r] = (OPER_SMEM || r0 + r < nb) ? arow[r0 + r] : mk<R2>(0.0, 0.0);
#pragma unroll
                        for (int c = 0; c < kTC; ++c) bv[c] = Ym[(size_t)b * P + c0 + c];
#pragma unroll
                        for (int r = 0; r < kTR; ++r)
#pragma unroll
                            for (int c = 0; c < kTC; ++c) cfma(acc[r][c], av[r], bv[c]);
                    }
                }
                // ---- delta band: list the (mode, tile) pairs that can hold an allowed triplet
                bool band = false;
                const R w_1 = active ? (R)d.omega[(size_t)q * nb + s0 + m1] : (R)0;
                if (active && w_1 > (R)0) {
                    R wlo = (R)1e30, whi = (R)-1e30, xlo = (R)1e30, xhi = (R)-1e30;
#pragma unroll
                    for (int r = 0; r < kTR; ++r) { wlo = fmin(wlo, wp[r0 + r]); whi = fmax(whi, wp[r0 + r]); }
#pragma unroll
                    for (int c = 0; c < kTC; ++c) { xlo = fmin(xlo, wpp[c0 + c]); xhi = fmax(xhi, wpp[c0 + c]); }
                    // w + w' - w'' in [w + wlo - xhi, w + whi - xlo]
                    // w - w' - w'' in [w - whi - xhi, w - wlo - xlo]
                    // w - w' + w'' in [w - whi + xlo, w - wlo + xhi] (orbits)
                    // (widened by 1e-4 of the cut and the rounding of sums of three
                    // frequencies, so that no tile is dropped here that the exact
                    // per-element test below would reach)
                    const R cb = cut * (R)1.0001 + (kPair ? (R)1e-6 : (R)1e-14) * (w_1 + whi + xhi);
                    band = ((w_1 + wlo - xhi < cb) && (w_1 + whi - xlo > -cb)) ||
                           ((w_1 - whi - xhi < cb) && (w_1 - wlo - xlo > -cb)) ||
                           (ORBIT && (w_1 - whi + xlo < cb) && (w_1 - wlo + xhi > -cb));
                }
                const unsigned bal = __ballot_sync(0xffffffffu, band);
                if (lane == 0) warp_cnt[warp] = __popc(bal);
                __syncthreads();
                if (active) {
                    R2 *Ym = Y + m1 * ysz;
#pragma unroll
                    for (int r = 0; r < kTR; ++r)
#pragma unroll
                        for (int c = 0; c < kTC; ++c)
                            Ym[(size_t)(c0 + c) * Q + r0 + r] = acc[r][c];   // T'^T(c, s')
                }
                if (band) {
                    int off = 0;
                    for (int w8 = 0; w8 < warp; ++w8) off += warp_cnt[w8];
                    tiles[off + __popc(bal & ((1u << lane) - 1u))] = tid;
                }
                if (tid == 0) {
                    int n = 0;
                    for (int w8 = 0; w8 < nwarps; ++w8) n += warp_cnt[w8];
                    n_act_sm = n;
                }
                __syncthreads();

                // ---- GEMM2 + epilogue on the listed tiles, K split over S lanes
                const int n_act = n_act_sm;
                int S = 1;
                while (S < 8 && n_act * S * 2 <= nthr) S <<= 1;
                const int per_pass = nthr / S;
                const int ks = tid & (S - 1);
                const int kc = (nb + S - 1) / S;
                const int kb0 = ks * kc, kb1 = min(nb, kb0 + kc);
                for (int base = 0; base < n_act; base += per_pass) {
                    // every lane runs every pass (the shuffles below need the
                    // whole warp); lanes past the list do no work
                    const int ti2 = base + tid / S;
                    const bool valid = tid / S < per_pass && ti2 < n_act;
                    const int code = valid ? tiles[ti2] : 0;
                    const int m = code / n_tiles, tt = code - m * n_tiles;
                    const R2 *Ym = Y + m * ysz;
                    r0 = (tt / tcols) * kTR;
                    c0 = (tt % tcols) * kTC;
#pragma unroll
                    for (int r = 0; r < kTR; ++r)
#pragma unroll
                        for (int c = 0; c < kTC; ++c) acc[r][c] = mk<R2>(0.0, 0.0);
                    const int ke = valid ? kb1 : kb0;
                    for (int c = kb0; c < ke; ++c) {
                        R2 av[kTR], bv[kTC];
#pragma unroll
                        for (int r = 0; r < kTR; ++r) av[r] = Ym[(size_t)c * Q + r0 + r];
                        if (OPER_SMEM) {
#pragma unroll
                            for (int k = 0; k < kTC; ++k) bv[k] = EppT[(size_t)c * P + c0 + k];
                        } else {
                            const R2 *brow = epsT_all + ((size_t)qpp * nb + c) * nb;
#pragma unroll
                            for (int k = 0; k < kTC; ++k) {
                                R2 v = (c0 + k < nb) ? brow[c0 + k] : mk<R2>(0.0, 0.0);
                                v.y = -v.y;
                                bv[k] = v;
                            }
                        }
#pragma unroll
                        for (int r = 0; r < kTR; ++r)
#pragma unroll
                            for (int k = 0; k < kTC; ++k) cfma(acc[r][k], av[r], bv[k]);
                    }
                    // add the S partial tiles (aligned lanes, fixed order)
                    for (int o = S >> 1; o > 0; o >>= 1) {
#pragma unroll
                        for (int r = 0; r < kTR; ++r)
#pragma unroll
                            for (int c = 0; c < kTC; ++c) {
                                acc[r][c].x += __shfl_xor_sync(0xffffffffu, acc[r][c].x, o);
                                acc[r][c].y += __shfl_xor_sync(0xffffffffu, acc[r][c].y, o);
                            }
                    }
                    if (!valid || ks != 0) continue;
                    const double w_s = d.omega[(size_t)q * nb + s0 + m];
                    const R w = (R)w_s;
                    F2 w0p, n0p;                              // FP32 pairs of w and n of (q, s)
                    R n0 = (R)0;
                    if constexpr (kPair) {
                        const float4 u = d.wn32[(size_t)q * nb + s0 + m];
                        w0p = F2{u.x, u.y};
                        n0p = F2{u.z, u.w};
                        n0 = u.z;
                    } else if (ORBIT) {
                        n0 = d.occ[(size_t)q * nb + s0 + m];
                    }
                    R part = (R)0, colsum[kTC];
#pragma unroll
                    for (int c = 0; c < kTC; ++c) colsum[c] = (R)0;
#pragma unroll
                    for (int r = 0; r < kTR; ++r) {
                        const R w1 = wp[r0 + r], n1 = np_[r0 + r];
                        R rowsum = (R)0;
                        if (w1 > (R)0) {
                            const R iw1 = (R)1 / w1;
                            F2 w1p, n1p, sp, sm;
                            if constexpr (kPair) {
                                w1p = F2{wp[r0 + r], wpl[r0 + r]};
                                n1p = F2{np_[r0 + r], npl[r0 + r]};
                                sp = f2_add(w0p, w1p);
                                sm = f2_add(w0p, f2_neg(w1p));
                            }
#pragma unroll
                            for (int c = 0; c < kTC; ++c) {
                                const R w2 = wpp[c0 + c];
                                if (w2 <= (R)0) continue;
                                const R n2 = npp[c0 + c];
                                F2 w2p, n2p;
                                if constexpr (kPair) {
                                    w2p = F2{wpp[c0 + c], wppl[c0 + c]};
                                    n2p = F2{npp[c0 + c], nppl[c0 + c]};
                                }
                                R dp, dm;
                                if constexpr (kPair) {
                                    dp = f2_diff(sp, w2p);
                                    dm = f2_diff(sm, w2p);
                                } else {
                                    dp = w + w1 - w2;
                                    dm = w - w1 - w2;
                                }
                                const bool hp = fabs(dp) < cut, hm = fabs(dm) < cut;
                                const R2 f = acc[r][c];
                                const R f2 = f.x * f.x + f.y * f.y;
                                R dn;                                        // n' - n''
                                if constexpr (kPair) dn = f2_diff(n1p, n2p);
                                else dn = n1 - n2;
                                if constexpr (ORBIT) {
                                    // positions 1 = (q, s), 2 = (q', s'), 3 = (-q'', s'')
                                    R d2, dn02, dn01;
                                    if constexpr (kPair) {
                                        d2 = f2_diff(sm, f2_neg(w2p));
                                        dn02 = f2_diff(n0p, n2p);
                                        dn01 = f2_diff(n0p, n1p);
                                    } else {
                                        d2 = w - w1 + w2;
                                        dn02 = n0 - n2;
                                        dn01 = n0 - n1;
                                    }
                                    const bool h2 = fabs(d2) < cut;
                                    const bool near_edge = fabs(fabs(dp) - cut) < edge || fabs(fabs(dm) - cut) < edge ||
                                                           fabs(fabs(d2) - cut) < edge;
                                    if (near_edge) {
                                        if constexpr (kPair) hits += window_hits6({w0p, w1p, w2p}, cut);
                                        else hits += window_hits6({w, w1, w2}, cut);
                                    } else {
                                        hits += 2u * ((unsigned)(hp || hm) + (unsigned)(hp || h2) + (unsigned)(hm || h2));
                                    }
                                    if (hp || hm || h2) {
                                        const R e3 = hp ? delta_shape(dp, p.shape, sig2inv) : (R)0;
                                        const R e1 = hm ? delta_shape(dm, p.shape, sig2inv) : (R)0;
                                        const R e2 = h2 ? delta_shape(d2, p.shape, sig2inv) : (R)0;
                                        const R iw2 = (R)1 / w2;
                                        part += f2 * (dn * (e3 - e2) + ((R)1 + n1 + n2) * e1) * iw1 * iw2;
                                        rowsum += f2 * (dn02 * (e3 - e1) + ((R)1 + n0 + n2) * e2) * iw2;
                                        colsum[c] += f2 * (dn01 * (e2 - e1) + ((R)1 + n0 + n1) * e3) * iw1;
                                    }
                                } else if (hp || hm) {
                                    const R gpv = hp ? dn * delta_shape(dp, p.shape, sig2inv) : (R)0;
                                    const R gmv = hm ? (R)0.5 * ((R)1 + n1 + n2) * delta_shape(dm, p.shape, sig2inv) : (R)0;
                                    ++hits;
                                    part += f2 * (gpv + gmv) * iw1 / w2;
                                    if constexpr (!kPair) {
                                        if (p.bte) {
                                            // rates into the BTE operator planes (FP64 atomics;
                                            // every (q, s) row is owned by this item)
                                            const double sc = p.bte_pref / (w_s * w_s);
                                            const size_t N = (size_t)p.nq * nb;
                                            const size_t row = ((size_t)q * nb + s0 + m) * N;
                                            atomicAdd(d.g1_a + row + (size_t)qp * nb + r0 + r, sc * f2 * gpv / w2);
                                            atomicAdd(d.g1_am + row + (size_t)d.qneg[qp] * nb + r0 + r, sc * f2 * gmv / w2);
                                            atomicAdd(d.g1_b + row + (size_t)qpp * nb + c0 + c, sc * f2 * (gpv + gmv) / w1);
                                        }
                                    }
                                }
                            }
                        }
                        if (ORBIT) prow[6 * ti2 + r] = (double)(rowsum / w);     // / w of position 1
                    }
                    psum[ti2] = (double)part;
                    if (ORBIT)
#pragma unroll
                        for (int c = 0; c < kTC; ++c) pcol[3 * ti2 + c] = (double)(colsum[c] / w);
                }
                __syncthreads();
                // ---- the tiles' sums per mode, in the order of the list: position 1 by the
                // mode, 2 by the row, 3 by the column
                for (int x = tid; x < (ORBIT ? ns + 2 * nb : ns); x += nthr) {
                    double v = 0.0;
                    if (x < ns) {
                        for (int y = 0; y < n_act; ++y)
                            if (tiles[y] / n_tiles == x) v += psum[y];
                        red[s0 + x] += v;
                    } else {
                        const bool row = x < ns + nb;
                        const int e = x - ns - (row ? 0 : nb);
                        const int ta = row ? e / kTR : e / kTC, tb = row ? e % kTR : e % kTC;
                        for (int y = 0; y < n_act; ++y) {
                            const int tt = tiles[y] % n_tiles;
                            if ((row ? tt / tcols : tt % tcols) == ta) v += row ? prow[6 * y + tb] : pcol[3 * y + tb];
                        }
                        red[(row ? nb : 2 * nb) + e] += v;
                    }
                }
            }
        }
        __syncthreads();
        if (ORBIT) {
            for (int x = tid; x < 3 * nb; x += nthr) t.out3[(size_t)item_all * 3 * nb + x] = red[x];
        } else {
            for (int s = sbeg + tid; s < send; s += nthr) d.partial[(size_t)item * nb + s] = red[s];
        }
        allowed += (unsigned long long)mult * hits;
        __syncthreads();
    }
    // delta-allowed triplet count (orbits: six times it)
    for (int o = 16; o > 0; o >>= 1) allowed += __shfl_xor_sync(0xffffffffu, allowed, o);
    if (lane == 0 && allowed) atomicAdd(d.allowed, allowed);
}

// gamma = pref / w * sum over chunks; then average over degenerate sets.
// Row j of gamma is q-point qout[j], j < n_out; its sums are in row qrow[j]
// of partial (those of q itself, or of -q).  One CTA per row, one thread per
// mode: the sums and the rank of each mode, then the thread of each set's first
// mode averages it in ascending order (a thread per row sorting its modes took
// 0.11 ms for 64 q-points of 96 modes).
__global__ void __launch_bounds__(kMaxNbSmall)
lw_finish_kernel(int nb, int n_chunks, const double *__restrict__ partial, const int *__restrict__ qout,
                 const int *__restrict__ qrow, const double *__restrict__ omega, const double *__restrict__ nu, double pref,
                 double degen_tol, double *__restrict__ gamma) {
    __shared__ double v[kMaxNbSmall], gs[kMaxNbSmall];
    __shared__ int order[kMaxNbSmall];
    const int j = blockIdx.x, s = threadIdx.x, q = qout[j];
    const size_t row = (size_t)qrow[j];
    if (s < nb) {
        double t = 0.0;
#pragma unroll 4
        for (int c = 0; c < n_chunks; ++c) t += partial[(row * n_chunks + c) * nb + s];
        const double w = omega[(size_t)q * nb + s];
        gs[s] = (w > 0.0) ? pref * t / w : 0.0;
        v[s] = nu[(size_t)q * nb + s];
    }
    __syncthreads();
    if (s < nb) {                                  // ascending, ties by index, NaN last
        const double x = v[s];
        int r = 0;
        for (int t = 0; t < nb; ++t) {
            const double y = v[t];
            const bool lt = y < x || (x != x && y == y);
            const bool gt = y > x || (y != y && x == x);
            r += lt || (!gt && t < s);
        }
        order[r] = s;
    }
    __syncthreads();
    // degenerate sets: chains of |d nu| < tol in ascending order of nu
    double *g = gamma + (size_t)j * nb;
    if (s < nb && (s == 0 || v[order[s]] - v[order[s - 1]] >= degen_tol)) {
        int end = s + 1;
        while (end < nb && !(v[order[end]] - v[order[end - 1]] >= degen_tol)) ++end;
        double t = 0.0;
        for (int b = s; b < end; ++b) t += gs[order[b]];
        if (end - s > 1) t /= (double)(end - s);
        for (int b = s; b < end; ++b) g[order[b]] = t;
    }
}

// The live modes of every q-point in ascending frequency (ties by index), then
// kNoMode as frequency: omega and n in FP64, or their FP32 pairs when wn is given.
constexpr float kNoMode = 1e30f;
__global__ void sort_modes_kernel(int nb, const double *__restrict__ omega, const double *__restrict__ occ,
                                  double2 *__restrict__ wn64, float4 *__restrict__ wn) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *w = reinterpret_cast<double *>(smem_raw);
    const size_t row = (size_t)blockIdx.x * nb;
    for (int x = threadIdx.x; x < nb; x += blockDim.x) w[x] = omega[row + x];
    __syncthreads();
    for (int x = threadIdx.x; x < nb; x += blockDim.x) {
        const double v = w[x];
        if (!(v > 0.0)) {                                // behind the live ones, in any order
            int r = nb - 1;
            for (int y = 0; y < x; ++y) r -= !(w[y] > 0.0);
            if (wn64) wn64[row + r] = make_double2(kNoMode, 0.0);
            if (wn) wn[row + r] = make_float4(kNoMode, 0.f, 0.f, 0.f);
            continue;
        }
        int r = 0;
        for (int y = 0; y < nb; ++y) r += w[y] > 0.0 && (w[y] < v || (w[y] == v && y < x));
        const double n = occ[row + x];
        if (wn64) wn64[row + r] = make_double2(v, n);
        if (wn) {
            const F2 a = f2_of(v), o = f2_of(n);
            wn[row + r] = make_float4(a.h, a.l, o.h, o.l);
        }
    }
}

// -q of a mesh point.
__device__ __forceinline__ int neg_point(const int *__restrict__ k, const int (&mesh)[3]) {
    const int a = k[0] ? mesh[0] - k[0] : 0, b = k[1] ? mesh[1] - k[1] : 0, c = k[2] ? mesh[2] - k[2] : 0;
    return (a * mesh[1] + b) * mesh[2] + c;
}
// *differ |= 1 unless every q-point has the frequencies w of -q, to 4e-13 of its largest
// (two diagonalisations of D(q) and of its conjugate agree to some 1e-14), 5e-12 sigma
// and 1e-11 w.  The sums of -q are then those of q to 1e-10: three frequencies change a
// Gaussian weight inside n_sigma sigma by 3 n_sigma / sigma times their difference (5e-11
// at 3 sigma) and an occupation of n >> 1 by a part in 1e11.
template <typename M>
__global__ void __launch_bounds__(128)
mirror_check_kernel(LwParams p, const int *__restrict__ qfrac, const M *__restrict__ modes, int *__restrict__ differ) {
    __shared__ double top[4];
    const int q = blockIdx.x, m = neg_point(qfrac + 3 * q, p.mesh);
    if (m <= q) return;
    auto freq = [&](int k, int x) {
        const M a = modes[(size_t)k * p.nb + x];
        if constexpr (std::is_same<M, float4>::value) return (double)a.x + (double)a.y;
        else return a.x;
    };
    double mx = 0.0;
    for (int x = threadIdx.x; x < p.nb; x += blockDim.x) {
        const double w = freq(q, x);
        if (w < (double)kNoMode) mx = fmax(mx, w);
    }
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) top[threadIdx.x >> 5] = mx;
    __syncthreads();
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mx = fmax(mx, top[w]);
    bool d = false;
    for (int x = threadIdx.x; x < p.nb; x += blockDim.x) {
        const double w = freq(q, x);
        d |= !(fabs(w - freq(m, x)) <= fmin(fmin(4e-13 * mx, 5e-12 * p.sigma_w), 1e-11 * w));
    }
    if (__syncthreads_or(d) && threadIdx.x == 0) atomicOr(differ, 1);
}

// Phase space per mode (the definition after Eq. delta_deconstructed, with
// the weights of Eq. phase_space and the readings of the linewidths: the 1/2
// on the - process, 1/N_k, masked modes):
//   g_mu = (1/N_k) sum_{q' s' s''} [(n' - n'') G(w + w' - w'') + 1/2 (1 + n' + n'') G(w - w' - w'')],
// q'' = q + q' for both processes (the - process of (q, -q') has the same
// frequencies, since w(-q) = w(q)); where the input says so (mirror_check_kernel), one
// q-point of each pair {q, -q}.  CTA = (q, block of s, chunk of q'), one
// thread per s, FP64 sums over q', one partial sum per chunk.  FP64, or FP32
// weights with the compensated differences.
//
// Bound: issue slots.  The modes of q' and q'' are staged in ascending order,
// so along w' the two windows of w'' slide one way each: a thread keeps their
// near ends and walks only the modes inside (about a seventh of them per
// window at 3 sigma = 0.15 THz of a 2 THz band); the exact test of the window
// decides, the walk is a little wider.  32 atoms, 6^3 mesh, FP32: 143 ms when
// every (s', s'') was tested by one thread per (q, s), 5.5 ms now (half of the q-points).
template <typename R>
__global__ void __launch_bounds__(128)
phase_space_kernel(LwParams p, LwDev d, const void *__restrict__ modes, const int *__restrict__ differ, int chunk,
                   double *__restrict__ partial) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr bool kPair = std::is_same<R, float>::value;
    const int nb = p.nb;
    const int per_q = (nb + blockDim.x - 1) / blockDim.x;          // CTAs per q and chunk
    const int q = (int)blockIdx.x / per_q;
    if (differ && *differ == 0 && neg_point(d.qfrac + 3 * q, p.mesh) < q) return;   // -q's sums are taken
    const int s = ((int)blockIdx.x % per_q) * blockDim.x + threadIdx.x;
    // modes of q' and q'': FP32 pairs (w hi, w lo, n hi, n lo), or FP64 (w, n)
    using M = typename std::conditional<kPair, float4, double2>::type;
    M *f1 = reinterpret_cast<M *>(smem_raw), *f2 = f1 + nb;
    const M *all = static_cast<const M *>(modes);
    const R a = (R)delta_param(p.shape, p.sigma_w);
    const R cut = (R)p.cut_w;
    const double w_s = s < nb ? d.omega[(size_t)q * nb + s] : 0.0;
    const F2 wsp = f2_of(w_s);
    const R w = (R)w_s;
    double sum = 0.0;
    const int qp1 = min(p.nq, ((int)blockIdx.y + 1) * chunk);
    for (int qp = blockIdx.y * chunk; qp < qp1; ++qp) {
        const int *kq = d.qfrac + 3 * q, *kp = d.qfrac + 3 * qp;
        const int qpp = (((kq[0] + kp[0]) % p.mesh[0]) * p.mesh[1] + (kq[1] + kp[1]) % p.mesh[1]) * p.mesh[2] +
                        (kq[2] + kp[2]) % p.mesh[2];
        int m1 = 0, m2 = 0;                    // live modes of q' and q''
        __syncthreads();
        for (int x0 = 0; x0 < nb; x0 += blockDim.x) {
            const int x = x0 + threadIdx.x;
            bool l1 = false, l2 = false;
            if (x < nb) {
                const M a1 = all[(size_t)qp * nb + x], a2 = all[(size_t)qpp * nb + x];
                f1[x] = a1;
                f2[x] = a2;
                l1 = a1.x < (R)kNoMode;
                l2 = a2.x < (R)kNoMode;
            }
            m1 += __syncthreads_count(l1);
            m2 += __syncthreads_count(l2);
        }
        if (!(w_s > 0.0) || m1 == 0 || m2 == 0) continue;
        // half width of the walk: the window, plus the rounding of sums of three frequencies
        const R wide = cut * (R)1.0001 + (kPair ? (R)1e-6 : (R)1e-14) * (w + f1[m1 - 1].x + f2[m2 - 1].x);
        R part = (R)0;
        int lo = 0, top = m2;                  // first w'' of the + window, one past the last of the - window
        for (int sp = 0; sp < m1; ++sp) {
            const M u = f1[sp];
            const R w1 = u.x;
            R n1;
            F2 n1p, sum_p, dif_p;
            if constexpr (kPair) {
                n1 = u.z;
                n1p = F2{u.z, u.w};
                sum_p = f2_add(wsp, F2{u.x, u.y});
                dif_p = f2_add(wsp, F2{-u.x, -u.y});
            } else {
                n1 = u.y;
            }
            R inner = (R)0;
            const R wp = w + w1, wm = w - w1;
            while (lo < m2 && wp - f2[lo].x >= wide) ++lo;
            for (int k = lo; k < m2; ++k) {
                const M v = f2[k];
                if (!(wp - v.x > -wide)) break;
                R dp, dn;
                if constexpr (kPair) {
                    dp = f2_diff(sum_p, F2{v.x, v.y});
                    dn = f2_diff(n1p, F2{v.z, v.w});
                } else {
                    dp = w_s + w1 - v.x;
                    dn = n1 - v.y;
                }
                if (fabs(dp) < cut) inner += dn * delta_shape(dp, p.shape, a);
            }
            while (top > 0 && f2[top - 1].x - wm >= wide) --top;
            for (int k = top - 1; k >= 0; --k) {
                const M v = f2[k];
                if (!(v.x - wm > -wide)) break;
                R dm, n2;
                if constexpr (kPair) {
                    dm = f2_diff(dif_p, F2{v.x, v.y});
                    n2 = v.z;
                } else {
                    dm = w_s - w1 - v.x;
                    n2 = v.y;
                }
                if (fabs(dm) < cut) inner += (R)0.5 * ((R)1 + n1 + n2) * delta_shape(dm, p.shape, a);
            }
            part += inner;
        }
        sum += (double)part;
    }
    if (s < nb) partial[((size_t)blockIdx.y * p.nq + q) * nb + s] = sum;
}

// g[x] = scale * sum of the chunks' partial sums in order (partial may be g); for a
// q-point left out, those of -q's mode of the same frequency.
__global__ void phase_space_sum_kernel(LwParams p, const int *__restrict__ qfrac, const double *__restrict__ omega,
                                       const int *__restrict__ differ, int n_chunks, const double *partial, double scale,
                                       double *g) {
    const size_t n = (size_t)p.nq * p.nb, x = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (x >= n) return;
    size_t y = x;
    if (differ && *differ == 0) {
        const int q = (int)(x / p.nb), m = neg_point(qfrac + 3 * q, p.mesh);
        if (m < q) {
            const double w = omega[x];
            double best = 1e300;
            for (size_t z = (size_t)m * p.nb; z < (size_t)(m + 1) * p.nb; ++z) {
                const double e = fabs(omega[z] - w);
                if (e < best) {
                    best = e;
                    y = z;
                }
            }
        }
    }
    double t = 0.0;
    for (int c = 0; c < n_chunks; ++c) t += partial[(size_t)c * n + y];
    g[x] = scale * t;
}

}  // namespace

cudaError_t launch_mode_prep(int n, const double *nu, double omega_min_w, double T, int classical,
                             double *omega, double *occ, cudaStream_t st) {
    mode_prep_kernel<<<counted((n + 255) / 256), 256, 0, st>>>(n, nu, omega_min_w, T, classical, omega, occ);
    return cudaGetLastError();
}

cudaError_t launch_lw_prep(const LwParams &p, const LwDev &d, int fp32, cudaStream_t st) {
    const int n = p.nq * p.nb;
    mode_prep_kernel<<<counted((n + 255) / 256), 256, 0, st>>>(n, d.nu, p.omega_min_w, p.T, p.classical,
                                                      d.omega, d.occ);
    const int nc = p.nq * p.n_rep;
    const size_t ne = (size_t)p.nq * p.nb * p.nb;
    const int grid = (int)std::min<size_t>((ne + 255) / 256, 4096);
    if (fp32) {
        wn_pair_kernel<<<counted((n + 255) / 256), 256, 0, st>>>(n, d.omega, d.occ, d.wn32);
        if (nc) chi_kernel<float2><<<counted((nc + 255) / 256), 256, 0, st>>>(p.nq, p.n_rep, d.qcart, d.rep_cart,
                                                             (float2 *)d.chi);
        eps_transpose_kernel<float2><<<counted(grid), 256, 0, st>>>(p.nq, p.nb, d.eig, (float2 *)d.eps_work);
    } else {
        if (nc) chi_kernel<double2><<<counted((nc + 255) / 256), 256, 0, st>>>(p.nq, p.n_rep, d.qcart, d.rep_cart,
                                                              (double2 *)d.chi);
        eps_transpose_kernel<double2><<<counted(grid), 256, 0, st>>>(p.nq, p.nb, d.eig, (double2 *)d.eps_work);
    }
    return cudaGetLastError();
}

template <typename R>
static void run_lw_tables(int nq, int n_rep, const LwTerms &t, const int4 *blkinfo, const R *fc3,
                          const typename C2<R>::T *chi, cudaStream_t st) {
    const size_t nt = (size_t)std::max({t.n_slot[0], t.n_slot[1], t.n_slot[2]}) * 27 * nq;
    if (nt)
        lw_tables_kernel<R><<<counted((unsigned)std::min<size_t>((nt + 255) / 256, 16384)), 256, 0, st>>>(nq, n_rep, t,
                                                                                                         blkinfo, fc3, chi);
}
cudaError_t launch_lw_same(int nb, int nq, const LwTerms &t, int n_rows, const int2 *rows, const void *epsT, int fp32,
                           cudaStream_t st) {
    if (!t.n_cg || !n_rows) return cudaSuccess;
    const dim3 grid(rows ? n_rows : nq, t.n_cg);
    const int threads = (nb + 31) / 32 * 32;
    if (fp32) lw_same_kernel<float><<<counted(grid), threads, 0, st>>>(nb, t, rows, static_cast<const float2 *>(epsT));
    else lw_same_kernel<double><<<counted(grid), threads, 0, st>>>(nb, t, rows, static_cast<const double2 *>(epsT));
    return cudaGetLastError();
}
cudaError_t launch_lw_tables_f32(int nq, int n_rep, const LwTerms &t, const int4 *blkinfo, const float *fc3,
                                 const float2 *chi, cudaStream_t st) {
    run_lw_tables<float>(nq, n_rep, t, blkinfo, fc3, chi, st);
    return cudaGetLastError();
}

// Modes per pass and threads of a CTA: up to 256 threads, and two CTAs per SM in
// shared memory where several modes run side by side.
template <typename R>
static void lw_shape(int nb, bool orbit, size_t smem_optin, int &sb, int &nthr) {
    const int P = (nb + kTR - 1) / kTR * kTR, n_tiles = (P / kTR) * (P / kTC);
    const size_t half = (smem_optin - 4096) / 2;
    auto threads = [&](int m) { return (m * n_tiles + 31) / 32 * 32; };
    sb = std::max(1, std::min(nb, 256 / n_tiles));
    while (sb > 1 && lw_smem_bytes<R>(nb, sb, threads(sb), true, orbit) > half) --sb;
    nthr = threads(sb);
}
// Blocks of modes per pair or q chunk: one, or as many as give every SM about
// eight items on a coarse mesh (from the mesh, not from the q-points of a call).
static int lw_mode_blocks(int nb, int sb, long long n_base, int sm_count) {
    const long long want = 8LL * std::max(1, sm_count);
    return (int)std::max(1LL, std::min<long long>((nb + sb - 1) / sb, (want + n_base - 1) / std::max(1LL, n_base)));
}
// Orbits of one launch: their positions' sums take at most kOrbitSums bytes (24 nb bytes
// per orbit, 26 GB for four atoms on 32^3), and the sums by q-point are formed after
// every launch, in one pass over all (q, q2) each.  Three atoms on 20^3, five launches
// in place of one: 0.390 -> 0.392 s in FP32, 3.55 s both ways in FP64.
constexpr size_t kOrbitSums = size_t(256) << 20;
static int lw_orbit_launch(int nb, int n_pairs) {
    const long long top = (long long)(kOrbitSums / (sizeof(double) * 3 * nb));
    const long long n = (n_pairs + top - 1) / top;
    return (int)((n_pairs + n - 1) / n);               // of about one size
}
template <typename R>
static int orbit_blocks(int nb, int n_pairs, int sm_count, size_t smem_optin) {
    int sb, nthr;
    lw_shape<R>(nb, true, smem_optin, sb, nthr);
    return lw_mode_blocks(nb, sb, n_pairs, sm_count);
}
// Values of an orbit run's out3: [pairs][blocks][3][nb], and [pairs][3][nb] after it when
// there are several blocks of modes (on coarse meshes, one launch).
size_t lw_orbit_sums(int nb, int n_pairs, int fp32, int sm_count, size_t smem_optin) {
    const int blocks = fp32 ? orbit_blocks<float>(nb, n_pairs, sm_count, smem_optin)
                            : orbit_blocks<double>(nb, n_pairs, sm_count, smem_optin);
    return 3 * (size_t)lw_orbit_launch(nb, n_pairs) * nb * (blocks > 1 ? blocks + 1 : 1);
}

template <typename R, bool ORBIT>
static cudaError_t run_lw_main(const LwParams &p, const LwDev &d, LwTerms t, int sm_count, size_t smem_optin,
                               cudaStream_t st) {
    using R2 = typename C2<R>::T;
    int sb, nthr;
    lw_shape<R>(p.nb, ORBIT, smem_optin, sb, nthr);
    // the eigenvectors in shared memory where they fit
    const bool oper = lw_smem_bytes<R>(p.nb, sb, nthr, true, ORBIT) <= smem_optin;
    const size_t smem = lw_smem_bytes<R>(p.nb, sb, nthr, oper, ORBIT);
    if (smem > smem_optin || nthr > kThreads) return cudaErrorInvalidValue;
    auto k = oper ? lw_main_kernel<R, true, ORBIT> : lw_main_kernel<R, false, ORBIT>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 1;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, nthr, smem);
    if (e != cudaSuccess) return e;
    run_lw_tables<R>(p.nq, p.n_rep, t, d.blkinfo, static_cast<const R *>(d.fc3), static_cast<const R2 *>(d.chi), st);
    // (an orbit's pair starts at any q of the mesh)
    e = launch_lw_same(p.nb, p.nq, t, ORBIT ? p.nq : p.nqc, ORBIT ? nullptr : d.qsel, d.eps_work, sizeof(R) == 4, st);
    if (e != cudaSuccess) return e;
    const int n_batch = (p.nb + sb - 1) / sb;
    t.n_sblk = ORBIT ? lw_mode_blocks(p.nb, sb, t.n_pairs, sm_count)
                     : lw_mode_blocks(p.nb, sb, (long long)(p.nq / 2 + 1) * p.n_chunks, sm_count);
    t.s_per = (n_batch + t.n_sblk - 1) / t.n_sblk * sb;
    auto launch = [&](const LwTerms &t) {
        const long long n_items = (ORBIT ? t.n_pairs : (long long)p.nqc * p.n_chunks) * t.n_sblk;
        if (n_items > 0x7fffffffLL - (1 << 20)) return cudaErrorInvalidValue;
        const cudaError_t r = cudaMemsetAsync(d.queue, 0, sizeof(int), st);
        if (r != cudaSuccess) return r;
        const int grid = (int)std::max(1LL, std::min<long long>(n_items, (long long)sm_count * std::max(1, per_sm)));
        ProfMark pm(p.prof, KALD_PROF_LW_MAIN, st);
        k<<<counted(grid), nthr, smem, st>>>(p, d, t, sb, static_cast<const R *>(d.fc3),
                                             static_cast<const R2 *>(d.eps_work), static_cast<const R2 *>(d.chi));
        pm.end();
        return cudaGetLastError();
    };
    if (!ORBIT) return launch(t);
    const int per = lw_orbit_launch(p.nb, t.n_pairs);
    for (int p0 = 0; p0 < t.n_pairs && e == cudaSuccess; p0 += per) {
        LwTerms c = t;
        c.n_pairs = std::min(per, t.n_pairs - p0);
        c.pairs += p0;
        c.orbit += p0;
        e = launch(c);
        const double *sums = c.out3;
        if (e == cudaSuccess && c.n_sblk > 1) {
            const size_t n = (size_t)c.n_pairs * 3 * p.nb;
            lw_block_sums_kernel<<<counted((unsigned)std::min<size_t>((n + 255) / 256, 4096)), 256, 0, st>>>(
                n, 3 * p.nb, c.n_sblk, c.out3, c.out3 + n * c.n_sblk);
            sums = c.out3 + n * c.n_sblk;
        }
        if (e == cudaSuccess) e = launch_orbit_class_sums(*t.plan, p.nb, p0, p0 + c.n_pairs, sums, d.partial, st);
    }
    return e;
}

cudaError_t launch_lw_main(const LwParams &p, const LwDev &d, const LwTerms &t, int fp32, int sm_count,
                           size_t smem_optin, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(d.allowed, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    if (t.n_pairs)
        return fp32 ? run_lw_main<float, true>(p, d, t, sm_count, smem_optin, st)
                    : run_lw_main<double, true>(p, d, t, sm_count, smem_optin, st);
    return fp32 ? run_lw_main<float, false>(p, d, t, sm_count, smem_optin, st)
                : run_lw_main<double, false>(p, d, t, sm_count, smem_optin, st);
}

// The fc3 blocks by group (j, k), class and home atom i: one table slot per
// (group, class < 3, i), one term per slot and per block of class 3 (every block
// without tables).
void plan_lw_terms(const HostSystem &h, bool tables, LwTermsHost &o) {
    const int na = h.n_atoms, ng = (int)h.pair3_j.size();
    o.group.assign((size_t)na * na, -1);
    o.term_start.assign(1, 0);
    o.term.clear();
    o.group_c.clear();
    o.cterm_start.assign(1, 0);
    o.cterm.clear();
    std::vector<std::vector<int>> slots[3];               // block lists, class by class
    for (int g = 0; g < ng; ++g) {
        o.group[(size_t)h.pair3_j[g] * na + h.pair3_k[g]] = g;
        std::vector<std::array<int, 3>> key;              // (class, i, block), the blocks of a slot in order
        std::vector<unsigned char> has(na, 0);            // classes in use, per i
        for (int pass = 0; pass < 2; ++pass)
            for (int b = h.pair3_start[g]; b < h.pair3_start[g + 1]; ++b) {
                const int *rj = &h.rep_int[3 * (size_t)h.fc3_rj[b]], *rk = &h.rep_int[3 * (size_t)h.fc3_rk[b]];
                const bool zj = !rj[0] && !rj[1] && !rj[2], zk = !rk[0] && !rk[1] && !rk[2];
                const int i = h.fc3_i[b];
                // a block with both at home has no phase: it joins a slot of its (i, j, k)
                // where there is one (class 2 where there is none and j = k: those blocks
                // are the ones that take many i)
                if (tables && pass == (zj && zk ? 0 : 1)) continue;
                if (!tables && pass) continue;
                const int cls = !tables      ? 3
                                : zj && zk   ? (has[i] & 1 ? 0 : has[i] & 2 ? 1 : has[i] & 4 || h.pair3_j[g] == h.pair3_k[g] ? 2 : 0)
                                : zk         ? 0
                                : zj         ? 1
                                : h.fc3_rj[b] == h.fc3_rk[b] ? 2 : 3;
                has[i] |= cls < 3 ? 1 << cls : 0;
                key.push_back({cls, i, b});
            }
        std::sort(key.begin(), key.end());
        for (size_t x = 0; x < key.size(); ++x) {
            const int cls = key[x][0], i = key[x][1], b = key[x][2];
            if (cls == 3) {
                o.term.push_back(make_int4(i, 3, b, 0));
            } else {
                if (x == 0 || key[x - 1][0] != cls || key[x - 1][1] != i) {
                    o.term.push_back(make_int4(i, cls, (int)slots[cls].size(), 0));
                    slots[cls].emplace_back();
                }
                slots[cls].back().push_back(b);
            }
        }
        // many class-2 terms are summed per q-point, not per pair (an atom paired with
        // itself has one per neighbour: a single thread walks a group's terms); two cost
        // what reading their sum does
        const size_t t0 = (size_t)o.term_start.back();
        const auto is2 = [](const int4 &t) { return t.y == 2; };
        const bool many = std::count_if(o.term.begin() + t0, o.term.end(), is2) >= 3;
        o.group_c.push_back(many ? (int)o.cterm_start.size() - 1 : -1);
        if (many) {
            for (size_t y = t0; y < o.term.size(); ++y)
                if (is2(o.term[y])) o.cterm.push_back(make_int2(o.term[y].x, o.term[y].z));
            o.term.erase(std::remove_if(o.term.begin() + t0, o.term.end(), is2), o.term.end());
            o.cterm_start.push_back((int)o.cterm.size());
        }
        o.term_start.push_back((int)o.term.size());
    }
    o.slot_start.assign(1, 0);
    o.slot_blk.clear();
    for (int c = 0; c < 3; ++c) {
        o.n_slot[c] = (int)slots[c].size();
        o.slot0[c] = (int)o.slot_start.size() - 1;
        for (const auto &v : slots[c]) {
            o.slot_blk.insert(o.slot_blk.end(), v.begin(), v.end());
            o.slot_start.push_back((int)o.slot_blk.size());
        }
    }
}

// q' chunks of the phase-space sum: about 26 CTAs per SM, two waves of three warps each
// (eight left the SMs uneven: 6.9 ms where 26 take 5.3 for 32 atoms on 6^3).
static int phase_space_chunks(int nb, int nq, int sm_count) {
    const long long rows = (long long)(nq / 2 + 1) * ((nb + 127) / 128);      // (half of the q-points as a rule)
    return (int)std::max(1LL, std::min<long long>(std::min(nq, 1024), (26LL * std::max(1, sm_count) + rows - 1) / rows));
}
// (lean: the sorted modes alone, one chunk straight into the result)
size_t phase_space_bytes(int nb, int nq, int sm_count, int lean) {
    const size_t n = (size_t)nb * nq;
    return ws_round(16 * n) +
           (lean ? 0 : ws_round(sizeof(int)) + ws_round(sizeof(double) * n * phase_space_chunks(nb, nq, sm_count)));
}

cudaError_t launch_phase_space(const LwParams &p, const LwDev &d, int fp32, int sm_count, void *work, int lean,
                               double *g_out, cudaStream_t st) {
    const size_t n = (size_t)p.nb * p.nq;
    char *w = static_cast<char *>(work);
    void *modes = w;
    int *differ = lean ? nullptr : reinterpret_cast<int *>(w + ws_round(16 * n));
    double *partial = lean ? g_out : reinterpret_cast<double *>(w + ws_round(16 * n) + ws_round(sizeof(int)));
    const int n_chunks0 = lean ? 1 : phase_space_chunks(p.nb, p.nq, sm_count);
    const int chunk = (p.nq + n_chunks0 - 1) / n_chunks0, n_chunks = (p.nq + chunk - 1) / chunk;
    const int threads = std::min(128, (p.nb + 31) / 32 * 32);
    const int per_q = (p.nb + threads - 1) / threads;
    const size_t ssort = sizeof(double) * (size_t)p.nb, smem = 2 * sizeof(float4) * (size_t)p.nb;
    cudaError_t e = cudaFuncSetAttribute(sort_modes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssort);
    if (e != cudaSuccess) return e;
    auto *wn64 = static_cast<double2 *>(modes);
    auto *wn32 = static_cast<float4 *>(modes);
    sort_modes_kernel<<<counted(p.nq), threads, ssort, st>>>(p.nb, d.omega, d.occ, fp32 ? nullptr : wn64,
                                                             fp32 ? wn32 : nullptr);
    if (differ) {
        e = cudaMemsetAsync(differ, 0, sizeof(int), st);
        if (e != cudaSuccess) return e;
        if (fp32) mirror_check_kernel<float4><<<counted(p.nq), threads, 0, st>>>(p, d.qfrac, wn32, differ);
        else mirror_check_kernel<double2><<<counted(p.nq), threads, 0, st>>>(p, d.qfrac, wn64, differ);
    }
    const double scale = delta_norm(p.shape, p.sigma_w) / (double)p.nq;
    auto k32 = phase_space_kernel<float>;
    auto k64 = phase_space_kernel<double>;
    e = cudaFuncSetAttribute(fp32 ? k32 : k64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)(p.nq * per_q), (unsigned)n_chunks);
    if (fp32) k32<<<counted(grid), threads, smem, st>>>(p, d, modes, differ, chunk, partial);
    else k64<<<counted(grid), threads, smem, st>>>(p, d, modes, differ, chunk, partial);
    phase_space_sum_kernel<<<counted((unsigned)((n + 255) / 256)), 256, 0, st>>>(p, d.qfrac, d.omega, differ, n_chunks,
                                                                               partial, scale, g_out);
    return cudaGetLastError();
}

cudaError_t launch_lw_finish(const LwParams &p, const LwDev &d, double degen_tol_thz,
                             double *gamma_out, cudaStream_t st) {
    const double pref = kHbarEvPs * kPi / 8.0 * kEvA2AmuPs2 * kEvA2AmuPs2 * kEvA2AmuPs2 /
                        (double)p.nq / (1.0 / delta_norm(p.shape, p.sigma_w));
    const int n_out = p.q1 - p.q0;
    lw_finish_kernel<<<counted(n_out), (p.nb + 31) / 32 * 32, 0, st>>>(p.nb, p.n_chunks, d.partial, d.qout, d.qrow,
                                                                       d.omega, d.nu, pref, degen_tol_thz, gamma_out);
    return cudaGetLastError();
}

}  // namespace kald
