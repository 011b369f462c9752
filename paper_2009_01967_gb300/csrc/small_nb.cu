// Crystal linewidths of one- and two-atom cells (nb = 3 or 6; paper Eq.
// projection_plus, gamma_operators, phase_space).  One thread per (pair,
// mode s): the contraction Y_s of the phase sums, both dense contractions
//   T'(s', c) = sum_b eps'(b, s') Y_s(b, c),  phi(s', s'') = sum_c T'(s', c) conj(eps''(c, s''))
// and the delta-weight epilogue run in registers (nb^2 complex values each).
// A tensor-core tile of 128 rows would be more than 70% padding here.
//
// The Bloch phase chi(q', Rj) conj(chi(q'', Rk)) of a block is
// exp(-2 pi i m / L) with m = kk(q').nj - kk(q'').nk (kk_d = k_d L / N_d,
// L = lcm of the mesh), read from a table of roots of unity.
//
// Three kinds of blocks have a phase of one q-point only (Rk = 0: q', Rj = 0:
// q'', Rj = Rk: q) and are summed once per q-point into tables.
//
// A Phi3 symmetric under permutations needs one projection per orbit of momentum
// triples (sn_orbit_kernel, sn_orbit32_kernel); otherwise sn_kernel:
// CTA = (q, chunk of q'), thread = (q' lane, mode s); every thread walks its
// q' of the chunk in order, the CTA adds the lanes of each mode in order and
// writes one FP64 partial per (q, chunk, s) for lw_finish.

#include <algorithm>
#include <type_traits>
#include <vector>

#include "kald_internal.h"
#include "wdiff.cuh"

namespace kald {

// Bytes of the orbits' sums (three positions per orbit) ...
size_t sn_orbit_bytes(int nb, int n_pairs, int fp32) {
    return (fp32 ? sizeof(float) : sizeof(double)) * 3 * (size_t)n_pairs * nb;
}
// ... and the packed eigenvectors of sn_orbit32_kernel after them.
size_t sn_orbit_work(int nb, int nq, int n_pairs, int fp32) {
    const size_t sums = ws_round(sn_orbit_bytes(nb, n_pairs, fp32));
    return sums + (fp32 ? ws_round(sizeof(float4) * (size_t)nq * nb * nb) +
                              ws_round(sizeof(float4) * (size_t)nq * nb * ((nb + 1) / 2))
                        : 0);
}

namespace {

template <typename R> struct Cx;
template <> struct Cx<float> { using T = float2; };
template <> struct Cx<double> { using T = double2; };

constexpr int kSnThreads = 256;

// FP64: scalar FMAs; FP32: packed FP32x2 FMAs (two lanes of the complex
// value per instruction).
__device__ __forceinline__ void cfma(double2 &acc, double2 a, double2 b) {      // acc += a b
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(-a.y, b.y, acc.x);
    acc.y = fma(a.x, b.y, acc.y);
    acc.y = fma(a.y, b.x, acc.y);
}
__device__ __forceinline__ void cfma(float2 &acc, float2 a, float2 b) {
    acc = __ffma2_rn(make_float2(a.x, a.x), b, acc);
    acc = __ffma2_rn(make_float2(-a.y, a.y), make_float2(b.y, b.x), acc);
}
__device__ __forceinline__ void cfma_conj(double2 &acc, double2 a, double2 b) { // acc += a conj(b)
    acc.x = fma(a.x, b.x, acc.x);
    acc.x = fma(a.y, b.y, acc.x);
    acc.y = fma(a.y, b.x, acc.y);
    acc.y = fma(-a.x, b.y, acc.y);
}
__device__ __forceinline__ void cfma_conj(float2 &acc, float2 a, float2 b) {
    acc = __ffma2_rn(make_float2(b.x, b.x), a, acc);
    acc = __ffma2_rn(make_float2(b.y, -b.y), make_float2(a.y, a.x), acc);
}
// roots[t] = exp(-2 pi i (t - m0) / L), argument reduced to [0, L) first.
__global__ void roots_kernel(int L, int m0, double2 *__restrict__ out) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t > 2 * m0) return;
    const int r = (((t - m0) % L) + L) % L;
    double sn, cs;
    sincospi(2.0 * (double)r / (double)L, &sn, &cs);
    out[t] = make_double2(cs, -sn);
}

// Sum over the blocks of one class and atom triple (CSR key) of Phi3~[al be ga]
// times the block's phase exp(-2 pi i m / L), m = x.nj - y.nk with x, y the
// scaled mesh coordinates of q' and q'' (one of them zero for a table); FP64.  Every
// step-th block from `first` on.
__device__ __forceinline__ double2 phase_sum(const SnTables &t, int key, int v, int x0, int x1, int x2, int y0, int y1,
                                             int y2, int first = 0, int step = 1) {
    double2 acc = make_double2(0.0, 0.0);
    const int b1 = t.start[key + 1];
#pragma unroll 4
    for (int bl = t.start[key] + first; bl < b1; bl += step) {
        const int4 nj = __ldg(t.bj + bl), nk = __ldg(t.bk + bl);
        const int m = x0 * nj.x + x1 * nj.y + x2 * nj.z - y0 * nk.x - y1 * nk.y - y2 * nk.z;
        const double2 ph = __ldg(t.roots + m + t.m0);
        const double f = __ldg(t.fc3 + (size_t)28 * bl + v);
        acc.x = fma(f, ph.x, acc.x);
        acc.y = fma(f, ph.y, acc.y);
    }
    return acc;
}

// Tables of the phase sums that depend on one q-point only, [nq][NB^3] each
// (index (a NB + b) NB + c): A(q') of the blocks with Rk = 0, B(q'') of those
// with Rj = 0, C(q) of those with Rj = Rk (chi(q', R) conj chi(q'', R) =
// conj chi(q, R), q'' = q + q').  One CTA per q-point, FP64 sums.
// PACKED: as float4 (re c, re c + 1, im c, im c + 1) for sn_orbit32_kernel.
template <typename R, int NB, bool PACKED = false>
__global__ void __launch_bounds__(kSnThreads)
sn_tables_kernel(int nq, SnTables t, typename Cx<R>::T *__restrict__ tab) {
    using R2 = typename Cx<R>::T;
    constexpr int N3 = NB * NB * NB, NA = NB / 3;
    // one atom: a sum runs over every block of its class, three threads share it
    constexpr int kParts = 3 * N3 * 3 <= kSnThreads ? 3 : 1;
    __shared__ double2 part[kParts > 1 ? 3 * N3 : 1][kParts];
    const int q = blockIdx.x;
    const int k0 = t.kk[3 * q], k1 = t.kk[3 * q + 1], k2 = t.kk[3 * q + 2];
    auto store = [&](int x, double2 s) {
        if constexpr (PACKED) {
            constexpr int C2 = (NB + 1) / 2;
            const int e = x % N3, c = e % NB;
            R *v = reinterpret_cast<R *>(tab) + (((size_t)(x / N3) * nq + q) * (NB * NB * C2) + e / NB * C2 + c / 2) * 4 +
                   c % 2;
            v[0] = (R)s.x;
            v[2] = (R)s.y;
            if (c == NB - 1 && NB % 2) v[1] = v[3] = (R)0;
        } else {
            R2 o;
            o.x = (R)s.x;
            o.y = (R)s.y;
            tab[((size_t)(x / N3) * nq + q) * N3 + x % N3] = o;
        }
    };
    for (int y = threadIdx.x; y < 3 * N3 * kParts; y += kSnThreads) {
        const int x = y / kParts, h = y - x * kParts;
        const int cls = x / N3, e = x - cls * N3;
        const int a = e / (NB * NB), b = (e / NB) % NB, c = e % NB;
        const int key = cls * NA * NA * NA + ((a / 3) * NA + b / 3) * NA + c / 3;
        const int v = 9 * (a % 3) + 3 * (b % 3) + c % 3;
        const double2 s = cls == 0 ? phase_sum(t, key, v, k0, k1, k2, 0, 0, 0, h, kParts)
                                   : phase_sum(t, key, v, 0, 0, 0, k0, k1, k2, h, kParts);
        if constexpr (kParts > 1) part[x][h] = s;
        else store(x, s);
    }
    if constexpr (kParts > 1) {
        __syncthreads();
        for (int x = threadIdx.x; x < 3 * N3; x += kSnThreads) {
            double2 s = part[x][0];
            for (int h = 1; h < kParts; ++h) {
                s.x += part[x][h].x;
                s.y += part[x][h].y;
            }
            store(x, s);
        }
    }
}

// BTE: each thread also scatters its (q', s) rates into the three operator
// planes (FP64 only; every plane entry has exactly one writer).
//
// Y_s(b, c) = sum_a eps_a(q s) W(a, b, c) with the mode-independent phase sums
// W = A(q') + B(q'') + C(q) + the blocks whose two cell vectors are non-zero
// and different (class 3, summed per pair).  The CTA forms W for its pairs one
// row a at a time in shared memory; every mode of the pair reads it from there.
//
// Bound: FMA issue, FP32 or FP64.  Phasing every block for every (pair, mode)
// cost 54 n_fc3 FMA (25,380 for the two-atom cell), fifteen times the two dense
// contractions; with the tables a (pair, mode) costs 3 nb^3 complex FMA in all.
// One call, two-atom cell, 24^3 mesh, FP32: 1367 ms before, 191 ms (34 with orbits).
template <typename R, int NB, bool BTE>
__global__ void __launch_bounds__(kSnThreads)
sn_kernel(LwParams p, LwDev d, SnTables t, const typename Cx<R>::T *__restrict__ tab,
          const typename Cx<R>::T *__restrict__ epsT) {
    using R2 = typename Cx<R>::T;
    constexpr int NA = NB / 3, N2 = NB * NB, N3 = N2 * NB;
    constexpr int JPC = kSnThreads / NB;           // q' lanes per CTA
    constexpr int WP = N2 + 1;                     // row pitch of W (odd: the pairs' rows start in other banks)
    __shared__ __align__(16) R2 W[JPC * WP];
    __shared__ __align__(16) R2 eq[N2], Cq[N3];    // eps(q)^T: eq[b * NB + s]
    __shared__ int qpp_sm[JPC];
    __shared__ double red[kSnThreads];

    const int qi = blockIdx.x, chunk = blockIdx.y;
    const int2 qm = d.qsel[qi];
    const int q = qm.x;
    const int tid = threadIdx.x;
    const bool tabs = tab != nullptr;
    const R2 *tabA = tab, *tabB = tab + (size_t)p.nq * N3, *tabC = tab + 2 * (size_t)p.nq * N3;
    for (int x = tid; x < N2; x += kSnThreads) eq[x] = epsT[(size_t)q * N2 + x];
    for (int x = tid; x < N3; x += kSnThreads)
        if (tabs) Cq[x] = tabC[(size_t)q * N3 + x];

    const int jl = tid / NB, s = tid - (tid / NB) * NB;
    const bool act = jl < JPC;
    const R w = act ? (R)d.omega[(size_t)q * NB + s] : (R)0;
    // FP32: omega and n as hi + lo pairs, so that w +- w' - w'' and n' - n''
    // keep their accuracy when the terms nearly cancel (wdiff.cuh)
    constexpr bool kPair = std::is_same<R, float>::value;
    const F2 wsp = act ? f2_of(d.omega[(size_t)q * NB + s]) : F2{0.f, 0.f};
    const R sig2inv = (R)delta_param(p.shape, p.sigma_w);   // the delta shape's parameter
    const R cut = (R)p.cut_w;
    const int *kq = d.qfrac + 3 * q;
    const int n_gen = t.start[4 * NA * NA * NA] - t.start[3 * NA * NA * NA];
    double sum = 0.0;
    unsigned long long allowed = 0;
    const int qp0 = chunk * p.qp_chunk, qp1 = min(p.nq, qp0 + p.qp_chunk);
    for (int qb = qp0; qb < qp1; qb += JPC) {
        const int n_p = min(JPC, qp1 - qb);        // pairs of this pass: q' = qb ..
        __syncthreads();                           // the last pass has read qpp_sm and W
        if (tid < n_p) {
            const int *kp = d.qfrac + 3 * (qb + tid);
            qpp_sm[tid] = (((kq[0] + kp[0]) % p.mesh[0]) * p.mesh[1] + (kq[1] + kp[1]) % p.mesh[1]) * p.mesh[2] +
                          (kq[2] + kp[2]) % p.mesh[2];
        }
        R2 Y[NB][NB];
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int c = 0; c < NB; ++c) Y[b][c].x = Y[b][c].y = (R)0;
        const int qp = qb + jl;
        const bool run = act && jl < n_p && w > (R)0;
#pragma unroll 1
        for (int a = 0; a < NB; ++a) {
            __syncthreads();
            for (int x = tid; x < n_p * N2; x += kSnThreads) {
                const int pj = x / N2, e = x - pj * N2;
                const size_t r1 = (size_t)(qb + pj) * N3 + a * N2 + e, r2 = (size_t)qpp_sm[pj] * N3 + a * N2 + e;
                R2 v;
                v.x = v.y = (R)0;
                if (tabs) {
                    const R2 u1 = __ldg(tabA + r1), u2 = __ldg(tabB + r2), u3 = Cq[a * N2 + e];
                    v.x = u1.x + u2.x + u3.x;
                    v.y = u1.y + u2.y + u3.y;
                }
                if (n_gen) {
                    const int b = e / NB, c = e - (e / NB) * NB;
                    const int *x1 = t.kk + 3 * (qb + pj), *x2 = t.kk + 3 * qpp_sm[pj];
                    const double2 g = phase_sum(t, 3 * NA * NA * NA + ((a / 3) * NA + b / 3) * NA + c / 3,
                                                9 * (a % 3) + 3 * (b % 3) + c % 3, x1[0], x1[1], x1[2], x2[0], x2[1],
                                                x2[2]);
                    v.x += (R)g.x;
                    v.y += (R)g.y;
                }
                W[pj * WP + e] = v;
            }
            __syncthreads();
            if (run) {
                const R2 ev = eq[a * NB + s];
                const R2 *Wj = W + jl * WP;
#pragma unroll
                for (int b = 0; b < NB; ++b)
#pragma unroll
                    for (int c = 0; c < NB; ++c) cfma(Y[b][c], ev, Wj[b * NB + c]);
            }
        }
        if (!run) continue;
        const int qpp = qpp_sm[jl];
        // ---- per s': the row T'(s', c) = sum_b eps'(b, s') Y(b, c), then
        // phi(s', s'') = sum_c T'(s', c) conj(eps''(c, s'')) and both weights
        const R2 *e1 = epsT + (size_t)qp * NB * NB;    // e1[b * NB + s']
        const R2 *e2 = epsT + (size_t)qpp * NB * NB;   // e2[c * NB + s'']
        R part = (R)0;
        R ap[BTE ? NB : 1], am[BTE ? NB : 1], bb[BTE ? NB : 1];
        if constexpr (BTE) {
#pragma unroll
            for (int x = 0; x < NB; ++x) ap[x] = am[x] = bb[x] = (R)0;
        }
#pragma unroll
        for (int sp = 0; sp < NB; ++sp) {
            const R w1 = (R)d.omega[(size_t)qp * NB + sp];
            if (!(w1 > (R)0)) continue;
            const R n1 = (R)d.occ[(size_t)qp * NB + sp];
            F2 n1p, sump, difp;
            if constexpr (kPair) {
                const float4 a = __ldg(d.wn32 + (size_t)qp * NB + sp);
                n1p = F2{a.z, a.w};
                sump = f2_add(wsp, F2{a.x, a.y});
                difp = f2_add(wsp, F2{-a.x, -a.y});
            }
            R2 T[NB];
#pragma unroll
            for (int c = 0; c < NB; ++c) T[c].x = T[c].y = (R)0;
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const R2 ev = __ldg(e1 + b * NB + sp);
#pragma unroll
                for (int c = 0; c < NB; ++c) cfma(T[c], ev, Y[b][c]);
            }
#pragma unroll
            for (int spp = 0; spp < NB; ++spp) {
                R w2, dp, dm, n2, dn;
                if constexpr (kPair) {
                    const float4 b = __ldg(d.wn32 + (size_t)qpp * NB + spp);
                    w2 = b.x;
                    if (!(w2 > 0.0f)) continue;
                    dp = f2_diff(sump, F2{b.x, b.y});
                    dm = f2_diff(difp, F2{b.x, b.y});
                    n2 = b.z;
                    dn = f2_diff(n1p, F2{b.z, b.w});
                } else {
                    w2 = d.omega[(size_t)qpp * NB + spp];
                    if (!(w2 > (R)0)) continue;
                    dp = w + w1 - w2;
                    dm = w - w1 - w2;
                    n2 = d.occ[(size_t)qpp * NB + spp];
                    dn = n1 - n2;
                }
                const bool hp = fabs(dp) < cut, hm = fabs(dm) < cut;
                if (!(hp || hm)) continue;
                R2 f;
                f.x = f.y = (R)0;
#pragma unroll
                for (int c = 0; c < NB; ++c) cfma_conj(f, T[c], __ldg(e2 + c * NB + spp));
                const R gpv = hp ? dn * delta_shape(dp, p.shape, sig2inv) : (R)0;
                const R gmv = hm ? (R)0.5 * ((R)1 + n1 + n2) * delta_shape(dm, p.shape, sig2inv) : (R)0;
                const R g = gpv + gmv;
                const R f2 = f.x * f.x + f.y * f.y;
                part += f2 * g / (w1 * w2);
                ++allowed;
                if constexpr (BTE) {
                    ap[sp] += f2 * gpv / w2;
                    am[sp] += f2 * gmv / w2;
                    bb[spp] += f2 * g / w1;
                }
            }
        }
        sum += (double)part;
        if constexpr (BTE) {
            // (w'/w) Gamma = pref |phi|^2 g / (w^2 w''), (w''/w) Gamma = pref |phi|^2 g / (w^2 w')
            const double sc = p.bte_pref / ((double)w * (double)w);
            const size_t N = (size_t)p.nq * NB;
            const size_t row = ((size_t)q * NB + s) * N;
            const int qm = d.qneg[qp];
#pragma unroll
            for (int x = 0; x < NB; ++x) {
                d.g1_a[row + (size_t)qp * NB + x] = sc * (double)ap[x];
                d.g1_am[row + (size_t)qm * NB + x] = sc * (double)am[x];
                d.g1_b[row + (size_t)qpp * NB + x] = sc * (double)bb[x];
            }
        }
    }
    red[tid] = sum;
    allowed *= (unsigned long long)qm.y;           // the count of -q too, where -q takes q's linewidths
    for (int o = 16; o > 0; o >>= 1) allowed += __shfl_xor_sync(0xffffffffu, allowed, o);
    if ((tid & 31) == 0 && allowed) atomicAdd(d.allowed, allowed);
    __syncthreads();
    if (tid < NB) {
        double r = 0.0;
        for (int x = 0; x < JPC; ++x) r += red[x * NB + tid];
        d.partial[((size_t)qi * p.n_chunks + chunk) * NB + tid] = r;
    }
}

// One projection per orbit of momentum triples (orbits.cu): Phi3 symmetric under
// permutations.  Thread = (pair lane, mode s of q), CTA = up to `passes` passes of
// kSnThreads / NB pairs.  phi(s, s', s'') gives three weights, one for each of its
// modes (positions 1 = (q, s), 2 = (q', s'), 3 = (-q'', s''), as in lw_main_kernel);
// the pair's sums of all three go to out3[pair][3][NB].
//
// FP64; bound by its units.  A sixth of the pairs of sn_kernel for three weights each.
// The CTA keeps eps(q')^T, conj eps(q'')^T and the frequencies of its pairs in shared
// memory next to W.  One-atom cell, 6^3 mesh (3,925 orbits): with the plan and the
// sums by row the whole calculation takes 0.63 ms, by sn_kernel 0.69.
template <int NB, int NT> struct SnOrb {
    static constexpr int kPairs = NT / NB, N2 = NB * NB, N3 = N2 * NB;
    static constexpr int WP = N3 + 2 - N3 % 2;         // pitches: even; the pairs of a warp start in other banks
    static constexpr int EP = 2 * N2 + 2;
    static constexpr int kFreq = 2 * 2 * NB + 1;       // per pair: (w, n) of q' and q''
    // W (then the pairs' sums) | eps(q')^T, conj eps(q'')^T | frequencies
    static constexpr size_t kW = sizeof(double2) * kPairs * WP;
    static constexpr size_t kE = sizeof(double2) * kPairs * EP;
    static constexpr size_t kBytes = kW + kE + sizeof(double) * kPairs * kFreq;
    // resident CTAs: registers for Y (2 NB^2 values) without spills
    static constexpr int kMin = (NB == 3 ? 384 : 256) / NT;
};

template <int NB, int NT>
__global__ void __launch_bounds__(NT, (SnOrb<NB, NT>::kMin))
sn_orbit_kernel(LwParams p, LwDev d, SnTables t, const double2 *__restrict__ tab, const double2 *__restrict__ epsT,
                int n_pairs, int passes, const int2 *__restrict__ pairs, const int *__restrict__ orbit,
                double *__restrict__ out3) {
    using S = SnOrb<NB, NT>;
    constexpr int NA = NB / 3, N2 = S::N2, N3 = S::N3, JPC = S::kPairs;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2 *W = reinterpret_cast<double2 *>(smem_raw);
    double *sums = reinterpret_cast<double *>(smem_raw);
    double2 *E = reinterpret_cast<double2 *>(smem_raw + S::kW);
    double *F = reinterpret_cast<double *>(smem_raw + S::kW + S::kE);
    __shared__ int q_sm[3][JPC];

    const int tid = threadIdx.x, jl = tid / NB, s = tid - jl * NB;
    const bool act = jl < JPC;
    const bool tabs = tab != nullptr;
    const int n_gen = t.start[4 * NA * NA * NA] - t.start[3 * NA * NA * NA];
    const double sig2inv = delta_param(p.shape, p.sigma_w);
    const double cut = p.cut_w;
    const double edge = cut * 1e-9 + 1e-12;
    unsigned long long allowed = 0;
    const long long first = (long long)blockIdx.x * passes * JPC;
    for (int pass = 0; pass < passes; ++pass) {
        const long long base = first + (long long)pass * JPC;
        if (base >= n_pairs) break;
        const int n_p = (int)min((long long)JPC, n_pairs - base);
        __syncthreads();                               // the last pass has read everything
        if (tid < n_p) {
            const int2 pr = pairs[base + tid];
            const int *kq = d.qfrac + 3 * pr.x, *kp = d.qfrac + 3 * pr.y;
            q_sm[0][tid] = pr.x;
            q_sm[1][tid] = pr.y;
            q_sm[2][tid] = (((kq[0] + kp[0]) % p.mesh[0]) * p.mesh[1] + (kq[1] + kp[1]) % p.mesh[1]) * p.mesh[2] +
                           (kq[2] + kp[2]) % p.mesh[2];
        }
        __syncthreads();
        // eps(q')(b, s') at E[pair][s' NB + b], conj eps(q'')(c, s'') at [N2 + s'' NB + c]
        for (int x = tid; x < n_p * 2 * N2; x += NT) {
            const int pj = x / (2 * N2), e = x - pj * 2 * N2, k = e / N2, f = e - k * N2;
            double2 v = __ldg(epsT + (size_t)q_sm[1 + k][pj] * N2 + f);
            if (k) v.y = -v.y;
            E[pj * S::EP + k * N2 + (f % NB) * NB + f / NB] = v;
        }
        for (int x = tid; x < n_p * 2 * NB; x += NT) {
            const int pj = x / (2 * NB), e = x - pj * 2 * NB, k = e / NB;
            const size_t o = (size_t)q_sm[1 + k][pj] * NB + e - k * NB;
            double *f = F + pj * S::kFreq + 2 * e;
            f[0] = d.omega[o];
            f[1] = d.occ[o];
        }
        const int q = act && jl < n_p ? q_sm[0][jl] : 0;
        const double w = act && jl < n_p ? d.omega[(size_t)q * NB + s] : 0.0;
        const bool run = w > 0.0;
        double2 Y[NB][NB];
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int c = 0; c < NB; ++c) Y[b][c].x = Y[b][c].y = 0.0;
        // W(a, b, c) of every pair: one pass over the tables, many loads in flight
#pragma unroll 4
        for (int x = tid; x < n_p * N3; x += NT) {
            const int pj = x / N3, o = x - pj * N3;
            double2 v;
            v.x = v.y = 0.0;
            if (tabs) {
                const double2 u1 = __ldg(tab + (size_t)q_sm[1][pj] * N3 + o);
                const double2 u2 = __ldg(tab + ((size_t)p.nq + q_sm[2][pj]) * N3 + o);
                const double2 u3 = __ldg(tab + (2 * (size_t)p.nq + q_sm[0][pj]) * N3 + o);
                v.x = u1.x + u2.x + u3.x;
                v.y = u1.y + u2.y + u3.y;
            }
            W[pj * S::WP + o] = v;
        }
        if (n_gen)                                     // uniform; each entry by the thread that wrote it
            for (int x = tid; x < n_p * N3; x += NT) {
                const int pj = x / N3, o = x - pj * N3, a = o / N2, b = o / NB % NB, c = o % NB;
                const int *x1 = t.kk + 3 * q_sm[1][pj], *x2 = t.kk + 3 * q_sm[2][pj];
                const double2 g = phase_sum(t, 3 * NA * NA * NA + ((a / 3) * NA + b / 3) * NA + c / 3,
                                            9 * (a % 3) + 3 * (b % 3) + c % 3, x1[0], x1[1], x1[2], x2[0], x2[1], x2[2]);
                double2 v = W[pj * S::WP + o];
                v.x += g.x;
                v.y += g.y;
                W[pj * S::WP + o] = v;
            }
        __syncthreads();
        if (run) {
            const double2 *Wj = W + jl * S::WP;
#pragma unroll 1
            for (int a = 0; a < NB; ++a) {
                const double2 ev = __ldg(epsT + (size_t)q * N2 + a * NB + s);
#pragma unroll
                for (int b = 0; b < NB; ++b)
#pragma unroll
                    for (int c = 0; c < NB; ++c) cfma(Y[b][c], ev, Wj[a * N2 + b * NB + c]);
            }
        }
        __syncthreads();                               // W is free: the pairs' sums take its place
        if (run) {
            const double2 *e1 = E + jl * S::EP, *e2 = e1 + N2;
            const double *f1 = F + jl * S::kFreq, *f2s = f1 + 2 * NB;
            const double n0 = d.occ[(size_t)q * NB + s];
            double part = 0.0;
            unsigned hits = 0;
            const double iw = 1.0 / w;
            double *out = sums + jl * (2 * NB + 1) * NB + s;
#pragma unroll
            for (int x = 0; x < NB; ++x) out[(NB + x) * NB] = 0.0;
            // (both loops rolled: unrolled they overflow the instruction cache)
#pragma unroll 1
            for (int sp = 0; sp < NB; ++sp) {
                const double w1 = f1[2 * sp], n1 = f1[2 * sp + 1];
                double row = 0.0;
                if (w1 > 0.0) {
                    const double iw1 = 1.0 / w1;
                    double2 T[NB];
#pragma unroll
                    for (int c = 0; c < NB; ++c) T[c].x = T[c].y = 0.0;
#pragma unroll
                    for (int b = 0; b < NB; ++b) {
                        const double2 ev = e1[sp * NB + b];
#pragma unroll
                        for (int c = 0; c < NB; ++c) cfma(T[c], ev, Y[b][c]);
                    }
#pragma unroll 1
                    for (int spp = 0; spp < NB; ++spp) {
                        const double w2 = f2s[2 * spp], n2 = f2s[2 * spp + 1];
                        if (!(w2 > 0.0)) continue;
                        double s3, s1, s2, dn12, dn02, dn01;
                        s3 = w + w1 - w2;
                        s1 = w - w1 - w2;
                        s2 = w - w1 + w2;
                        // (the edges of the windows lie within cut + edge)
                        if (fabs(s3) >= cut + edge && fabs(s1) >= cut + edge && fabs(s2) >= cut + edge) continue;
                        const bool h3 = fabs(s3) < cut, h1 = fabs(s1) < cut, h2 = fabs(s2) < cut;
                        if (fabs(fabs(s3) - cut) < edge || fabs(fabs(s1) - cut) < edge || fabs(fabs(s2) - cut) < edge) {
                            hits += window_hits6({w, w1, w2}, cut);
                        } else {
                            hits += 2u * ((unsigned)(h3 || h1) + (unsigned)(h3 || h2) + (unsigned)(h1 || h2));
                        }
                        if (!(h3 || h1 || h2)) continue;
                        dn12 = n1 - n2;
                        dn02 = n0 - n2;
                        dn01 = n0 - n1;
                        double2 f;
                        f.x = f.y = 0.0;
#pragma unroll
                        for (int c = 0; c < NB; ++c) cfma(f, T[c], e2[spp * NB + c]);
                        const double ff = f.x * f.x + f.y * f.y, iw2 = 1.0 / w2;
                        const double g3 = h3 ? delta_shape(s3, p.shape, sig2inv) : 0.0;
                        const double g1 = h1 ? delta_shape(s1, p.shape, sig2inv) : 0.0;
                        const double g2 = h2 ? delta_shape(s2, p.shape, sig2inv) : 0.0;
                        part += ff * (dn12 * (g3 - g2) + (1.0 + n1 + n2) * g1) * iw1 * iw2;
                        row += ff * (dn02 * (g3 - g1) + (1.0 + n0 + n2) * g2) * iw2;
                        out[(NB + spp) * NB] += iw * ff * (dn01 * (g2 - g1) + (1.0 + n0 + n1) * g3) * iw1;
                    }
                }
                out[sp * NB] = row * iw;               // / w of position 1
            }
            out[2 * NB * NB] = part;
            allowed += (unsigned long long)orbit[base + jl] * hits;
        } else if (act && jl < n_p) {
            double *out = sums + jl * (2 * NB + 1) * NB + s;
            for (int x = 0; x <= 2 * NB; ++x) out[x * NB] = 0.0;
        }
        __syncthreads();
        for (int x = tid; x < n_p * 3 * NB; x += NT) {
            const int pj = x / (3 * NB), e = x - pj * 3 * NB;
            const double *v = sums + pj * (2 * NB + 1) * NB;
            double r;
            if (e < NB) {
                r = v[2 * NB * NB + e];
            } else {
                r = v[(e - NB) * NB];
#pragma unroll
                for (int y = 1; y < NB; ++y) r += v[(e - NB) * NB + y];
            }
            out3[(size_t)base * 3 * NB + x] = r;
        }
    }
    for (int o = 16; o > 0; o >>= 1) allowed += __shfl_xor_sync(0xffffffffu, allowed, o);
    if ((tid & 31) == 0 && allowed) atomicAdd(d.allowed, allowed);
}

// The same for FP32, without the repacking of complex operands that the packed
// FP32x2 FMAs need there: two columns c, c + 1 of every complex array stand together
// as float4 (re, re, im, im), so that one FMA pair takes the real and the imaginary
// parts of two columns; eps(q') comes doubled, (x, x, y, y).  C2 column pairs (the
// last column of three branches is padded).  Per q-point, made by sn_pack_kernel:
//   e1 [NB s'][NB b]   eps(q)(b, s') doubled     e2 [NB s''][C2]  conj eps(q)(c, s'')
// and the phase-sum tables as [NB a][NB b][C2].
//
// Only about a third of the (s, s', s'') lie in a window, but in a warp of 32 (pair, s)
// hardly any (s', s'') is free of them: T' goes to shared memory, a first loop marks a
// thread's hits (high parts, widened), a second one takes them one by one.
//
// Bound: issue, then shared memory (issue 40%, L1 53%).  Two-atom cell, 24^3 mesh
// (15.9 M orbits): 193 ms by sn_kernel, 60 ms with complex values as they stand and
// every (s', s'') in turn, 34.4 ms so.
template <int NB, int NT> struct SnOrb32 {
    static constexpr int C2 = (NB + 1) / 2, N2P = NB * C2, N3P = NB * N2P;
    static constexpr int kPairs = NT / NB;
    static constexpr int TP = N2P + 1 - N2P % 2;       // odd pitches in float4: other banks for each thread or pair
    static constexpr int WP = (NB * TP > N3P ? NB * TP : N3P) | 1;
    static constexpr int EP = (NB * NB + N2P) | 1;
    static constexpr int FP = 2 * NB | 1;
    static constexpr int SP = (2 * NB + 1) | 1;        // floats per thread: rows, columns, position 1
    static constexpr size_t kBytes = sizeof(float4) * kPairs * (WP + EP + FP) + sizeof(float) * (2 * NB * kPairs + NT * SP);
    static constexpr int kMin = 384 / NT;
};

template <int NB>
__global__ void __launch_bounds__(128)
sn_pack_kernel(int nq, const float2 *__restrict__ epsT, float4 *__restrict__ e1, float4 *__restrict__ e2) {
    constexpr int C2 = (NB + 1) / 2, N2 = NB * NB;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x < nq * N2) {
        const int q = x / N2, sp = x % N2 / NB, b = x % NB;
        const float2 v = epsT[(size_t)q * N2 + b * NB + sp];
        e1[x] = make_float4(v.x, v.x, v.y, v.y);
    }
    if (x < nq * NB * C2) {
        const int q = x / (NB * C2), s = x % (NB * C2) / C2, c = 2 * (x % C2);
        const float2 u = epsT[(size_t)q * N2 + c * NB + s];
        const float2 v = c + 1 < NB ? epsT[(size_t)q * N2 + (c + 1) * NB + s] : make_float2(0.f, 0.f);
        e2[x] = make_float4(u.x, v.x, -u.y, -v.y);
    }
}

template <int NB, int NT, int SHAPE>
__global__ void __launch_bounds__(NT, (SnOrb32<NB, NT>::kMin))
sn_orbit32_kernel(LwParams p, LwDev d, SnTables t, const float4 *__restrict__ tab, const float2 *__restrict__ epsT,
                  const float4 *__restrict__ e1_all, const float4 *__restrict__ e2_all, int n_pairs, int passes,
                  const int2 *__restrict__ pairs, const int *__restrict__ orbit, float *__restrict__ out3) {
    using S = SnOrb32<NB, NT>;
    constexpr int NA = NB / 3, N2 = NB * NB, C2 = S::C2, N2P = S::N2P, N3P = S::N3P, JPC = S::kPairs;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float4 *W = reinterpret_cast<float4 *>(smem_raw), *E = W + JPC * S::WP, *F = E + JPC * S::EP;
    float *IW = reinterpret_cast<float *>(F + JPC * S::FP), *sums = IW + 2 * NB * JPC;
    __shared__ int q_sm[3][JPC];

    const int tid = threadIdx.x, jl = tid / NB, s = tid - jl * NB;
    const bool act = jl < JPC;
    const bool tabs = tab != nullptr;
    const int n_gen = t.start[4 * NA * NA * NA] - t.start[3 * NA * NA * NA];
    const float par = delta_param2(SHAPE, (float)delta_param(SHAPE, p.sigma_w));
    const float cut = (float)p.cut_w;
    const float edge = cut * 1e-4f + 1e-5f;
    unsigned long long allowed = 0;
    const long long first = (long long)blockIdx.x * passes * JPC;
    for (int pass = 0; pass < passes; ++pass) {
        const long long base = first + (long long)pass * JPC;
        if (base >= n_pairs) break;
        const int n_p = (int)min((long long)JPC, n_pairs - base);
        __syncthreads();                               // the last pass has read everything
        if (tid < n_p) {
            const int2 pr = pairs[base + tid];
            const int *kq = d.qfrac + 3 * pr.x, *kp = d.qfrac + 3 * pr.y;
            q_sm[0][tid] = pr.x;
            q_sm[1][tid] = pr.y;
            q_sm[2][tid] = (((kq[0] + kp[0]) % p.mesh[0]) * p.mesh[1] + (kq[1] + kp[1]) % p.mesh[1]) * p.mesh[2] +
                           (kq[2] + kp[2]) % p.mesh[2];
        }
        __syncthreads();
        // W(a, b, c) of every pair
#pragma unroll 4
        for (int x = tid; x < n_p * N3P; x += NT) {
            const int pj = x / N3P, o = x - pj * N3P;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (tabs) {
                const float4 u1 = __ldg(tab + (size_t)q_sm[1][pj] * N3P + o);
                const float4 u2 = __ldg(tab + ((size_t)p.nq + q_sm[2][pj]) * N3P + o);
                const float4 u3 = __ldg(tab + (2 * (size_t)p.nq + q_sm[0][pj]) * N3P + o);
                const float2 re = __fadd2_rn(__fadd2_rn(make_float2(u1.x, u1.y), make_float2(u2.x, u2.y)),
                                             make_float2(u3.x, u3.y));
                const float2 im = __fadd2_rn(__fadd2_rn(make_float2(u1.z, u1.w), make_float2(u2.z, u2.w)),
                                             make_float2(u3.z, u3.w));
                v = make_float4(re.x, re.y, im.x, im.y);
            }
            W[pj * S::WP + o] = v;
        }
        if (n_gen)                                     // uniform; each entry by the thread that wrote it
            for (int x = tid; x < n_p * N3P; x += NT) {
                const int pj = x / N3P, o = x - pj * N3P, a = o / N2P, b = o / C2 % NB, c = 2 * (o % C2);
                const int *x1 = t.kk + 3 * q_sm[1][pj], *x2 = t.kk + 3 * q_sm[2][pj];
                float4 v = W[pj * S::WP + o];
                const int key = 3 * NA * NA * NA + ((a / 3) * NA + b / 3) * NA, f = 9 * (a % 3) + 3 * (b % 3);
                const double2 g = phase_sum(t, key + c / 3, f + c % 3, x1[0], x1[1], x1[2], x2[0], x2[1], x2[2]);
                v.x += (float)g.x;
                v.z += (float)g.y;
                if (c + 1 < NB) {
                    const double2 h = phase_sum(t, key + (c + 1) / 3, f + (c + 1) % 3, x1[0], x1[1], x1[2], x2[0],
                                                x2[1], x2[2]);
                    v.y += (float)h.x;
                    v.w += (float)h.y;
                }
                W[pj * S::WP + o] = v;
            }
#pragma unroll 2
        for (int x = tid; x < n_p * (N2 + N2P); x += NT) {
            const int pj = x / (N2 + N2P), o = x - pj * (N2 + N2P);
            E[pj * S::EP + o] = o < N2 ? __ldg(e1_all + (size_t)q_sm[1][pj] * N2 + o)
                                       : __ldg(e2_all + (size_t)q_sm[2][pj] * N2P + o - N2);
        }
        for (int x = tid; x < n_p * 2 * NB; x += NT) {
            const int pj = x / (2 * NB), e = x - pj * 2 * NB, k = e / NB;
            const float4 v = __ldg(d.wn32 + (size_t)q_sm[1 + k][pj] * NB + e - k * NB);
            F[pj * S::FP + e] = v;
            IW[x] = v.x > 0.f ? 1.0f / v.x : 0.f;
        }
        const int q = act && jl < n_p ? q_sm[0][jl] : 0;
        const float4 own = act && jl < n_p ? __ldg(d.wn32 + (size_t)q * NB + s) : make_float4(0.f, 0.f, 0.f, 0.f);
        const bool run = own.x > 0.f;
        __syncthreads();
        float2 Yr[NB][C2], Yi[NB][C2];
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int c = 0; c < C2; ++c) Yr[b][c] = Yi[b][c] = make_float2(0.f, 0.f);
        if (run) {
            const float4 *Wj = W + jl * S::WP;
#pragma unroll 1
            for (int a = 0; a < NB; ++a) {
                const float2 ev = __ldg(epsT + (size_t)q * N2 + a * NB + s);
                const float2 ex = make_float2(ev.x, ev.x), ey = make_float2(ev.y, ev.y), en = make_float2(-ev.y, -ev.y);
#pragma unroll
                for (int b = 0; b < NB; ++b)
#pragma unroll
                    for (int c = 0; c < C2; ++c) {
                        const float4 v = Wj[a * N2P + b * C2 + c];
                        const float2 vr = make_float2(v.x, v.y), vi = make_float2(v.z, v.w);
                        Yr[b][c] = __ffma2_rn(ex, vr, Yr[b][c]);
                        Yi[b][c] = __ffma2_rn(ex, vi, Yi[b][c]);
                        Yr[b][c] = __ffma2_rn(en, vi, Yr[b][c]);
                        Yi[b][c] = __ffma2_rn(ey, vr, Yi[b][c]);
                    }
            }
        }
        __syncthreads();                               // W has been read: T' takes its place
        float *out = sums + tid * S::SP;
#pragma unroll
        for (int x = 0; x <= 2 * NB; ++x) out[x] = 0.f;
        if (run) {
            float4 *Tt = W + jl * S::WP + s * S::TP;
            const float4 *e1 = E + jl * S::EP, *e2 = e1 + N2;
            const float4 *f1 = F + jl * S::FP, *f2 = f1 + NB;
            const float *i1 = IW + jl * 2 * NB, *i2 = i1 + NB;
            const F2 w0p{own.x, own.y}, n0p{own.z, own.w};
            unsigned long long todo = 0;
#pragma unroll 1
            for (int sp = 0; sp < NB; ++sp) {
                // T'(s', c) = sum_b eps'(b, s') Y(b, c)
                float2 ta[C2], tb[C2], ti[C2];
#pragma unroll
                for (int c = 0; c < C2; ++c) ta[c] = tb[c] = ti[c] = make_float2(0.f, 0.f);
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    const float4 v = e1[sp * NB + b];
                    const float2 vx = make_float2(v.x, v.y), vy = make_float2(v.z, v.w);
#pragma unroll
                    for (int c = 0; c < C2; ++c) {
                        ta[c] = __ffma2_rn(vx, Yr[b][c], ta[c]);
                        tb[c] = __ffma2_rn(vy, Yi[b][c], tb[c]);
                        ti[c] = __ffma2_rn(vx, Yi[b][c], ti[c]);
                        ti[c] = __ffma2_rn(vy, Yr[b][c], ti[c]);
                    }
                }
#pragma unroll
                for (int c = 0; c < C2; ++c)
                    Tt[sp * C2 + c] = make_float4(ta[c].x - tb[c].x, ta[c].y - tb[c].y, ti[c].x, ti[c].y);
                // the s'' near a window: high parts only, the window widened by more
                // than the low parts and the roundings
                const float w1 = f1[sp].x;
                if (!(w1 > 0.f)) continue;
                const float a = own.x + w1, b = own.x - w1, mc = cut + edge + 1e-6f * a;
#pragma unroll
                for (int spp = 0; spp < NB; ++spp) {
                    const float w2 = f2[spp].x;
                    const bool near = w2 > 0.f && (fabsf(a - w2) < mc || fabsf(b - w2) < mc || fabsf(b + w2) < mc);
                    todo |= (unsigned long long)near << (sp * NB + spp);
                }
            }
            const float iw = 1.0f / own.x;
            unsigned hits = 0;
            float part = 0.f;
            while (todo) {
                const int e = __ffsll((long long)todo) - 1;
                todo &= todo - 1;
                const int sp = e / NB, spp = e - sp * NB;
                const float4 a = f1[sp], b = f2[spp];
                const F2 w1p{a.x, a.y}, w2p{b.x, b.y}, n1p{a.z, a.w}, n2p{b.z, b.w};
                const F2 sump = f2_add(w0p, w1p), difp = f2_add(w0p, f2_neg(w1p));
                const float s3 = f2_diff(sump, w2p), s1 = f2_diff(difp, w2p), s2 = f2_diff(difp, f2_neg(w2p));
                const bool h3 = fabsf(s3) < cut, h1 = fabsf(s1) < cut, h2 = fabsf(s2) < cut;
                if (fabsf(fabsf(s3) - cut) < edge || fabsf(fabsf(s1) - cut) < edge || fabsf(fabsf(s2) - cut) < edge)
                    hits += window_hits6({w0p, w1p, w2p}, cut);
                else
                    hits += 2u * ((unsigned)(h3 || h1) + (unsigned)(h3 || h2) + (unsigned)(h1 || h2));
                if (!(h3 || h1 || h2)) continue;
                // phi(s', s'') = sum_c T'(s', c) conj eps''(c, s'')
                float2 fa = make_float2(0.f, 0.f), fb = fa, fi = fa;
#pragma unroll
                for (int c = 0; c < C2; ++c) {
                    const float4 u = Tt[sp * C2 + c], v = e2[spp * C2 + c];
                    const float2 ur = make_float2(u.x, u.y), ui = make_float2(u.z, u.w);
                    const float2 vr = make_float2(v.x, v.y), vi = make_float2(v.z, v.w);
                    fa = __ffma2_rn(ur, vr, fa);
                    fb = __ffma2_rn(ui, vi, fb);
                    fi = __ffma2_rn(ur, vi, fi);
                    fi = __ffma2_rn(ui, vr, fi);
                }
                const float fr = (fa.x + fa.y) - (fb.x + fb.y), fm = fi.x + fi.y;
                const float ff = fr * fr + fm * fm;
                const float2 g31 = delta_shape2<SHAPE>(make_float2(s3, s1), par);
                const float g3 = h3 ? g31.x : 0.f, g1 = h1 ? g31.y : 0.f;
                const float g2 = h2 ? delta_shape2<SHAPE>(make_float2(s2, s2), par).x : 0.f;
                const float j1 = i1[sp], j2 = i2[spp];
                part += ff * (f2_diff(n1p, n2p) * (g3 - g2) + (1.f + a.z + b.z) * g1) * j1 * j2;
                out[sp] += iw * ff * (f2_diff(n0p, n2p) * (g3 - g1) + (1.f + own.z + b.z) * g2) * j2;
                out[NB + spp] += iw * ff * (f2_diff(n0p, n1p) * (g2 - g1) + (1.f + own.z + a.z) * g3) * j1;
            }
            out[2 * NB] = part;
            allowed += (unsigned long long)orbit[base + jl] * hits;
        }
        __syncthreads();
        for (int x = tid; x < n_p * 3 * NB; x += NT) {
            const int pj = x / (3 * NB), e = x - pj * 3 * NB;
            const float *v = sums + pj * NB * S::SP;
            float r;
            if (e < NB) {
                r = v[e * S::SP + 2 * NB];
            } else {
                r = v[e - NB];
#pragma unroll
                for (int y = 1; y < NB; ++y) r += v[y * S::SP + e - NB];
            }
            out3[(size_t)base * 3 * NB + x] = r;
        }
    }
    for (int o = 16; o > 0; o >>= 1) allowed += __shfl_xor_sync(0xffffffffu, allowed, o);
    if ((tid & 31) == 0 && allowed) atomicAdd(d.allowed, allowed);
}

template <int NB, int NT, int SHAPE>
cudaError_t run_sn_orbit32(const LwParams &p, const LwDev &d, const SnTables &t, const OrbitPlan &o, float *out3, int sms,
                           const float4 *e1, const float4 *e2, cudaStream_t st) {
    using S = SnOrb32<NB, NT>;
    auto k = sn_orbit32_kernel<NB, NT, SHAPE>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kBytes);
    if (e != cudaSuccess) return e;
    // up to 16 passes per CTA, fewer where that leaves less than 16 CTAs per SM
    const long long all = ((long long)o.n_pairs + S::kPairs - 1) / S::kPairs;
    const int passes = (int)std::max(1LL, std::min(16LL, all / (16LL * std::max(1, sms))));
    k<<<counted((unsigned)((all + passes - 1) / passes)), NT, S::kBytes, st>>>(
        p, d, t, static_cast<const float4 *>(t.tab), static_cast<const float2 *>(d.eps_work), e1, e2, o.n_pairs, passes,
        o.pairs, o.orbit, out3);
    return cudaGetLastError();
}
template <int NB, int NT>
cudaError_t run_sn_orbit32(const LwParams &p, const LwDev &d, const SnTables &t, const OrbitPlan &o, float *out3, int sms,
                           cudaStream_t st) {
    float4 *e1 = reinterpret_cast<float4 *>(out3 + ws_round(sn_orbit_bytes(NB, o.n_pairs, 1)) / sizeof(float));
    float4 *e2 = e1 + ws_round(sizeof(float4) * (size_t)p.nq * NB * NB) / sizeof(float4);
    sn_pack_kernel<NB><<<counted((unsigned)(((size_t)p.nq * NB * NB + 127) / 128)), 128, 0, st>>>(
        p.nq, static_cast<const float2 *>(d.eps_work), e1, e2);
    return p.shape == kDeltaGauss     ? run_sn_orbit32<NB, NT, kDeltaGauss>(p, d, t, o, out3, sms, e1, e2, st)
           : p.shape == kDeltaLorentz ? run_sn_orbit32<NB, NT, kDeltaLorentz>(p, d, t, o, out3, sms, e1, e2, st)
                                      : run_sn_orbit32<NB, NT, kDeltaTriangle>(p, d, t, o, out3, sms, e1, e2, st);
}

template <int NB, int NT>
cudaError_t run_sn_orbits_nt(const LwParams &p, const LwDev &d, const SnTables &t, const OrbitPlan &o, double *out3,
                             int sms, cudaStream_t st) {
    using S = SnOrb<NB, NT>;
    auto k = sn_orbit_kernel<NB, NT>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kBytes);
    if (e != cudaSuccess) return e;
    // up to 16 passes per CTA, fewer where that leaves less than 16 CTAs per SM
    const long long all = ((long long)o.n_pairs + S::kPairs - 1) / S::kPairs;
    const int passes = (int)std::max(1LL, std::min(16LL, all / (16LL * std::max(1, sms))));
    k<<<counted((unsigned)((all + passes - 1) / passes)), NT, S::kBytes, st>>>(
        p, d, t, static_cast<const double2 *>(t.tab), static_cast<const double2 *>(d.eps_work), o.n_pairs, passes,
        o.pairs, o.orbit, out3);
    return cudaGetLastError();
}
template <typename R, int NB>
cudaError_t run_sn_orbits(const LwParams &p, const LwDev &d, const SnTables &t, const OrbitPlan &o, R *out3, int sms,
                          cudaStream_t st) {
    using R2 = typename Cx<R>::T;
    R2 *tab = static_cast<R2 *>(t.tab);
    constexpr bool f32 = sizeof(R) == 4;
    if (tab) sn_tables_kernel<R, NB, f32><<<counted(p.nq), kSnThreads, 0, st>>>(p.nq, t, tab);
    ProfMark pm(p.prof, KALD_PROF_SMALL_NB, st);
    // 128 threads; 64 where the pairs are too few for two such CTAs per SM
    const bool many = (long long)o.n_pairs * NB >= 256LL * std::max(1, sms);
    cudaError_t e;
    if constexpr (f32)
        e = many ? run_sn_orbit32<NB, 128>(p, d, t, o, out3, sms, st) : run_sn_orbit32<NB, 64>(p, d, t, o, out3, sms, st);
    else
        e = many ? run_sn_orbits_nt<NB, 128>(p, d, t, o, out3, sms, st)
                 : run_sn_orbits_nt<NB, 64>(p, d, t, o, out3, sms, st);
    if (e == cudaSuccess) e = launch_orbit_class_sums(o, p.nb, out3, d.partial, st);
    pm.end();
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename R, int NB, bool BTE = false>
cudaError_t run_sn(const LwParams &p, const LwDev &d, const SnTables &t, cudaStream_t st) {
    using R2 = typename Cx<R>::T;
    R2 *tab = static_cast<R2 *>(t.tab);
    if (tab) sn_tables_kernel<R, NB><<<counted(p.nq), kSnThreads, 0, st>>>(p.nq, t, tab);
    ProfMark pm(p.prof, KALD_PROF_SMALL_NB, st);
    sn_kernel<R, NB, BTE><<<counted(dim3(p.nqc, p.n_chunks)), kSnThreads, 0, st>>>(
        p, d, t, tab, static_cast<const R2 *>(d.eps_work));
    pm.end();
    return cudaGetLastError();
}

}  // namespace

bool sn_supported(int nb) { return nb == 3 || nb == 6; }

// q' per CTA: up to eight passes over the CTA's lanes, fewer where the mesh is
// too coarse to give every SM about four CTAs.  From the mesh alone, not from the
// q-points of a call: a q-point's sums do not depend on the call.
int sn_chunk(int nb, int nq, int sm_count) {
    const int lanes = kSnThreads / nb;
    const long long rows = nq / 2 + 1, passes = (nq + lanes - 1) / lanes;
    const long long ctas = 4LL * std::max(1, sm_count);
    return lanes * (int)std::max(1LL, std::min(8LL, rows * passes / ctas));
}
size_t sn_table_bytes(int nb, int nq, int fp32) {
    // (FP32: columns in pairs, the last one of three branches padded)
    const size_t cols = fp32 ? (nb + 1) / 2 * 2 : nb;
    return (fp32 ? sizeof(float2) : sizeof(double2)) * 3 * (size_t)nq * nb * nb * cols;
}

// The blocks ordered by class (0: Rk = 0, 1: Rj = 0, 2: Rj = Rk, 3: the rest)
// and, inside a class, by the atom triple (i, j, k); start [4 n_atoms^3 + 1].
// Without tables every block is of class 3.
void plan_sn(const HostSystem &h, bool tables, std::vector<int> &order, std::vector<int> &start) {
    const int na = h.n_atoms, n = (int)h.fc3_i.size(), keys = 4 * na * na * na;
    std::vector<int> key(n);
    start.assign(keys + 1, 0);
    for (int b = 0; b < n; ++b) {
        const int *rj = &h.rep_int[3 * (size_t)h.fc3_rj[b]], *rk = &h.rep_int[3 * (size_t)h.fc3_rk[b]];
        const bool zj = !rj[0] && !rj[1] && !rj[2], zk = !rk[0] && !rk[1] && !rk[2];
        const int cls = !tables ? 3 : zk ? 0 : zj ? 1 : h.fc3_rj[b] == h.fc3_rk[b] ? 2 : 3;
        key[b] = ((cls * na + h.fc3_i[b]) * na + h.fc3_atoms[3 * (size_t)b + 1]) * na + h.fc3_atoms[3 * (size_t)b + 2];
        ++start[key[b] + 1];
    }
    for (int k = 0; k < keys; ++k) start[k + 1] += start[k];
    std::vector<int> at(start.begin(), start.end() - 1);
    order.resize(n);
    for (int b = 0; b < n; ++b) order[at[key[b]]++] = b;
}

cudaError_t launch_lw_small(const LwParams &p, const LwDev &d, const SnTables &t, int fp32, const OrbitPlan *orb,
                            void *out3, int sms, cudaStream_t st) {
    if (!sn_supported(p.nb) || t.L < 1 || t.m0 < 0) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(d.allowed, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    roots_kernel<<<counted((2 * t.m0 + 1 + 255) / 256), 256, 0, st>>>(t.L, t.m0, t.roots);
    if (orb) {
        if (fp32)
            return p.nb == 3 ? run_sn_orbits<float, 3>(p, d, t, *orb, static_cast<float *>(out3), sms, st)
                             : run_sn_orbits<float, 6>(p, d, t, *orb, static_cast<float *>(out3), sms, st);
        return p.nb == 3 ? run_sn_orbits<double, 3>(p, d, t, *orb, static_cast<double *>(out3), sms, st)
                         : run_sn_orbits<double, 6>(p, d, t, *orb, static_cast<double *>(out3), sms, st);
    }
    if (fp32) return p.nb == 3 ? run_sn<float, 3>(p, d, t, st) : run_sn<float, 6>(p, d, t, st);
    if (p.bte) return p.nb == 3 ? run_sn<double, 3, true>(p, d, t, st) : run_sn<double, 6, true>(p, d, t, st);
    return p.nb == 3 ? run_sn<double, 3>(p, d, t, st) : run_sn<double, 6>(p, d, t, st);
}

}  // namespace kald
