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
// CTA = (q, chunk of q'), thread = (q' lane, mode s); every thread walks its
// q' of the chunk in order, the CTA adds the lanes of each mode in order and
// writes one FP64 partial per (q, chunk, s) for lw_finish.

#include <algorithm>
#include <type_traits>
#include <vector>

#include "kald_internal.h"
#include "wdiff.cuh"

namespace kald {
namespace {

template <typename R> struct Cx;
template <> struct Cx<float> { using T = float2; };
template <> struct Cx<double> { using T = double2; };

constexpr int kSnThreads = 256;

template <typename R2>
__device__ __forceinline__ R2 cmul(R2 a, R2 b) {
    R2 r;
    r.x = a.x * b.x - a.y * b.y;
    r.y = a.x * b.y + a.y * b.x;
    return r;
}
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
// acc += v * e (v real)
__device__ __forceinline__ void rfma(double2 &acc, double v, double2 e) {
    acc.x = fma(v, e.x, acc.x);
    acc.y = fma(v, e.y, acc.y);
}
__device__ __forceinline__ void rfma(float2 &acc, float v, float2 e) {
    acc = __ffma2_rn(make_float2(v, v), e, acc);
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
// scaled mesh coordinates of q' and q'' (one of them zero for a table); FP64.
__device__ __forceinline__ double2 phase_sum(const SnTables &t, int key, int v, int x0, int x1, int x2, int y0, int y1,
                                             int y2) {
    double2 acc = make_double2(0.0, 0.0);
    for (int bl = t.start[key]; bl < t.start[key + 1]; ++bl) {
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
template <typename R, int NB>
__global__ void __launch_bounds__(kSnThreads)
sn_tables_kernel(int nq, SnTables t, typename Cx<R>::T *__restrict__ tab) {
    using R2 = typename Cx<R>::T;
    constexpr int N3 = NB * NB * NB, NA = NB / 3;
    const int q = blockIdx.x;
    const int k0 = t.kk[3 * q], k1 = t.kk[3 * q + 1], k2 = t.kk[3 * q + 2];
    for (int x = threadIdx.x; x < 3 * N3; x += kSnThreads) {
        const int cls = x / N3, e = x - cls * N3;
        const int a = e / (NB * NB), b = (e / NB) % NB, c = e % NB;
        const int key = cls * NA * NA * NA + ((a / 3) * NA + b / 3) * NA + c / 3;
        const int v = 9 * (a % 3) + 3 * (b % 3) + c % 3;
        const double2 s = cls == 0 ? phase_sum(t, key, v, k0, k1, k2, 0, 0, 0)
                                   : phase_sum(t, key, v, 0, 0, 0, k0, k1, k2);
        R2 o;
        o.x = (R)s.x;
        o.y = (R)s.y;
        tab[((size_t)cls * nq + q) * N3 + e] = o;
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
// One call, two-atom cell, 24^3 mesh, FP32: 1367 ms before, 191 ms now.
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
    return (fp32 ? sizeof(float2) : sizeof(double2)) * 3 * (size_t)nq * nb * nb * nb;
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

cudaError_t launch_lw_small(const LwParams &p, const LwDev &d, const SnTables &t, int fp32, cudaStream_t st) {
    if (!sn_supported(p.nb) || t.L < 1 || t.m0 < 0) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(d.allowed, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    roots_kernel<<<counted((2 * t.m0 + 1 + 255) / 256), 256, 0, st>>>(t.L, t.m0, t.roots);
    if (fp32) return p.nb == 3 ? run_sn<float, 3>(p, d, t, st) : run_sn<float, 6>(p, d, t, st);
    if (p.bte) return p.nb == 3 ? run_sn<double, 3, true>(p, d, t, st) : run_sn<double, 6, true>(p, d, t, st);
    return p.nb == 3 ? run_sn<double, 3>(p, d, t, st) : run_sn<double, 6>(p, d, t, st);
}

}  // namespace kald
