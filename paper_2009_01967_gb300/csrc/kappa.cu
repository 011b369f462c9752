// Thermal conductivity on the GPU, FP64 throughout.
//
// BTE-RTA (paper Eq. RTA, Eq. heat_capacity): kappa = 1/(N_k V) sum c tau v v,
// tau = 1/(2 gamma), c = kB x^2 e^x/(e^x - 1)^2; inside a degenerate set D of
// one q, v_a v_b -> sum_{s,s' in D} Re(V^a_{ss'} conj(V^b_{ss'})) with
// V^a_{ss'} = eta_s^dagger dD/dq_a eta_s' / (2 sqrt(w_s w_s')).
//
// QHGK (Eq. conductivity_amorphous, twod_heat_capacity, generalized_velocity,
// lorentzian_amorphous) for Gamma-only systems: W_a = E^T A_a E / (2 sqrt(w w')),
// A_a(i, j) = sum_L (x_i - x_j - L)_a Phi2(i, jL)/sqrt(mi mj), then
// kappa_ab = 1/V sum_{mu mu'} c_{mu mu'} tau_{mu mu'} W_a W_b.

#include <algorithm>

#include "kald_internal.h"

namespace kald {
namespace {

__device__ __forceinline__ double2 cmulc(double2 a, double2 b) {   // conj(a) * b
    return make_double2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}

__device__ __forceinline__ double heat_cap(double w, double T, int classical) {
    if (!(w > 0.0)) return 0.0;
    if (classical) return kKbJK;
    const double x = kHbarEvPs * w / (kKbEvK * T);
    const double ex = exp(-x);
    const double den = 1.0 - ex;
    return kKbJK * x * x * ex / (den * den);
}

__device__ __forceinline__ double bose(double w, double T, int classical) {
    if (!(w > 0.0)) return 0.0;
    const double x = kHbarEvPs * w / (kKbEvK * T);
    return classical ? 1.0 / x : 1.0 / expm1(fmin(x, 700.0));
}

// Fixed-order block reduction of 9 values; result valid in thread 0.
__device__ void block_reduce9(double v[9], double *sm /*[nwarps][9]*/) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    for (int a = 0; a < 9; ++a) {
        double x = v[a];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) sm[warp * 9 + a] = x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int a = 0; a < 9; ++a) {
            double t = 0.0;
            for (int w = 0; w < nw; ++w) t += sm[w * 9 + a];
            v[a] = t;
        }
    }
    __syncthreads();
}

constexpr int kRtaThreads = 128;
constexpr int kRtaChunk = 256;       // fc2 blocks staged per pass
constexpr int kRtaTasks = 1024;      // (s, s') pairs per round (8 per thread)

// One CTA per q.  Thread 0 sorts the modes, forms the degenerate sets and
// lists the (s, s') pairs inside each participating set; the pairs are
// dealt to threads (8 each per round), and each thread accumulates
// V^a_{ss'} over the fc2 blocks, staged in chunks with their phases.
__global__ void __launch_bounds__(kRtaThreads)
kappa_rta_kernel(DevFc2 f, int nb, const double *__restrict__ qcart, const double *__restrict__ nu,
                 const double2 *__restrict__ eig, const double *__restrict__ gamma, double T,
                 int classical, double omega_min_thz, double degen_tol, double *__restrict__ partial) {
    __shared__ int order[kMaxNbSmall];
    __shared__ int set_start[kMaxNbSmall + 1];
    __shared__ int set_id[kMaxNbSmall];
    __shared__ double ct[kMaxNbSmall];
    __shared__ double2 ph[kRtaChunk];
    __shared__ double rc[kRtaChunk][3];
    __shared__ int bi[kRtaChunk], bj[kRtaChunk];
    __shared__ short2 task[kRtaTasks];
    __shared__ int n_task_sm, n_sets_sm;
    __shared__ double red[(kRtaThreads / 32) * 9];
    const int q = blockIdx.x, tid = threadIdx.x;
    const double *v = nu + (size_t)q * nb;
    const double *g = gamma + (size_t)q * nb;
    if (tid == 0) {
        for (int s = 0; s < nb; ++s) order[s] = s;
        for (int a = 1; a < nb; ++a) {
            const int x = order[a];
            int b = a - 1;
            while (b >= 0 && v[order[b]] > v[x]) { order[b + 1] = order[b]; --b; }
            order[b + 1] = x;
        }
        int start = 0, sid = 0;
        set_start[0] = 0;
        for (int a = 1; a <= nb; ++a) {
            if (a == nb || v[order[a]] - v[order[a - 1]] >= degen_tol) {
                double acc = 0.0;
                int cnt = 0;
                for (int b = start; b < a; ++b) {
                    const int s = order[b];
                    const bool ok = (v[s] > omega_min_thz) && (g[s] > 0.0);
                    set_id[s] = ok ? sid : -1;
                    if (ok) { acc += heat_cap(kTwoPi * v[s], T, classical) / (2.0 * g[s]); ++cnt; }
                }
                ct[sid] = cnt ? acc / cnt : 0.0;
                ++sid;
                set_start[sid] = a;
                start = a;
            }
        }
        n_sets_sm = sid;
    }
    __syncthreads();
    const int n_sets = n_sets_sm;
    const double qx = qcart[3 * q], qy = qcart[3 * q + 1], qz = qcart[3 * q + 2];
    const double2 *E = eig + (size_t)q * nb * nb;
    const int n_blk = f.pair_start[f.n_pairs];
    double acc[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    int skip = 0;                                 // tasks already done in earlier rounds
    for (;;) {
        if (tid == 0) {
            int n = 0, seen = 0;
            for (int d = 0; d < n_sets && n < kRtaTasks; ++d)
                for (int a = set_start[d]; a < set_start[d + 1] && n < kRtaTasks; ++a)
                    for (int b = set_start[d]; b < set_start[d + 1] && n < kRtaTasks; ++b) {
                        const int s = order[a], t = order[b];
                        if (set_id[s] < 0 || set_id[t] < 0) continue;
                        if (seen++ < skip) continue;
                        task[n++] = make_short2((short)s, (short)t);
                    }
            n_task_sm = n;
        }
        __syncthreads();
        const int n_task = n_task_sm;
        if (n_task == 0) break;
        double2 V[8][3];
        for (int u = 0; u < 8; ++u)
            for (int a = 0; a < 3; ++a) V[u][a] = make_double2(0.0, 0.0);
        for (int c0 = 0; c0 < n_blk; c0 += kRtaChunk) {
            const int c1 = min(n_blk, c0 + kRtaChunk);
            __syncthreads();
            for (int b = c0 + tid; b < c1; b += kRtaThreads) {
                const double *R = f.rcart + 3 * b;
                double sn, cn;
                sincos(qx * R[0] + qy * R[1] + qz * R[2], &sn, &cn);
                ph[b - c0] = make_double2(cn, -sn);
                rc[b - c0][0] = R[0]; rc[b - c0][1] = R[1]; rc[b - c0][2] = R[2];
                int lo = 0, hi = f.n_pairs - 1;           // block -> atom pair
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (f.pair_start[mid] <= b) lo = mid; else hi = mid - 1;
                }
                bi[b - c0] = f.pair_i[lo];
                bj[b - c0] = f.pair_j[lo];
            }
            __syncthreads();
            for (int u = 0; u < 8; ++u) {
                const int x = tid + u * kRtaThreads;
                if (x >= n_task) break;
                const double2 *es = E + (size_t)task[x].x * nb;
                const double2 *et = E + (size_t)task[x].y * nb;
                for (int b = c0; b < c1; ++b) {
                    const int i = bi[b - c0], j = bj[b - c0];
                    double2 h = make_double2(0.0, 0.0);
                    for (int a = 0; a < 3; ++a) {
                        double2 t = make_double2(0.0, 0.0);
                        for (int c = 0; c < 3; ++c) {
                            const double bv = f.blk[9 * b + 3 * a + c];
                            const double2 ej = et[3 * j + c];
                            t.x += bv * ej.x; t.y += bv * ej.y;
                        }
                        const double2 r = cmulc(es[3 * i + a], t);
                        h.x += r.x; h.y += r.y;
                    }
                    const double2 z = make_double2(ph[b - c0].x * h.x - ph[b - c0].y * h.y,
                                                   ph[b - c0].x * h.y + ph[b - c0].y * h.x);
                    // dD/dq_a carries (-i R_a): (-i R_a) z = R_a (z.y - i z.x)
                    for (int a = 0; a < 3; ++a) {
                        V[u][a].x += rc[b - c0][a] * z.y;
                        V[u][a].y -= rc[b - c0][a] * z.x;
                    }
                }
            }
        }
        for (int u = 0; u < 8; ++u) {
            const int x = tid + u * kRtaThreads;
            if (x >= n_task) break;
            const int s = task[x].x, t = task[x].y;
            const double ws = kTwoPi * v[s], wt = kTwoPi * v[t];
            const double sc = kEvA2AmuPs2 / (2.0 * sqrt(ws * wt));
            const double w8 = ct[set_id[s]] * sc * sc;
            for (int a = 0; a < 3; ++a)
                for (int b = 0; b < 3; ++b)
                    acc[3 * a + b] += w8 * (V[u][a].x * V[u][b].x + V[u][a].y * V[u][b].y);
        }
        skip += n_task;
        __syncthreads();
        if (n_task < kRtaTasks) break;
    }
    block_reduce9(acc, red);
    if (tid == 0)
        for (int a = 0; a < 9; ++a) partial[(size_t)q * 9 + a] = acc[a];
}

// kappa_RTA of one q per CTA from the diagonal elements: ranks, degenerate
// sets and their mean c tau formed by one thread per mode; the elements
// between different modes of one set (rare in disordered cells) over ordered
// atom pairs whose blocks are summed once, in shared memory, for all pairs of modes.
// One thread sorting the modes and every (s, s') running over all blocks took
// 12.2 ms for 32 atoms and 512 q-points; with velocity.cu 2.6 ms now.
constexpr int kRtaPairs = 8;         // ordered atom pairs per pass
__global__ void __launch_bounds__(kRtaThreads)
kappa_rta_diag_kernel(DevFc2 f, int nb, const double *__restrict__ qcart, const double *__restrict__ nu,
                      const double2 *__restrict__ eig, const double *__restrict__ gamma, const int *__restrict__ src,
                      const double *__restrict__ vre, const double *__restrict__ vim,
                      const double2 *__restrict__ phases, int n_blk, double T, int classical, double omega_min_thz,
                      double degen_tol, double *__restrict__ partial) {
    __shared__ double v[kMaxNbSmall], ct[kMaxNbSmall];
    __shared__ int order[kMaxNbSmall], set_of[kMaxNbSmall], start[kMaxNbSmall + 1];   // set_of[s]: -1 takes no part
    __shared__ unsigned starts[kRtaThreads / 32];
    __shared__ short2 task[kRtaTasks];
    __shared__ double2 M[kRtaPairs * 27];
    __shared__ int n_task_sm;
    __shared__ double red[(kRtaThreads / 32) * 9];
    const int q = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double *g = gamma + (size_t)q * nb;
    if (tid < nb) v[tid] = nu[(size_t)q * nb + tid];
    __syncthreads();
    if (tid < nb) {                                // ascending, ties by index, NaN last
        const double x = v[tid];
        int r = 0;
        for (int t = 0; t < nb; ++t) {
            const double y = v[t];
            const bool lt = y < x || (x != x && y == y);
            const bool gt = y > x || (y != y && x == x);
            r += lt || (!gt && t < tid);
        }
        order[r] = tid;
    }
    __syncthreads();
    const bool first = tid < nb && (tid == 0 || v[order[tid]] - v[order[tid - 1]] >= degen_tol);
    const unsigned bal = __ballot_sync(0xffffffffu, first);
    if (lane == 0) starts[warp] = bal;
    __syncthreads();
    int sid = __popc(starts[warp] & (0xffffffffu >> (31 - lane))) - 1, n_sets = 0;
    for (int w = 0; w < kRtaThreads / 32; ++w) {
        if (w < warp) sid += __popc(starts[w]);
        n_sets += __popc(starts[w]);
    }
    if (first) start[sid] = tid;
    if (tid == 0) start[n_sets] = nb;
    __syncthreads();
    int many = 0;
    if (tid < n_sets) {
        double acc = 0.0;
        int cnt = 0;
        for (int b = start[tid]; b < start[tid + 1]; ++b) {
            const int s = order[b];
            const bool ok = (v[s] > omega_min_thz) && (g[s] > 0.0);
            set_of[s] = ok ? tid : -1;
            if (ok) { acc += heat_cap(kTwoPi * v[s], T, classical) / (2.0 * g[s]); ++cnt; }
        }
        ct[tid] = cnt ? acc / cnt : 0.0;
        many = cnt > 1;
    }
    many = __syncthreads_or(many);
    double acc[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    if (tid < nb && set_of[tid] >= 0) {
        const size_t o = ((size_t)src[q] * nb + tid) * 3;
        const double sc = kEvA2AmuPs2 / (2.0 * (kTwoPi * v[tid]));
        const double w8 = ct[set_of[tid]] * sc * sc;
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b)
                acc[3 * a + b] = w8 * (vre[o + a] * vre[o + b] + (vim ? vim[o + a] * vim[o + b] : 0.0));
    }
    if (many) {
        // pairs of different modes inside a set: s < s' counted twice when dD is
        // Hermitian (symmetric Phi2), every ordered pair otherwise
        const bool herm = vim == nullptr;
        const double qx = qcart[3 * q], qy = qcart[3 * q + 1], qz = qcart[3 * q + 2];
        const double2 *E = eig + (size_t)q * nb * nb;
        for (int skip = 0;;) {
            if (tid == 0) {
                int n = 0, seen = 0;
                for (int d = 0; d < n_sets && n < kRtaTasks; ++d)
                    for (int a = start[d]; a < start[d + 1] && n < kRtaTasks; ++a)
                        for (int b = herm ? a + 1 : start[d]; b < start[d + 1] && n < kRtaTasks; ++b) {
                            const int s = order[a], t = order[b];
                            if (a == b || set_of[s] < 0 || set_of[t] < 0) continue;
                            if (seen++ < skip) continue;
                            task[n++] = make_short2((short)s, (short)t);
                        }
                n_task_sm = n;
            }
            __syncthreads();
            const int n_task = n_task_sm;
            if (n_task == 0) break;
            double2 V[8][3];
            for (int u = 0; u < 8; ++u)
                for (int a = 0; a < 3; ++a) V[u][a] = make_double2(0.0, 0.0);
            for (int p0 = 0; p0 < f.n_pairs; p0 += kRtaPairs) {
                const int n_p = min(kRtaPairs, f.n_pairs - p0);
                __syncthreads();
                // (several threads per pair and element where there are few pairs)
                const int parts = max(1, min(kRtaThreads / (9 * n_p), kRtaPairs / n_p));
                for (int x = tid; x < 9 * n_p * parts; x += kRtaThreads) {
                    const int pp = x / 9, part = pp / n_p, p = pp - part * n_p, ab = x - 9 * pp;
                    double2 m[3];
                    for (int a = 0; a < 3; ++a) m[a] = make_double2(0.0, 0.0);
                    for (int b = f.pair_start[p0 + p] + part; b < f.pair_start[p0 + p + 1]; b += parts) {
                        const double *R = f.rcart + 3 * (size_t)b;
                        double sn, cn;
                        if (phases) {
                            const double2 z = phases[(size_t)q * n_blk + b];
                            cn = z.x;
                            sn = -z.y;
                        } else {
                            sincos(qx * R[0] + qy * R[1] + qz * R[2], &sn, &cn);
                        }
                        const double bv = f.blk[9 * (size_t)b + ab];
                        // (-i R_a) exp(-i q.R) = -R_a sin - i R_a cos
                        for (int a = 0; a < 3; ++a) {
                            m[a].x -= R[a] * (bv * sn);
                            m[a].y -= R[a] * (bv * cn);
                        }
                    }
                    for (int a = 0; a < 3; ++a) M[27 * pp + 3 * ab + a] = m[a];
                }
                __syncthreads();
                if (parts > 1) {
                    for (int x = tid; x < 27 * n_p; x += kRtaThreads) {
                        double2 m = M[x];
                        for (int k = 1; k < parts; ++k) {
                            const double2 z = M[27 * n_p * k + x];
                            m.x += z.x;
                            m.y += z.y;
                        }
                        M[x] = m;
                    }
                    __syncthreads();
                }
                for (int u = 0; u < 8; ++u) {
                    const int x = tid + u * kRtaThreads;
                    if (x >= n_task) break;
                    const double2 *es = E + (size_t)task[x].x * nb, *et = E + (size_t)task[x].y * nb;
                    for (int p = 0; p < n_p; ++p) {
                        const double2 *ei = es + 3 * f.pair_i[p0 + p], *ej = et + 3 * f.pair_j[p0 + p];
                        for (int a = 0; a < 3; ++a)
                            for (int b = 0; b < 3; ++b) {
                                const double2 P = cmulc(ei[a], ej[b]);
                                for (int c = 0; c < 3; ++c) {
                                    const double2 z = M[27 * p + 3 * (3 * a + b) + c];
                                    V[u][c].x += P.x * z.x - P.y * z.y;
                                    V[u][c].y += P.x * z.y + P.y * z.x;
                                }
                            }
                    }
                }
            }
            for (int u = 0; u < 8; ++u) {
                const int x = tid + u * kRtaThreads;
                if (x >= n_task) break;
                const int s = task[x].x, t = task[x].y;
                const double sc = kEvA2AmuPs2 / (2.0 * sqrt((kTwoPi * v[s]) * (kTwoPi * v[t])));
                const double w8 = (herm ? 2.0 : 1.0) * ct[set_of[s]] * sc * sc;
                for (int a = 0; a < 3; ++a)
                    for (int b = 0; b < 3; ++b)
                        acc[3 * a + b] += w8 * (V[u][a].x * V[u][b].x + V[u][a].y * V[u][b].y);
            }
            skip += n_task;
            __syncthreads();
            if (n_task < kRtaTasks) break;
        }
    }
    block_reduce9(acc, red);
    if (tid == 0)
        for (int a = 0; a < 9; ++a) partial[(size_t)q * 9 + a] = acc[a];
}

// out[a] = scale * sum of n partial sums: one warp per component, every lane
// its share in order, then a fixed tree (one thread per component took 12 us
// for 216 partial sums and grew with their number).
__global__ void __launch_bounds__(288)
sum_partials_kernel(int n, const double *__restrict__ partial, double scale, double *__restrict__ out) {
    const int a = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double t = 0.0;
#pragma unroll 4
    for (int x = lane; x < n; x += 32) t += partial[(size_t)x * 9 + a];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) out[a] = t * scale;
}

// ---------------------------------------------------------------- QHGK
// B_a[mu][d] = sum_e A_a[d][e] E[mu][e], rows d = 3 i + a' gathered over the
// blocks of atom i (CSR).  CTA = MU modes, their eigenvectors in shared memory
// so that a block's values are read once for all of them; one thread per row,
// three outputs (a) per mode.  Bound: FP64 units, 6 FMA per (block, row, mode).
// (SMEM false: one mode per CTA read from global memory, for eigenvectors that
// do not fit.)
template <int MU, bool SMEM = true>
__global__ void __launch_bounds__(256)
sparse_ae_kernel(DevFc2Dist f, int nb, const double2 *__restrict__ eig, double *__restrict__ B) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *E = reinterpret_cast<double *>(smem_raw);          // [MU][nb]
    const int mu0 = blockIdx.x * MU;
    for (int m = 0; m < (SMEM ? MU : 0); ++m)
        for (int x = threadIdx.x; x < nb; x += blockDim.x)
            E[m * nb + x] = mu0 + m < nb ? eig[(size_t)(mu0 + m) * nb + x].x : 0.0;
    __syncthreads();
    for (int ra = threadIdx.x; ra < 3 * f.n_rows; ra += blockDim.x) {       // 3 i + a'
        const int i = ra / 3, ap = ra - 3 * i;
        double s[MU][3];
#pragma unroll
        for (int m = 0; m < MU; ++m) s[m][0] = s[m][1] = s[m][2] = 0.0;
        for (int b = f.row_start[i]; b < f.row_start[i + 1]; ++b) {
            const int j = 3 * f.col_j[b];
            const double *blk = f.blk + 9 * (size_t)b + 3 * ap, *R = f.dist + 3 * (size_t)b;
            const double v0 = blk[0], v1 = blk[1], v2 = blk[2], r0 = R[0], r1 = R[1], r2 = R[2];
#pragma unroll
            for (int m = 0; m < MU; ++m) {
                double e0, e1, e2;
                if constexpr (SMEM) {
                    const double *e = E + m * nb + j;
                    e0 = e[0]; e1 = e[1]; e2 = e[2];
                } else {
                    const double2 *e = eig + (size_t)(mu0 + m) * nb + j;
                    e0 = e[0].x; e1 = e[1].x; e2 = e[2].x;
                }
                const double t = fma(v2, e2, fma(v1, e1, v0 * e0));
                s[m][0] = fma(r0, t, s[m][0]);
                s[m][1] = fma(r1, t, s[m][1]);
                s[m][2] = fma(r2, t, s[m][2]);
            }
        }
#pragma unroll
        for (int m = 0; m < MU; ++m)
            if (mu0 + m < nb)
#pragma unroll
                for (int a = 0; a < 3; ++a) B[((size_t)a * nb + mu0 + m) * nb + ra] = s[m][a];
    }
}

// Per mode: omega (rad/ps, 0 for a masked mode nu <= omega_min), n, c and the
// factor sqrt(C / (2 omega)) whose product over two modes scales W_a (0 masked).
__global__ void qhgk_modes_kernel(int nb, const double *__restrict__ nu, double omega_min_thz, double T, int classical,
                                  QhgkModes q) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= nb) return;
    const double w = (nu[x] > omega_min_thz) ? kTwoPi * nu[x] : 0.0;
    q.omega[x] = w;
    q.occ[x] = bose(w, T, classical);
    q.heat[x] = heat_cap(w, T, classical);
    q.fac[x] = w > 0.0 ? sqrt(0.5 * kEvA2AmuPs2 / w) : 0.0;
}

// Pair sum over the rows mu = blockIdx.x, blockIdx.x + gridDim.x, .. of the CTA,
// threads over mu'; per-CTA partial [9].  half: W is antisymmetric and formed
// on and above the diagonal only, so each pair mu < mu' counts twice (its weight
// is symmetric and W vanishes on the diagonal).  n and c come from tables per
// mode, and c tau is one quotient: an exponential and two divisions per pair
// bound this sum before (1.3 ms for 2,592 modes, 0.24 ms now).
__global__ void __launch_bounds__(256)
qhgk_pairsum_kernel(int nb, const double *__restrict__ W, QhgkModes q, const double *__restrict__ gamma, double T,
                    double degen_tol_w, double bandwidth_w, double threshold_w, int half,
                    double *__restrict__ partial) {
    __shared__ double red[8 * 9];
    double acc[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    const double mult = half ? 2.0 : 1.0;
    for (int m = blockIdx.x; m < nb; m += gridDim.x) {
        const double w1 = q.omega[m];
        const double g1 = gamma[m];
        // with a bandwidth the linewidths are not used (Allen-Feldman)
        if (!(w1 > 0.0) || (!(bandwidth_w > 0.0) && !(g1 > 0.0))) continue;
        const double n1 = q.occ[m], c1 = q.heat[m];
        // hbar w w' / T in J, ps: 1e24 from the two frequencies, 1e-12 from their difference
        const double k1 = mult * (kHbarJs * 1e12 / T) * w1;
        const double *W0 = W + (size_t)m * nb;
        const double *W1 = W + ((size_t)nb + m) * nb;
        const double *W2 = W + ((size_t)2 * nb + m) * nb;
        for (int n = (half ? m + 1 : 0) + threadIdx.x; n < nb; n += blockDim.x) {
            const double w2 = q.omega[n];
            if (!(w2 > 0.0) || (!(bandwidth_w > 0.0) && !(gamma[n] > 0.0))) continue;
            const double dw = w1 - w2;
            if (threshold_w > 0.0 && fabs(dw) > threshold_w) continue;
            const double gs = bandwidth_w > 0.0 ? bandwidth_w : g1 + gamma[n];
            const double den = fma(dw, dw, gs * gs);
            const double wgt = fabs(dw) < degen_tol_w ? 0.5 * mult * (c1 + q.heat[n]) * gs / den
                                                      : k1 * w2 * (q.occ[n] - n1) * gs / (dw * den);
            const double x0 = W0[n], x1 = W1[n], x2 = W2[n];
            const double y0 = wgt * x0, y1 = wgt * x1, y2 = wgt * x2;
            acc[0] = fma(y0, x0, acc[0]); acc[1] = fma(y0, x1, acc[1]); acc[2] = fma(y0, x2, acc[2]);
            acc[4] = fma(y1, x1, acc[4]); acc[5] = fma(y1, x2, acc[5]); acc[8] = fma(y2, x2, acc[8]);
        }
    }
    acc[3] = acc[1]; acc[6] = acc[2]; acc[7] = acc[5];
    block_reduce9(acc, red);
    if (threadIdx.x == 0)
        for (int a = 0; a < 9; ++a) partial[(size_t)blockIdx.x * 9 + a] = acc[a];
}

// Mode diffusivity (Eq. diffusivity_per_mode, read as the Allen-Feldman
// diffusivity averaged over the three directions):
//   D_mu = 1/3 sum_a sum_mu' W_a(mu, mu')^2 tau_{mu mu'},
// tau as in the QHGK pair sum; modes with w <= 0 or gamma <= 0 get 0 and take
// no part as mu'.  One CTA per mu, threads over mu', fixed-order reduction.
__global__ void __launch_bounds__(256)
diffusivity_kernel(int nb, const double *__restrict__ W, const double *__restrict__ omega,
                   const double *__restrict__ gamma, double bandwidth_w, double threshold_w, double *__restrict__ D) {
    __shared__ double red[8];
    const int m = blockIdx.x;
    const double w1 = omega[m], g1 = gamma[m];
    const bool bw = bandwidth_w > 0.0;
    const bool ok = w1 > 0.0 && (bw || g1 > 0.0);
    double acc = 0.0;
    if (ok) {
        const double *W0 = W + (size_t)m * nb;
        const double *W1 = W + ((size_t)nb + m) * nb;
        const double *W2 = W + ((size_t)2 * nb + m) * nb;
        for (int n = threadIdx.x; n < nb; n += blockDim.x) {
            const double w2 = omega[n], g2 = gamma[n];
            if (!(w2 > 0.0) || (!bw && !(g2 > 0.0))) continue;
            const double dw = w1 - w2, gs = bw ? bandwidth_w : g1 + g2;
            if (threshold_w > 0.0 && fabs(dw) > threshold_w) continue;
            const double tau = gs / (dw * dw + gs * gs);
            const double x0 = W0[n], x1 = W1[n], x2 = W2[n];
            acc += (x0 * x0 + x1 * x1 + x2 * x2) * tau;
        }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += red[k];
        D[m] = ok ? t / 3.0 : 0.0;
    }
}

}  // namespace

cudaError_t launch_kappa_rta(const DevFc2 &f, int nb, int nq, const double *qcart,
                             const double *nu_thz, const double2 *eig, const double *gamma,
                             double T, int classical, double omega_min_thz, double degen_tol_thz,
                             double *partial, double *kappa_out, double scale, cudaStream_t st) {
    kappa_rta_kernel<<<counted(nq), kRtaThreads, 0, st>>>(f, nb, qcart, nu_thz, eig, gamma, T, classical,
                                                omega_min_thz, degen_tol_thz, partial);
    sum_partials_kernel<<<counted(1), 288, 0, st>>>(nq, partial, scale, kappa_out);
    return cudaGetLastError();
}

cudaError_t launch_kappa_rta_diag(const DevFc2 &f, int nb, int nq, const double *qcart, const double *nu_thz,
                                  const double2 *eig, const double *gamma, const int *src, const double *vre,
                                  const double *vim, const double2 *phases, int n_blk, double T, int classical, double omega_min_thz,
                                  double degen_tol_thz, double *partial, double *kappa_out, double scale,
                                  cudaStream_t st) {
    kappa_rta_diag_kernel<<<counted(nq), kRtaThreads, 0, st>>>(f, nb, qcart, nu_thz, eig, gamma, src, vre, vim,
                                                               phases, n_blk, T, classical, omega_min_thz,
                                                               degen_tol_thz, partial);
    sum_partials_kernel<<<counted(1), 288, 0, st>>>(nq, partial, scale, kappa_out);
    return cudaGetLastError();
}

// W [3][nb][nb] of a Gamma-only system (over B), and the modes' tables.
static cudaError_t launch_velocity_w(const DevFc2Dist &f, int nb, const double *nu_thz, const double2 *eig, double T,
                                     int classical, double omega_min_thz, int antisym, int fill, const QhgkWork &w,
                                     size_t smem_optin, uint32_t wait_limit, cudaStream_t st) {
    qhgk_modes_kernel<<<counted((nb + 255) / 256), 256, 0, st>>>(nb, nu_thz, omega_min_thz, T, classical, w.modes);
    // modes per CTA: four, fewer where their eigenvectors do not fit
    const size_t row = sizeof(double) * (size_t)nb;
    cudaError_t e = cudaSuccess;
    auto sparse = [&](auto kern, int mu) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(mu * row));
        if (e == cudaSuccess) kern<<<counted((nb + mu - 1) / mu), 256, mu * row, st>>>(f, nb, eig, w.W);
    };
    if (4 * row <= smem_optin) sparse(sparse_ae_kernel<4>, 4);
    else if (2 * row <= smem_optin) sparse(sparse_ae_kernel<2>, 2);
    else sparse_ae_kernel<1, false><<<counted(nb), 256, 0, st>>>(f, nb, eig, w.W);
    if (e != cudaSuccess) return e;
    return launch_oz_gemm(nb, eig, w.W, w.modes.fac, antisym, fill, w.oz, w.dirs, w.err, wait_limit, st);
}

cudaError_t launch_diffusivity(const DevFc2Dist &f, int nb, const double *nu_thz, const double2 *eig,
                               const double *gamma, double omega_min_thz, double bandwidth_w, double threshold_w,
                               int antisym, const QhgkWork &w, double *D, size_t smem_optin, uint32_t wait_limit,
                               cudaStream_t st) {
    cudaError_t e = launch_velocity_w(f, nb, nu_thz, eig, 1.0, 1, omega_min_thz, antisym, 1, w, smem_optin, wait_limit, st);
    if (e != cudaSuccess) return e;
    diffusivity_kernel<<<counted(nb), 256, 0, st>>>(nb, w.W, w.modes.omega, gamma, bandwidth_w, threshold_w, D);
    return cudaGetLastError();
}

cudaError_t launch_qhgk(const DevFc2Dist &f, int nb, const double *nu_thz, const double2 *eig,
                        const double *gamma, double T, int classical, double omega_min_thz,
                        double degen_tol_thz, double bandwidth_w, double threshold_w, int antisym, int fill,
                        const QhgkWork &w, double *partial, int n_partial, double *kappa_out, double scale,
                        size_t smem_optin, uint32_t wait_limit, cudaStream_t st) {
    cudaError_t e = launch_velocity_w(f, nb, nu_thz, eig, T, classical, omega_min_thz, antisym, fill, w, smem_optin,
                                      wait_limit, st);
    if (e != cudaSuccess) return e;
    qhgk_pairsum_kernel<<<counted(n_partial), 256, 0, st>>>(nb, w.W, w.modes, gamma, T, kTwoPi * degen_tol_thz,
                                                            bandwidth_w, threshold_w, antisym, partial);
    sum_partials_kernel<<<counted(1), 288, 0, st>>>(n_partial, partial, scale, kappa_out);
    return cudaGetLastError();
}

}  // namespace kald
