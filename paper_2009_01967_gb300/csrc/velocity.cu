// Diagonal velocity matrix elements eta_s^dagger (dD/dq_a) eta_s of crystals
// with nb <= 96 branches (paper Eq. velocity_crystal, read with the conjugate
// and the -i R of chi = exp(-i q.R)), FP64: the group velocities of
// kald_phonons and kald_kappa_bte and the diagonal of kappa_RTA.
//
//   dD_a(i, j) = sum_b (-i R_a) Phi2~_b exp(-i q.R_b)   (blocks b of atoms i, j)
//   e^dagger dD_a e = sum_{i <= j} sum_{al be} P [ dD_a(i,j)_{al be} + conj dD_a(j,i)_{be al} ],
//   P = conj(e_{i al}) e_{j be}, its real part; the imaginary part takes the
//   difference instead and vanishes for a symmetric Phi2.
//
// Bound: FP64 units.  The blocks of an atom pair are summed once per q (with
// phases from a table made once per (q, block)) instead of once per mode, and
// the two orders of a pair share the products P: 90 FP64 operations per mode
// and unordered atom pair, where phasing every block for every mode took a
// sincos and 45 operations per block.  32 atoms, 512 q-points: 17.8 ms before,
// 2.5 ms now (one q-point of each pair {q, -q}).

#include <algorithm>

#include "kald_internal.h"

namespace kald {
namespace {

constexpr int kVelPairs = 32;                    // unordered atom pairs per pass
constexpr size_t kVelTableBytes = size_t(64) << 20;   // phases of one batch of q-points (stays in L2)

// ph[q][b] = exp(-i q.R_b) of the q-points of a batch.
__global__ void phase_kernel(size_t n, int n_blk, const double *__restrict__ qcart, const double *__restrict__ rcart,
                             double2 *__restrict__ ph) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < n; x += (size_t)gridDim.x * blockDim.x) {
        const size_t q = x / n_blk;
        const int b = (int)(x - q * n_blk);
        const double *k = qcart + 3 * q, *R = rcart + 3 * (size_t)b;
        double s, c;
        sincos(k[0] * R[0] + k[1] * R[1] + k[2] * R[2], &s, &c);
        ph[x] = make_double2(c, -s);
    }
}

size_t vel_smem(int nb, int groups) {
    return sizeof(double2) * ((size_t)nb * (nb | 1) + kVelPairs * 27) +
           sizeof(double) * std::max<size_t>((size_t)groups * nb * 6, 1);
}

// CTA = q-point q0 + blockIdx.x, threads = (mode s, group of atom pairs).
// out_re/out_im [nq][nb][3]: the elements (eV/A^2/amu A); with nu given, out_re
// is the group velocity in A/ps instead.  src (may be NULL): a q-point whose
// inverse -q = neg[q] has the smaller index, equal frequencies and conjugate
// eigenvectors takes src[q] = neg[q] and no elements of its own (its diagonal
// elements are those of -q with the other sign); src[q] = q otherwise.
template <bool IMAG>
__global__ void __launch_bounds__(384)
vel_kernel(DevFc2 f, int nb, int nbp, int q0, const double2 *__restrict__ ph_all, const double *__restrict__ nu,
           const double *__restrict__ nu_cmp, const double2 *__restrict__ eig, const int *__restrict__ neg,
           int *__restrict__ src, double *__restrict__ out_re, double *__restrict__ out_im) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int ld = nb | 1;                                       // odd pitch: the transposing stores spread over the banks
    double2 *Et = reinterpret_cast<double2 *>(smem_raw);         // [dof][s]
    double2 *N = Et + (size_t)nb * ld;                           // [pair][al be][direction]
    double *red = reinterpret_cast<double *>(N + kVelPairs * 27);
    const int q = q0 + blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    const int n_blk = f.pair_start[f.n_pairs];
    const double2 *e = eig + (size_t)q * nb * nb;
    if (src) {
        const int qn = neg[q];
        if (qn < q) {
            int differ = 0;
            const double2 *en = eig + (size_t)qn * nb * nb;
            for (int x = tid; x < nb * nb; x += nt) {
                const double2 u = e[x], v = en[x];
                differ |= !(u.x == v.x && u.y == -v.y);
            }
            for (int x = tid; x < nb; x += nt) differ |= !(nu_cmp[(size_t)q * nb + x] == nu_cmp[(size_t)qn * nb + x]);
            differ = __syncthreads_or(differ);
            if (tid == 0) src[q] = differ ? q : qn;
            if (!differ) return;
        } else if (tid == 0) {
            src[q] = q;
        }
    }
    for (int x = tid; x < nb * nb; x += nt) Et[(x % nb) * ld + x / nb] = e[x];
    const double2 *ph = ph_all + (size_t)blockIdx.x * n_blk;
    const int groups = nt / nbp, g = tid / nbp, s = tid % nbp;
    const bool act = s < nb;
    double re[3] = {0.0, 0.0, 0.0}, im[3] = {0.0, 0.0, 0.0};
    for (int c0 = 0; c0 < f.n_up; c0 += kVelPairs) {
        const int n_c = min(kVelPairs, f.n_up - c0);
        __syncthreads();
        // sums of the blocks: `parts` threads per (pair, al be) where the cell has few
        // pairs of many blocks each, three directions; the combination for the
        // imaginary part is formed in a second pass (IMAG) over the same storage
        const int parts = max(1, min(min(nt / (9 * n_c), kVelPairs / n_c), 8));
        for (int pass = 0; pass < (IMAG ? 2 : 1); ++pass) {
            if (pass) __syncthreads();
            const double sg = pass ? -1.0 : 1.0;
            for (int x = tid; x < 9 * n_c * parts; x += nt) {
                const int pp = x / 9, part = pp / n_c, p = pp - part * n_c;
                const int ab = x - 9 * pp, ba = 3 * (ab % 3) + ab / 3;
                const int4 u = f.up[c0 + p];
                double2 m[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) m[a] = make_double2(0.0, 0.0);
                if (u.z >= 0)
                    for (int b = f.pair_start[u.z] + part; b < f.pair_start[u.z + 1]; b += parts) {
                        const double2 z = ph[b];
                        const double v = f.blk[9 * (size_t)b + ab], vx = v * z.y, vy = -v * z.x;
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            const double R = f.rcart[3 * (size_t)b + a];
                            m[a].x = fma(R, vx, m[a].x);
                            m[a].y = fma(R, vy, m[a].y);
                        }
                    }
                if (u.w >= 0)
                    for (int b = f.pair_start[u.w] + part; b < f.pair_start[u.w + 1]; b += parts) {
                        const double2 z = ph[b];
                        const double v = sg * f.blk[9 * (size_t)b + ba], vx = v * z.y, vy = v * z.x;
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            const double R = f.rcart[3 * (size_t)b + a];
                            m[a].x = fma(R, vx, m[a].x);
                            m[a].y = fma(R, vy, m[a].y);
                        }
                    }
                const double h = u.x == u.y ? 0.5 : 1.0;         // (i, i) is its own other order
#pragma unroll
                for (int a = 0; a < 3; ++a) N[27 * pp + 3 * ab + a] = make_double2(h * m[a].x, h * m[a].y);
            }
            __syncthreads();
            if (parts > 1) {
                for (int x = tid; x < 27 * n_c; x += nt) {
                    double2 m = N[x];
                    for (int k = 1; k < parts; ++k) {
                        const double2 z = N[27 * n_c * k + x];
                        m.x += z.x;
                        m.y += z.y;
                    }
                    N[x] = m;
                }
                __syncthreads();
            }
            if (act)
                for (int p = g; p < n_c; p += groups) {
                    const int4 u = f.up[c0 + p];
                    double2 ei[3], ej[3];
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        ei[a] = Et[(3 * u.x + a) * ld + s];
                        ej[a] = Et[(3 * u.y + a) * ld + s];
                    }
                    const double2 *Np = N + 27 * p;
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int b = 0; b < 3; ++b) {
                            const double pr = fma(ei[a].x, ej[b].x, ei[a].y * ej[b].y);
                            const double pi = fma(ei[a].x, ej[b].y, -(ei[a].y * ej[b].x));
#pragma unroll
                            for (int d = 0; d < 3; ++d) {
                                const double2 v = Np[3 * (3 * a + b) + d];
                                if (pass == 0) {
                                    re[d] = fma(pr, v.x, re[d]);
                                    re[d] = fma(-pi, v.y, re[d]);
                                } else {
                                    im[d] = fma(pr, v.y, im[d]);
                                    im[d] = fma(pi, v.x, im[d]);
                                }
                            }
                        }
                }
        }
    }
    // the groups' sums in order
    __syncthreads();
    if (act)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            red[((size_t)g * nb + s) * 6 + d] = re[d];
            red[((size_t)g * nb + s) * 6 + 3 + d] = im[d];
        }
    __syncthreads();
    for (int x = tid; x < 3 * nb; x += nt) {
        const int m = x / 3, d = x - 3 * m;
        double r = 0.0, i = 0.0;
        for (int k = 0; k < groups; ++k) {
            r += red[((size_t)k * nb + m) * 6 + d];
            if (IMAG) i += red[((size_t)k * nb + m) * 6 + 3 + d];
        }
        const size_t o = ((size_t)q * nb + m) * 3 + d;
        if (nu) {
            const double w = kTwoPi * nu[(size_t)q * nb + m];
            r *= (w > 0.0) ? kEvA2AmuPs2 / (2.0 * w) : 0.0;
        }
        out_re[o] = r;
        if (IMAG) out_im[o] = i;
    }
}

}  // namespace

// q-points per batch of the phase table.
int vel_batch(int nq, size_t n_blk) {
    return (int)std::max<size_t>(1, std::min<size_t>(nq, kVelTableBytes / (sizeof(double2) * std::max<size_t>(n_blk, 1))));
}
size_t vel_table_bytes(int nq, size_t n_blk) {
    return ws_round(sizeof(double2) * std::max<size_t>(n_blk, 1) * vel_batch(nq, n_blk));
}

cudaError_t launch_vel_diag(const DevFc2 &f, int nb, int nq, size_t n_blk, const double *qcart, const double *nu_scale,
                            const double *nu_cmp, const double2 *eig, const int *neg, int *src, void *table,
                            size_t table_bytes, double *out_re, double *out_im, cudaStream_t st) {
    const int nbp = (nb + 31) / 32 * 32, groups = std::min(384 / nbp, 4);
    const size_t smem = vel_smem(nb, groups);
    auto k0 = vel_kernel<false>;
    auto k1 = vel_kernel<true>;
    cudaError_t e = cudaFuncSetAttribute(out_im ? k1 : k0, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    double2 *ph = static_cast<double2 *>(table);
    const int batch = (int)std::max<size_t>(1, std::min<size_t>(nq, table_bytes / (sizeof(double2) * std::max<size_t>(n_blk, 1))));
    for (int q0 = 0; q0 < nq; q0 += batch) {
        const int n = std::min(batch, nq - q0);
        const size_t np = (size_t)n * n_blk;
        if (np)
            phase_kernel<<<counted((unsigned)std::min<size_t>((np + 255) / 256, 8192)), 256, 0, st>>>(
                np, (int)n_blk, qcart + 3 * (size_t)q0, f.rcart, ph);
        if (out_im)
            k1<<<counted(n), nbp * groups, smem, st>>>(f, nb, nbp, q0, ph, nu_scale, nu_cmp, eig, neg, src, out_re, out_im);
        else
            k0<<<counted(n), nbp * groups, smem, st>>>(f, nb, nbp, q0, ph, nu_scale, nu_cmp, eig, neg, src, out_re, out_im);
    }
    return cudaGetLastError();
}

}  // namespace kald
