// Internal declarations shared by the translation units of libkald.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include <memory>
#include <string>
#include <vector>

#include "../../include/kald.h"

// ---- physical constants (CODATA 2018) ---------------------------------------
namespace kald {
constexpr double kEvJ = 1.602176634e-19;     // J / eV
constexpr double kAmuKg = 1.66053906660e-27; // kg / amu
constexpr double kHbarJs = 1.054571817e-34;  // J s
constexpr double kKbJK = 1.380649e-23;       // J / K
// 1 eV/(A^2 amu) in ps^-2
constexpr double kEvA2AmuPs2 = kEvJ / (1e-20 * kAmuKg) * 1e-24;
constexpr double kHbarEvPs = kHbarJs / kEvJ * 1e12;   // eV ps
constexpr double kKbEvK = kKbJK / kEvJ;                // eV / K
constexpr double kPi = 3.14159265358979323846;
constexpr double kTwoPi = 2.0 * kPi;
// (J/K) (A/ps)^2 ps / A^3 -> W/(m K)
constexpr double kKappaSI = 1e4 * 1e-12 / 1e-30;

constexpr int kMaxNbSmall = 96;    // largest nb of the per-q dense kernels
constexpr uint32_t kDefaultWaitPolls = 1u << 22;   // polls of a bounded device wait
constexpr int kMaxDegen = 96;      // largest degenerate set handled
}  // namespace kald

// ---- per-launch timing of named kernels (kald_profile_*) ----------------------
namespace kald {
struct HostSystem;
// CUDA events around individual launches, on the launching stream; folded
// into per-kernel totals once the call has synchronised (fold()).
struct Prof {
    bool on = false;
    std::vector<cudaEvent_t> pool;          // created on demand, reused
    size_t used = 0;
    struct Rec { int kind; cudaEvent_t a, b; };
    std::vector<Rec> recs;
    double total_ms[KALD_PROF_COUNT] = {};
    uint64_t count[KALD_PROF_COUNT] = {};
    cudaEvent_t take();
    void fold();                             // stream(s) already synchronised
    void reset();
    void destroy();
};
// Records the start event at construction and the stop event at end() when
// profiling is on (prof may be NULL).
struct ProfMark {
    Prof *p;
    int kind;
    cudaStream_t st;
    cudaEvent_t a = nullptr;
    ProfMark(Prof *prof, int k, cudaStream_t s) : p(prof && prof->on ? prof : nullptr), kind(k), st(s) {
        if (p) { a = p->take(); if (a) cudaEventRecord(a, st); }
    }
    void end() {
        if (!p || !a) return;
        cudaEvent_t b = p->take();
        if (b) { cudaEventRecord(b, st); p->recs.push_back({kind, a, b}); }
        p = nullptr;
    }
};
}

// ---- context -----------------------------------------------------------------
struct kald_ctx {
    int device = 0;
    cudaStream_t own_stream = nullptr;
    cudaStream_t stream = nullptr;
    char *ws = nullptr;          // device workspace
    size_t ws_cap = 0;
    size_t ws_used = 0;
    std::string err;
    int sm_count = 0;
    size_t smem_optin = 0;
    uint32_t wait_limit = kald::kDefaultWaitPolls;   // polls of the pipeline waits
    size_t ws_limit = 0;                           // workspace cap in bytes (0: none)
    kald::Prof prof;                               // optional per-launch timing
    std::vector<cudaStream_t> lanes;               // extra streams for concurrent systems (lazy)
    // host plans of recently seen systems, keyed by a 128-bit hash of their
    // whole content (oldest first)
    struct Plan {
        uint64_t k0, k1;
        std::shared_ptr<const kald::HostSystem> h;
        size_t bytes;
    };
    std::vector<Plan> plans;
};

namespace kald {

// Kernel launches made by the library in this process (a diagnostic read
// through kald_kernel_launches): every launch passes its grid through counted().
extern std::atomic<unsigned long long> g_launches;
inline dim3 counted(dim3 grid) {
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return grid;
}

// Set ctx->err and return `st`.
kald_status fail(kald_ctx *ctx, kald_status st, const std::string &msg);

// Check a CUDA call; on error record it (with `what`) and return KALD_E_CUDA.
kald_status cuda_check(kald_ctx *ctx, cudaError_t e, const char *what);

// Workspace: reserve(total) grows the buffer (synchronising first); take()
// carves 256-byte aligned pieces until the next reset().
kald_status ws_reserve(kald_ctx *ctx, size_t bytes);
void *ws_take(kald_ctx *ctx, size_t bytes);
inline size_t ws_round(size_t b) { return (b + 255) & ~size_t(255); }

// Pointer kind: true if `p` is device (or managed) memory usable on ctx->device.
bool is_device_ptr(const void *p);

// (j, k) groups of more blocks than this take a warp each in the Gamma-only Y build.
constexpr int kYLong = 8;

// ---- host-side plan of a system ---------------------------------------------
struct LwTermsHost;
struct TcxPlanHost;
struct HostSystem {
    int n_atoms = 0;
    int nb = 0;
    double lattice[3][3];
    double volume = 0;
    std::vector<double> masses, positions;
    // fc2 grouped by (i, j) atom pair (CSR over pairs)
    std::vector<int> pair2_i, pair2_j, pair2_start;   // pairs, start offsets (n_pairs+1)
    std::vector<int> fc2_rep;                          // replica index per block (sorted order)
    std::vector<double> fc2_blk;                       // [n_fc2][9] Phi2 (eV/A^2), grouped, not mass-scaled
    std::vector<int> fc2_atoms;                        // [n_fc2][2] (i, j) of each block
    std::vector<double> fc2_rcart;                     // [n_fc2][3] Cartesian R
    std::vector<double> fc2_dist;                      // [n_fc2][3] x_i - x_j - R
    std::vector<int4> pair2_up;                        // DevFc2::up (nb <= 96)
    mutable int fc2_symmetric = -1;                    // Phi2(i, jR) = Phi2(j, i-R)^T (lazy)
    // fc3 grouped by (j, k) atom pair (CSR over output pairs)
    std::vector<int> pair3_j, pair3_k, pair3_start;
    // the groups of each k (first block, end, j, 0), those of more than kYLong blocks
    // first, then by falling length, and where each k's begin with how many of the long
    // ones it has (the Y build of the Gamma-only tensor-core path)
    std::vector<int2> pair3_kstart;
    std::vector<int4> pair3_grp;
    std::vector<int> fc3_i, fc3_rj, fc3_rk;            // per block (sorted order)
    std::vector<double> fc3_blk;                       // [n_fc3][27] Phi3 (eV/A^3), grouped, not mass-scaled
    std::vector<int> fc3_atoms;                        // [n_fc3][3] (i, j, k) of each block
    // distinct replica vectors (Cartesian) referenced by fc3 / fc2
    std::vector<double> rep_cart;                      // [n_rep][3]
    std::vector<int> rep_int;                          // [n_rep][3] integer cell vectors
    int n_rep = 0;
    mutable int fc3_symmetric = -1;                    // Phi3 symmetric in its last two indices (lazy)
    mutable int fc3_perm_symmetric = -1;               // ... under every permutation of its indices (lazy)
    mutable std::shared_ptr<const LwTermsHost> lw_terms;   // plan_lw_terms with tables (lazy)
    mutable std::shared_ptr<const TcxPlanHost> tcx_plan;   // plan_tcx_gather of those terms (lazy)
};

// Validate and plan one kald_system (host).  Returns KALD_OK or an error.
kald_status plan_system(kald_ctx *ctx, const kald_system *s, HostSystem &h);
// The same through the context's plan cache: a system whose content (sizes,
// geometry, masses, force constants) hashes to a cached plan reuses it.
kald_status plan_system_cached(kald_ctx *ctx, const kald_system *s, std::shared_ptr<const HostSystem> &h);

kald_status check_mesh(kald_ctx *ctx, const int32_t mesh[3]);

// ---- kernels (launch wrappers) ----------------------------------------------
// phonons.cu
struct DevFc2 {
    int n_pairs;
    const int *pair_i, *pair_j, *pair_start;
    const double *blk;        // [n][9]
    const double *rcart;      // [n][3]
    // unordered atom pairs i <= j: (i, j, pair of (i, j), pair of (j, i)), -1 where
    // there is none (crystals; n_up = 0 otherwise)
    int n_up = 0;
    const int4 *up = nullptr;
};
// Mass-scaled copy of force-constant blocks on the device (Phi / sqrt of the
// product of the n_at masses of each block): raw [n_blk][nval] FP64, atoms
// [n_blk][n_at], out [n_blk][out_stride] (zero padding past nval), FP64 or FP32.
cudaError_t launch_mass_scale(int n_blk, int nval, int n_at, const double *raw, const int *atoms,
                              const double *masses, int out_stride, int f32, void *out, cudaStream_t st);
cudaError_t launch_mirror_phonons(int nq, int nb, const int *row, const int *conj, const double *nu_c,
                                  const double2 *eig_c, const double *vel_c, double *nu, double2 *eig, double *vel,
                                  cudaStream_t st);
cudaError_t launch_dynmat(const DevFc2 &f, int nb, int nq, size_t n_blk, const double *qcart, double2 *D,
                          cudaStream_t st);
size_t jacobi_scratch(int nb);
cudaError_t launch_jacobi(int nb, int nq, double2 *A, double2 *V, double *nu_thz,
                          double2 *eig_out, int *nonconv, size_t smem_optin, cudaStream_t st);
// eigh_large.cu: one real symmetric matrix (the Gamma-only D), n up to about
// 9600 (three length-n FP64 vectors per CTA in shared memory)
size_t eigh_large_scratch_bytes(int n);
// n >= 3 and three length-n FP64 vectors fit in one CTA's shared memory
bool eigh_large_supported(int n, size_t smem_optin);
// One system of a batched large eigensolve: D [n][n] in, scratch of
// eigh_large_scratch_bytes(n), frequencies (THz) and row-major eigenvectors out.
struct EighJob {
    int n;
    const double2 *D;
    double *scratch;
    double *nu_out;
    double2 *eig_out;
};
// Device records of a batch (eigh_batch_records_bytes(n_sys) of workspace).
size_t eigh_batch_records_bytes(int n_sys);
// The eigensolves of n_sys (<= 64) systems as one launch sequence; each
// system's results equal those of a solve of it alone.
cudaError_t launch_eigh_large_batch(int n_sys, const EighJob *jobs, void *records, int sms, size_t smem_optin,
                                    cudaStream_t st);
cudaError_t launch_velocity_diag(const DevFc2 &f, int nb, int nq, const double *qcart,
                                 const double *nu_thz, const double2 *eig, double *vel,
                                 cudaStream_t st);

// velocity.cu: diagonal velocity elements (nb <= 96); table of vel_table_bytes.
size_t vel_table_bytes(int nq, size_t n_blk);
int vel_batch(int nq, size_t n_blk);   // q-points of one batch: the table holds them all when this is nq
cudaError_t launch_vel_diag(const DevFc2 &f, int nb, int nq, size_t n_blk, const double *qcart, const double *nu_scale,
                            const double *nu_cmp, const double2 *eig, const int *neg, int *src, void *table, size_t table_bytes,
                            double *out_re, double *out_im, cudaStream_t st);

// linewidths.cu
struct LwParams {
    int nb, nq, mesh[3];
    int n_rep;
    double sigma_w;           // 2 pi sigma (rad/ps)
    double cut_w;             // n_sigma * sigma_w
    int shape;                // energy-delta shape (kald_options.delta_shape)
    double T;
    int classical;
    double omega_min_w;       // 2 pi omega_min (rad/ps)
    int qp_chunk;             // q' per work item
    int n_chunks;             // ceil(nq / qp_chunk)
    int q0, q1;               // q-points whose linewidths are returned: [q0, q1)
    int nqc;                  // q-points projected (rows of LwDev::partial), <= q1 - q0
    int bte;                  // 1: also scatter the rates into the BTE operator planes (FP64 paths)
    double bte_pref;          // hbar pi / (8 N_k) (eV/A^2 amu -> ps^-2)^3 x delta normalisation
    uint32_t wait_limit;      // polls of the tensor-core pipeline waits
    Prof *prof;               // per-launch timing (NULL: off); host pointer, never read on the device
};
struct LwDev {
    const int4 *blkinfo;      // [n_fc3] (i, rep(Rj), rep(Rk), 0), HostSystem order
    const void *fc3;          // [n_fc3][28] float or double, Phi3 / sqrt(mi mj mk), padded
    const double *rep_cart;   // [n_rep][3]
    const double *qcart;      // [nq][3]
    const int *qfrac;         // [nq][3]
    const double *nu;         // [nq][nb] THz
    const double2 *eig;       // [nq][nb][nb]
    // derived (filled by prep kernels)
    double *omega;            // [nq*nb] rad/ps (0 if masked)
    double *occ;              // [nq*nb] Bose n (0 if masked)
    float4 *wn32;             // [nq*nb] (w hi, w lo, n hi, n lo) FP32 pairs of omega and occ
                              // (FP32 and BF16-split paths; see wdiff.cuh)
    void *eps_work;           // [nq][nb][nb] eps^T in the working precision
    void *chi;                // [nq][n_rep] exp(-i q.R) in the working precision
    double *partial;          // [nqc][n_chunks][nb] FP64 partial sums
    // returned q-points qout[j], j < q1 - q0 (gamma row j), and the projected
    // ones qsel[i] = (q, number of returned q-points it stands for), i < nqc;
    // qrow[j] = the row i of partial that holds the sums of qout[j] (those of
    // qout[j] itself or of -qout[j])
    const int *qout;
    const int2 *qsel;
    const int *qrow;
    // full-BTE assembly (p.bte): three [N][N] planes, N = nq nb, row mu = q nb + s:
    //   g1_a  (w'/w) Gamma^+ summed over s'' at column (q', s')
    //   g1_am (w'/w) Gamma^- summed over s'' at column (-q', s')
    //   g1_b  (w''/w) (Gamma^+ + Gamma^-) summed over s' at column (q + q', s'')
    double *g1_a, *g1_am, *g1_b;
    const int *qneg;          // [nq] flat index of -q
    unsigned long long *allowed;   // [1] delta-allowed triplet count
    int *queue;               // [1] work counter
};
// orbits.cu: orbits of momentum triples on a whole mesh, enumerated on the
// device.  rows: the lower index of each pair {q, -q}, ascending; row_of [nq]: the
// row of a q-point that has one.
struct OrbitPlan {
    int n_pairs = 0, n_rows = 0, nq = 0;
    int mesh[3] = {0, 0, 0};
    const int2 *pairs = nullptr;    // [n_pairs] (q1, q2), by row
    const int *orbit = nullptr;     // [n_pairs] ordered triples in the orbit
    const uint2 *bits = nullptr;    // [n_rows][words] (canonical q2, canonical ones before)
    const int *start = nullptr;     // [n_rows + 1] first pair of a row
    const int *rows = nullptr, *row_of = nullptr;
};
int orbit_pairs(const int32_t mesh[3]);           // number of orbits, -1: too many to index
size_t orbit_bytes(const int32_t mesh[3], int n_rows);
cudaError_t launch_orbit_plan(const int32_t mesh[3], int n_rows, const int *rows, const int *row_of, void *work,
                              OrbitPlan &o, cudaStream_t st);
// out [n_rows][nb]: sums of each row's q from the positions' sums out3
// [n_pairs][3][nb] (nb <= 96) of its orbits.
cudaError_t launch_orbit_class_sums(const OrbitPlan &o, int nb, const float *out3, double *out, cudaStream_t st);
cudaError_t launch_orbit_class_sums(const OrbitPlan &o, int nb, const double *out3, double *out, cudaStream_t st);
// The same from the orbits p0 .. p1 - 1 (out3 from p0 on), added to out when p0 > 0.
cudaError_t launch_orbit_class_sums(const OrbitPlan &o, int nb, int p0, int p1, const double *out3, double *out,
                                    cudaStream_t st);

// The phase sums of the CUDA-core kernel (plan_lw_terms): per (j, k) group its
// terms (i, class, slot) -- phase sums of class 0, 1 or 2 from tables per q', q''
// or q -- or (i, 3, block), phased per pair.  n_pairs > 0: one projection per
// orbit (pairs, orbit of the OrbitPlan `plan`), the positions' sums through out3 into
// LwDev::partial.
struct LwTermsHost {
    std::vector<int> group, term_start, slot_start, slot_blk;
    std::vector<int4> term;
    int n_slot[3] = {0, 0, 0}, slot0[3] = {0, 0, 0};
    // groups with three or more class-2 terms: their index (-1: none) and those terms
    // (i, slot), which are not among the others (launch_lw_same sums them per q)
    std::vector<int> group_c, cterm_start;
    std::vector<int2> cterm;
};
struct LwTerms {
    const int *group = nullptr;        // [n_atoms^2] group of (j, k), -1: none
    const int *term_start = nullptr;   // [n_groups + 1]
    const int4 *term = nullptr;
    const int *slot_start = nullptr;   // blocks of each slot, the classes' slots one after another
    const int *slot_blk = nullptr;
    int n_slot[3] = {0, 0, 0}, slot0[3] = {0, 0, 0};
    void *tab[3] = {nullptr, nullptr, nullptr};   // [nq][n_slot][27] complex
    int n_cg = 0;
    const int *group_c = nullptr, *cterm_start = nullptr;
    const int2 *cterm = nullptr;
    void *yc = nullptr;                // [nq][n_cg][9][nb] complex
    int n_pairs = 0;
    const int2 *pairs = nullptr;
    const int *orbit = nullptr;
    double *out3 = nullptr;            // lw_orbit_sums values: [pairs of a launch][blocks][3][nb] ..
    const OrbitPlan *plan = nullptr;
    int n_sblk = 1, s_per = 0;         // blocks of modes per item, modes per block (set by the launch)
};
size_t lw_orbit_sums(int nb, int n_pairs, int fp32, int sm_count, size_t smem_optin);
void plan_lw_terms(const HostSystem &h, bool tables, LwTermsHost &o);
cudaError_t launch_lw_tables_f32(int nq, int n_rep, const LwTerms &t, const int4 *blkinfo, const float *fc3,
                                 const float2 *chi, cudaStream_t st);
// Y_s(3j + beta, 3k + gamma) of the class-2 terms set apart, into t.yc, for the n_rows
// q-points rows[.].x (rows null: q-points 0 .. n_rows - 1).
cudaError_t launch_lw_same(int nb, int nq, const LwTerms &t, int n_rows, const int2 *rows, const void *epsT, int fp32,
                           cudaStream_t st);
cudaError_t launch_lw_prep(const LwParams &p, const LwDev &d, int fp32, cudaStream_t st);
cudaError_t launch_lw_main(const LwParams &p, const LwDev &d, const LwTerms &t, int fp32, int sm_count,
                           size_t smem_optin, cudaStream_t st);
cudaError_t launch_lw_finish(const LwParams &p, const LwDev &d, double degen_tol_thz,
                             double *gamma_out, cudaStream_t st);

cudaError_t launch_mode_prep(int n, const double *nu, double omega_min_w, double T, int classical,
                             double *omega, double *occ, cudaStream_t st);

// gamma_only.cu: Gamma-only linewidths of a system with nb > kMaxNbSmall
struct GammaPlan {
    int n_groups = 0;
    size_t n_fc3 = 0;                // fc3 blocks
    int n_part = 0;                  // epilogue CTAs (partial sums) per mode
    std::vector<double> omega_h;     // [nb] rad/ps, 0 for a masked mode
    // tensor-core path: delta-band tiles (tm, tn) of each mode, CSR by mode
    std::vector<int2> tiles;
    std::vector<int> tile_start;     // [nb + 1]
    int symmetric = 0;               // Phi3 symmetric in its last two indices
    int sym3 = 0;                    // ... and under every permutation: each triple of modes projected once
    int row_entries = 1;             // largest number of entries of a row of Y_mu^T
    int mb_max = 1;                  // largest modes per launch that the scratch holds
    int sms = 1;                     // SMs of the device (modes per tensor-core launch)
    int mb = 0;                      // modes per tensor-core launch (0: tc_gamma_batch; autotuned)
};
struct GammaDev {
    const int *group_jk, *group_start, *blk_i;   // (j, k) groups of fc3 blocks
    const int2 *k_start;             // HostSystem::pair3_kstart, pair3_grp (tensor-core path)
    const int4 *k_grp;
    const double *fc3;               // [n_fc3][27] Phi3 / sqrt(mi mj mk)
    const double2 *eig;              // [nb][nb] (real parts used)
    const double *nu;                // [nb] THz
    double *omega, *occ;             // [nb]
    void *E, *Y, *T, *PHI;           // [nb][nb] in the working precision
    double *partial;                 // [nb][n_part]
    int *order;                      // [nb]
    unsigned long long *allowed;
    // tensor-core path
    void *tc_scratch;                // tc_gamma_scratch_bytes(nb, sms)
    int2 *tiles_dev;                 // [tiles]
    double *partial_tc;              // [tiles]
    int *err;                        // bounded-wait failures
};
// mode: 0 FP64 CUDA cores, 1 FP32 CUDA cores, 2 BF16-split tensor cores
cudaError_t launch_gamma_only(const GammaPlan &gp, const GammaDev &d, const LwParams &p, int mode,
                              double degen_tol_thz, double *gamma_out, cudaStream_t st);
// Modes per launch of the Gamma-only tensor-core path for this system (the
// autotuner's choice for (nb, SMs), timed on first use; tc_gamma_batch
// before that).  The timing runs use the system's own buffers.
int tune_gamma_batch(const GammaPlan &gp, const GammaDev &d, const LwParams &p, cudaStream_t st);
// modes per launch of the tensor-core Gamma-only path and its scratch bytes
int tc_gamma_batch(int nb, int sms, int sym3);
int tc_gamma_batch_max(int nb, int sms, int sym3);
size_t tc_gamma_scratch_bytes(int nb, int mb_max, size_t n_fc3, int sym3, size_t n_tiles);
int tc_tile(void);
cudaError_t launch_gamma_only_tc(const GammaPlan &gp, const GammaDev &d, const LwParams &p, void *scratch,
                                 const std::vector<int2> &tiles, const std::vector<int> &tile_start,
                                 int2 *tiles_dev, int symmetric, double *partial_tc, int *err, int sms,
                                 cudaStream_t st, int mode_limit, const double **gacc_out);

// small_nb.cu: crystal linewidths of one- and two-atom cells (nb = 3 or 6),
// one thread per (pair, mode), the projection in registers.  The Bloch phase
// of a block is a root of unity of order L = lcm(mesh), taken from a table:
// q.R = 2 pi sum_d k_d n_d / N_d for q = sum_d (k_d / N_d) b_d, R = sum_d n_d a_d.
struct SnTables {
    int L, m0;                        // root order, index offset of the table
    const int *kk;                    // [nq][3] k_d L / N_d
    const int *start;                 // [4 n_atoms^3 + 1] blocks of each (class, i, j, k) (plan_sn)
    const int4 *bj, *bk;              // [n_fc3] Rj and Rk in cells, plan_sn order
    const double *fc3;                // [n_fc3][28] Phi3 / sqrt(mi mj mk), plan_sn order
    double2 *roots;                   // [2 m0 + 1] exp(-2 pi i (t - m0) / L)
    void *tab;                        // phase-sum tables A, B, C [3][nq][nb^3] in the working
                                      // precision, or NULL: every block summed per pair
};
bool sn_supported(int nb);
int sn_chunk(int nb, int nq, int sm_count);
size_t sn_table_bytes(int nb, int nq, int fp32);
void plan_sn(const HostSystem &h, bool tables, std::vector<int> &order, std::vector<int> &start);
// orb: one projection per orbit (Phi3 symmetric under permutations, the whole mesh),
// the positions' sums through out3 (sn_orbit_work bytes).
size_t sn_orbit_bytes(int nb, int n_pairs, int fp32);
size_t sn_orbit_work(int nb, int nq, int n_pairs, int fp32);
struct OrbitPlan;
cudaError_t launch_lw_small(const LwParams &p, const LwDev &d, const SnTables &t, int fp32, const OrbitPlan *orb,
                            void *out3, int sms, cudaStream_t st);

// tc_crystal.cu: crystal linewidth sums on tensor cores (BF16 split, nb <= 96).
// The gather runs over the fc3 blocks grouped by (j, k) atom pair (the order
// of HostSystem), the groups dealt to the gather's warps by plan_tcx_gather.
// Tables of the tensor-core phase sum (tcx_y_kernel): the fc3 blocks of each
// (j, k) group ordered by the home atom i.
struct TcxYTables {
    int n_at = 0;                     // atoms of the cell (nb / 3)
    int n_groups = 0;                 // (j, k) groups with blocks, HostSystem order
    const int *gi_start = nullptr;    // [n_groups][n_at + 1] first block of (group, i) in fc3 / rep
    const float4 *fc3 = nullptr;      // [n_fc3][7] Phi3 / sqrt(mi mj mk), FP32, 27 values + 1 pad
    const int2 *rep = nullptr;        // [n_fc3] (rep(Rj), rep(Rk))
    const int2 *gjk = nullptr;        // [n_groups] atoms (j, k)
};
struct TcxGroups {
    TcxYTables y;                     // the same blocks for the tensor-core phase sum
    int n_groups = 0;
    const int2 *gjk = nullptr;        // [n_groups] atoms (j, k)
    const int4 *blkinfo = nullptr;    // [n_fc3] (i, rep(Rj), rep(Rk), 0), group order
    const float *fc3 = nullptr;       // [n_fc3][28] Phi3 / sqrt(mi mj mk), FP32, padded
    const float2 *tab[3] = {nullptr, nullptr, nullptr};   // [nq][n_slot][27] phase sums per class
    int n_slot[3] = {0, 0, 0};
    // the gather's lists: see TcxPlanHost
    const int *term_start = nullptr, *list_start = nullptr, *glist = nullptr, *tblk = nullptr;
    const int4 *term = nullptr;
    int n_cg = 0;
    const float2 *yc = nullptr;       // [nq][n_cg][9][nb] (LwTerms::yc)
};
// Lists of the gather.  Terms of list x: term[term_start[x]..], each (i, class, slot
// or start in blk, blocks), class 0..2 (a table's slot), 3 (blocks blk[..]) or 4
// (nothing to add), plus 8 at the last term of a group; the list's groups in order:
// glist[list_start[x]..], each j + (k << 8) + ((c + 1) << 16), c = LwTermsHost::group_c.
struct TcxPlanHost {
    std::vector<int> term_start, list_start, glist, blk;
    std::vector<int4> term;
};
void plan_tcx_gather(const HostSystem &h, const LwTermsHost &lt, TcxPlanHost &o);
bool tcx_y_wanted(size_t n_fc3, size_t n_groups);   // the phase sum on tensor cores is considered
size_t tcx_sym_bytes(int nb, int batch, int n_pairs);
bool tcx_supported(int nb);           // 65 <= nb <= 96 (one tile width, N = K = 192)
int tcx_half(int nb);
int tcx_batch(int nb, int nq, int sm_count);
int tcx_batch_max(int nb, int nq, int sm_count);
size_t tcx_scratch_bytes(int nb, int nq, int batch);
cudaError_t launch_lw_tensor(const LwParams &p, const LwDev &d, const TcxGroups &g, void *scratch, int batch,
                             int sms, int *err, cudaStream_t st, const OrbitPlan *sym = nullptr,
                             void *sym_scratch = nullptr);

// ifc.cu: finite-difference force constants of a pair potential.  Neighbours
// of each basis atom k within the cutoff (infinite lattice), CSR over k:
// basis atom, cell offset n and the vector x_b + n A - x_k.
struct IfcNeighbours {
    const int *start;        // [n_atoms + 1]
    const int *basis;        // [n]
    const int3 *cell;        // [n]
    const double3 *vec;      // [n]
};
cudaError_t launch_fd_force_constants(int n_fc2, const int *fc2_idx, int n_fc3, const int *fc3_idx,
                                      const IfcNeighbours &nb, double h, double eps, double sig, double *fc2_out,
                                      double *fc3_out, cudaStream_t st);

// bte.cu: the full linearised BTE on the assembled operator
size_t bte_work_bytes(int N);
cudaError_t bte_combine(size_t NN, double *a, const double *am, const double *b, cudaStream_t st);
// method 0: Jacobi-preconditioned BiCGSTAB, 1: the self-consistent series;
// writes kappa (9 values, scale = KAPPA_SI / (N_k V)) on the device.
cudaError_t bte_solve(int N, const double *G1, const double *g0, const double *nu, const double *vel,
                      double omega_min_thz, double T, int classical, int method, double tol, int max_iter,
                      void *work, double scale, double *kappa_out, int &iters, bool &converged, cudaStream_t st);

// kappa.cu
// From the diagonal elements vre (vim: NULL for a symmetric Phi2) of
// launch_vel_diag; src[q]: the q-point whose elements q takes; phases: its
// table exp(-i q.R) [nq][n_blk], or NULL.
cudaError_t launch_kappa_rta_diag(const DevFc2 &f, int nb, int nq, const double *qcart, const double *nu_thz,
                                  const double2 *eig, const double *gamma, const int *src, const double *vre,
                                  const double *vim, const double2 *phases, int n_blk, double T, int classical, double omega_min_thz,
                                  double degen_tol_thz, double *partial, double *kappa_out, double scale,
                                  cudaStream_t st);
// Without scratch beyond the partial sums (kald_kappa_rta_noalloc).
cudaError_t launch_kappa_rta(const DevFc2 &f, int nb, int nq, const double *qcart,
                             const double *nu_thz, const double2 *eig, const double *gamma,
                             double T, int classical, double omega_min_thz, double degen_tol_thz,
                             double *partial /*[nq][9]*/, double *kappa_out /*[9]*/,
                             double scale, cudaStream_t st);
struct DevFc2Dist {
    int n_rows;               // atoms i
    const int *row_start;     // CSR by i over blocks
    const int *col_j;         // [n] atom j
    const double *blk;        // [n][9] Phi2/sqrt(mi mj)
    const double *dist;       // [n][3] x_i - x_j - L
};
// Tables per mode and work buffers of the generalised velocities.
struct QhgkModes {
    double *omega, *occ, *heat, *fac;   // [nb] each
};
struct QhgkWork {
    QhgkModes modes;
    double *W;                // [3][nb][nb]
    void *oz;                 // oz_work_bytes(nb, dirs)
    int dirs;                 // directions whose slices are held at once: 3, or 1 (and 128 rows)
    int *err;                 // bounded-wait failures
};
// qhgk_gemm.cu: W_a = E B_a^T scaled by fac per mode, over B_a [3][n][n] in BW;
// antisym: the tiles on and above the diagonal only, mirrored when fill.
size_t oz_work_bytes(int n, int dirs);
cudaError_t launch_oz_gemm(int n, const double2 *E, double *BW, const double *fac, int antisym, int fill, void *work,
                           int dirs, int *err, uint32_t wait_limit, cudaStream_t st);
// Mode diffusivity D [nb] (A^2/ps) of a Gamma-only system (generalised
// velocity as for QHGK, then the per-mode sum).
// bandwidth_w > 0: fixed width in place of gamma + gamma'; threshold_w > 0:
// pairs with |d omega| > threshold left out (rad/ps, as for launch_qhgk).
cudaError_t launch_diffusivity(const DevFc2Dist &f, int nb, const double *nu_thz, const double2 *eig,
                               const double *gamma, double omega_min_thz, double bandwidth_w, double threshold_w,
                               int antisym, const QhgkWork &w, double *D, size_t smem_optin, uint32_t wait_limit,
                               cudaStream_t st);
// Phase space per mode (linewidths.cu): g [nq * nb] in ps; work of
// phase_space_bytes (sorted modes, counts, partial sums of the q' chunks).
size_t phase_space_bytes(int nb, int nq, int sm_count, int lean);
cudaError_t launch_phase_space(const LwParams &p, const LwDev &d, int fp32, int sm_count, void *work, int lean,
                               double *g_out, cudaStream_t st);
cudaError_t launch_qhgk(const DevFc2Dist &f, int nb, const double *nu_thz, const double2 *eig,
                        const double *gamma, double T, int classical, double omega_min_thz,
                        double degen_tol_thz, double bandwidth_w, double threshold_w, int antisym, int fill,
                        const QhgkWork &w, double *partial /*[n_partial][9]*/, int n_partial,
                        double *kappa_out /*[9]*/, double scale, size_t smem_optin, uint32_t wait_limit,
                        cudaStream_t st);
// gamma(nu) by a not-a-knot cubic spline through the valid source modes
// (interp.cu); work of interp_work_bytes(n_src).
size_t interp_work_bytes(int n_src);
cudaError_t launch_interpolate_gamma(int n_src, const double *nu_src, const double *g_src, int n_dst,
                                     const double *nu_dst, double *g_dst, double omega_min_thz, double degen_tol_thz,
                                     void *work, cudaStream_t st);

}  // namespace kald
