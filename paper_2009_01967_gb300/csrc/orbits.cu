// Orbits of momentum triples (q1, q2, q3), q1 + q2 + q3 = 0 on the mesh, under
// the six permutations and inversion, enumerated on the GPU, and the sums of the
// linewidths from one projection per orbit (Eq. gamma_operators with Phi3
// symmetric under permutations).
//
// An orbit is represented by its lexicographically smallest ordered triple; its
// first member is then the lower index of a pair {q, -q} (a row).  Rows keep a
// bit per q2 (canonical or not) and prefix counts per 32 bits, so that the index
// of the orbit of any pair (q, q2) is a few integer operations and one bit
// count: no list per q-point is kept or sorted.  On the host the same
// enumeration took a loop over all pairs (5 ms for 512 q-points, seconds for
// 13,824).

#include <algorithm>

#include "kald_internal.h"

namespace kald {
namespace {

struct Mesh3 {
    int m0, m1, m2;
    __device__ int flat(int a, int b, int c) const { return (a * m1 + b) * m2 + c; }
};

// The triple of (q1, q2): indices of q1, q2, q3 and of their inverses.
struct Triple {
    int q[3], n[3];
};
__device__ __forceinline__ void split(const Mesh3 &m, int q, int &a, int &b, int &c) {
    c = q % m.m2;
    const int t = q / m.m2;
    b = t % m.m1;
    a = t / m.m1;
}
__device__ __forceinline__ int neg1(int x, int m) { return x ? m - x : 0; }
__device__ __forceinline__ Triple triple_of(const Mesh3 &m, int q1, int q2) {
    int a1, b1, c1, a2, b2, c2;
    split(m, q1, a1, b1, c1);
    split(m, q2, a2, b2, c2);
    int a = a1 + a2, b = b1 + b2, c = c1 + c2;         // q1 + q2 = -q3
    if (a >= m.m0) a -= m.m0;
    if (b >= m.m1) b -= m.m1;
    if (c >= m.m2) c -= m.m2;
    Triple t;
    t.q[0] = q1;
    t.q[1] = q2;
    t.n[2] = m.flat(a, b, c);
    t.n[0] = m.flat(neg1(a1, m.m0), neg1(b1, m.m1), neg1(c1, m.m2));
    t.n[1] = m.flat(neg1(a2, m.m0), neg1(b2, m.m1), neg1(c2, m.m2));
    t.q[2] = m.flat(neg1(a, m.m0), neg1(b, m.m1), neg1(c, m.m2));
    return t;
}
// The smallest image (first two members as one key), the place in it of the
// triple's first member, and how many of the twelve images equal the triple.
__device__ __forceinline__ unsigned long long canonical(const Triple &t, unsigned nq, int &place, int &stab) {
    unsigned long long best = ~0ull;
    const unsigned long long self = (unsigned long long)t.q[0] * nq + t.q[1];
    place = 0;
    stab = 0;
#pragma unroll
    for (int x = 0; x < 3; ++x)
#pragma unroll
        for (int y = 0; y < 3; ++y) {
            if (x == y) continue;
            const int pl = x == 0 ? 0 : y == 0 ? 1 : 2;          // where member 0 went
            const unsigned long long k0 = (unsigned long long)t.q[x] * nq + t.q[y];
            const unsigned long long k1 = (unsigned long long)t.n[x] * nq + t.n[y];
            stab += (k0 == self) + (k1 == self);
            if (k0 < best) { best = k0; place = pl; }
            if (k1 < best) { best = k1; place = pl; }
        }
    return best;
}

// Row i (q1 = rows[i]): one bit per q2, the number of canonical q2 before each
// 32-bit word, and the row's count.  One CTA per row.
__global__ void __launch_bounds__(256)
orbit_rows_kernel(Mesh3 m, int nq, int words, const int *__restrict__ rows, uint2 *__restrict__ bits,
                  int *__restrict__ count) {
    __shared__ int warp_sum[8], base_sm;
    const int i = blockIdx.x, q1 = rows[i], lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) base_sm = 0;
    __syncthreads();
    for (int q0 = 0; q0 < words * 32; q0 += 256) {
        const int q2 = q0 + threadIdx.x;
        bool c = false;
        if (q2 >= q1 && q2 < nq) {
            int place, stab;
            c = canonical(triple_of(m, q1, q2), (unsigned)nq, place, stab) == (unsigned long long)q1 * nq + q2;
        }
        const unsigned b = __ballot_sync(0xffffffffu, c);
        if (lane == 0) warp_sum[warp] = __popc(b);
        __syncthreads();
        int before = base_sm;
        for (int w = 0; w < warp; ++w) before += warp_sum[w];
        const int word = (q0 >> 5) + warp;
        if (lane == 0 && word < words) bits[(size_t)i * words + word] = make_uint2(b, (unsigned)before);
        __syncthreads();
        if (threadIdx.x == 0)
            for (int w = 0; w < 8; ++w) base_sm += warp_sum[w];
        __syncthreads();
    }
    if (threadIdx.x == 0) count[i] = base_sm;
}

// start[i] = sum of the counts before row i, i <= n.  One CTA.
__global__ void __launch_bounds__(1024)
orbit_scan_kernel(int n, const int *__restrict__ count, int *__restrict__ start) {
    __shared__ int part[1024];
    const int per = (n + 1023) / 1024, a = threadIdx.x * per, b = min(n, a + per);
    int s = 0;
    for (int i = a; i < b; ++i) s += count[i];
    part[threadIdx.x] = s;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const int v = threadIdx.x >= o ? part[threadIdx.x - o] : 0;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    int base = threadIdx.x ? part[threadIdx.x - 1] : 0;
    for (int i = a; i < b; ++i) {
        start[i] = base;
        base += count[i];
    }
    if (threadIdx.x == 1023) start[n] = part[1023];
}

// The pairs (q1, q2) in row order and their orbit sizes.
__global__ void __launch_bounds__(256)
orbit_fill_kernel(Mesh3 m, int nq, int words, const int *__restrict__ rows, const uint2 *__restrict__ bits,
                  const int *__restrict__ start, int2 *__restrict__ pairs, int *__restrict__ orbit) {
    const int i = blockIdx.x, q1 = rows[i], s0 = start[i];
    for (int q2 = threadIdx.x; q2 < nq; q2 += 256) {
        const uint2 w = bits[(size_t)i * words + (q2 >> 5)];
        if (!((w.x >> (q2 & 31)) & 1u)) continue;
        int place, stab;
        canonical(triple_of(m, q1, q2), (unsigned)nq, place, stab);
        const int at = s0 + (int)w.y + __popc(w.x & ((1u << (q2 & 31)) - 1u));
        pairs[at] = make_int2(q1, q2);
        orbit[at] = 12 / stab;
    }
}

// out[i][s] = 1/2 sum over q2 of the sums of q = rows[i] in the orbit of
// (q, q2, -(q + q2)): out3[pair - p0][place][s] (FP64 here; a fixed order: every lane
// group its q2 in steps, then the groups in order), of the pairs p0 .. p1 - 1 alone;
// `add`: on top of what out holds.  CTA = row, threads (group, s).
template <typename T>
__global__ void __launch_bounds__(256)
orbit_class_sums_kernel(Mesh3 m, int nq, int nb, int words, const int *__restrict__ rows, const int *__restrict__ row_of,
                        const uint2 *__restrict__ bits, const int *__restrict__ start, int p0, int p1, int add,
                        const T *__restrict__ out3, double *__restrict__ out) {
    __shared__ int ent[256];
    __shared__ double red[256];
    const int i = blockIdx.x, q = rows[i], tid = threadIdx.x;
    const int groups = 256 / nb, g = tid / nb, s = tid - g * nb;
    double sum = 0.0;
    for (int q0 = 0; q0 < nq; q0 += 256) {
        __syncthreads();
        const int q2 = q0 + tid;
        if (q2 < nq) {
            int place, stab;
            const unsigned long long key = canonical(triple_of(m, q, q2), (unsigned)nq, place, stab);
            const int c1 = (int)(key / (unsigned)nq), c2 = (int)(key - (unsigned long long)c1 * nq);
            const int r = row_of[c1];
            const uint2 w = bits[(size_t)r * words + (c2 >> 5)];
            const int pair = start[r] + (int)w.y + __popc(w.x & ((1u << (c2 & 31)) - 1u));
            ent[tid] = pair >= p0 && pair < p1 ? 3 * (pair - p0) + place : -1;
        }
        __syncthreads();
        if (g < groups)
            for (int x = g; x < min(256, nq - q0); x += groups)
                if (ent[x] >= 0) sum += (double)out3[(size_t)ent[x] * nb + s];
    }
    red[tid] = sum;
    __syncthreads();
    if (tid < nb) {
        double t = 0.0;
        for (int x = 0; x < groups; ++x) t += red[x * nb + tid];
        double *o = out + (size_t)i * nb + tid;
        *o = (add ? *o : 0.0) + 0.5 * t;
    }
}

}  // namespace

// Orbits of pairs (q1, q2), by Burnside's lemma over the twelve operations:
// the identity fixes N^2 pairs, inversion s^2 (s q-points with -q = q), each of
// the three exchanges N, each with inversion N (q1 = -q2, q3 = 0), the two
// 3-cycles the q with 3 q = 0, each with inversion q = 0 alone.
int orbit_pairs(const int32_t mesh[3]) {
    long long n = 1, s = 1, c = 1;
    for (int a = 0; a < 3; ++a) {
        n *= mesh[a];
        s *= mesh[a] % 2 == 0 ? 2 : 1;
        c *= mesh[a] % 3 == 0 ? 3 : 1;
    }
    const long long total = (n * n + s * s + 6 * n + 2 * c + 2) / 12;
    return total > 0x7fffffffLL / 3 ? -1 : (int)total;
}

static int orbit_words(int nq) { return (nq + 31) / 32; }

size_t orbit_bytes(const int32_t mesh[3], int n_rows) {
    const int nq = mesh[0] * mesh[1] * mesh[2];
    const size_t np = (size_t)orbit_pairs(mesh);
    return ws_round(sizeof(uint2) * (size_t)n_rows * orbit_words(nq)) + 2 * ws_round(sizeof(int) * ((size_t)n_rows + 1)) +
           ws_round(sizeof(int2) * np) + ws_round(sizeof(int) * np);
}

cudaError_t launch_orbit_plan(const int32_t mesh[3], int n_rows, const int *rows, const int *row_of, void *work,
                              OrbitPlan &o, cudaStream_t st) {
    const int nq = mesh[0] * mesh[1] * mesh[2], words = orbit_words(nq);
    o.n_pairs = orbit_pairs(mesh);
    o.n_rows = n_rows;
    o.nq = nq;
    for (int a = 0; a < 3; ++a) o.mesh[a] = mesh[a];
    char *b = static_cast<char *>(work);
    auto take = [&](size_t bytes) { char *r = b; b += ws_round(bytes); return r; };
    uint2 *bits = reinterpret_cast<uint2 *>(take(sizeof(uint2) * (size_t)n_rows * words));
    int *count = reinterpret_cast<int *>(take(sizeof(int) * ((size_t)n_rows + 1)));
    int *start = reinterpret_cast<int *>(take(sizeof(int) * ((size_t)n_rows + 1)));
    int2 *pairs = reinterpret_cast<int2 *>(take(sizeof(int2) * (size_t)o.n_pairs));
    int *orbit = reinterpret_cast<int *>(take(sizeof(int) * (size_t)o.n_pairs));
    const Mesh3 m{mesh[0], mesh[1], mesh[2]};
    orbit_rows_kernel<<<counted(n_rows), 256, 0, st>>>(m, nq, words, rows, bits, count);
    orbit_scan_kernel<<<counted(1), 1024, 0, st>>>(n_rows, count, start);
    orbit_fill_kernel<<<counted(n_rows), 256, 0, st>>>(m, nq, words, rows, bits, start, pairs, orbit);
    o.bits = bits;
    o.start = start;
    o.pairs = pairs;
    o.orbit = orbit;
    o.rows = rows;
    o.row_of = row_of;
    return cudaGetLastError();
}

template <typename T>
static cudaError_t class_sums(const OrbitPlan &o, int nb, int p0, int p1, const T *out3, double *out, cudaStream_t st) {
    const Mesh3 m{o.mesh[0], o.mesh[1], o.mesh[2]};
    orbit_class_sums_kernel<T><<<counted(o.n_rows), 256, 0, st>>>(m, o.nq, nb, orbit_words(o.nq), o.rows, o.row_of, o.bits,
                                                                  o.start, p0, p1, p0 > 0, out3, out);
    return cudaGetLastError();
}
cudaError_t launch_orbit_class_sums(const OrbitPlan &o, int nb, const float *out3, double *out, cudaStream_t st) {
    return class_sums(o, nb, 0, o.n_pairs, out3, out, st);
}
cudaError_t launch_orbit_class_sums(const OrbitPlan &o, int nb, const double *out3, double *out, cudaStream_t st) {
    return class_sums(o, nb, 0, o.n_pairs, out3, out, st);
}
cudaError_t launch_orbit_class_sums(const OrbitPlan &o, int nb, int p0, int p1, const double *out3, double *out,
                                    cudaStream_t st) {
    return class_sums(o, nb, p0, p1, out3, out, st);
}

}  // namespace kald
