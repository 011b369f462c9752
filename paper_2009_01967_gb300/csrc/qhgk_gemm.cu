// The dense product of the generalised velocities of Gamma-only systems (paper
// Eq. generalized_velocity),
//   W_a(mu, mu') = sum_d E(mu, d) B_a(mu', d) x scale(mu) scale(mu'),  B_a = E A_a^T,
// to FP64 accuracy on the BF16 tensor cores (an exact slicing of both operands,
// after Ozaki, Ogita, Oishi and Rump, "Error-free transformations of matrix
// multiplication by using fast routines of matrix multiplication", Numerical
// Algorithms 59, 2012).
//
// Every row of an operand is scaled by a power of two so that its largest
// element is below 64, and cut into kOz = 8 signed digits of base 2^7,
// x = sum_i d_i 2^(-7 i), |d_i| <= 64, exact in BF16.  Digit products are
// integers of at most 2^12; those of level i + j = l (up to eight pairs) over
// kOzChunk = 512 values of d sum to at most 2^24, so that the FP32 accumulators
// hold them exactly.  After every chunk the epilogue adds the eight levels
// into two 64-bit integers per element (levels 0-3 and 4-7), and only the end
// converts to FP64.  What is lost: each operand's rounding, 2^-56 of its row's
// largest element, and the levels above 7, of which the first holds seven digit
// products of up to 2^-56 of the product of the row maxima for every d -- together
// at most about 9 n 2^-56 of that product (3e-13 for 2,592 modes), and some
// sqrt(n) of it as a rule: 2e-15 to 4e-15 of the product of the row maxima for 324
// and 768 modes, where FP64 sums have 2e-15 to 1e-14.  It is relative to the rows'
// largest elements, not to sum |E B|: an element between two modes whose vectors
// hardly overlap carries the absolute error of its rows (5e-14 of sum |E B| for
// elements spread over e^-20, where an FP64 sum has 2e-15).
//
// Bound: L2 to shared memory, 98 KB per stage of 32 values of d (36 digit
// pairs, 1,152 MMA cycles).  The FP64 units made the same product the time of
// the whole call: 88 ms for 2,592 modes as a tiled FP64 kernel (at the FP64
// peak), 2.3 ms here, slicing included.  A_a is antisymmetric for a symmetric Phi2, and W with it, so only
// the tiles on and above the diagonal are formed then.
//
// Tile 128 x 64, 320 threads: warps 0-7 epilogue (TMEM lane quadrant warp % 4,
// column half warp / 4), warp 8 TMA (two stages, 64-byte swizzle), warp 9 MMA.
// The eight levels take all 512 TMEM columns.  Every wait is bounded.

#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "kald_internal.h"
#include "tc_common.cuh"

namespace kald {
namespace {
using namespace tc;

constexpr int kOz = 8, kOzBM = 128, kOzBN = 64, kOzBK = 32, kOzChunk = 512;
constexpr int kOzA = kOzBM * kOzBK * 2, kOzB = kOzBN * kOzBK * 2;       // one digit plane of a stage
constexpr int kOzStage = kOz * (kOzA + kOzB);
constexpr int kOzThreads = 320;
constexpr size_t kOzSmem = 2 * (size_t)kOzStage + 1024;

// K-major operand, 64-byte swizzle: SBO = 512 B between 8-row groups.
__device__ __forceinline__ uint64_t smem_desc64(const void *p) {
    const uint64_t a = smem_u32(p);
    return ((a >> 4) & 0x3FFFull) | (1ull << 16) | ((uint64_t)(512 >> 4) << 32) | (1ull << 46) | (4ull << 61);
}

// Digits of one row per CTA, row r0 + blockIdx.x: src row (stride in elements of T; the
// real part of a double2) -> row blockIdx.x of the planes [kOz][rows][ld], zero past n
// and for rows past n.  The row's scale: 2^(exponent) x fac[row] (NaN when the row holds
// a value that is not finite, so that the product does not hide it).
template <typename T>
__global__ void __launch_bounds__(256)
oz_slice_kernel(int n, int r0, int rows, int ld, const T *__restrict__ src_all, const double *__restrict__ fac,
                __nv_bfloat16 *__restrict__ out_all, double *__restrict__ scale_all) {
    __shared__ double red[8];
    __shared__ int bad;
    const int row = r0 + blockIdx.x, dir = blockIdx.y, tid = threadIdx.x;
    const T *src = src_all + ((size_t)dir * n + row) * n;
    __nv_bfloat16 *out = out_all + ((size_t)dir * kOz * rows + blockIdx.x) * ld;
    const size_t plane = (size_t)rows * ld;
    auto val = [&](int c) {
        if constexpr (sizeof(T) == 16) return src[c].x;
        else return src[c];
    };
    double m = 0.0;
    int inf = 0;
    if (row < n)
        for (int c = tid; c < n; c += 256) {
            const double x = fabs(val(c));
            inf |= !(x <= 1.7976931348623157e308);
            m = fmax(m, x);
        }
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (tid == 0) bad = 0;
    if ((tid & 31) == 0) red[tid >> 5] = m;
    __syncthreads();
    if (inf) bad = 1;
    for (int w = 0; w < 8; ++w) m = fmax(m, red[w]);
    __syncthreads();
    int k = 0;
    const bool live = m > 0.0 && !bad;
    if (live) frexp(m, &k);                          // m = f 2^k, 0.5 <= f < 1
    if (tid == 0 && row < n) scale_all[(size_t)dir * n + row] = bad ? nan("") : live ? scalbn(fac[row], k - 6) : 0.0;
    for (int c = 2 * tid; c < ld; c += 512) {
        long long v[2];
        for (int u = 0; u < 2; ++u)                  // 55 - k: the row's largest value becomes < 2^55
            v[u] = (live && c + u < n) ? llrint(scalbn(val(c + u), 55 - k)) : 0;
#pragma unroll
        for (int i = kOz - 1; i >= 0; --i) {
            uint32_t w = 0;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                // signed digit of base 128 in [-64, 63]; the first takes what is left
                const int d = i ? (int)((v[u] + 64) & 127) - 64 : (int)v[u];
                v[u] = (v[u] - d) >> 7;
                w |= (uint32_t)__bfloat16_as_ushort(__int2bfloat16_rn(d)) << (16 * u);
            }
            *reinterpret_cast<uint32_t *>(out + i * plane + c) = w;
        }
    }
}

// The rows [128 tm0, 128 (tm0 + gridDim.y)) of W; mA holds their digits from row 0 on.
// (What a box reaches past the planes' rows and columns is zero.)
__global__ void __launch_bounds__(kOzThreads, 1)
oz_gemm_kernel(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB, int n, int n_st,
               int tm0, int antisym, const double *__restrict__ sa, const double *__restrict__ sb, double *__restrict__ W,
               int *err, uint32_t wait_limit) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *base = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full[2], empty[2], tfull, tempty, drain;
    __shared__ uint32_t tmem_base_sm;
    __shared__ int fail_sm;
    const int tn = blockIdx.x, tm = tm0 + blockIdx.y, dir = blockIdx.z;
    if (antisym && (tn + 1) * kOzBN <= tm * kOzBM) return;       // below the diagonal
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int spc = kOzChunk / kOzBK;                         // stages per chunk
    const int n_chunks = (n_st + spc - 1) / spc;
    if (threadIdx.x == 0) {
        for (int s = 0; s < 2; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        mbar_init(&tfull, 1);
        mbar_init(&tempty, 8);
        mbar_init(&drain, 1);
        fail_sm = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 9) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(&tmem_base_sm)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_sm;

    int issued = 0;                                  // stages handed to TMA (drain bookkeeping)
    if (warp == 8) {
        if (lane == 0)
            for (int it = 0; it < n_st; ++it) {
                const int s = it & 1;
                if (it >= 2 && !mbar_wait(&empty[s], ((it >> 1) - 1) & 1, wait_limit)) fail_sm = 1;
                if (*(volatile int *)&fail_sm) break;
                unsigned char *st = base + (size_t)s * kOzStage;
                mbar_expect_tx(&full[s], kOzStage);
                tma_load_3d(st, &mA, &full[s], it * kOzBK, (int)blockIdx.y * kOzBM, 0);
                tma_load_3d(st + kOz * kOzA, &mB, &full[s], it * kOzBK, tn * kOzBN, dir * kOz);
                ++issued;
            }
    } else if (warp == 9) {
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_bf16(kOzBN);
            for (int it = 0; it < n_st && !*(volatile int *)&fail_sm; ++it) {
                const int s = it & 1, ic = it % spc;
                // the epilogue has read the previous chunk
                if (ic == 0 && it > 0 && !mbar_wait(&tempty, (it / spc - 1) & 1, wait_limit)) { fail_sm = 1; break; }
                if (!mbar_wait(&full[s], (it >> 1) & 1, wait_limit) || *(volatile int *)&fail_sm) { fail_sm = 1; break; }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                unsigned char *st = base + (size_t)s * kOzStage;
                const uint64_t a0 = smem_desc64(st), b0 = smem_desc64(st + kOz * kOzA);
#pragma unroll
                for (int l = 0; l < kOz; ++l)
#pragma unroll
                    for (int i = 0; i <= l; ++i)
#pragma unroll
                        for (int k = 0; k < kOzBK / 16; ++k)
                            mma_bf16(tmem + (uint32_t)(l * kOzBN), a0 + (uint64_t)((i * kOzA + k * 32) >> 4),
                                     b0 + (uint64_t)(((l - i) * kOzB + k * 32) >> 4), idesc,
                                     (ic > 0 || i > 0 || k > 0) ? 1u : 0u);
                mma_commit(&empty[s]);
                if (ic == spc - 1 || it == n_st - 1) mma_commit(&tfull);
            }
            mma_commit(&drain);
        }
    } else {
        const int qd = warp & 3, half = warp >> 2;
        long long hi[32], lo[32];
#pragma unroll
        for (int x = 0; x < 32; ++x) hi[x] = lo[x] = 0;
        bool ok = true;
        for (int c = 0; c < n_chunks && ok; ++c) {
            ok = !*(volatile int *)&fail_sm && mbar_wait(&tfull, c & 1, wait_limit);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) { fail_sm = 1; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t t0 = tmem + ((uint32_t)(qd * 32) << 16) + (uint32_t)(half * 32);
#pragma unroll
            for (int l = 0; l < kOz; ++l) {
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    float v[16];
                    tmem_ld16(t0 + (uint32_t)(l * kOzBN + 16 * g), v);
#pragma unroll
                    for (int x = 0; x < 16; ++x) {
                        const long long d = (long long)__float2int_rn(v[x]) * (1 << (7 * (3 - (l & 3))));
                        if (l < 4) hi[16 * g + x] += d;
                        else lo[16 * g + x] += d;
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty);
        }
        const int m = tm * kOzBM + qd * 32 + lane;
        if (ok && m < n) {
            const double s1 = sa[m];
            double *out = W + ((size_t)dir * n + m) * n;
            const int c0 = tn * kOzBN + half * 32;
#pragma unroll
            for (int x = 0; x < 32; ++x)
                if (c0 + x < n)
                    out[c0 + x] = ((double)hi[x] * 0x1p-21 + (double)lo[x] * 0x1p-49) * (s1 * sb[(size_t)dir * n + c0 + x]);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (*(volatile int *)&fail_sm && threadIdx.x == 256) {       // the TMA thread: its copies land before the CTA exits
        atomicOr(err, 1);
        for (int s = 0; s < 2; ++s) {
            int last = -1;
            for (int it = s; it < issued; it += 2) last = it;
            if (last >= 0) mbar_wait(&full[s], (last >> 1) & 1);
        }
    }
    if (warp == 9) {
        if (lane == 0) mbar_wait(&drain, 0);
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
    __syncthreads();
}

// W(mu', mu) = -W(mu, mu') below the diagonal tiles (antisymmetric A_a).
__global__ void __launch_bounds__(256)
antisym_fill_kernel(int n, double *__restrict__ W_all) {
    __shared__ double tile[32][33];
    if (blockIdx.x > blockIdx.y) return;                          // source tile (x, y) is above or on the diagonal
    double *W = W_all + (size_t)blockIdx.z * n * n;
    const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int r = ty; r < 32; r += 8)
        if (r0 + r < n && c0 + tx < n) tile[r][tx] = W[(size_t)(r0 + r) * n + c0 + tx];
    __syncthreads();
    for (int r = ty; r < 32; r += 8)
        if (c0 + r < n && r0 + tx < n && c0 + r > r0 + tx) W[(size_t)(c0 + r) * n + r0 + tx] = -tile[tx][r];
}

int oz_ld(int n) { return (n + 7) / 8 * 8; }          // (16-byte rows)
size_t oz_planes(int n, int rows) { return sizeof(__nv_bfloat16) * kOz * (size_t)rows * oz_ld(n); }
// Rows of E whose digits are held at once: all of them, or those of one row of tiles.
int oz_rows(int n, int dirs) { return dirs == 3 ? n : std::min(n, kOzBM); }

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// Digit planes [planes][rows][ld], box 32 x box_rows x kOz, 64-byte swizzle.
bool oz_map(CUtensorMap *map, const void *ptr, int ld, int rows, int planes, int box_rows) {
    static EncodeTiledFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        return cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                           cudaSuccess &&
                       q == cudaDriverEntryPointSuccess
                   ? reinterpret_cast<EncodeTiledFn>(p)
                   : nullptr;
    }();
    if (!fn) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)ld, (cuuint64_t)rows, (cuuint64_t)planes};
    const cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)ld * 2 * rows};
    const cuuint32_t box[3] = {(cuuint32_t)kOzBK, (cuuint32_t)box_rows, (cuuint32_t)kOz};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ptr), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

size_t oz_work_bytes(int n, int dirs) {
    return ws_round(oz_planes(n, oz_rows(n, dirs))) + ws_round(dirs * oz_planes(n, n)) +
           ws_round(sizeof(double) * 4 * (size_t)n);
}

cudaError_t launch_oz_gemm(int n, const double2 *E, double *BW, const double *fac, int antisym, int fill, void *work,
                           int dirs, int *err, uint32_t wait_limit, cudaStream_t st) {
    const int rows = oz_rows(n, dirs), ld = oz_ld(n);
    char *w = static_cast<char *>(work);
    auto *pa = reinterpret_cast<__nv_bfloat16 *>(w);
    auto *pb = reinterpret_cast<__nv_bfloat16 *>(w + ws_round(oz_planes(n, rows)));
    double *sa = reinterpret_cast<double *>(w + ws_round(oz_planes(n, rows)) + ws_round(dirs * oz_planes(n, n)));
    double *sb = sa + n;
    CUtensorMap mA, mB;
    if (!oz_map(&mA, pa, ld, rows, kOz, kOzBM) || !oz_map(&mB, pb, ld, n, dirs * kOz, kOzBN))
        return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(oz_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOzSmem);
    if (e != cudaSuccess) return e;
    // all directions and rows at once, or one direction and 128 rows in a small workspace
    const int n_tm = (n + kOzBM - 1) / kOzBM, tms = (rows + kOzBM - 1) / kOzBM;
    for (int d = 0; d < 3; d += dirs) {
        double *bw = BW + (size_t)d * n * n;
        oz_slice_kernel<double><<<counted(dim3(n, dirs)), 256, 0, st>>>(n, 0, n, ld, bw, fac, pb, sb);
        for (int tm = 0; tm < n_tm; tm += tms) {
            oz_slice_kernel<double2><<<counted(dim3(rows, 1)), 256, 0, st>>>(n, tm * kOzBM, rows, ld, E, fac, pa, sa);
            oz_gemm_kernel<<<counted(dim3((n + kOzBN - 1) / kOzBN, tms, dirs)), kOzThreads, kOzSmem, st>>>(
                mA, mB, n, (n + kOzBK - 1) / kOzBK, tm, antisym, sa, sb, bw, err, wait_limit);
        }
    }
    if (antisym && fill) {
        const unsigned nt = (unsigned)((n + 31) / 32);
        antisym_fill_kernel<<<counted(dim3(nt, nt, 3)), 256, 0, st>>>(n, BW);
    }
    return cudaGetLastError();
}

}  // namespace kald
