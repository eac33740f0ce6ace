// roks_noalloc.cu -- roks_orthonormalize_noalloc: Cholesky orthonormalisation
// of a band block (overlap S = 1) that allocates no device memory.
//
// Who needs it: callers that cannot call cudaMalloc, e.g. code running
// inside a framework that has reserved the GPU's memory for its own caching
// allocator, or an embedded solver loop that must not allocate once it is
// running.  The scratch of this entry point (split-K partial sums, the
// overlap matrix, L^{-H} and a status flag) lives in one file-scope
// __device__ array of fixed size, reserved when the library is loaded; every
// GPU that loads the library holds it until the process exits.
#include <cooperative_groups.h>

#include <atomic>
#include <cstddef>

#include "../../include/roks.h"
#include "roks_chol.cuh"
#include "roks_impl.cuh"

using namespace roks;

namespace {

constexpr int kNaMaxBands = 64;    // largest band count accepted
constexpr int kNaMaxChunks = 64;   // K chunks of the overlap contraction
constexpr size_t kNaPart = (size_t)kNaMaxChunks * kNaMaxBands * kNaMaxBands;   // double2
constexpr size_t kNaMat = (size_t)kNaMaxBands * kNaMaxBands;                   // double2
// layout (double2 units): partials | O | LinvH | L | flag (int, 256-byte slot)
constexpr size_t kNaBytes = sizeof(double2) * (kNaPart + 3 * kNaMat) + 256;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaBytes];

// Device address of the scratch array on the current device (the host name
// g_noalloc_scratch is only a stand-in and must never reach a kernel).  It
// is resolved on every call: the lookup is cheap next to the synchronising
// call, and a cached address would go stale if the module were reloaded
// (after cudaDeviceReset, for instance).
cudaError_t scratch_address(unsigned char** out) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    *out = static_cast<unsigned char*>(p);
    return cudaSuccess;
}

// psi <- psi U in place, U upper triangular (nb x nb, FP64, column major).
// A block owns 64 rows: it reads them into shared memory before writing.
template <typename T>
__global__ void __launch_bounds__(256) k_rows_times_upper(int npw, int nb, c2<T>* psi, int64_t ld,
                                                          const double2* __restrict__ U) {
    using V = c2<T>;
    constexpr int RT = 64;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V* tile = reinterpret_cast<V*>(smem_raw);       // [nb][RT]
    V* Us = tile + (size_t)nb * RT;                 // [nb][nb] column major
    const int g0 = blockIdx.x * RT;
    for (int idx = threadIdx.x; idx < nb * RT; idx += blockDim.x) {
        const int r = idx % RT, j = idx / RT;
        const int g = g0 + r;
        tile[idx] = g < npw ? psi[(int64_t)j * ld + g] : mk<T>(T(0), T(0));
    }
    for (int idx = threadIdx.x; idx < nb * nb; idx += blockDim.x) {
        const double2 u = U[idx];
        Us[idx] = mk<T>(T(u.x), T(u.y));
    }
    __syncthreads();
    const int r = threadIdx.x % RT;
    const int g = g0 + r;
    if (g >= npw) return;
    for (int j = threadIdx.x / RT; j < nb; j += blockDim.x / RT) {
        T sr = T(0), si = T(0);
        for (int k = 0; k <= j; ++k) {
            const V a = tile[k * RT + r], b = Us[j * nb + k];
            sr += a.x * b.x - a.y * b.y;
            si += a.x * b.y + a.y * b.x;
        }
        psi[(int64_t)j * ld + g] = mk<T>(sr, si);
    }
}

// All of it in one cluster of eight blocks, for blocks small enough: a block
// keeps its share of the rows in shared memory, sums its part of the overlap
// (a warp per element, lanes over rows), the parts meet through distributed
// shared memory in block order, every block takes the Cholesky inverse
// (chol_inverse_block) and multiplies its rows, unless a pivot failed.  The
// launch chain of the kernels above, 102 us for 6 bands x 1045 rows in FP64,
// is the cost it removes: 55 us.  Up to 7 bands (8 in FP32), where the kernels
// above fill few threads and the Cholesky is short (times of the chain and
// here, in us: FP64 1000 x 6 71 and 44, 3000 x 6 109 and 65, 1000 x 8 58 and 65,
// 1000 x 12 63 and 99; FP32 1000 x 8 46 and 41, 10000 x 6 72 and 53, 700 x 12 48
// and 52, 6000 x 10 47 and 77), and in FP64 up to 250,000 multiply-adds (rows x
// bands^2), beyond which eight SMs' FP64 pipes take longer than the chain.
constexpr int kNaCluster = 8, kNaThreads = 256;
constexpr size_t kNaSmem = 200 * 1024;
template <typename T> size_t cluster_smem(int npw, int nb) {
    const size_t rows = (size_t)(npw + kNaCluster - 1) / kNaCluster;
    return sizeof(double2) * 3 * (size_t)nb * nb + sizeof(c2<T>) * rows * nb;
}
template <typename T> bool cluster_takes(int npw, int nb) {
    return nb <= (sizeof(T) == 8 ? 7 : 8) && cluster_smem<T>(npw, nb) <= kNaSmem &&
           (sizeof(T) == 4 || (int64_t)npw * nb * nb <= 250000);
}

template <typename T>
__global__ void __cluster_dims__(kNaCluster, 1, 1) __launch_bounds__(kNaThreads)
    k_orth_cluster(int npw, int nb, c2<T>* psi, int64_t ld, int* flag) {
    using V = c2<T>;
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2* part = reinterpret_cast<double2*>(smem_raw);   // this block's part of O (lower triangle)
    double2* L = part + nb * nb;
    double2* X = L + nb * nb;
    V* tile = reinterpret_cast<V*>(X + nb * nb);             // [nb][rows]
    __shared__ double dinv[kNaMaxBands];
    const int rank = (int)cluster.block_rank(), tid = threadIdx.x;
    const int rows = (npw + kNaCluster - 1) / kNaCluster, r0 = rank * rows, nr = max(0, min(rows, npw - r0));
    for (int idx = tid; idx < nb * nr; idx += kNaThreads) {
        const int j = idx / nr, r = idx - j * nr;
        tile[j * rows + r] = psi[(int64_t)j * ld + r0 + r];
    }
    for (int idx = tid; idx < nb * nb; idx += kNaThreads) X[idx] = make_double2(0.0, 0.0);
    __syncthreads();
    const int warp = tid >> 5, lane = tid & 31;
    for (int e = warp; e < nb * nb; e += kNaThreads / 32) {
        const int j = e / nb, i = e - j * nb;
        if (i < j) continue;
        const V *a = tile + i * rows, *b = tile + j * rows;
        T sr = T(0), si = T(0);   // conj(a) b
        for (int r = lane; r < nr; r += 32) {
            sr += a[r].x * b[r].x + a[r].y * b[r].y;
            si += a[r].x * b[r].y - a[r].y * b[r].x;
        }
        double dr = double(sr), di = double(si);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            dr += __shfl_xor_sync(0xffffffffu, dr, o);
            di += __shfl_xor_sync(0xffffffffu, di, o);
        }
        if (lane == 0) part[e] = make_double2(dr, di);
    }
    cluster.sync();
    for (int e = tid; e < nb * nb; e += kNaThreads) {
        const int j = e / nb, i = e - j * nb;
        if (i < j) continue;
        double2 s = make_double2(0.0, 0.0);
        for (int q = 0; q < kNaCluster; ++q) {
            const double2 v = cluster.map_shared_rank(part, q)[e];
            s.x += v.x;
            s.y += v.y;
        }
        L[e] = s;
    }
    cluster.sync();   // (no block ends while its part is read)
    const int bad = chol_inverse_block<kNaThreads>(nb, L, X, dinv);
    if (rank == 0 && tid == 0) *flag = bad;
    if (bad) return;
    // psi_j = sum_{k <= j} psi_k U_kj, U = L^{-H}: U_kj = conj X_jk
    for (int idx = tid; idx < nb * nr; idx += kNaThreads) {
        const int j = idx / nr, r = idx - j * nr;
        T sr = T(0), si = T(0);
        for (int k = 0; k <= j; ++k) {
            const V a = tile[k * rows + r];
            const double2 x = X[k * nb + j];
            const T ux = T(x.x), uy = T(-x.y);
            sr += a.x * ux - a.y * uy;
            si += a.x * uy + a.y * ux;
        }
        psi[(int64_t)j * ld + r0 + r] = mk<T>(sr, si);
    }
}

// The call's status once its work is done.  The flag is zero between calls, as
// the array is when it is loaded: whatever may have left it set clears it.
roks_status broken(int* flag, cudaStream_t st) {
    cudaMemsetAsync(flag, 0, sizeof(int), st);
    return ROKS_ECUDA;
}
roks_status result(int* flag, cudaStream_t st) {
    int h = 0;
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpyAsync(&h, flag, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return broken(flag, st);
    if (!h) return ROKS_OK;
    if (cudaMemsetAsync(flag, 0, sizeof(int), st) != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess)
        return ROKS_ECUDA;
    return ROKS_ENOTPOSDEF;
}

// The product of the last call may still read the scratch when that call has
// returned.  On the same stream this one comes after it; on another the device
// is waited for.  (Streams are told apart by their number, never used twice.)
bool after_earlier_calls(cudaStream_t st) {
    static std::atomic<unsigned long long> last{0};   // 1 + the number, 0: no call yet
    unsigned long long id = 0;
    if (cudaStreamGetId(st, &id) != cudaSuccess) return false;
    const unsigned long long was = last.exchange(id + 1);
    return was == 0 || was == id + 1 || cudaDeviceSynchronize() == cudaSuccess;
}

template <typename T>
roks_status run(int npw, int nb, void* psi, int64_t ld, cudaStream_t st, unsigned char* base) {
    using V = c2<T>;
    double2* part = reinterpret_cast<double2*>(base);
    double2* O = part + kNaPart;
    double2* LinvH = O + kNaMat;
    double2* Lw = LinvH + kNaMat;
    int* flag = reinterpret_cast<int*>(Lw + kNaMat);
    if (cluster_takes<T>(npw, nb)) {
        const size_t sm = cluster_smem<T>(npw, nb);
        if (allow_smem(k_orth_cluster<T>, kNaSmem) != cudaSuccess) return ROKS_ECUDA;
        count_launch();
        k_orth_cluster<T><<<kNaCluster, kNaThreads, sm, st>>>(npw, nb, static_cast<V*>(psi), ld, flag);
        return result(flag, st);
    }
    if (!after_earlier_calls(st)) return ROKS_ECUDA;
    V* X = static_cast<V*>(psi);
    gemm_cn_capped<T>(nb, nb, npw, X, ld, X, ld, O, nb, part, kNaMaxChunks, st);
    cholesky_inverse(nb, O, Lw, LinvH, flag, st);
    // psi is touched only if all before it was launched (the scratch holds an
    // earlier call's L^{-H} otherwise) and no pivot failed.  The status is read
    // before the product, which runs while the caller goes on (FP64, 8 bands x
    // 19,672 and 9 x 6245: 110 and 78 us, with the status last 124 and 91).
    if (cudaGetLastError() != cudaSuccess) return broken(flag, st);
    const roks_status status = result(flag, st);
    if (status != ROKS_OK) return status;
    const size_t sm = sizeof(V) * ((size_t)nb * 64 + (size_t)nb * nb);
    if (allow_smem(k_rows_times_upper<T>, sizeof(V) * kNaMaxBands * (64 + kNaMaxBands)) != cudaSuccess)
        return broken(flag, st);
    count_launch();
    k_rows_times_upper<T><<<(npw + 63) / 64, 256, sm, st>>>(npw, nb, X, ld, LinvH);
    return cudaGetLastError() == cudaSuccess ? ROKS_OK : ROKS_ECUDA;
}

}  // namespace

extern "C" roks_status roks_orthonormalize_noalloc(int precision, int npw, int nbands, void* psi, int64_t ld,
                                                   void* cuda_stream) {
    if (precision != ROKS_FP64 && precision != ROKS_MIXED) return ROKS_EINVAL;
    if (!psi || npw <= 0 || nbands <= 0 || ld < npw) return ROKS_EINVAL;
    if (nbands > kNaMaxBands) return ROKS_EINVAL;     // beyond the fixed scratch
    unsigned char* base = nullptr;
    if (scratch_address(&base) != cudaSuccess) return ROKS_ECUDA;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    return precision == ROKS_FP64 ? run<double>(npw, nbands, psi, ld, st, base)
                                  : run<float>(npw, nbands, psi, ld, st, base);
}
