// fw_energy_noalloc: the objective E(U) -- the Laplacian quadratic form
// 1/2 <U, L U>, plus the penalty (1/eps) sum u (1 - u), plus the fidelity
// term 1/2 sum_i omega_i ||u_hat_i - u_i||^2 -- of a graph and an iterate
// that live in the caller's device memory, with no device allocation by the
// call.  The paper has no counterpart to this entry point: it is a service
// of the library.
//
// This is the allocation-free variant of the handle's objective evaluation
// (k_objective, which takes its fresh L U product and its partial sums from
// memory owned by a handle).  Here the only scratch is the file-scope array
// g_noalloc_scratch below: FW_NOALLOC_MAX_N degrees (FP64) plus 256 bytes of
// accumulator words.  Callers that cannot allocate are the reason it exists:
//  * a process whose device memory is already held by another allocator
//    (a serving framework's caching allocator that reserved the free HBM),
//    where cudaMalloc would fail even though the evaluation needs little;
//  * a latency-bound loop that must not call cudaMalloc / cudaFree, which
//    may synchronise the device.
// Nothing here calls cudaMalloc, cudaMallocAsync, cudaFree or any library
// routine that allocates device memory.
//
// Set-up: the first call on each device, with that device current, looks the
// scratch array up with cudaGetSymbolAddress (which may load the module's
// device data), sets the energy kernel's shared-memory limit, and caches the
// address together with the identity of the current CUDA context.  A later call in another context of that device (for
// instance after cudaDeviceReset) looks the address up again.  Make the first
// call on a device before any stream capture.
//
// Calls share the one scratch array of their device: two calls that overlap
// in time on the same device (from two host threads, or on two streams
// without an ordering between them) race on it and may return wrong values.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cmath>
#include <mutex>
#include <string>

#include "fw_device.cuh"
#include "fw_internal.h"

namespace fw {
namespace {

constexpr int64_t kNaMaxN = FW_NOALLOC_MAX_N;
constexpr int kNaErrWord = kAccWords;           // graph / label error bits
constexpr int kNaAccWords = 32;                 // 256 bytes of accumulator words
static_assert(kNaErrWord < kNaAccWords, "accumulators exceed the scratch words");
constexpr size_t kNaScratchBytes = size_t(kNaAccWords) * 8 + size_t(kNaMaxN) * 8;
constexpr int kNaMaxBlocks = 1024;              // < 2^11 block totals (fx_add range)
constexpr int kNaMaxDevices = 64;

// error bits of the graph / label word
constexpr unsigned long long kNaBadRowPtr = 1, kNaBadCol = 2, kNaIsolated = 4, kNaBadLabel = 8;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaScratchBytes];

// d_i = sum_j w_ij in CSR order (FP64).  Rows with an out-of-range extent or
// column, or with no positive degree, raise an error bit; nothing outside
// [0, nnz) or [0, n) is read.
__global__ void __launch_bounds__(kBlock)
k_na_degrees(int64_t n, int64_t nnz, const int32_t* __restrict__ rp,
             const int32_t* __restrict__ col, const double* __restrict__ w,
             double* __restrict__ deg, unsigned long long* acc) {
    const int64_t stride = int64_t(gridDim.x) * kBlock;
    for (int64_t i = blockIdx.x * int64_t(kBlock) + threadIdx.x; i < n; i += stride) {
        const int64_t e0 = rp[i], e1 = rp[i + 1];
        double d = 0.0;
        if (e0 < 0 || e1 > nnz || e1 < e0) {
            atomicOr(&acc[kNaErrWord], kNaBadRowPtr);
        } else {
            for (int64_t e = e0; e < e1; ++e) {
                const int32_t j = col[e];
                if (j < 0 || j >= n) {
                    atomicOr(&acc[kNaErrWord], kNaBadCol);
                    continue;
                }
                d += w[e];
            }
            if (!(d > 0.0)) atomicOr(&acc[kNaErrWord], kNaIsolated);
        }
        deg[i] = d;
    }
}

// One row's energy from its products s_k = sum_j w_ij u_jk, k in steps of `ks`.
__device__ __forceinline__ double na_row_energy(int K, const double* __restrict__ ui,
                                                const double* s, int ks, double di, int f,
                                                double inv_eps, double omega0, int comb) {
    double quad = 0.0, pen = 0.0, fidt = 0.0;
    for (int k = 0; k < K; ++k) {
        const double u = ui[k];
        const double lu = (comb ? di : 1.0) * u - s[k * ks];
        quad += u * lu;
        pen += u * (1.0 - u);
        if (f >= 0) {
            const double dlt = (k == f ? 1.0 : 0.0) - u;
            fidt += dlt * dlt;
        }
    }
    return 0.5 * quad + inv_eps * pen + (f >= 0 ? 0.5 * omega0 * fidt : 0.0);
}

// Entries of a warp's 32 rows normalised at a time.
constexpr int kNaChunk = 256;
// Dynamic shared memory of one warp: the chunk's weights and columns, the
// rows' products.
__host__ __device__ constexpr size_t na_warp_smem(int K) {
    return size_t(kNaChunk) * (sizeof(double) + sizeof(int32_t)) + size_t(32) * K * sizeof(double);
}
constexpr int kNaMaxK = 32;
// A block's, for the limit that k_na_energy is given (88 KB).  It is the same
// for every K: what a kernel gets without asking, 48 KB, counts its 3,168
// static bytes too and ends at K = 10.
constexpr size_t kNaSmemMax = (kBlock / 32) * na_warp_smem(kNaMaxK);

// Per row i (FP64): 1/2 sum_k u_ik (L u)_ik + 1/eps sum_k u_ik (1 - u_ik)
// + 1/2 omega_i sum_k (uhat_ik - u_ik)^2, with (L u)_ik = u_ik - sum_j
// w_ij u_jk / sqrt(d_i d_j) (L_s) or d_i u_ik - sum_j w_ij u_jk (L = D - W).
// Threads add their rows in order; the block adds its threads in a fixed
// order and adds its total into the exact fixed-point accumulator, so the
// result does not depend on the order in which blocks finish.
//
// FP64 issue bounds this kernel (an FP64 instruction holds a scheduler for 64
// cycles; a square root and a division are about 35 of them), so every entry
// is normalised once, not once per class, and by the next free lane: a warp
// takes the contiguous entries of its 32 rows kNaChunk at a time, its lanes
// normalise 32 entries together whatever rows they belong to, then take one
// (row, class) each and add that row's entries of the chunk in CSR order (the
// sums of one thread per row, in the same order).  300,007 rows, 14 entries
// each, K = 6: 310 us a call, 1,720 us with the square root and the division
// per entry and class and one thread per row.
__global__ void __launch_bounds__(kBlock)
k_na_energy(int64_t n, int64_t nnz, int K, const int32_t* __restrict__ rp,
            const int32_t* __restrict__ col, const double* __restrict__ w,
            const double* __restrict__ deg, const double* __restrict__ U, int64_t ldu,
            const int32_t* __restrict__ labels, double inv_eps, double omega0, int comb,
            unsigned long long* acc) {
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int32_t s_rp[kBlock / 32][33];
    __shared__ double s_deg[kBlock];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double* const sw = reinterpret_cast<double*>(smraw + warp * na_warp_smem(K));
    double* const ss = sw + kNaChunk;                              // [32][K]
    int32_t* const sc = reinterpret_cast<int32_t*>(ss + 32 * K);   // columns, -1: out of range
    const int64_t stride = int64_t(gridDim.x) * kBlock;
    double e_thr = 0.0;
    for (int64_t i0 = blockIdx.x * int64_t(kBlock) + (threadIdx.x & ~31); i0 < n; i0 += stride) {
        const int64_t i = i0 + lane;
        const bool in = i < n;
        const int32_t e0 = in ? rp[i] : 0, e1 = in ? rp[i + 1] : 0;
        const double di = in ? deg[i] : 0.0;
        const bool ok = in && !(e0 < 0 || e1 > nnz || e1 < e0 || !(di > 0.0));   // else flagged by k_na_degrees
        int f = -1;
        if (ok && labels) {
            f = labels[i];
            if (f < -1 || f >= K) {
                atomicOr(&acc[kNaErrWord], kNaBadLabel);
                f = -1;
            }
        }
        if (!__all_sync(0xffffffffu, ok || !in)) {
            // a flagged row: the call fails, whatever the energy; rows one by one
            if (ok) {
                for (int k = 0; k < K; ++k) {
                    double s = 0.0;
                    for (int32_t e = e0; e < e1; ++e) {
                        const int32_t j = col[e];
                        if (j < 0 || j >= n) continue;
                        const double wij = comb ? w[e] : w[e] / sqrt(di * deg[j]);
                        s += wij * U[j * ldu + k];
                    }
                    ss[lane * K + k] = s;
                }
                e_thr += na_row_energy(K, U + i * ldu, ss + lane * K, 1, di, f, inv_eps, omega0, comb);
            }
            __syncwarp();
            continue;
        }
        const int rows = __popc(__ballot_sync(0xffffffffu, in));
        s_rp[warp][lane] = e0;
        if (lane == rows - 1) s_rp[warp][rows] = e1;
        s_deg[threadIdx.x] = di;
        for (int k = 0; k < K; ++k) ss[lane * K + k] = 0.0;
        __syncwarp();
        const int32_t* const q = s_rp[warp];
        const int64_t last = q[rows];
        for (int64_t b = q[0]; b < last; b += kNaChunk) {
            const int cnt = last - b < kNaChunk ? int(last - b) : kNaChunk;
            for (int t = lane; t < cnt; t += 32) {
                const int64_t e = b + t;
                const int32_t j = col[e];
                const bool good = j >= 0 && j < n;
                double v = w[e];
                if (!comb && good) {
                    int lo = 0, hi = rows - 1;   // the row that holds e
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (q[mid] <= e) lo = mid;
                        else hi = mid - 1;
                    }
                    v = v / sqrt(s_deg[(threadIdx.x & ~31) + lo] * deg[j]);
                }
                sw[t] = v;
                sc[t] = good ? j : -1;
            }
            __syncwarp();
            for (int t = lane; t < rows * K; t += 32) {
                const int r = t / K, k = t - r * K;
                const int a0 = q[r] > b ? int(q[r] - b) : 0;
                const int a1 = q[r + 1] - b < cnt ? int(q[r + 1] - b) : cnt;
                double s = ss[t];
                for (int x = a0; x < a1; ++x) {
                    const int32_t j = sc[x];
                    if (j >= 0) s += sw[x] * U[j * ldu + k];
                }
                ss[t] = s;
            }
            __syncwarp();
        }
        if (in)
            e_thr += na_row_energy(K, U + i * ldu, ss + lane * K, 1, di, f, inv_eps, omega0, comb);
        __syncwarp();
    }
    const double v[1] = {e_thr};
    block_accumulate<double, 1>(v, acc, 0, int(blockIdx.x % kAccCopies));
}

std::mutex g_na_mu;
struct NaCache {
    unsigned long long ctx = 0;   // unique id of the context the address belongs to
    void* ptr = nullptr;
};
NaCache g_na_cache[kNaMaxDevices];

// Unique id of the current CUDA context (the driver's cuCtxGetCurrent and
// cuCtxGetId, reached through the runtime's entry-point query, so the library
// needs no link against the driver library).  0 when it cannot be read: the
// caller then looks the address up on every call.
unsigned long long current_ctx_id() {
    typedef CUresult (*get_current_fn)(CUcontext*);
    typedef CUresult (*get_id_fn)(CUcontext, unsigned long long*);
    static get_current_fn get_current = nullptr;
    static get_id_fn get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 4000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<get_current_fn>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<get_id_fn>(f);
        cudaGetLastError();
    });
    if (!get_current || !get_id) return 0;
    CUcontext c = nullptr;
    unsigned long long id = 0;
    if (get_current(&c) != CUDA_SUCCESS || !c) return 0;
    if (get_id(c, &id) != CUDA_SUCCESS) return 0;
    return id;
}

// Device address of this device's scratch array, looked up once per device
// and context, together with the energy kernel's shared-memory limit.
fw_status na_scratch(void** out) {
    int dev = 0;
    FW_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kNaMaxDevices) {
        set_error("fw_energy_noalloc: device ordinal out of the supported range");
        return FW_ERR_UNSUPPORTED;
    }
    // before the process's first CUDA work no context is current yet (id 0):
    // the lookup below then creates it, and the next call caches its id
    const unsigned long long ctx = current_ctx_id();
    std::lock_guard<std::mutex> lock(g_na_mu);
    NaCache& c = g_na_cache[dev];
    if (!c.ptr || ctx == 0 || c.ctx != ctx) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
        FW_CUDA(cudaFuncSetAttribute(k_na_energy, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     int(kNaSmemMax)));
        c.ptr = p;
        c.ctx = ctx;
    }
    *out = c.ptr;
    return FW_OK;
}

fw_status na_invalid(const char* m) {
    set_error(m);
    return FW_ERR_INVALID_ARG;
}

}  // namespace
}  // namespace fw

using namespace fw;

extern "C" fw_status fw_energy_noalloc(int64_t n, int32_t K, const int32_t* row_ptr_dev,
                                       const int32_t* col_dev, const double* w_dev, int64_t nnz,
                                       const double* U_dev, int64_t ldu,
                                       const int32_t* labels_dev, double eps, double omega0,
                                       int32_t laplacian, void* cuda_stream, double* E_host) {
    if (!E_host) return na_invalid("fw_energy_noalloc: E_host is NULL");
    if (n < 1) return na_invalid("fw_energy_noalloc: n must be >= 1");
    if (n > kNaMaxN) {
        set_error("fw_energy_noalloc: n = " + std::to_string(n) +
                  " exceeds the static scratch limit FW_NOALLOC_MAX_N = " +
                  std::to_string(kNaMaxN) + " rows");
        return FW_ERR_UNSUPPORTED;
    }
    if (K < 2 || K > kNaMaxK) return na_invalid("fw_energy_noalloc: K must be in [2, 32]");
    if (nnz < 0 || nnz >= (int64_t(1) << 31))
        return na_invalid("fw_energy_noalloc: nnz must be in [0, 2^31)");
    if (!row_ptr_dev || !U_dev || (nnz > 0 && (!col_dev || !w_dev)))
        return na_invalid("fw_energy_noalloc: NULL device pointer");
    if (ldu < K) return na_invalid("fw_energy_noalloc: ldu must be >= K");
    if (!(eps > 0.0)) return na_invalid("fw_energy_noalloc: eps must be > 0 (or +inf)");
    if (!(omega0 >= 0.0) || std::isinf(omega0))
        return na_invalid("fw_energy_noalloc: omega0 must be finite and >= 0");
    if (laplacian != FW_LAPLACIAN_SYM && laplacian != FW_LAPLACIAN_COMB)
        return na_invalid("fw_energy_noalloc: bad laplacian");

    void* base = nullptr;
    const fw_status ss = na_scratch(&base);
    if (ss != FW_OK) return ss;
    unsigned long long* acc = static_cast<unsigned long long*>(base);
    double* deg = reinterpret_cast<double*>(static_cast<unsigned char*>(base) + kNaAccWords * 8);
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);

    // the accumulators and error words must start at zero; the degrees are
    // written in full before they are read
    FW_CUDA(cudaMemsetAsync(acc, 0, kNaAccWords * 8, s));
    const int64_t want = (n + kBlock - 1) / kBlock;
    const int blocks = int(want < kNaMaxBlocks ? want : kNaMaxBlocks);
    k_na_degrees<<<blocks, kBlock, 0, s>>>(n, nnz, row_ptr_dev, col_dev, w_dev, deg, acc);
    FW_CUDA(cudaGetLastError());
    const size_t smem = size_t(kBlock / 32) * na_warp_smem(K);
    k_na_energy<<<blocks, kBlock, smem, s>>>(n, nnz, K, row_ptr_dev, col_dev, w_dev, deg, U_dev,
                                          ldu, labels_dev, std::isinf(eps) ? 0.0 : 1.0 / eps,
                                          omega0, laplacian == FW_LAPLACIAN_COMB ? 1 : 0, acc);
    FW_CUDA(cudaGetLastError());
    unsigned long long h[kNaAccWords];
    FW_CUDA(cudaMemcpyAsync(h, acc, sizeof(h), cudaMemcpyDeviceToHost, s));
    FW_CUDA(cudaStreamSynchronize(s));

    const unsigned long long err = h[kNaErrWord];
    if (err & (kNaBadRowPtr | kNaBadCol)) {
        set_error("fw_energy_noalloc: row_ptr extent or column index out of range");
        return FW_ERR_GRAPH;
    }
    if (err & kNaIsolated) {
        set_error("fw_energy_noalloc: a node has degree 0");
        return FW_ERR_ISOLATED;
    }
    if (err & kNaBadLabel) return na_invalid("fw_energy_noalloc: label outside [-1, K)");
    if (h[kAccFlag]) {
        set_error("fw_energy_noalloc: non-finite or out-of-range partial energy");
        return FW_ERR_NUMERIC;
    }
    // exact 128-bit total of the accumulator copies of quantity 0
    unsigned long long lo = 0ull, hi = 0ull;
    for (int c = 0; c < kAccCopies; ++c) {
        const unsigned long long l = h[c * kNumR * kAccLine], hw = h[c * kNumR * kAccLine + 1];
        const unsigned long long lo2 = lo + l;
        hi += hw + (lo2 < lo ? 1ull : 0ull);
        lo = lo2;
    }
    *E_host = double(static_cast<long long>(hi)) + std::ldexp(double(lo), -64);
    return FW_OK;
}
