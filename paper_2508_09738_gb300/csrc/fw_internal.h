// Host-side internals shared by the translation units of the library.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <algorithm>
#include <string>
#include <vector>

#include "../../include/fw_seg.h"
#include "fw_types.h"

namespace fw {

// Thread-local error text behind fw_seg_last_error().
void set_error(const std::string& msg);
fw_status cuda_fail(cudaError_t e, const char* what);

#define FW_CUDA(call)                                         \
    do {                                                      \
        cudaError_t e_ = (call);                              \
        if (e_ != cudaSuccess) return fw::cuda_fail(e_, #call); \
    } while (0)

// Streams and events as the runtime makes them, NULL when it cannot: what a
// failed call leaves in the handle is not one to wait for or destroy.
inline cudaError_t make_stream(cudaStream_t* s) {
    const cudaError_t e = cudaStreamCreateWithFlags(s, cudaStreamNonBlocking);
    if (e != cudaSuccess) *s = nullptr;
    return e;
}
inline cudaError_t make_event(cudaEvent_t* ev, unsigned flags) {
    const cudaError_t e = cudaEventCreateWithFlags(ev, flags);
    if (e != cudaSuccess) *ev = nullptr;
    return e;
}

// Kernel launchers for one (iterate type, weight type, class bound) choice.
// Every launcher takes the problem's descriptor (device pointers inside).
class Ops {
public:
    virtual ~Ops() {}
    virtual size_t elem() const = 0;    // sizeof(T)
    virtual size_t welem() const = 0;   // sizeof(WT)
    virtual int kmax() const = 0;
    // fin: take the previous iteration's step decision inside this pass (the
    // previous iteration then has no k_finish); 0: apply the stored step
    virtual void passA(const ProbDesc& pd, ProbState* st, cudaStream_t s, int fin) = 0;
    virtual void passB(const ProbDesc& pd, ProbState* st, cudaStream_t s) = 0;
    // one thread: read the exact totals, stop test, step
    virtual void finish(const ProbDesc& pd, ProbState* st, cudaStream_t s) = 0;
    virtual void flush(const ProbDesc& pd, ProbState* st, cudaStream_t s) = 0;
    virtual void grad(const ProbDesc& pd, ProbState* st, void* Gout, uint8_t* chout,
                      cudaStream_t s) = 0;
    virtual void spmm(const ProbDesc& pd, const void* X, void* out, cudaStream_t s) = 0;
    // out = L U_hat, valid while U holds U_hat (right after reinit)
    virtual void spmm_hat(const ProbDesc& pd, void* out, cudaStream_t s) = 0;
    // classic FW gap partials per row block (fresh LUf)
    virtual void lmo_gap(const ProbDesc& pd, const void* LUf, double* part, cudaStream_t s) = 0;
    // One-Shot Frank-Wolfe labels (Alg. 4) of rows [first, last) in one CSR pass
    virtual void oneshot(const ProbDesc& pd, int32_t* labels, int first, int last,
                         cudaStream_t s) = 0;
    virtual void build(int64_t n, const int32_t* rp, const int32_t* col, const double* w,
                       const double* deg, const int32_t* rpp, int32_t* colp, void* valp,
                       void* diag, int comb, int col16, cudaStream_t s) = 0;
    virtual void reinit(const ProbDesc& pd, cudaStream_t s) = 0;
    // out[(i - r0) K + k] = X[k npad + i] for rows i of [r0, r0 + rows)
    virtual void rowmajor(const void* X, int64_t npad, int K, int64_t r0, int64_t rows, double* out,
                          cudaStream_t s) = 0;
    virtual void labels(const ProbDesc& pd, int32_t* out, cudaStream_t s) = 0;
    virtual void objective(const ProbDesc& pd, const void* LUf, double* part, cudaStream_t s) = 0;
    // Whether pass B has a form for pattern problems of K classes, and the
    // search for the patterns of n rows (col: kPatRow 16-bit offsets each).
    virtual bool pattern_kernels(int K) const = 0;
    virtual void patterns(int n, const void* col, unsigned long long* keys, int* rep, uint8_t* pat,
                          int16_t* ptab, int* fail, cudaStream_t s) = 0;
    virtual cudaError_t configure() = 0;   // dynamic shared-memory limits
    // Dynamic shared memory of k_passB_tab for this many lanes per row and
    // rows; 0 when the instantiation has no such form (FP64 iterate, K > 16).
    virtual size_t tab_smem(int lanes, int64_t n) const = 0;
};

// The resident kernel's launch of one problem (fw_resident.cuh).
struct ResPlan {
    int32_t group = 0;     // blocks that share the problem (0: the kernel does not apply)
    int32_t cluster = 0;   // 1: they are one thread-block cluster, 0: a cooperative grid
    int32_t layers = 0;    // 512-row layers of the fullest block
    int32_t form = 0;      // kResShared, kResNarrow or kResWide
    size_t smem = 0;       // dynamic shared memory of a block
    int32_t direct = 0;    // rows walked in place (ResProb::direct)
    int64_t slack = 0;     // entries added to each block's range of the slices
    int64_t entries = 0;   // entries of the slices
    size_t welem = 0;      // bytes of a weight
};
struct ResArgs;
struct ResProb;
class ResKern {
public:
    virtual ~ResKern() {}
    // Whether (and how) the kernel takes this problem on the current device;
    // maxrow: entries of the longest row.  share: layers a block should hold
    // where other problems run beside this one (0: it has the device to itself).
    virtual bool plan(const ProbDesc& pd, int maxrow, int64_t nnz_pad, int sms, int share,
                      ResPlan& p) = 0;
    // Fill the slices `prob` names.
    virtual cudaError_t slice(const ResProb& prob, const ResPlan& p, cudaStream_t s) = 0;
    // After the slices are built: most chunks of a block, from ResSlices::chunks.
    virtual void sliced(ResPlan& p, int chunks) = 0;
    virtual cudaError_t launch(const ResArgs& a, const ResPlan& p, cudaStream_t s) = 0;
};
// NULL when no resident kernel is compiled for K classes.
ResKern* make_res(int weight_dtype, int K);

// A state as copied from the device.  `err` says that a wait ran out in some
// block; the decision of a block that saw none may have been stored beside it.
inline void settle(ProbState& s) {
    if (!s.err) return;
    s.done = 1;
    s.status = FW_ERR_TIMEOUT;
}
constexpr const char* kTimeoutText = "a wait between the blocks of a launch ran out of its budget";

// Non-template kernels (defined in fw_seg.cu).
__global__ void k_validate(int64_t n, const int32_t* rp, const int32_t* col, const double* w,
                           double* deg, int* err, int* band);
__global__ void k_state_init(ProbState* st, const double* part, int nb);
__global__ void k_fid(int64_t n, const int32_t* labels, int8_t* fid);

// Factories, one per translation unit.  kmax in {4, 8, 10, 12, 16, 32}.
Ops* make_ops_f32(int kmax);
Ops* make_ops_bf16(int kmax);
Ops* make_ops_f64(int kmax);
Ops* make_ops(int weight_dtype, int K);
int kmax_for(int K);

// A graph on the host, as passed to the C ABI.
struct HostGraph {
    int64_t n;
    const int32_t* rp;
    const int32_t* col;
    const double* w;
    int32_t K;
    const int32_t* labels;
};

// Host-side layout of one problem: sizes, tiles and the padded row_ptr.
struct ProbLayout {
    int64_t n = 0, nnz = 0, nnz_pad = 0, npad = 0;
    int32_t K = 0, tile_rows = 0, ntiles = 0, lanes = 1;
    int32_t maxrow = 0;    // entries of the longest row
    int32_t padw = kPadW;  // rows padded to a multiple of this many entries
    // keep the 4-bit class array (ProbDesc::cls4): set by the two-kernel
    // single-problem path for K <= 16; the persistent kernels do not use it
    bool cls4 = false;
    // store columns as 16-bit offsets when the graph allows (fw_seg_opts::index_width)
    bool allow16 = true;
    // pass B with the class table in shared memory (fw_seg_opts::class_table)
    int32_t tab_mode = FW_TABLE_AUTO;
};

// Host checks (options, row_ptr, labels) and the padded layout.
fw_status check_opts(const fw_seg_opts& o);
fw_status plan_problem(const HostGraph& g, const fw_seg_opts& o, ProbLayout& lay);
// Device bytes of one problem's persistent arrays (256-byte aligned pieces).
size_t problem_bytes(const ProbLayout& lay, size_t te, size_t we, bool comb);
// Carve the problem's arrays out of [base, base + problem_bytes) and fill pd.
void place_problem(char* base, const ProbLayout& lay, size_t te, size_t we, const fw_seg_opts& o,
                   ProbDesc& pd);
// Stream-ordered device allocation from the library's per-device pool (freed
// with cudaFreeAsync on a stream ordered after every use).  FW_ERR_NO_MEMORY
// with the message set on failure.
fw_status pool_alloc(void** out, size_t bytes, cudaStream_t s);

// Stream-ordered temporaries, released (stream-ordered) when the object dies.
struct Temps {
    cudaStream_t s;
    std::vector<void*> ptrs;
    explicit Temps(cudaStream_t st) : s(st) {}
    ~Temps() {
        for (void* p : ptrs) cudaFreeAsync(p, s);
    }
    template <typename P>
    fw_status get(P** out, size_t bytes) {
        void* q = nullptr;
        const fw_status st = pool_alloc(&q, bytes, s);
        if (st != FW_OK) return st;
        ptrs.push_back(q);
        *out = reinterpret_cast<P*>(q);
        return FW_OK;
    }
};

// Touch the pages of a host output buffer, unless all of them have been.
void touch_pages(void* p, size_t bytes);

// Copy a class-major array X[K][npad] (n rows) to the host as row-major doubles;
// `scratch` (device, `bytes` long) holds as many rows at a time as it can.
// Waits for the stream.
fw_status rowmajor_to_host(Ops* ops, const void* X, int64_t n, int64_t npad, int K, double* out,
                           void* scratch, size_t bytes, cudaStream_t s);
// The same for small arrays: one copy of X as it lies, put in row order on the
// host, which saves the kernel, its scratch and the bytes of the wider type.
// Below kHostRowsMax values (handle, us, host against device): 972 values 22
// against 47, 24,300 35 against 51, 64,800 45 against 53; 131,072 80 against
// 44, 1,572,528 890 against 135.
constexpr int64_t kHostRowsMax = int64_t(1) << 16;
fw_status soa_to_host(const void* X, size_t te, int64_t n, int64_t npad, int K, double* out,
                      cudaStream_t s);

// Device copies of a caller's input arrays (row_ptr, col, w, labels).
struct Upload {
    Temps t;
    int64_t n = 0, nnz = 0;
    int32_t *rp = nullptr, *col = nullptr, *lab = nullptr;
    double* w = nullptr;
    explicit Upload(cudaStream_t s) : t(s) {}
};
// The O(1) checks the upload relies on: n, K, pointers, row_ptr[0] and nnz.
fw_status check_graph_args(const HostGraph& g);
// Enqueue the copies of g's arrays on up's stream (asynchronous from pinned
// host memory; the caller's arrays must stay valid until the stream passes).
fw_status upload_inputs(const HostGraph& g, Upload& up);
// Upload, validate and build the problem into pd's arrays; U_0, L U_0 and the
// fresh state *st.  Temporaries are stream-ordered (pool_alloc).  Waits
// for the validation result on `s`.
fw_status assemble_problem(Ops* ops, const HostGraph& g, const ProbLayout& lay, ProbDesc& pd,
                           ProbState* st, cudaStream_t s);
// The same from inputs already uploaded (or in flight) on stream s.
// Sets pd.col16 from the validated graph.
fw_status assemble_uploaded(Ops* ops, Upload& up, const ProbLayout& lay, ProbDesc& pd,
                            ProbState* st, cudaStream_t s);
// Restart pd at U_0 (or at its current U when from_current) with a fresh state.
fw_status restart_problem(Ops* ops, const ProbDesc& pd, ProbState* st, bool from_current,
                          cudaStream_t s);

// Geometry helpers.
inline int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }
int tile_rows_for(int64_t n);
int default_lanes(double avg_padded_degree);

}  // namespace fw
