// Resident kernel: a whole run of GFW iterations of one problem in one launch,
// with U and L U in registers and the row sums of the one-hot product in
// shared memory from the first iteration to the last.
#pragma once
#include <algorithm>

#include "fw_internal.h"
#include "fw_kernels.cuh"
#include "fw_step.cuh"

namespace fw {

constexpr int kResThreads = 512;
constexpr int kResWarps = kResThreads / 32;
constexpr int kResRing = 32;                      // iterations between statistics
// Most iterations of one launch: a launch cannot be interrupted (this many
// take a few tens of ms at most), and the arrival count of the grid barrier
// (two per block and iteration) stays far below 2^32.
constexpr int kResIters = 4096;
constexpr int kResTilesPerLayer = kResThreads / kBlock;   // row tiles per layer of a block
constexpr int kResMaxCluster = 16;
constexpr int kResMaxGrid = 160;                  // blocks of a grid group
constexpr int kResMaxLen = 255;                   // chunks of 4 entries in the longest row
constexpr int kResSmemMax = 220 * 1024;           // dynamic shared memory (227 KB less the static)

// Layers (512 rows each) a block holds at most: 2 * KMAX values per layer and
// thread have to stay in registers (128 a thread) next to the working set.
template <typename T, int KMAX>
__host__ __device__ constexpr int res_layers() {
    return sizeof(T) == 8 ? 1 : KMAX <= 8 ? 4 : KMAX <= 10 ? 3 : 2;
}

// The forms of the kernel (see k_resident).
enum { kResShared = 0, kResNarrow = 1, kResWide = 2 };

struct ResSlot {   // a block's exact total of one quantity (Q64.64)
    unsigned long long lo, hi;
};
// hi of a slot whose total is not finite or out of range (no sum of totals
// below 2^52 reaches it)
constexpr unsigned long long kResBad = 0x4000000000000000ull;

// One problem's sliced copy of its CSR rows for a group of `group` blocks
// (k_res_slice).  A block sorts its rows by length, longest first, and gives
// 32 rows at a time to its warps; slice (w, l) holds warp w's l-th 32 rows as
// chunk-major runs of 4 entries per lane, so that a warp reads 32 lanes' next
// 4 columns and 4 weights with one coalesced load each.  With L lanes per row
// in the problem's summation order, the chunks c = 0, L, 2L, ... come first,
// then 1, L + 1, ... (the entries lane 0, 1, ... of csr_bins adds).  Columns
// are row numbers relative to the block's class table.
struct ResSlices {
    void* col;            // uint16 (narrow) or int32 (wide), 4 per lane and chunk
    void* val;            // weights, likewise
    uint16_t* perm;       // [group][layers * 512]: local row of a (warp, layer, lane) position
    uint16_t* len;        // [group][layers * 16]: chunks of slice (w, l)
    int* chunks;          // most chunks of a block (atomicMax)
};

struct ResProb {          // what the kernel needs besides ProbDesc
    ProbDesc pd;
    ResSlices sl;
    int64_t slack;        // entries between blocks' slice ranges (beyond their rows'
    int32_t layers;       // layers of the block with the most tiles
    int32_t direct;       // 1: rows are not sorted (and L = 1): they are walked in place
};

// The launch's parameter block (constant bank: the problem's fields cost the
// kernel no registers).
struct ResArgs {
    ResProb p;
    ProbState* state;
    int32_t group;           // blocks that work on the problem: the cluster, or the grid
    int32_t cluster;         // 1: the group is a thread-block cluster, 0: the whole grid
    int32_t iters;           // iterations of this launch
    int32_t expect_extra;    // test hook: every wait is for this much that never arrives
    unsigned long long wait_ns;   // bound of one wait inside the kernel
    // Grid group, > 0: an ordinary launch whose blocks first meet, for at most
    // this long; if some find no SM meanwhile, all leave and the state says so
    // (unstarted).  0: a cooperative launch, which starts when every block can.
    unsigned long long meet_ns;
    uint32_t* bar;           // grid group: arrivals, blocks that met; zero at launch
    ResSlot* slots;          // grid group: [kNumR][group]
};

// The block's part of the problem.
struct ResSpan {
    int t0, ntl, row0, first, window;   // tiles, first row, class table start and rows
    __device__ __forceinline__ ResSpan(const ProbDesc& pd, int rank, int group, int cluster) {
        t0 = int(unsigned(rank * pd.ntiles) / unsigned(group));   // < 2^31: at most 1216 tiles
        ntl = int(unsigned((rank + 1) * pd.ntiles) / unsigned(group)) - t0;
        row0 = t0 * kBlock;
        first = 0;
        window = pd.ntiles * kBlock;   // cluster: every unit of every block, padding rows included
        if (!cluster) {                // grid: the rows the block's columns can name
            first = max(0, row0 - pd.band) & ~31;
            const int64_t end = int64_t(row0) + ntl * kBlock + pd.band;
            window = ((end < pd.n ? int(end) : pd.n) - first + 31) & ~31;
        }
    }
    // first entry of the block's slices
    __device__ __forceinline__ int64_t entry0(const ResProb& rp, int rank) const {
        const int64_t own = rp.direct ? 0 : __ldg(rp.pd.rp + min(rp.pd.n, row0));
        return ((own + 127) & ~int64_t(127)) + rank * rp.slack;
    }
};
// Entries a block's slices can take beyond its rows' own (whole multiples of
// 128): a sorted slice is no longer than the shortest row of the one before
// it, and the first no longer than the longest row.
inline int64_t res_slack(int64_t maxlen) { return 32 * 4 * maxlen + 128; }

// Shared memory of one block: row sums of `layers` layers, the threads'
// private bins, row permutation, slice lengths, class table.
__host__ __device__ inline size_t res_smem(size_t elem, int K, int layers, size_t tab) {
    return size_t(K) * kResThreads * elem * size_t(layers + 1) +
           2 * (size_t(layers) * kResThreads + size_t(layers) * kResWarps) + tab;
}

// ------------------------------------------------------------------ slices
// Builds ResSlices: one block per block of the group.  Unless the rows are
// walked in place they are ordered by a stable counting sort of their lengths.
// Padding entries add weight 0 to the class of the lane's own row.
template <typename WT, bool WIDE>
__global__ void __launch_bounds__(kResThreads)
    k_res_slice(const __grid_constant__ ResProb s_rp, int group, int cluster) {
    __shared__ uint16_t s_cnt[64][kResMaxLen + 1];   // rows of each length in each 32-row unit
    __shared__ int s_base[kResMaxLen + 1];
    __shared__ uint16_t s_perm[4 * kResThreads];
    __shared__ int s_off[64];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = int(blockIdx.x);
    const ProbDesc& pd = s_rp.pd;
    const ResSpan sp(pd, rank, group, cluster);
    const int layers = s_rp.layers, rows = layers * kResThreads, units = layers * kResWarps;
    for (int i = tid; i < 64 * (kResMaxLen + 1); i += kResThreads)
        s_cnt[i / (kResMaxLen + 1)][i % (kResMaxLen + 1)] = 0;
    __syncthreads();
    auto length = [&](int lr) {   // chunks of local row lr
        const int row = sp.row0 + lr;
        if (lr >= sp.ntl * kBlock || row >= pd.n) return 0;
        return min((__ldg(pd.rp + row + 1) - __ldg(pd.rp + row)) >> 2, kResMaxLen);
    };
    for (int lr = tid; lr < rows; lr += kResThreads) {
        const int len = length(lr);
        const unsigned same = __match_any_sync(0xffffffffu, len);
        if ((same & ((1u << lane) - 1)) == 0) s_cnt[lr >> 5][len] = uint16_t(__popc(same));
    }
    __syncthreads();
    if (tid <= kResMaxLen) {   // exclusive sums over the units; total per length
        int run = 0;
        for (int u = 0; u < units; ++u) {
            const int c = s_cnt[u][tid];
            s_cnt[u][tid] = uint16_t(run);
            run += c;
        }
        s_base[tid] = run;
    }
    __syncthreads();
    if (tid == 0) {   // longest first
        int run = 0;
        for (int l = kResMaxLen; l >= 0; --l) {
            const int c = s_base[l];
            s_base[l] = run;
            run += c;
        }
    }
    __syncthreads();
    for (int lr = tid; lr < rows; lr += kResThreads) {
        const int len = length(lr);
        const unsigned same = __match_any_sync(0xffffffffu, len);
        const int pos = s_base[len] + s_cnt[lr >> 5][len] + __popc(same & ((1u << lane) - 1));
        s_perm[s_rp.direct ? lr : pos] = uint16_t(lr);
    }
    __syncthreads();
    // sorted run s goes to warp s % 16, layer s / 16; slices are stored warp by
    // warp, so that a warp reads one contiguous stream
    for (int s = warp; s < units; s += kResWarps) {
        const int len = length(s_perm[s * 32 + lane]);
        const int mx = __reduce_max_sync(0xffffffffu, len);
        if (lane == 0) s_off[(s % kResWarps) * layers + s / kResWarps] = mx;
    }
    __syncthreads();
    if (tid == 0) {
        int run = 0;
        for (int i = 0; i < units; ++i) {
            const int c = s_off[i];
            s_rp.sl.len[size_t(rank) * units + i] = uint16_t(c);
            s_off[i] = run;
            run += c;
        }
        atomicMax(s_rp.sl.chunks, run);
    }
    __syncthreads();
    const int64_t e0 = sp.entry0(s_rp, rank);
    const WT* val = static_cast<const WT*>(pd.val);
    const int16_t* col16 = reinterpret_cast<const int16_t*>(pd.col);
    for (int s = warp; s < units; s += kResWarps) {
        const int slot = (s % kResWarps) * layers + s / kResWarps;
        const int lr = s_perm[s * 32 + lane];
        s_rp.sl.perm[size_t(rank) * rows + size_t(slot) * 32 + lane] = uint16_t(lr);
        const int row = sp.row0 + lr;
        const bool held = lr < sp.ntl * kBlock && row < pd.n;
        const int len = length(lr);
        const int mx = __reduce_max_sync(0xffffffffu, len);
        const int L = pd.lanes;
        for (int i = 0; i < mx; ++i) {
            // i-th stored chunk: set j, then c = j + L * (its rank in the set)
            int c = i, j = 0;
            for (int cnt = (mx + L - 1) / L; c >= cnt; cnt = (mx - j + L - 1) / L) {
                c -= cnt;
                ++j;
            }
            c = j + L * c;
            const int64_t o = e0 + (int64_t(s_off[slot] + i) * 32 + lane) * 4;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                int j = held ? row : sp.first;
                WT w = WT(0.0f);
                if (c < len) {
                    const int e = __ldg(pd.rp + row) + 4 * c + t;
                    j = pd.col16 ? row + col16[e] : pd.col[e];
                    w = val[e];
                }
                if (WIDE) static_cast<int32_t*>(s_rp.sl.col)[o + t] = j - sp.first;
                else static_cast<uint16_t*>(s_rp.sl.col)[o + t] = uint16_t(j - sp.first);
                static_cast<WT*>(s_rp.sl.val)[o + t] = w;
            }
        }
    }
}

// ------------------------------------------------------- cluster exchange
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// 16 bytes into another block's shared memory, counted by its mbarrier.
__device__ __forceinline__ void st_async(uint32_t dst, uint32_t bar, const uint4& v) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], "
                 "{%1, %2, %3, %4}, [%5];" ::"r"(dst), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w),
                 "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// mbar_wait with the acquire scope that st_async from other blocks needs,
// bounded by `limit` ns.
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity,
                                                  unsigned long long limit) {
    uint32_t ok = 0;
    unsigned long long t0 = 0;
    for (;;) {
        asm volatile(
            "{\n .reg .pred p;\n"
            " mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n"
            " selp.u32 %0, 1, 0, p;\n}"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity), "r"(20000u)
            : "memory");
        if (ok) return true;
        const unsigned long long t = globaltimer_ns();
        if (!t0) t0 = t;
        else if (t - t0 > limit) return false;
    }
}

// Barrier over the grid: arrival count with release / acquire at GPU scope,
// the wait bounded by `limit` ns.  False when it ran out.
__device__ __forceinline__ bool grid_barrier(uint32_t* bar, uint32_t target,
                                             unsigned long long limit) {
    __syncthreads();
    bool late = false;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        unsigned long long t0 = 0;
        for (;;) {
            uint32_t v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if (int32_t(v - target) >= 0) break;
            const unsigned long long t = globaltimer_ns();
            if (!t0) t0 = t;
            else if (t - t0 > limit) {
                late = true;
                break;
            }
        }
    }
    return !__syncthreads_or(late);
}

// Whether all blocks of an ordinary grid launch are on the device: each has
// added itself to *word, and they wait for the last one for at most `limit`
// ns.  The block that gives up first sets the top bit in exchange for a count
// below `group`: a word holds either the bit or the full count, never both in
// doubt, so all blocks leave, late ones included, or all go on (and then
// they are resident together, and their barriers can be met).
__device__ __forceinline__ bool grid_meet(uint32_t* word, uint32_t group, unsigned long long limit,
                                          ProbState* st) {
    int out = 0;
    if (threadIdx.x == 0) {
        unsigned long long t0 = 0;
        for (;;) {
            const uint32_t v = *reinterpret_cast<volatile uint32_t*>(word);
            if (v >> 31) {
                out = 1;
                break;
            }
            if (v >= group) break;
            const unsigned long long t = globaltimer_ns();
            if (!t0) t0 = t;
            else if (t - t0 > limit && atomicCAS(word, v, v | 0x80000000u) == v) {
                st->unstarted = 1;
                out = 1;
                break;
            }
        }
    }
    return !__syncthreads_or(out);
}

// ------------------------------------------------------------------ warps
// 128-bit sums over the lanes l, l ^ off, l ^ off/2, ... down to l ^ last
template <int OFF, int LAST>
__device__ __forceinline__ void warp_sum128(unsigned long long& lo, unsigned long long& hi) {
#pragma unroll
    for (int off = OFF; off >= LAST; off >>= 1) {
        const unsigned long long l2 = __shfl_xor_sync(0xffffffffu, lo, off);
        const unsigned long long h2 = __shfl_xor_sync(0xffffffffu, hi, off);
        add128(lo, hi, l2, h2);
    }
}

// Tests of the row evaluation.  For FP64 they work on the bits: an FP64
// compare holds the scheduler for 64 cycles, as any other FP64 instruction.
__device__ __forceinline__ bool is_one(float u) { return u == 1.0f; }
__device__ __forceinline__ bool is_one(double u) {
    return __double_as_longlong(u) == 0x3ff0000000000000ll;
}
__device__ __forceinline__ bool is_binary(float u) { return u == 0.0f || u == 1.0f; }
__device__ __forceinline__ bool is_binary(double u) {
    return is_one(u) || (__double_as_longlong(u) << 1) == 0ll;
}
__device__ __forceinline__ bool is_pos(float u) { return u > 0.0f; }
__device__ __forceinline__ bool is_pos(double u) {
    return __double_as_longlong(u) > 0ll && __double_as_longlong(u) <= 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool less(float a, float b) { return a < b; }
__device__ __forceinline__ bool less(double a, double b) {   // b is not NaN
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    const long long inf = 0x7ff0000000000000ll, mag = 0x7fffffffffffffffll;
    // order of the bits with negative values mirrored; -0 counts as +0
    const long long kx = x < 0 ? -(x & mag) : x, ky = y < 0 ? -(y & mag) : y;
    return (x & mag) <= inf && kx < ky;
}
// L S and D at class k of a row: only the entry of class s takes arithmetic,
// done once by the caller (ss = diag - b_s, ds = 1 - u_s) where FP64 is slow.
template <typename T>
__device__ __forceinline__ T ls_of(bool at, T diag, T bk, T ss) {
    if constexpr (sizeof(T) == 8) return at ? ss : -bk;
    else return at ? sub_(diag, bk) : -bk;
}
template <typename T>
__device__ __forceinline__ T d_of(bool at, T u, T ds) {
    if constexpr (sizeof(T) == 8) return at ? ds : -u;
    else return sub_(at ? T(1) : T(0), u);
}

// Four weights as loaded, widened when they are used.
template <typename WT> struct Weights4;
template <> struct Weights4<float> {
    float4 q;
    __device__ __forceinline__ void load(const float* p) {
        q = ld_stream(reinterpret_cast<const float4*>(p));
    }
    __device__ __forceinline__ void get(float (&v)[4]) const {
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    }
};
template <> struct Weights4<__nv_bfloat16> {
    uint2 q;
    __device__ __forceinline__ void load(const __nv_bfloat16* p) {
        q = ld_stream(reinterpret_cast<const uint2*>(p));
    }
    __device__ __forceinline__ void get(float (&v)[4]) const {
        v[0] = __uint_as_float(q.x << 16); v[1] = __uint_as_float(q.x & 0xffff0000u);
        v[2] = __uint_as_float(q.y << 16); v[3] = __uint_as_float(q.y & 0xffff0000u);
    }
};
template <> struct alignas(16) Weights4<double> {
    double2 a, b;
    __device__ __forceinline__ void load(const double* p) {
        a = ld_stream(reinterpret_cast<const double2*>(p));
        b = ld_stream(reinterpret_cast<const double2*>(p) + 1);
    }
    __device__ __forceinline__ void get(double (&v)[4]) const {
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    }
};

// Four columns as loaded.
template <bool WIDE> struct Cols4;
template <> struct Cols4<false> {
    uint2 q;
    __device__ __forceinline__ void load(const void* p) {
        q = ld_stream(static_cast<const uint2*>(p));
    }
    __device__ __forceinline__ uint32_t get(int t) const {
        const uint32_t w = t < 2 ? q.x : q.y;
        return t & 1 ? w >> 16 : w & 0xffffu;
    }
};
template <> struct Cols4<true> {
    int4 q;
    __device__ __forceinline__ void load(const void* p) {
        q = ld_stream(static_cast<const int4*>(p));
    }
    __device__ __forceinline__ uint32_t get(int t) const {
        return uint32_t(t == 0 ? q.x : t == 1 ? q.y : t == 2 ? q.z : q.w);
    }
};

// One chunk of a slice, as loaded from global or shared memory.
template <typename WT, bool WIDE, bool SHARED>
struct Chunk {
    Cols4<WIDE> c;
    Weights4<WT> w;
    static constexpr int kColBytes = WIDE ? 16 : 8;
    __device__ __forceinline__ void load(const char* col, const WT* val, int i) {
        if constexpr (SHARED) {
            c.q = *reinterpret_cast<const decltype(c.q)*>(col + i * (32 * kColBytes));
            w = *reinterpret_cast<const Weights4<WT>*>(val + i * 128);
        } else {
            c.load(col + size_t(i) * (32 * kColBytes));
            w.load(val + size_t(i) * 128);
        }
    }
    // the classes of its four columns
    __device__ __forceinline__ void gather(uint32_t tab, uint32_t (&s)[4]) const {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const uint32_t i = c.get(t);
            if (WIDE) s[t] = (uint32_t(ld_shared_u8(tab + (i >> 1))) >> ((i & 1) << 2)) & 15u;
            else s[t] = uint32_t(ld_shared_u8(tab + i));
        }
    }
    // Its four entries into the lane's bins, in entry order.  From shared
    // memory (where a warp's walk is one dependent chain) the four bins are
    // loaded together and equal classes resolved in registers, so a chunk
    // waits for its bins once, not four times; the walks from L2, which wait
    // for the slices, take the fewest instructions instead.
    template <typename T>
    __device__ __forceinline__ void add(const uint32_t (&s)[4], T* bins) const {
        T v[4];
        w.get(v);
        if constexpr (SHARED) {
            T b[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) b[t] = bins[s[t] * kResThreads];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
#pragma unroll
                for (int p = 0; p < t; ++p)
                    if (s[p] == s[t]) b[t] = b[p];
                b[t] = add_(b[t], v[t]);
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) bins[s[t] * kResThreads] = b[t];
        } else {
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                T* const p = bins + s[t] * kResThreads;
                *p = add_(*p, v[t]);
            }
        }
    }
};

// Exact objective after `cnt` steps whose totals are in ring[], one lane per
// step; the last step's q and a are returned too.  Called by one warp.
__device__ __forceinline__ void ring_energy(const ResSlot (*ring)[kNumR], int cnt,
                                            const StepCfg& cfg, double& E, double& last_q,
                                            double& last_a) {
    const int lane = threadIdx.x & 31;
    double g = 1.0, q = 0.0, a = 1.0;
    if (lane < cnt) {
        const ResSlot* S = ring[lane];
        g = fx_double(S[0].lo, S[0].hi);
        q = curvature(fx_double(S[5].lo, S[5].hi), fx_double(S[3].lo, S[3].hi),
                      fx_double(S[2].lo, S[2].hi), fx_double(S[1].lo, S[1].hi), cfg.inv_eps);
        a = step_length(g, q, cfg.step_rule);
    }
    for (int i = 0; i < cnt; ++i) {
        last_q = __shfl_sync(0xffffffffu, q, i);
        last_a = __shfl_sync(0xffffffffu, a, i);
        E = next_energy(E, __shfl_sync(0xffffffffu, g, i), last_q, last_a);
    }
}

// A slot's totals as decide() takes them: word l in lane l, then the flag.
__device__ __forceinline__ unsigned long long ring_word(const ResSlot* tot, int bad) {
    const int lane = threadIdx.x & 31;
    if (lane < kAccFlag) return lane & 1 ? tot[lane >> 1].hi : tot[lane >> 1].lo;
    return lane == kAccFlag && bad ? 1ull : 0ull;
}

// One group of blocks (a thread-block cluster, or the whole cooperative grid)
// iterates one problem.  Block `rank` holds a contiguous run of 256-row tiles,
// one row per thread and layer (local row layer * 512 + thread), whose U and
// L U stay in registers for the whole launch.  An iteration is
//   A  apply the step, choose the classes (the arithmetic of passA_staged) and
//      publish them: into every block's table (cluster), or through choice /
//      cls4 and a grid barrier, after which a block copies the rows its
//      columns can name (its own and the graph's bandwidth around them);
//   B  walk the slices, one row per lane, into the thread's bins; after each
//      of the L sets of chunks the bins are added to the row's sums (the order
//      of csr_bins with L lanes);
//   C  the per-row pieces of g, ||D||^2, <D,LU> and <D,LS>, tile totals (8
//      warp sums in warp order, as in block_accumulate) added exactly over the
//      block in 128 bits and exchanged; every block sums the blocks' totals
//      and takes the same step (quick_step, or decide()).
// L S is never stored: it follows from the row sums.  The totals of the last
// iterations stay in a ring from which rank 0 forms the objective in FP64
// every kResRing iterations.  Every sum has the order of the two-kernel path,
// so the iterates and statistics are bitwise the same.
//
// What bounds it: chains of dependent instructions (a warp issues about every
// tenth cycle, four warps a scheduler), for small problems the exchange, the
// longest row of the graph and the one-warp decision; registers (two values
// per row and class) allow no more warps.  Two launches an iteration took
// 14.3 us where this takes 4.7 (2,000-point k-NN graph, K = 5), 14.4 -> 8.4
// (22,470 points, K = 7), 24.0 -> 10.6 (613 x 487 image, K = 6) and 31.8 ->
// 21.4 (200,000-node block model, K = 10: the walk waits on L2 there).
//
// FORM kResWide: 4-bit class table and 32-bit columns; else one byte per row
// and 16-bit columns (a table of at most 65,536 rows), with kResShared the
// block's slices in shared memory for the whole launch.  EXACT: K == KMAX.
template <typename T, typename WT, int KMAX, bool EXACT, int FORM>
__global__ void __launch_bounds__(kResThreads, 1) k_resident(const __grid_constant__ ResArgs a) {
    constexpr int R = res_layers<T, KMAX>();
    constexpr bool WIDE = FORM == kResWide, SHARED = FORM == kResShared;
    // a cluster can have blocks without rows (plan(): FP64 alone takes more
    // blocks than pairs of tiles rounded up to a power of two)
    constexpr bool empties = sizeof(T) == 8;
    extern __shared__ __align__(128) unsigned char smraw[];
    __shared__ __align__(16) ResSlot s_slot[kResMaxCluster][kNumR];
    __shared__ __align__(16) ResSlot s_ring[kResRing][kNumR];   // totals of iteration it % kResRing
    __shared__ __align__(16) T s_part[kNumR][R * kResWarps];
    __shared__ __align__(16) uint4 s_note;      // from blocks without rows, never read
    __shared__ __align__(8) uint64_t bars[2];   // classes, totals from the cluster's blocks
    __shared__ int s_bad;                       // a total is not finite
    __shared__ T s_alpha;
    __shared__ int s_done, s_fail;
    __shared__ QuickCfg s_quick;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = int(blockIdx.x);
    ProbState* const st = a.state;
    const ResProb& s_rp = a.p;
    const ProbDesc& pd = a.p.pd;
    if (tid == 64) {
        s_done = ld_cg(&st->done);
        s_fail = s_bad = 0;
        mbar_init(&bars[0], 1);
        mbar_init(&bars[1], 1);
    }
    __syncthreads();
    if (s_done) return;   // the same in every block of the group
    if (a.meet_ns && tid == 0) atomicAdd(a.bar + 1, 1u);   // see grid_meet
    const int K = EXACT ? KMAX : pd.K, n = pd.n, L = pd.lanes;
    const int64_t np = pd.npad;
    const int layers = s_rp.layers;
    const ResSpan sp(pd, rank, a.group, a.cluster);
    const int nu = sp.ntl * (kBlock / 32);
    const bool multi = a.cluster && a.group > 1;
    const T* __restrict__ diag = static_cast<const T*>(pd.diag);
    const T c2 = c2_of<T>(pd), om = om_of<T>(pd);
    const bool greedy = pd.oracle == 0;   // admissible classes: u > 0 (greedy), or all

    // ------------------------------------------------------- shared memory
    T* const slab = reinterpret_cast<T*>(smraw);            // [layers][K][512]: row sums
    T* const bins = slab + size_t(layers) * K * kResThreads;   // [K][512]
    uint16_t* const s_perm = reinterpret_cast<uint16_t*>(bins + size_t(K) * kResThreads);
    uint16_t* const s_len = s_perm + layers * kResThreads;
    uint8_t* const tab = reinterpret_cast<uint8_t*>(s_len + layers * kResWarps);
    const int units = layers * kResWarps;
    for (int i = tid; i < layers * kResThreads / 8; i += kResThreads)
        reinterpret_cast<uint4*>(s_perm)[i] =
            reinterpret_cast<const uint4*>(s_rp.sl.perm + size_t(rank) * layers * kResThreads)[i];
    for (int i = tid; i < units; i += kResThreads) s_len[i] = s_rp.sl.len[size_t(rank) * units + i];

    // ---- the rows of this thread, with a pending step of an earlier launch applied
    T U[R][KMAX], LU[R][KMAX];
    T best[R];     // G' of the chosen class
    int meta[R];   // class | moved << 7 | (fidelity class + 1) << 8
    T alpha = alpha_of<T>(st), oma = sub_(T(1), alpha);
    {
        const T* __restrict__ Ub = static_cast<const T*>(pd.U);
        const T* __restrict__ LUb = static_cast<const T*>(pd.LU);
        const T* __restrict__ LSb = static_cast<const T*>(pd.LS);
        const bool upd = ld_cg(&st->has_update) != 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int lr = r * kResThreads + tid, row = sp.row0 + lr;
            meta[r] = 0;
            if (lr < sp.ntl * kBlock && row < n) {
                const int sv = ld_cg(pd.choice + row);
                meta[r] = sv | ((int(__ldg(pd.fid + row)) + 1) << 8);
#pragma unroll
                for (int k = 0; k < KMAX; ++k)
                    if (k < K) {
                        U[r][k] = ld_cg(Ub + k * np + row);
                        LU[r][k] = ld_cg(LUb + k * np + row);
                    }
                if (upd) {   // as in phase A
                    const bool mv = (sv & kActiveBit) != 0;
                    const T um = mv ? oma : T(1), ua = mv ? alpha : T(0);
#pragma unroll
                    for (int k = 0; k < KMAX; ++k)
                        if (k < K) {
                            LU[r][k] = fma_(alpha, ld_cg(LSb + k * np + row), mul_(oma, LU[r][k]));
                            U[r][k] = fma_(um, U[r][k], k == (sv & 0x7f) ? ua : T(0));
                        }
                }
            }
        }
    }
    const int cur = ld_cg(&st->cur);
    StepIn in;     // warp 0: inputs of the next decision, E as of the last statistics
    in.E = ld_cg(&st->in[cur].E);
    in.g0 = ld_cg(&st->in[cur].g0);
    in.iter = ld_cg(&st->in[cur].iter);
    in.g0_set = ld_cg(&st->in[cur].g0_set);
    const int err0 = ld_cg(&st->err);
    if (tid == 0) s_quick = quick_cfg(step_cfg(pd), in.g0);
    double last_q = 0.0, last_a = 0.0;
    __syncthreads();   // s_len
    // this warp's stream of chunks, 32 lanes x 4 entries each
    int chunks = 0, before = 0;
    for (int l = 0; l < layers; ++l) chunks += s_len[warp * layers + l];
    for (int i = 0; i < warp * layers; ++i) before += s_len[i];
    constexpr int kColBytes = WIDE ? 16 : 8;
    const int64_t ent0 = sp.entry0(s_rp, rank);
    const char* col0 = static_cast<const char*>(s_rp.sl.col) + ent0 / 4 * kColBytes;
    const WT* val0 = static_cast<const WT*>(s_rp.sl.val) + ent0;
    if constexpr (SHARED) {   // the block's slices after the class table
        int all = 0;
        for (int i = 0; i < units; ++i) all += s_len[i];
        WT* const sv = reinterpret_cast<WT*>(tab + sp.window);
        char* const sc = reinterpret_cast<char*>(sv + size_t(all) * 128);
        for (int i = tid; i < all * 32; i += kResThreads) {
            reinterpret_cast<uint2*>(sc)[i] = __ldg(reinterpret_cast<const uint2*>(col0) + i);
            Weights4<WT> w;
            w.load(val0 + size_t(i) * 4);
            reinterpret_cast<Weights4<WT>*>(sv)[i] = w;
        }
        col0 = sc;
        val0 = sv;
    }
    col0 += (size_t(before) * 32 + lane) * kColBytes;
    val0 += (size_t(before) * 32 + lane) * 4;
    uint32_t target = 0;
    if (a.cluster) cluster_barrier();   // every block's shared memory can be written
    // nothing but loads so far: without its blocks the launch leaves no trace
    if (a.meet_ns && !grid_meet(a.bar + 1, uint32_t(a.group), a.meet_ns, st)) return;
    __syncthreads();

    for (int it = 0;;) {
        if (multi && tid == 0) {
            const int others = pd.ntiles * (kBlock / 32) - nu;
            const int notes = empties ? max(a.group - pd.ntiles, 0) - (nu == 0 ? 1 : 0) : 0;
            mbar_expect_tx(&bars[0], uint32_t(others) * (WIDE ? 16u : 32u) +
                                         uint32_t(notes + a.expect_extra) * 16u);
            mbar_expect_tx(&bars[1], uint32_t(a.group - 1) * kNumR * 16u);
        }
        // A block's classes also say that it has read the last totals, so that
        // the next may overwrite them.  A block without rows (fewer tiles than
        // blocks) has none to send: it sends a note instead.
        if (empties && multi && nu == 0 && warp == 0 && lane < a.group && lane != rank)
            st_async(map_rank(smem_u32(&s_note), uint32_t(lane)),
                     map_rank(smem_u32(&bars[0]), uint32_t(lane)), make_uint4(0u, 0u, 0u, 0u));
        // ---------------------------------------------------------- phase A
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int u0 = r * kResWarps + warp;   // local 32-row unit
            if (u0 >= nu) continue;
            const int row = sp.row0 + u0 * 32 + lane;
            int s = 0;
            if (row < n) {
                const int f = (meta[r] >> 8) - 1;
                const int sv = meta[r] & 0x7f;
                bool one = false;
                if (it > 0) {
                    const T* b = slab + size_t(r) * K * kResThreads + tid;
                    const T dg = pd.comb ? __ldg(diag + row) : T(1);
                    const bool mv = (meta[r] & kActiveBit) != 0;
                    // rows that stay: u = 1 u + 0; moved rows: fma(oma, u, 0) is oma u
                    const T um = mv ? oma : T(1), ua = mv ? alpha : T(0);
                    T ss = T(0);
                    if constexpr (sizeof(T) == 8) ss = sub_(dg, b[sv * kResThreads]);
#pragma unroll
                    for (int k = 0; k < KMAX; ++k)
                        if (k < K) {
                            const T ls = ls_of(k == sv, dg, b[k * kResThreads], ss);
                            LU[r][k] = fma_(alpha, ls, mul_(oma, LU[r][k]));
                            U[r][k] = fma_(um, U[r][k], k == sv ? ua : T(0));
                            one = one || is_one(U[r][k]);
                        }
                }
                // a row is binary only if one of its entries is 1
                bool binary = false;
                int at = sv;
                if (it == 0 || one) {
                    binary = true;
                    int f1 = -1;
#pragma unroll
                    for (int k = 0; k < KMAX; ++k)
                        if (k < K) {
                            const T u = U[r][k];
                            binary = binary && is_binary(u);
                            if (f1 < 0 && is_one(u)) f1 = k;
                        }
                    at = f1 < 0 ? 0 : f1;
                }
                if (greedy && binary) {
                    s = at;
                    meta[r] = (meta[r] & ~0xff) | s;
                } else {
                    T gs = inf_<T>();
                    s = -1;
                    if (f < 0) {
#pragma unroll
                        for (int k = 0; k < KMAX; ++k)
                            if (k < K) {
                                const T u = U[r][k];
                                const T gk = fma_(-c2, u, LU[r][k]);
                                if ((!greedy || is_pos(u)) && less(gk, gs)) {
                                    gs = gk;
                                    s = k;
                                }
                            }
                    } else {
#pragma unroll
                        for (int k = 0; k < KMAX; ++k)
                            if (k < K) {
                                const T u = U[r][k];
                                const T gk = fma_(om, sub_(u, k == f ? T(1) : T(0)),
                                                  fma_(-c2, u, LU[r][k]));
                                if ((!greedy || is_pos(u)) && less(gk, gs)) {
                                    gs = gk;
                                    s = k;
                                }
                            }
                    }
                    if (s < 0) {   // no finite candidate: the gap becomes NaN
#pragma unroll
                        for (int k = KMAX - 1; k >= 0; --k)
                            if (k < K && (!greedy || is_pos(U[r][k]))) s = k;
                        if (s < 0) s = 0;
                        gs = CUDART_NAN_F;
                    }
                    best[r] = gs;
                    bool at_vertex = false;
                    if (binary) {
#pragma unroll
                        for (int k = 0; k < KMAX; ++k)
                            if (k < K && k == s) at_vertex = is_one(U[r][k]);
                    }
                    meta[r] = (meta[r] & ~0xff) | s | (at_vertex ? 0 : int(kActiveBit));
                }
            }
            // publish the unit's classes
            const int gu = sp.t0 * (kBlock / 32) + u0;
            if (!WIDE) {
                if (a.cluster) {
                    uint8_t* const t = tab + gu * 32;
                    t[lane] = uint8_t(s);
                    if (multi) {
                        __syncwarp();
                        if (lane < a.group && lane != rank) {
                            const uint4 v0 = reinterpret_cast<const uint4*>(t)[0];
                            const uint4 v1 = reinterpret_cast<const uint4*>(t)[1];
                            const uint32_t dst = map_rank(smem_u32(t), uint32_t(lane));
                            const uint32_t bar = map_rank(smem_u32(&bars[0]), uint32_t(lane));
                            st_async(dst, bar, v0);
                            st_async(dst + 16, bar, v1);
                        }
                    }
                } else if (row < n) {
                    pd.choice[row] = uint8_t(meta[r] & 0xff);
                }
            } else {   // 32 classes in 16 bytes
                const uint32_t nib = uint32_t(s) << (4 * (lane & 7));
                uint4 v;
                v.x = __reduce_or_sync(0xffffffffu, lane < 8 ? nib : 0u);
                v.y = __reduce_or_sync(0xffffffffu, (lane >> 3) == 1 ? nib : 0u);
                v.z = __reduce_or_sync(0xffffffffu, (lane >> 3) == 2 ? nib : 0u);
                v.w = __reduce_or_sync(0xffffffffu, (lane >> 3) == 3 ? nib : 0u);
                if (a.cluster) {
                    uint4* const t = reinterpret_cast<uint4*>(tab) + gu;
                    if (lane == rank) *t = v;
                    else if (lane < a.group)
                        st_async(map_rank(smem_u32(t), uint32_t(lane)),
                                 map_rank(smem_u32(&bars[0]), uint32_t(lane)), v);
                } else if (lane == 0 && gu * 32 < n) {
                    reinterpret_cast<uint4*>(pd.cls4)[gu] = v;
                }
            }
        }
        // from L2 the walk's first chunks are on their way while the classes
        // are exchanged
        Chunk<WT, WIDE, SHARED> P, Q;
        if (!SHARED && chunks > 0) P.load(col0, val0, 0);
        if (!SHARED && chunks > 1) Q.load(col0, val0, 1);
        bool alive = true;
        if (a.cluster) {
            const bool got = !multi || mbar_wait_cluster(&bars[0], uint32_t(it & 1), a.wait_ns);
            alive = !__syncthreads_or(!got);
        } else {
            target += uint32_t(a.group);
            alive = grid_barrier(a.bar, target + uint32_t(a.expect_extra), a.wait_ns);
            if (!WIDE) {
                const uint4* src = reinterpret_cast<const uint4*>(pd.choice + sp.first);
                for (int i = tid; i < sp.window / 16; i += kResThreads) {
                    uint4 v = __ldcg(src + i);
                    v.x &= 0x7f7f7f7fu;
                    v.y &= 0x7f7f7f7fu;
                    v.z &= 0x7f7f7f7fu;
                    v.w &= 0x7f7f7f7fu;
                    reinterpret_cast<uint4*>(tab)[i] = v;
                }
            } else {
                const uint4* src = reinterpret_cast<const uint4*>(pd.cls4) + sp.first / 32;
#pragma unroll 8
                for (int i = tid; i < sp.window / 32; i += kResThreads)
                    reinterpret_cast<uint4*>(tab)[i] = __ldcg(src + i);
            }
            __syncthreads();
        }
        if (!alive) {   // a wait ran out (the same in all threads)
            if (tid == 0) s_fail = 1;
            break;
        }

        // ---------------------------------------------------------- phase B
        {
            const uint32_t tb = smem_u32(tab);
            // a set's bins added to the row's sums (position l of this warp), and cleared
            auto flush = [&](T* my, int l, int j) {
                const int lr = s_perm[(warp * layers + l) * 32 + lane];
                T* const out = slab + size_t(lr >> 9) * K * kResThreads + (lr & (kResThreads - 1));
#pragma unroll
                for (int k = 0; k < KMAX; ++k)
                    if (k < K) {
                        const T b = my[k * kResThreads];
                        out[k * kResThreads] = j == 0 ? b : add_(out[k * kResThreads], b);
                        my[k * kResThreads] = T(0);
                    }
            };
            auto clear = [&](T* my) {
#pragma unroll
                for (int k = 0; k < KMAX; ++k)
                    if (k < K) my[k * kResThreads] = T(0);
            };
            if constexpr (SHARED) {
                const char* cp = col0;
                const WT* vp = val0;
                // the next chunk and its classes are loaded before one is added
                auto walk = [&](T* my, int cnt) {
                    if (cnt <= 0) return;
                    Chunk<WT, WIDE, SHARED> A, B;
                    uint32_t sa[4], sb[4];
                    A.load(cp, vp, 0);
                    A.gather(tb, sa);
                    int i = 0;
                    for (; i + 2 < cnt; i += 2) {
                        B.load(cp, vp, i + 1);
                        B.gather(tb, sb);
                        A.add(sa, my);
                        A.load(cp, vp, i + 2);
                        A.gather(tb, sa);
                        B.add(sb, my);
                    }
                    if (i + 1 < cnt) {
                        B.load(cp, vp, i + 1);
                        B.gather(tb, sb);
                    }
                    A.add(sa, my);
                    if (i + 1 < cnt) B.add(sb, my);
                    cp += cnt * (32 * kColBytes);
                    vp += cnt * 128;
                };
                if (s_rp.direct) {   // rows in place: the bins are the row's sums
                    for (int l = 0; l < layers; ++l) {
                        T* const my = slab + size_t(l) * K * kResThreads + tid;
                        clear(my);
                        walk(my, s_len[warp * layers + l]);
                    }
                } else {
                    T* const my = bins + tid;
                    clear(my);
                    for (int l = 0; l < layers; ++l) {
                        const int len = s_len[warp * layers + l];
                        for (int j = 0; j < L; ++j) {
                            walk(my, (len - j + L - 1) / L);
                            flush(my, l, j);
                        }
                    }
                }
            } else {
                T* const my = bins + tid;
                int pos = 0, l = 0, j = 0, len = s_len[warp * layers];
                int rem = (len + L - 1) / L;   // chunks left in set j of slice l
                clear(my);
                // set j of slice l is complete: go on to the next set that has chunks
                auto next = [&] {
                    do {
                        flush(my, l, j);
                        if (++j == L) {
                            j = 0;
                            if (++l == layers) return;
                            len = s_len[warp * layers + l];
                        }
                        rem = (len - j + L - 1) / L;
                    } while (rem <= 0);
                };
                if (rem == 0) next();
                while (pos < chunks) {
                    uint32_t sc[4];
                    P.gather(tb, sc);
                    P.add(sc, my);
                    if (pos + 2 < chunks) P.load(col0, val0, pos + 2);
                    ++pos;
                    if (--rem == 0) next();
                    if (pos == chunks) break;
                    Q.gather(tb, sc);
                    Q.add(sc, my);
                    if (pos + 2 < chunks) Q.load(col0, val0, pos + 2);
                    ++pos;
                    if (--rem == 0) next();
                }
            }
        }
        __syncthreads();

        // ---------------------------------------------------------- phase C
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int u0 = r * kResWarps + warp;
            if (u0 >= nu) continue;
            const int row = sp.row0 + u0 * 32 + lane;
            T x[kNumR] = {T(0), T(0), T(0), T(0), T(0), T(0)};
            if (row < n && (meta[r] & kActiveBit)) {
                const int s = meta[r] & 0x7f, f = (meta[r] >> 8) - 1;
                const T* b = slab + size_t(r) * K * kResThreads + tid;
                const T dg = pd.comb ? __ldg(diag + row) : T(1);
                T ss = T(0), ds = T(0);
                if constexpr (sizeof(T) == 8) {
                    ss = sub_(dg, b[s * kResThreads]);
#pragma unroll
                    for (int k = 0; k < KMAX; ++k)
                        if (k < K) ds = k == s ? U[r][k] : ds;
                    ds = sub_(T(1), ds);
                }
#pragma unroll
                for (int k = 0; k < KMAX; ++k)
                    if (k < K) {
                        const T u = U[r][k], lu = LU[r][k];
                        T gk = fma_(-c2, u, lu);
                        if (f >= 0) gk = fma_(om, sub_(u, k == f ? T(1) : T(0)), gk);
                        const T d = d_of(k == s, u, ds);
                        const T ls = ls_of(k == s, dg, b[k * kResThreads], ss);
                        x[0] = fma_(u, sub_(gk, best[r]), x[0]);
                        x[1] = fma_(d, d, x[1]);
                        x[3] = fma_(d, lu, x[3]);
                        x[5] = fma_(d, ls, x[5]);
                    }
                x[4] = T(1);
                if (f >= 0) x[2] = fma_(om, x[1], T(0));
            }
            const T z = warp_sum6(x);
            if (sum6_lane(lane)) s_part[sum6_index(lane)][u0] = z;
        }
        __syncthreads();
        ResSlot* const tot = s_ring[it % kResRing];
        if (warp < kNumR) {
            unsigned long long lo = 0ull, hi = 0ull;
            bool ok = true;
            if (lane < sp.ntl) {
                T sum = T(0);
#pragma unroll
                for (int w = 0; w < kBlock / 32; ++w)
                    sum = add_(sum, s_part[warp][lane * (kBlock / 32) + w]);
                ok = fx_total_split(sum, lo, hi);
            }
            static_assert(R * kResTilesPerLayer <= 8, "tiles of a block");
            if (__any_sync(0xffffffffu, !ok)) {
                lo = 0ull;
                hi = kResBad;
            } else {
                warp_sum128<4, 1>(lo, hi);   // lanes 0..7 hold the tiles
                lo = __shfl_sync(0xffffffffu, lo, 0);
                hi = __shfl_sync(0xffffffffu, hi, 0);
            }
            if (a.cluster) {
                if (lane == rank) s_slot[rank][warp] = ResSlot{lo, hi};
                else if (lane < a.group)
                    st_async(map_rank(smem_u32(&s_slot[rank][warp]), uint32_t(lane)),
                             map_rank(smem_u32(&bars[1]), uint32_t(lane)),
                             make_uint4(uint32_t(lo), uint32_t(lo >> 32), uint32_t(hi),
                                        uint32_t(hi >> 32)));
            } else if (lane == 0) {
                reinterpret_cast<ulonglong2*>(a.slots)[warp * a.group + rank] = make_ulonglong2(lo, hi);
            }
        }
        if (a.cluster) {
            __syncthreads();   // the block's own slots
            if (warp == 0) {
                // lane (p, q): quantity q of the blocks p, p + 4, ...
                const int q = lane & 7, p = lane >> 3;
                alive = !multi || mbar_wait_cluster(&bars[1], uint32_t(it & 1), a.wait_ns);
                alive = __all_sync(0xffffffffu, alive);
                unsigned long long lo = 0ull, hi = 0ull;
                bool bad = false;
                if (alive && q < kNumR)
                    for (int d = p; d < a.group; d += 4) {
                        const ResSlot v = s_slot[d][q];
                        bad |= v.hi == kResBad;
                        add128(lo, hi, v.lo, v.hi);
                    }
                bad = __any_sync(0xffffffffu, bad);
                warp_sum128<16, 8>(lo, hi);
                if (lane < kNumR) tot[lane] = ResSlot{lo, hi};
                if (lane == 0 && bad) s_bad = 1;
                __syncwarp();
            }
        } else {
            target += uint32_t(a.group);
            alive = grid_barrier(a.bar, target + uint32_t(a.expect_extra), a.wait_ns);
            if (warp < kNumR) {
                unsigned long long lo = 0ull, hi = 0ull;
                bool bad = false;
                // all loads first: one round trip to L2 for up to kResMaxGrid blocks
                ulonglong2 v[kResMaxGrid / 32];
#pragma unroll
                for (int i = 0; i < kResMaxGrid / 32; ++i) {
                    const int d = lane + 32 * i;
                    v[i] = make_ulonglong2(0ull, 0ull);
                    if (d < a.group)
                        v[i] = __ldcg(reinterpret_cast<const ulonglong2*>(a.slots) + warp * a.group + d);
                }
#pragma unroll
                for (int i = 0; i < kResMaxGrid / 32; ++i) {
                    bad |= v[i].y == kResBad;
                    add128(lo, hi, v[i].x, v[i].y);
                }
                bad = __any_sync(0xffffffffu, bad);
                warp_sum128<16, 1>(lo, hi);
                if (lane == 0) {
                    tot[warp] = ResSlot{lo, hi};
                    if (bad) s_bad = 1;
                }
            }
            __syncthreads();
        }
        if (warp == 0) {
            float af = 0.f;
            T step = T(0);
            int done = 0;
            const StepCfg cfg = step_cfg(pd);
            bool quick = false;
            if (sizeof(T) == 4 && err0 == 0 && in.g0_set) {
                ResSlot v = tot[min(lane, kNumR - 1)];
                if (lane == 6) {
                    const ResSlot nW = tot[2], tLU = tot[3];   // v is tot[5]
                    add128(v.lo, v.hi, ~tLU.lo, ~tLU.hi);
                    add128(v.lo, v.hi, 1ull, 0ull);
                    add128(v.lo, v.hi, nW.lo, nW.hi);
                }
                quick = quick_step(v.lo, v.hi, s_bad != 0, in.iter, s_quick, af);
            }
            if (quick) {
                step = T(af);
            } else {
                const Decision d = decide(ring_word(tot, s_bad), in, err0, cfg);
                if (!in.g0_set && lane == 0) s_quick = quick_cfg(cfg, d.g0);
                in.g0 = d.g0;
                in.g0_set = 1;
                done = d.done;
                step = T(d.a);
            }
            if (lane == 0) {
                s_alpha = step;
                s_done = done;
                if (!alive) s_fail = 1;
            }
            ++in.iter;
        }
        __syncthreads();
        const bool end = s_done || s_fail || ++it >= a.iters;
        if (!end) {
            alpha = s_alpha;
            oma = sub_(T(1), alpha);
        }
        // the ring is full, and at least one more iteration follows
        if (!end && it % kResRing == 0 && rank == 0 && warp == 0)
            ring_energy(s_ring, kResRing, step_cfg(pd), in.E, last_q, last_a);
        if (end) {
            if (s_fail) break;
            // statistics: the steps since the last ones, then this decision
            if (rank == 0 && warp == 0) {
                const StepCfg cfg = step_cfg(pd);
                const int done = s_done;
                if (done) ++it;   // counted above otherwise
                const int lastslot = (it - 1) % kResRing;
                ring_energy(s_ring, lastslot, cfg, in.E, last_q, last_a);
                StepIn di = in;
                di.iter = in.iter - 1;
                const Decision d = decide(ring_word(s_ring[lastslot], s_bad), di, err0, cfg);
                commit_decision(st, d, next_in(di, d), cur);
                if (d.done && it > 1 && lane == 0) {   // q and alpha of the last step taken
                    st->q = last_q;
                    st->alpha = last_a;
                    st->alpha_f = float(last_a);
                }
            }
            break;
        }
    }

    __syncthreads();
    // A wait ran out: this block writes no row back.  Another may have finished
    // its last exchange and store its rows and the decision: `err`, which only
    // a restart clears, then overrules them (settle).
    if (s_fail) {
        if (tid == 0) {
            atomicExch(&st->err, 1);
            st->status = -7;   // FW_ERR_TIMEOUT
            st->done = 1;
        }
        // what other blocks have sent here, and nobody waits for now, arrives
        // before this block lets the cluster end (a few microseconds at most)
        if (a.cluster) {
            const unsigned long long t0 = globaltimer_ns();
            while (globaltimer_ns() - t0 < 100000ull) {
            }
        }
    } else {
        // ---- write the iterate back; the last evaluation's choice and L S with it
        T* __restrict__ Ub = static_cast<T*>(pd.U);
        T* __restrict__ LUb = static_cast<T*>(pd.LU);
        T* __restrict__ LSb = static_cast<T*>(pd.LS);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int u0 = r * kResWarps + warp;
            const int row = sp.row0 + u0 * 32 + lane;
            if (u0 >= nu) continue;
            const int s = meta[r] & 0x7f;
            const int hi = __shfl_down_sync(0xffffffffu, s, 1);
            if (row >= n) continue;
            const T* b = slab + size_t(r) * K * kResThreads + tid;
            const T dg = pd.comb ? __ldg(diag + row) : T(1);
            pd.choice[row] = uint8_t(meta[r] & 0xff);
            if ((lane & 1) == 0) pd.cls4[row >> 1] = uint8_t(s | (hi << 4));
#pragma unroll
            for (int k = 0; k < KMAX; ++k)
                if (k < K) {
                    const T bk = b[k * kResThreads];
                    Ub[k * np + row] = U[r][k];
                    LUb[k * np + row] = LU[r][k];
                    LSb[k * np + row] = (k == s) ? sub_(dg, bk) : -bk;
                }
        }
    }
    if (a.cluster) cluster_barrier();   // no block leaves while another may write its shared memory
}

// -------------------------------------------------------------- launchers
// Device bytes of a planned problem's slices, slots and counters.
inline size_t res_up(size_t x) { return (x + 255) / 256 * 256; }
inline size_t res_bytes(const ResPlan& p) {
    return res_up(256 + sizeof(ResSlot) * kNumR * size_t(p.group)) +
           res_up(2 * size_t(p.group) * p.layers * kResThreads) +
           res_up(2 * size_t(p.group) * p.layers * kResWarps) +
           res_up(size_t(p.entries) * (p.form == kResWide ? 4 : 2)) +
           res_up(size_t(p.entries) * p.welem);
}
// The launch parameters (but the iteration count) with those arrays at m.
inline ResArgs res_args(const ResPlan& p, const ProbDesc& pd, ProbState* st, char* m,
                        unsigned long long wait_ns, int expect_extra) {
    ResArgs a{};
    a.state = st;
    a.wait_ns = wait_ns;
    a.expect_extra = std::max(expect_extra, 0);
    a.group = p.group;
    a.cluster = p.cluster;
    a.p.pd = pd;
    a.p.slack = p.slack;
    a.p.layers = p.layers;
    a.p.direct = p.direct;
    a.bar = reinterpret_cast<uint32_t*>(m);
    a.p.sl.chunks = reinterpret_cast<int*>(m + 128);
    a.slots = reinterpret_cast<ResSlot*>(m + 256);
    m += res_up(256 + sizeof(ResSlot) * kNumR * size_t(p.group));
    a.p.sl.perm = reinterpret_cast<uint16_t*>(m);
    m += res_up(2 * size_t(p.group) * p.layers * kResThreads);
    a.p.sl.len = reinterpret_cast<uint16_t*>(m);
    m += res_up(2 * size_t(p.group) * p.layers * kResWarps);
    a.p.sl.col = m;
    m += res_up(size_t(p.entries) * (p.form == kResWide ? 4 : 2));
    a.p.sl.val = m;
    return a;
}
// Build the slices a names, wait for them, and choose the form that their
// size allows.
inline cudaError_t res_build(ResKern* k, const ResArgs& a, ResPlan& p, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(a.bar, 0, 256, s);
    if (e == cudaSuccess) e = k->slice(a.p, p, s);
    int chunks = 0;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&chunks, a.p.sl.chunks, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess) k->sliced(p, chunks);
    return e;
}
// Enqueue up to `iters` iterations, and no more than kResIters and one last
// evaluation: callers with more to do launch again.
inline cudaError_t res_launch(ResKern* k, ResArgs a, const ResPlan& p, int iters, cudaStream_t s) {
    a.iters = std::min(iters, kResIters + 1);
    const cudaError_t e =
        a.cluster ? cudaSuccess : cudaMemsetAsync(a.bar, 0, 2 * sizeof(uint32_t), s);
    return e == cudaSuccess ? k->launch(a, p, s) : e;
}

template <typename T, typename WT, int KMAX, bool EXACT>
class ResKernImpl final : public ResKern {
public:
    static constexpr int R = res_layers<T, KMAX>();

    bool plan(const ProbDesc& pd, int maxrow, int64_t nnz_pad, int sms, int share,
              ResPlan& p) override {
        p = ResPlan();
        if (!pd.cls4 || pd.tile_rows != kBlock) return false;
        const int maxlen = (maxrow + 3) / 4;
        if (maxlen > kResMaxLen) return false;
        const int nt = pd.ntiles;
        const int pairs = (nt + kResTilesPerLayer - 1) / kResTilesPerLayer;
        sms = std::min(sms, kResMaxGrid);
        auto cluster_of = [](int blocks) {
            int c = 1;
            while (c < blocks) c *= 2;
            return c;
        };
        // fewest blocks first when the problem shares the device: a block's
        // iteration takes 4.8 us with one layer, 7 with two, 12 with four
        for (int t = std::min(share, R); t > 0; --t) {
            const int blocks = (pairs + t - 1) / t;
            const int c = cluster_of(blocks);
            if (c <= kResMaxCluster && attempt(pd, nt, c, 1, p, maxlen, nnz_pad)) return true;
            if (blocks <= sms && attempt(pd, nt, blocks, 0, p, maxlen, nnz_pad)) return true;
        }
        if (sizeof(T) == 8) {   // FP64 issue bounds it: one tile a block, as many SMs as that takes
            const int ct = cluster_of(nt);
            if (ct <= kResMaxCluster && attempt(pd, nt, ct, 1, p, maxlen, nnz_pad)) return true;
            if (nt <= sms && attempt(pd, nt, nt, 0, p, maxlen, nnz_pad)) return true;
        }
        // All SMs, though fewer would do for the fullest block's tiles: 131 and 146
        // blocks in place of 152 took 1 to 2% more (sbm200k, 613 x 487 image).
        const int c = std::min(kResMaxCluster, cluster_of(pairs)), g = std::min(sms, pairs);
        // A cluster exchanges in 400 cycles what the grid barrier takes 2,300
        // for, but has 16 SMs: with more than two layers a block the grid's
        // SMs win (k-NN graphs, K = 7: 12,000 rows 7.0 us an iteration against
        // 9.7, 22,470 rows 12.2 against 8.5).
        const bool small = pairs <= 2 * kResMaxCluster;
        return (small && attempt(pd, nt, c, 1, p, maxlen, nnz_pad)) ||
               attempt(pd, nt, g, 0, p, maxlen, nnz_pad) ||
               attempt(pd, nt, c, 1, p, maxlen, nnz_pad);
    }
    bool attempt(const ProbDesc& pd, int nt, int group, int cluster, ResPlan& p, int maxlen,
                 int64_t nnz_pad) {
        const int per = (nt + group - 1) / group;
        const int l = (per + kResTilesPerLayer - 1) / kResTilesPerLayer;
        if (l > R) return false;
        // rows of nearly one length (pixel grids) are walked in place
        const int direct = pd.lanes == 1 && 4.0 * maxlen * pd.n <= 1.15 * double(nnz_pad);
        int64_t win = int64_t(nt) * kBlock;   // ResSpan::window of the largest block
        if (!cluster)
            win = std::min(win, (int64_t(per) * kBlock + 2 * int64_t(pd.band) + 95) / 32 * 32);
        for (int form : {int(kResNarrow), int(kResWide)}) {
            const bool wide = form == kResWide;
            if (!wide && win > 65536) continue;
            const size_t sm = res_smem(sizeof(T), pd.K, l, size_t(wide ? win / 2 : win) + 32);
            if (sm > size_t(kResSmemMax)) continue;
            p.group = group;
            p.cluster = cluster;
            p.layers = l;
            p.form = form;
            p.smem = sm;
            p.direct = direct;
            p.slack = direct ? int64_t(l) * kResThreads * 4 * maxlen : res_slack(maxlen);
            p.entries = (direct ? 0 : nnz_pad + 128) + p.slack * group;
            p.welem = sizeof(WT);
            if (fits(p)) return true;
        }
        p = ResPlan();
        return false;
    }
    void sliced(ResPlan& p, int chunks) override {
        if (p.form != kResNarrow) return;
        const size_t sm = p.smem + size_t(chunks) * 128 * (2 + sizeof(WT));
        if (sm > size_t(kResSmemMax)) return;
        ResPlan q = p;
        q.form = kResShared;
        q.smem = sm;
        if (fits(q)) p = q;
    }
    template <typename F>
    auto with(int form, F f) {
        return form == kResWide     ? f(k_resident<T, WT, KMAX, EXACT, kResWide>)
               : form == kResNarrow ? f(k_resident<T, WT, KMAX, EXACT, kResNarrow>)
                                    : f(k_resident<T, WT, KMAX, EXACT, kResShared>);
    }
    // The device can hold the whole group at once.
    bool fits(const ResPlan& p) {
        return with(p.form, [&](auto kern) {
            int got = 0;
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 kResSmemMax);
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e == cudaSuccess && p.cluster) {
                cudaLaunchConfig_t cfg = {};
                cudaLaunchAttribute attr[1];
                config(cfg, attr, p.group, 1, p.smem, nullptr);
                e = cudaOccupancyMaxActiveClusters(&got, kern, &cfg);
            } else if (e == cudaSuccess) {
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&got, kern, kResThreads, p.smem);
            }
            if (e != cudaSuccess) cudaGetLastError();
            return e == cudaSuccess && got > 0;
        });
    }
    static void config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, int group, int cluster,
                       size_t smem, cudaStream_t s) {
        cfg.gridDim = dim3(unsigned(group));
        cfg.blockDim = dim3(kResThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        if (cluster) {
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = unsigned(group);
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
        } else {
            attr[0].id = cudaLaunchAttributeCooperative;
            attr[0].val.cooperative = 1;
        }
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    cudaError_t slice(const ResProb& prob, const ResPlan& p, cudaStream_t s) override {
        if (p.form == kResWide) k_res_slice<WT, true><<<p.group, kResThreads, 0, s>>>(prob, p.group, p.cluster);
        else k_res_slice<WT, false><<<p.group, kResThreads, 0, s>>>(prob, p.group, p.cluster);
        return cudaGetLastError();
    }
    cudaError_t launch(const ResArgs& a, const ResPlan& p, cudaStream_t s) override {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        config(cfg, attr, p.group, p.cluster, p.smem, s);
        if (a.meet_ns) cfg.numAttrs = 0;
        return with(p.form, [&](auto kern) { return cudaLaunchKernelEx(&cfg, kern, a); });
    }
};

}  // namespace fw
