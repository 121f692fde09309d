// __global__ kernels of the single-problem path and of graph assembly.
#pragma once
#include "fw_step.cuh"

namespace fw {

// ---------------------------------------------------------------- hot loop
// The previous iteration's decision as the blocks of a fused pass A need it
// (warp 0 of each): the step *alpha, or true when the solve stops.  quick_step
// where it decides, else the full decision; nothing is committed.
template <typename T>
__device__ __forceinline__ bool fused_step(const ProbDesc& pd, ProbState* st, int c, T* alpha) {
    const unsigned long long* accb = pd.acc + c * kAccBank;
    if constexpr (sizeof(T) == 4) {
        const int lane = threadIdx.x & 31;
        const ulonglong2* S = reinterpret_cast<const ulonglong2*>(accb);
        ulonglong2 v = __ldcg(S + min(lane, kNumR - 1));
        const ulonglong2 nW = __ldcg(S + 2), tLU = __ldcg(S + 3);
        const bool flag = __ldcg(accb + kAccFlag) != 0ull || __ldcg(&st->err) != 0;
        const double g0 = __ldcg(&st->in[c].g0);
        const int iter = __ldcg(&st->in[c].iter), g0_set = __ldcg(&st->in[c].g0_set);
        if (lane == 6) {   // S5 - S3 + S2; v is S5
            add128(v.x, v.y, ~tLU.x, ~tLU.y);
            add128(v.x, v.y, 1ull, 0ull);
            add128(v.x, v.y, nW.x, nW.y);
        }
        float af;
        if (g0_set && quick_step(v.x, v.y, flag, iter, quick_cfg(step_cfg(pd), g0), af)) {
            *alpha = af;
            return false;
        }
    }
    double a;
    const int stop = warp_decide(accb, st, c, step_cfg(pd), false, &a);
    *alpha = T(a);
    return stop != 0;
}

// Step pass A of one tile (k_passA, k_passA_exact).  With `fin` the block first
// takes the previous iteration's step decision itself (no k_finish between
// the passes; see ProbState); otherwise it applies the step k_finish stored.
// `tile`: the problem's row tile this block works on (its block index in the
// single-problem launch, its work item's tile in a batched item launch).  A
// fused launch has one block more, with no tile (tile == ntiles): it takes the
// decision in full and commits it, so that no block with rows waits for FP64.
template <typename T, int KMAX, bool EXACT>
__device__ __forceinline__ void passA_step(const ProbDesc& pd, ProbState* st, int fin, T* stage,
                                           int tile) {
    __shared__ __align__(8) uint64_t bars[2];
    __shared__ T s_alpha;
    __shared__ int s_stop, s_done, s_cur;
    // The committing block may store a stop (done = 1) while other blocks
    // start: one thread reads the flag (and the parity) and the whole block
    // follows it, so no block splits between leaving and waiting on the bulk
    // copies; that thread issues the copies as soon as it knows.
    if (threadIdx.x == 0) {
        const int d = ld_cg(&st->done);
        const int c0 = ld_cg(&st->cur);
        s_done = d;
        s_cur = c0;
        if (!d) {
            mbar_init(&bars[0], 1);
            mbar_init(&bars[1], 1);
            if (tile == pd.ntiles) {
            } else if (fin) {   // the first copies go out at once (a step is always pending)
                const int r0 = tile * pd.tile_rows;
                stage_issue<T, KMAX>(pd, r0, min(kBlock, pd.n - r0), true, stage, &bars[0]);
            } else if (tile == 0) {
                st->cur_b = c0;
            }
        }
    }
    __syncthreads();
    if (s_done) return;
    const int c = s_cur;
    if (tile == pd.ntiles) {
        double a;
        if (threadIdx.x < 32) warp_decide(pd.acc + c * kAccBank, st, c, step_cfg(pd), true, &a);
        return;
    }
    if (fin && threadIdx.x < 32) {
        // warp 0 takes the previous iteration's decision while the copies are
        // in flight
        T a;
        const bool stop = fused_step<T>(pd, st, c, &a);
        if (threadIdx.x == 0) {
            s_stop = stop;
            s_alpha = a;
            if (tile == 0) st->cur_b = c ^ 1;
        }
    }
    const bool upd = fin ? true : ld_cg(&st->has_update) != 0;
    const T alpha = fin ? T(0) : alpha_of<T>(st);
    __syncthreads();
    uint32_t phases = 0;
    const int nst = (pd.tile_rows > kBlock && max_stages<T, KMAX>() == 2) ? 2 : 1;
    const int bank = fin ? (c ^ 1) : c;
    tile_A<T, KMAX, EXACT>(pd, st, tile, upd, alpha, FuseCtl{fin != 0, &s_stop, &s_alpha},
                           pd.acc + bank * kAccBank, stage, nst, bars, phases);
}

// Pass B entry: this iteration's bank (set by pass A); block 0 makes it the
// pending bank and clears the other one, which the next pass A will fill.
__device__ __forceinline__ unsigned long long* passB_bank(const ProbDesc& pd, ProbState* st,
                                                          bool& done, int tile) {
    const int b = ld_cg(&st->cur_b);
    done = ld_cg(&st->done) != 0;
    if (tile == 0 && threadIdx.x == 0) {
        st->cur = b;
        unsigned long long* z = pd.acc + (b ^ 1) * kAccBank;
#pragma unroll
        for (int w = 0; w < kAccWords; ++w) z[w] = 0ull;
    }
    return pd.acc + b * kAccBank;
}

// Blocks of pass A that one SM holds by shared memory (one stage buffer; at
// most 8, or 5 for an FP64 iterate, whose rows need more registers): the
// register budget is set to match, so that the fused step decision does not
// lower the occupancy.
template <typename T, int KMAX>
constexpr int passA_min_blocks() {
    constexpr int cap = sizeof(T) == 8 ? 5 : 8;
    constexpr int b = (227 * 1024) / (3 * kBlock * KMAX * int(sizeof(T)) + 1024);
    return b < 1 ? 1 : (b > cap ? cap : b);
}

// Pass A: one block per row tile.
//   MODE_STEP applies the pending step and evaluates (passA_step);
//   MODE_FLUSH applies a pending step only; MODE_GRAD writes G' and the choice.
template <typename T, int KMAX, int MODE>
__global__ void __launch_bounds__(kBlock, MODE == MODE_STEP ? passA_min_blocks<T, KMAX>() : 1)
    k_passA(ProbDesc pd, ProbState* st, T* Gout, uint8_t* chout, int fin) {
    if constexpr (MODE == MODE_STEP) {
        extern __shared__ __align__(128) unsigned char smraw[];
        passA_step<T, KMAX, false>(pd, st, fin, reinterpret_cast<T*>(smraw), blockIdx.x);
    } else {
        if (MODE != MODE_GRAD && ld_cg(&st->done)) return;
        const bool upd = ld_cg(&st->has_update) != 0;
        const T alpha = alpha_of<T>(st);
        const int r0 = blockIdx.x * pd.tile_rows;
        const int r1 = min(pd.n, r0 + pd.tile_rows);
        AccA<T> acc{T(0), T(0), T(0), T(0), T(0)};
        passA_rows<T, KMAX, MODE>(pd, r0, r1, upd, alpha, acc, Gout, chout);
        if (MODE == MODE_FLUSH) {
            if (last_to_arrive(&st->cntF, pd.ntiles) && threadIdx.x == 0) {
                st->has_update = 0;
                st->cntF = 0;
            }
        }
    }
}

// Pass A (step) for exactly K <= 8 classes with an FP32 iterate: the class loop
// is fully known at compile time, which removes the per-class guards, and the
// registers are bounded by the blocks whose two stage buffers (of K classes,
// not of the class bound) one SM holds.
template <int K>
constexpr int passA_exact_blocks() {
    constexpr int b = (227 * 1024) / (2 * 3 * kBlock * K * 4 + 1024);
    return b > 8 ? 8 : b;
}
template <typename T, int K>
__global__ void __launch_bounds__(kBlock, passA_exact_blocks<K>())
    k_passA_exact(ProbDesc pd, ProbState* st, int fin) {
    extern __shared__ __align__(128) unsigned char smraw[];
    passA_step<T, K, true>(pd, st, fin, reinterpret_cast<T*>(smraw), blockIdx.x);
}

// Pass B: one block per row tile; each adds its tile total to the exact
// accumulators (no block waits for another).
template <typename T, typename WT, int KMAX>
__global__ void __launch_bounds__(kBlock) k_passB(ProbDesc pd, ProbState* st) {
    bool done;
    unsigned long long* accb = passB_bank(pd, st, done, blockIdx.x);
    if (done) return;
    extern __shared__ __align__(128) unsigned char smraw[];
    T* sm_lane = reinterpret_cast<T*>(smraw);
    T* sm_row = sm_lane + kBlock * (KMAX | 1);
    tile_B<T, WT, KMAX, true, false>(pd, st, blockIdx.x, sm_lane, sm_row,
                                     sm_row + kBlock * (KMAX | 1), accb, nullptr);
}

// Pass B with LC lanes per row known at compile time (1 for low-degree graphs
// such as images, 2 or 4 for denser ones); EXACT for exactly KMAX classes.
// Same sums, in the same order, as k_passB.
template <typename T, typename WT, int KMAX, int LC, bool EXACT>
__device__ __forceinline__ void passB_lc_body(const ProbDesc& pd, ProbState* st) {
    bool done;
    unsigned long long* accb = passB_bank(pd, st, done, blockIdx.x);
    if (done) return;
    extern __shared__ __align__(128) unsigned char smraw[];
    T* sm_lane = reinterpret_cast<T*>(smraw);
    T* sm_row = sm_lane + kBlock * (KMAX | 1);
    tile_B<T, WT, KMAX, true, false, LC, EXACT>(pd, st, blockIdx.x, sm_lane, sm_row,
                                                sm_row + kBlock * (KMAX | 1), accb, nullptr);
}

template <typename T, typename WT, int KMAX, int LC, bool EXACT>
__global__ void __launch_bounds__(kBlock) k_passB_lc(ProbDesc pd, ProbState* st) {
    passB_lc_body<T, WT, KMAX, LC, EXACT>(pd, st);
}

// The 2- and 4-lane forms for 5 to 12 classes of FP32 need 44-48 registers,
// i.e. 5 blocks per SM, and a problem with more tiles than 5 x 152 then runs
// a second wave (sbm200k: 782 tiles).  Held to 40 registers (6 blocks per SM,
// a few spilled words) they measured 7% faster there.
template <typename T, typename WT, int KMAX, int LC, bool EXACT>
__global__ void __launch_bounds__(kBlock, 6) k_passB_lc6(ProbDesc pd, ProbState* st) {
    passB_lc_body<T, WT, KMAX, LC, EXACT>(pd, st);
}

// Pass B with the class table in shared memory (see passB_unit): one block
// of kTabThreads threads per SM over a contiguous run of at most
// kTabMaxTiles 256-row tiles.  The table arrives by bulk copies while the
// block starts; a copy that does not arrive within the bounded wait raises
// the problem's error flag and the block adds nothing.
template <typename T, typename WT, int KMAX, int LC, bool EXACT>
__global__ void __launch_bounds__(kTabThreads, 1) k_passB_tab(ProbDesc pd, ProbState* st) {
    __shared__ __align__(8) uint64_t bar;
    __shared__ T s_part[kTabMaxTiles * (kBlock / 32)];
    const int G = gridDim.x;
    const int t0 = int(int64_t(blockIdx.x) * pd.ntiles / G);
    const int t1 = int(int64_t(blockIdx.x + 1) * pd.ntiles / G);
    bool done;
    unsigned long long* accb = passB_bank(pd, st, done, t0);   // block 0 holds tile 0
    if (done) return;
    extern __shared__ __align__(128) unsigned char smraw[];
    T* sm_lane = reinterpret_cast<T*>(smraw);
    T* sm_row = sm_lane + kTabThreads * (KMAX | 1);   // unused with one lane per row
    uint8_t* tab = smraw + tab_bins_bytes<T, KMAX>(LC);
    if (threadIdx.x == 0) {
        const uint32_t tb = tab_bytes(pd.n);
        mbar_init(&bar, 1);
        fence_proxy_async();
        mbar_expect_tx(&bar, tb);
        for (uint32_t o = 0; o < tb; o += 32768u)
            bulk_g2s(tab + o, pd.cls4 + o, min(32768u, tb - o), &bar);
    }
    {
        // while the table arrives, pull the block's CSR slice (row offsets,
        // columns, weights) into L2, so the warps' dependent loads below wait
        // on L2 rather than DRAM
        const int rb = t0 * kBlock, re = min(pd.n, t1 * kBlock);
        const int e0 = __ldg(pd.rp + rb), e1 = __ldg(pd.rp + re);
        const int cw = pd.col16 ? 2 : 4;
        prefetch_l2_range(reinterpret_cast<const char*>(pd.col) + int64_t(e0) * cw,
                          int64_t(e1 - e0) * cw);
        prefetch_l2_range(static_cast<const WT*>(pd.val) + e0, int64_t(e1 - e0) * sizeof(WT));
        prefetch_l2_range(pd.rp + rb, int64_t(re - rb + 1) * 4);
    }
    __syncthreads();   // the barrier is initialised before any thread waits on it
    const bool got = mbar_wait(&bar, 0);
    if (__syncthreads_or(!got)) {
        if (!got) mbar_wait(&bar, 0);   // bounded: let copies still in flight land
        __syncthreads();
        if (threadIdx.x == 0) atomicExch(&st->err, 1);
        return;
    }
    // warp w takes units w, w + 32, ...; unit u is warp (u % 8) of tile t0 + u / 8
    const int nunits = (t1 - t0) * (kBlock / 32);
    for (int u = threadIdx.x >> 5; u < nunits; u += kTabThreads / 32) {
        const int tile = t0 + u / (kBlock / 32);
        const int row0 = tile * kBlock + (u % (kBlock / 32)) * 32;
        const int r_end = min(pd.n, tile * kBlock + kBlock);
        T x = passB_unit<T, WT, KMAX, LC, EXACT>(pd, row0, r_end, sm_lane, sm_row, tab);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) x = add_(x, __shfl_xor_sync(0xffffffffu, x, off));
        if ((threadIdx.x & 31) == 0) s_part[u] = x;
    }
    __syncthreads();
    // each tile's total: its 8 warp sums in warp order (block_accumulate's order)
    if (threadIdx.x < t1 - t0) {
        T sum = T(0);
#pragma unroll
        for (int w = 0; w < kBlock / 32; ++w) sum = add_(sum, s_part[threadIdx.x * (kBlock / 32) + w]);
        fx_add(acc_slot(accb, (t0 + int(threadIdx.x)) % kAccCopies, kNumA), accb + kAccFlag,
               sum);
    }
}

// Eight weights of a row of a pattern problem: one 256-bit load (FP32; it may
// leave L2 first, the iterate arrays are read again sooner) or one 128-bit
// load (BF16).
__device__ __forceinline__ void ld_w8(const float* p, float (&v)[8]) {
    asm volatile("ld.global.nc.L1::no_allocate.L2::evict_first.v8.f32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]),
                   "=f"(v[6]), "=f"(v[7])
                 : "l"(p));
}
__device__ __forceinline__ void ld_w8(const __nv_bfloat16* p, float (&v)[8]) {
    const int4 t = ld_stream(reinterpret_cast<const int4*>(p));
    const int w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[2 * i] = __uint_as_float(uint32_t(w[i]) << 16);
        v[2 * i + 1] = __uint_as_float(uint32_t(w[i]) & 0xffff0000u);
    }
}

// a += v where c holds (a predicated add: written with a branch, the compiler
// turns sums selected by a class into an array indexed by it, in local memory).
__device__ __forceinline__ void add_if(float& a, bool c, float v) {
    asm("{\n .reg .pred p;\n setp.ne.s32 p, %1, 0;\n @p add.rn.f32 %0, %0, %2;\n}"
        : "+f"(a)
        : "r"(int(c)), "f"(v));
}

// Pass B of a pattern problem (ProbDesc::pat): one lane per row, exactly K <= 8
// classes, every row kPatRow slots.  A row's columns follow from its pattern
// byte, so neither row offsets nor columns are read (images: 21% of pass B's
// bytes); its weights are one load and its class sums stay in registers (the
// same sums in the same order as csr_bins).  Each block takes whole row
// tiles, kPatSubs 256-row sub-tiles side by side; the threads' <D, L S> of up
// to kPatGroup sub-tiles wait in shared memory and are added in ascending
// order, as passB_rows adds them; the sub-tiles themselves run in descending
// order, from the rows pass A wrote last (no gain measured over ascending).
// Bound by HBM at 5 TB/s (275 MB an iteration at 2048 x 2048); before and
// after: 69.5 -> 52.0 us (K = 4, FP32), 64.9 -> 48.1 (BF16), 35.1 -> 21.6
// (1411 x 940, K = 6).
constexpr int kPatThreads = 512;
constexpr int kPatSubs = kPatThreads / kBlock;
constexpr int kPatGroup = 16;
template <typename WT, int K>
__global__ void __launch_bounds__(kPatThreads, 2) k_passB_pat(ProbDesc pd, ProbState* st) {
    __shared__ __align__(16) int16_t s_tab[kPatterns][kPatRow];
    __shared__ float s_q[kPatGroup][kBlock];
    __shared__ float s_red[kBlock / 32];
    bool done;
    unsigned long long* accb = passB_bank(pd, st, done, blockIdx.x);   // block 0 holds tile 0
    if (done) return;
    const int tid = threadIdx.x, t = tid & (kBlock - 1), sub = tid / kBlock;
    if (tid < kPatterns * kPatRow / 8)
        reinterpret_cast<uint4*>(s_tab)[tid] = __ldg(reinterpret_cast<const uint4*>(pd.ptab) + tid);
    __syncthreads();
    const int64_t np = pd.npad;
    const float* __restrict__ Ub = static_cast<const float*>(pd.U);
    float* __restrict__ LSb = static_cast<float*>(pd.LS);
    const float* __restrict__ diag = static_cast<const float*>(pd.diag);
    const WT* __restrict__ val = static_cast<const WT*>(pd.val);
    const uint8_t* __restrict__ choice = pd.choice;
    const int n = pd.n;
    for (int tile = blockIdx.x; tile < pd.ntiles; tile += gridDim.x) {
        const int r0 = tile * pd.tile_rows, r1 = min(n, r0 + pd.tile_rows);
        const int subs = (r1 - r0 + kBlock - 1) / kBlock;
        float accq = 0.f;   // threads below kBlock: their rows' sum so far
        for (int g0 = 0; g0 < subs; g0 += kPatGroup) {
            const int cnt = min(kPatGroup, subs - g0);
            int j = cnt - 1 - sub;   // this thread's sub-tile of the group
            int r = r0 + (g0 + j) * kBlock + t;
            int pid = j >= 0 && r < r1 ? int(__ldg(pd.pat + r)) : 0;
            for (; j >= 0; j -= kPatSubs) {
                const bool in = r < r1;
                const int rn = r - kPatSubs * kBlock;
                float q = 0.f;
                int pid_next = 0;
                if (in) {
                    float w[kPatRow], u[K];
                    ld_w8(val + int64_t(r) * kPatRow, w);
                    const uint8_t sv = __ldg(choice + r);
#pragma unroll
                    for (int k = 0; k < K; ++k) u[k] = ld_cg(Ub + k * np + r);
                    if (j >= kPatSubs) pid_next = __ldg(pd.pat + rn);   // the row below is in range
                    const uint4 o4 = *reinterpret_cast<const uint4*>(s_tab[pid]);
                    const uint32_t ow[4] = {o4.x, o4.y, o4.z, o4.w};
                    int s[kPatRow];
#pragma unroll
                    for (int i = 0; i < kPatRow; ++i) {
                        const int off = i & 1 ? int(ow[i / 2]) >> 16 : int(ow[i / 2] << 16) >> 16;
                        s[i] = __ldg(choice + uint32_t(r + off)) & 0x7f;
                    }
                    float b[K];
#pragma unroll
                    for (int k = 0; k < K; ++k) b[k] = 0.f;
#pragma unroll
                    for (int i = 0; i < kPatRow; ++i)
#pragma unroll
                        for (int k = 0; k < K; ++k)
                            add_if(b[k], s[i] == k, w[i]);
                    const int si = sv & 0x7f;
                    const float dg = pd.comb ? __ldg(diag + r) : 1.f;
#pragma unroll
                    for (int k = 0; k < K; ++k) {
                        const float ls = k == si ? sub_(dg, b[k]) : -b[k];
                        LSb[k * np + r] = ls;
                        q = fma_(sub_(k == si ? 1.f : 0.f, u[k]), ls, q);
                    }
                    if (!(sv & kActiveBit)) q = 0.f;
                } else if (j >= kPatSubs) {
                    pid_next = __ldg(pd.pat + rn);
                }
                s_q[j][t] = q;
                pid = pid_next;
                r = rn;
            }
            __syncthreads();
            if (sub == 0)
                for (int i = 0; i < cnt; ++i) accq = add_(accq, s_q[i][t]);
            __syncthreads();
        }
        // the tile's total: butterfly and warp order of block_accumulate
        if (sub == 0) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1)
                accq = add_(accq, __shfl_xor_sync(0xffffffffu, accq, off));
            if ((tid & 31) == 0) s_red[tid >> 5] = accq;
        }
        __syncthreads();
        if (tid == 0) {
            float sum = 0.f;
#pragma unroll
            for (int w = 0; w < kBlock / 32; ++w) sum = add_(sum, s_red[w]);
            fx_add(acc_slot(accb, tile % kAccCopies, kNumA), accb + kAccFlag, sum);
        }
    }
}

// One thread after pass B: read the iteration's totals (complete after the
// kernel boundary, in bank cur), run the stop test and the step.  Inside a
// captured graph only the last iteration ends with it; the others leave the
// decision to the next pass A.  (Doing it in the last block of pass B instead
// costs every block a fence and an arrival, which measured slower.)
static __global__ void k_finish(ProbDesc pd, ProbState* st) {   // one warp
    if (ld_cg(&st->done)) return;
    warp_finish(pd, st, pd.acc + ld_cg(&st->cur) * kAccBank);
}

// One-Shot Frank-Wolfe (Alg. 4): labels of U_1 = GLMO(grad E(U_hat)) in one
// CSR pass; the iterate arrays are not touched.  There is no reduction, so
// each block takes one 256-row sub-tile (fine-grained, no tail wave).
template <typename T, typename WT, int KMAX>
__global__ void __launch_bounds__(kBlock) k_osfw(ProbDesc pd, int32_t* labels, int first, int last) {
    extern __shared__ __align__(128) unsigned char smraw[];
    T* sm_lane = reinterpret_cast<T*>(smraw);
    T* sm_row = sm_lane + kBlock * (KMAX | 1);
    const int r0 = first + blockIdx.x * kBlock;
    const int r1 = min(last, r0 + kBlock);
    osfw_rows<T, WT, KMAX>(pd, labels, r0, r1, sm_lane, sm_row);
}

// The same for a pattern problem with exactly K <= 8 classes (see
// k_passB_pat): no row offsets or columns are read, and the sums stay in
// registers.  A labelled neighbour of class c adds fma(v, 1, .) to c and
// fma(v, 0, .) to the others, an unlabelled one fma(v, 1/K, .) to every class:
// the sums of csr_bins, branch-free.  Bound by its 37 bytes a row (FP32) from
// HBM and its instructions; the general kernel took 91 us on the 2048 x 2048
// image (K = 4), issue-bound on columns, bins and guards; this takes about 50 in
// two parts.
template <typename WT, int K>
__global__ void __launch_bounds__(kBlock) k_osfw_pat(ProbDesc pd, int32_t* labels, int first,
                                                     int last) {
    __shared__ __align__(16) int16_t s_tab[kPatterns][kPatRow];
    if (threadIdx.x < kPatterns * kPatRow / 8)
        reinterpret_cast<uint4*>(s_tab)[threadIdx.x] =
            __ldg(reinterpret_cast<const uint4*>(pd.ptab) + threadIdx.x);
    const int r = first + blockIdx.x * kBlock + threadIdx.x;
    const bool in = r < last;
    float w[kPatRow];
    int pid = 0, f = -1;
    if (in) {
        pid = __ldg(pd.pat + r);
        f = __ldg(pd.fid + r);
        ld_w8(static_cast<const WT*>(pd.val) + int64_t(r) * kPatRow, w);
    }
    __syncthreads();
    if (!in) return;
    const uint4 o4 = *reinterpret_cast<const uint4*>(s_tab[pid]);
    const uint32_t ow[4] = {o4.x, o4.y, o4.z, o4.w};
    int fj[kPatRow];
#pragma unroll
    for (int i = 0; i < kPatRow; ++i) {
        const int off = i & 1 ? int(ow[i / 2]) >> 16 : int(ow[i / 2] << 16) >> 16;
        fj[i] = __ldg(pd.fid + uint32_t(r + off));
    }
    const float unif = 1.f / float(K);
    float b[K];
#pragma unroll
    for (int k = 0; k < K; ++k) b[k] = 0.f;
#pragma unroll
    for (int i = 0; i < kPatRow; ++i) {
        const float other = fj[i] < 0 ? unif : 0.f;
#pragma unroll
        for (int k = 0; k < K; ++k) b[k] = fma_(w[i], fj[i] == k ? 1.f : other, b[k]);
    }
    const float c2 = pd.c2f, om = pd.omf;
    const bool greedy = pd.oracle == 0;
    const float dg = pd.comb ? static_cast<const float*>(pd.diag)[r] : 1.f;
    int s = f;   // a labelled row is binary: the greedy rule keeps its class
    if (f < 0 || !greedy) {
        float best = CUDART_INF_F;
        s = -1;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const float u = uhat_val<float>(f, k, unif);
            float gk = fma_(-c2, u, sub_(mul_(dg, u), b[k]));
            if (f >= 0) gk = fma_(om, sub_(u, k == f ? 1.f : 0.f), gk);
            if (gk < best) {   // unlabelled rows admit every class, the full LMO too
                best = gk;
                s = k;
            }
        }
        if (s < 0) s = 0;
    }
    labels[r] = s;
}

// OUT = L X (initial L U_0, refresh, direct objective).
template <typename T, typename WT, int KMAX>
__global__ void __launch_bounds__(kBlock) k_spmm(ProbDesc pd, const T* X, T* OUT) {
    extern __shared__ __align__(128) unsigned char smraw[];
    T* sm_lane = reinterpret_cast<T*>(smraw);
    T* sm_row = sm_lane + kBlock * (KMAX | 1);
    const int r0 = blockIdx.x * pd.tile_rows;
    const int r1 = min(pd.n, r0 + pd.tile_rows);
    spmm_rows<T, WT, KMAX>(pd, X, OUT, r0, r1, sm_lane, sm_row);
}

// L U_0 for U_0 = U_hat (the state reinit writes): the off-diagonal product
// from the fidelity bytes (an unlabelled neighbour adds w/K to every class, a
// labelled one w to its class), bitwise the dense SpMM of U_hat and without
// its K gathers per entry.
template <typename T, typename WT, int KMAX>
__global__ void __launch_bounds__(kBlock) k_spmm_hat(ProbDesc pd, T* OUT) {
    extern __shared__ __align__(128) unsigned char smraw[];
    T* sm_lane = reinterpret_cast<T*>(smraw);
    T* sm_row = sm_lane + kBlock * (KMAX | 1);
    const int r0 = blockIdx.x * pd.tile_rows;
    const int r1 = min(pd.n, r0 + pd.tile_rows);
    spmm_rows<T, WT, KMAX, kSrcUhat>(pd, static_cast<const T*>(pd.U), OUT, r0, r1, sm_lane,
                                     sm_row);
}

// ------------------------------------------------------------ read-outs
// labels[i] = argmax_k u_ik, lowest index on ties.
template <typename T>
__global__ void k_labels(ProbDesc pd, int32_t* out) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= pd.n) return;
    const T* Ub = static_cast<const T*>(pd.U);
    T best = Ub[r];
    int b = 0;
    for (int k = 1; k < pd.K; ++k) {
        const T x = Ub[(int64_t)k * pd.npad + r];
        if (x > best) {
            best = x;
            b = k;
        }
    }
    out[r] = b;
}

// Rows [r0, r0 + rows) of a class-major array as row-major doubles, 64 rows a
// block: read a class at a time, written as one contiguous run.
constexpr int kRmRows = 64;
template <typename T>
__global__ void __launch_bounds__(kBlock) k_rowmajor(const T* X, int64_t npad, int K, int64_t r0,
                                                     int64_t rows, double* out) {
    __shared__ T s[32 * (kRmRows + 1)];
    const int64_t b = blockIdx.x * int64_t(kRmRows);
    const int cnt = rows - b < kRmRows ? int(rows - b) : kRmRows;
    for (int e = threadIdx.x; e < K * kRmRows; e += kBlock) {
        const int k = e / kRmRows, i = e % kRmRows;
        if (i < cnt) s[k * (kRmRows + 1) + i] = X[k * npad + r0 + b + i];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < cnt * K; e += kBlock) {
        const int i = e / K, k = e - i * K;
        out[b * K + e] = double(s[k * (kRmRows + 1) + i]);
    }
}

// Per-block FP64 partials of E(U) with a freshly computed LUf = L U
// (eq. gradgl_vv2): 1/2 <U, L U> + 1/eps sum u(1-u) + 1/2 sum w_i ||u_hat_i - u_i||^2.
template <typename T>
__global__ void __launch_bounds__(kBlock) k_objective(ProbDesc pd, const T* LUf, double* part) {
    // per row in the iterate type (FP64 per element was the bulk of this
    // kernel on GB300), across rows in FP64
    const int r = blockIdx.x * kBlock + threadIdx.x;
    double e = 0.0;
    if (r < pd.n) {
        const T* Ub = static_cast<const T*>(pd.U);
        const int f = pd.fid[r];
        T quad = T(0), pen = T(0), fidt = T(0);
        for (int k = 0; k < pd.K; ++k) {
            const T u = Ub[(int64_t)k * pd.npad + r];
            quad = fma_(u, LUf[(int64_t)k * pd.npad + r], quad);
            pen = fma_(u, sub_(T(1), u), pen);
            if (f >= 0) {
                const T d = sub_(k == f ? T(1) : T(0), u);
                fidt = fma_(d, d, fidt);
            }
        }
        e = 0.5 * double(quad) + pd.inv_eps * double(pen) + 0.5 * pd.omega0 * double(fidt);
    }
    const double v[1] = {e};
    block_partials<double, 1>(v, part + blockIdx.x);
}

// Classic (full-LMO) FW gap at U (Alg. 2), the stationarity measure over
// Sigma: per row sum_k u_ik (G'_ik - min_j G'_ij) with G' from a freshly
// computed LUf = L U (the constant 1/eps term cancels); FP64 block partials.
template <typename T, int KMAX>
__global__ void __launch_bounds__(kBlock) k_lmo_gap(ProbDesc pd, const T* LUf, double* part) {
    const int r = blockIdx.x * kBlock + threadIdx.x;
    double e = 0.0;
    if (r < pd.n) {
        const T* Ub = static_cast<const T*>(pd.U);
        const int f = pd.fid[r];
        const T c2 = c2_of<T>(pd);
        const T om = om_of<T>(pd);
        T u[KMAX], g[KMAX];
        T mn = inf_<T>();
#pragma unroll
        for (int k = 0; k < KMAX; ++k)
            if (k < pd.K) {
                u[k] = Ub[(int64_t)k * pd.npad + r];
                T gk = fma_(-c2, u[k], LUf[(int64_t)k * pd.npad + r]);
                if (f >= 0) gk = fma_(om, sub_(u[k], k == f ? T(1) : T(0)), gk);
                g[k] = gk;
                mn = gk < mn ? gk : mn;
            }
        T acc = T(0);
#pragma unroll
        for (int k = 0; k < KMAX; ++k)
            if (k < pd.K) acc = fma_(u[k], sub_(g[k], mn), acc);
        e = double(acc);
    }
    const double v[1] = {e};
    block_partials<double, 1>(v, part + blockIdx.x);
}

// Fresh iteration state: E_0 = fixed-order sum of the objective partials,
// everything else zero, status FW_PENDING (one block).
__global__ void __launch_bounds__(kBlock) k_state_init(ProbState* st, const double* part, int nb);

// ------------------------------------------------------------- assembly
// Padded CSR of the off-diagonal operator: sym: W^_ij = w_ij / sqrt(d_i d_j)
// rounded to WT (bf16 via float, both nearest-even); comb: w_ij.  Padding
// entries point at the row itself with weight 0.  diag (comb only) = d_i.
template <typename WT, typename T>
__global__ void k_build(int64_t n, const int32_t* rp, const int32_t* col, const double* w,
                        const double* deg, const int32_t* rpp, int32_t* colp, WT* valp, T* diag,
                        int comb, int col16) {
    // deg holds d_i for L = D - W and d_i^{-1/2} for L_s (k_inv_sqrt): the
    // normalised weight is then two FP64 products per entry, since FP64
    // square roots and divisions per entry dominated this kernel on GB300
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int e0 = rp[i], e1 = rp[i + 1];
    int p = rpp[i];
    const int pend = rpp[i + 1];
    const double di = deg[i];
    int16_t* colp16 = reinterpret_cast<int16_t*>(colp);
    for (int e = e0; e < e1; ++e, ++p) {
        const int j = col[e];
        const double x = comb ? w[e] : (w[e] * di) * deg[j];
        if (col16) colp16[p] = int16_t(j - int(i));   // |j - i| < 2^15 (checked)
        else colp[p] = j;
        if constexpr (sizeof(WT) == 2)
            valp[p] = __float2bfloat16_rn(__double2float_rn(x));
        else if constexpr (sizeof(WT) == 4)
            valp[p] = __double2float_rn(x);
        else
            valp[p] = x;
    }
    for (; p < pend; ++p) {
        if (col16) colp16[p] = 0;
        else colp[p] = int32_t(i);
        valp[p] = WT(0.0f);
    }
    if (comb) diag[i] = T(di);
}

// ------------------------------------------------------- offset patterns
// Key of a row's offset list (an FNV-style hash of its kPatRow offsets; equal
// keys are compared offset by offset before they count as equal).  0 marks an
// empty table entry.
__device__ __forceinline__ unsigned long long pat_key(const uint4& o) {
    unsigned long long h = 1469598103934665603ull;
    const uint32_t w[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) h = (h ^ w[i]) * 1099511628211ull;
    h ^= h >> 29;
    return h ? h : 1ull;
}
// Collect the distinct offset lists (col: int16 offsets, kPatRow per row) in an
// open-addressing table; *fail when there are more than the table holds.
static __global__ void k_pat_find(int n, const int16_t* col, unsigned long long* keys, int* rep,
                                  int* fail) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n || *reinterpret_cast<volatile int*>(fail)) return;
    const unsigned long long key = pat_key(reinterpret_cast<const uint4*>(col)[r]);
    for (int i = 0, h = int(key % kPatterns); i < kPatterns; ++i, h = (h + 1) % kPatterns) {
        unsigned long long have = *reinterpret_cast<volatile unsigned long long*>(keys + h);
        if (have == 0ull) {
            have = atomicCAS(keys + h, 0ull, key);
            if (have == 0ull) {
                rep[h] = r;
                return;
            }
        }
        if (have == key) return;
    }
    *fail = 1;
}
// Every row's pattern; *fail when two lists share a key.
static __global__ void k_pat_assign(int n, const int16_t* col, const unsigned long long* keys,
                                    const int* rep, uint8_t* pat, int16_t* ptab, int* fail) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    const uint4* rows = reinterpret_cast<const uint4*>(col);
    if (blockIdx.x == 0 && threadIdx.x < kPatterns)
        reinterpret_cast<uint4*>(ptab)[threadIdx.x] =
            keys[threadIdx.x] ? rows[rep[threadIdx.x]] : make_uint4(0, 0, 0, 0);
    if (r >= n || *fail) return;
    const uint4 o = rows[r];
    const unsigned long long key = pat_key(o);
    for (int i = 0, h = int(key % kPatterns); i < kPatterns; ++i, h = (h + 1) % kPatterns) {
        if (keys[h] != key) continue;
        const uint4 p = rows[rep[h]];
        if (p.x != o.x || p.y != o.y || p.z != o.z || p.w != o.w) *fail = 1;
        pat[r] = uint8_t(h);
        return;
    }
    *fail = 1;
}

// U_0 = U_hat (Sec. 5.1): e_c on fidelity rows, 1/K elsewhere; choice reset.
template <typename T>
__global__ void k_reinit(ProbDesc pd) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;   // blockDim.x = kBlock
    int cls = 0;
    if (r < pd.n) {
        const int c = pd.fid[r];
        const T unif = T(1) / T(pd.K);
        T* Ub = static_cast<T*>(pd.U);
        for (int k = 0; k < pd.K; ++k)
            Ub[(int64_t)k * pd.npad + r] = c >= 0 ? (k == c ? T(1) : T(0)) : unif;
        cls = c >= 0 ? c : 0;
        pd.choice[r] = uint8_t(cls);
    }
    if (pd.cls4) {
        const int hi = __shfl_down_sync(0xffffffffu, cls, 1);
        if ((r & 1) == 0 && r < pd.n) pd.cls4[r >> 1] = uint8_t(cls | (hi << 4));
    }
}

}  // namespace fw
