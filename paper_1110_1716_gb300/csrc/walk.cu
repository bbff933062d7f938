// Direct scans: every start is walked from q0 by one lane, without filter
// tables, tiles or queues. For machines whose starts mostly report or live a
// few symbols (a filter would pass nearly all of them) and whose transition
// table is small: DFAs by their table, NFAs of at most 64 states by bitset
// (the set after a symbol is the OR of one table word per eight states).
//
// A warp owns a range of consecutive starts; a lane whose instance died takes
// the next one of the range. Every round loads the next eight text bytes of
// each lane (through L1) and steps them without a branch: the dead state is a
// row of its own that leads to itself, symbols past the end of the text are
// stepped and their matches dropped. Only then are the round's matches placed
// (one prefix sum over the lanes) in a per-warp buffer in shared memory, which
// leaves with one atomic per few hundred. The last CTA to end writes the
// status out and clears the stream's counters, so a scan is one launch.
//
// Measured on GB300 against the tile kernel with its prefix records, queues
// and carry kernel, which such scans took before (device time per scan):
// 64-state DNA DFA, 4 KB 25 -> 8.2 us, 1 MiB (1.07 M matches) 43 -> 18.5 us,
// 16,384-state DFA, 1 MB 36 -> 23 us; bound by instruction issue (58 %) and the
// latency of each lane's chain of table reads. Rounds of 4, 6 and 8 symbols
// measured within 5 % on those; 8 is the fastest on long-lived instances.
#include <algorithm>
#include <atomic>

#include "walk.cuh"

namespace pfsm {

constexpr int kWalkThreads = 512;
constexpr uint32_t kWalkStage = 192;       // staged matches per warp and half
constexpr uint32_t kWalkTabSmem = 32768;   // tables up to this size are copied to shared memory

// The CTA's part of a scan's starts: a warp takes a range of consecutive ones.
template <class I, bool TAB_SMEM, bool SEG>
__device__ __forceinline__ void walk_starts(const WalkArgs &a, uint8_t *smem) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
    if (TAB_SMEM) {
        uint4 *d = reinterpret_cast<uint4 *>(smem);
        const uint4 *g = reinterpret_cast<const uint4 *>(a.tab);
        for (uint32_t i = tid; i < (a.tab_bytes + 15) / 16; i += blockDim.x) d[i] = __ldg(g + i);
        __syncthreads();
    }
    WalkOut<3, kWalkStage> out{reinterpret_cast<uint32_t *>(smem + a.sm_stage) + wid * (2 * 3 * kWalkStage), 0u, 0u, 0u,
                               0ull};
    const uint64_t lo = (static_cast<uint64_t>(blockIdx.x) * nw + wid) * a.range;
    const uint32_t head = lo < a.n ? static_cast<uint32_t>(lo) : a.n;
    const uint32_t stop = lo + a.range < a.n ? static_cast<uint32_t>(lo + a.range) : a.n;
    bool bad = false;
    walk_range<I, SEG>(a, smem, head, stop, out, bad, lane);
    out.finish(a, lane);
    if (bad) atomicOr(&a.status[1], ERR_SYMBOL);
}

template <class I, bool TAB_SMEM>
__global__ void __launch_bounds__(kWalkThreads, 2) walk(const WalkArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    walk_starts<I, TAB_SMEM, false>(a, smem);
    scan_status_out(a.status, a.status_out, a.done, nullptr);
}

// ------------------------------------------------------------ long-lived instances
// Machines of at most 64 states whose instances live on and on (the paper's
// quadratic case): one lane per start would take as many dependent steps as
// the text has symbols. The text is cut into segments of kSegment symbols.
// The set after a segment, and the final states on the way, are the unions of
// those of the single states it was entered with, so `long_walk` runs every
// segment from every single state (Q lanes per segment) beside every start to
// the end of its own segment, and `long_finish` follows each start from
// segment to segment by unions of those results, a warp per start and a lane
// per position. A DFA is run as the NFA of single successors. Measured: 6-state
// DFA without a dead state, 6001 symbols (3.4 M matches) 3.5 ms -> 81 us (440
// us with one lane per start to the end), 8-state NFA with a live core 101 ms
// -> 160 us (609 us); bound by the chain of reads from segment to segment.
template <int W>
__global__ void __launch_bounds__(kWalkThreads, 2) long_walk(const WalkArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    if (blockIdx.x < a.start_ctas) {
        walk_starts<WalkNfa<W>, true, true>(a, smem);
        return;
    }
    for (uint32_t i = threadIdx.x; i < (a.tab_bytes + 15) / 16; i += blockDim.x)
        reinterpret_cast<uint4 *>(smem)[i] = __ldg(reinterpret_cast<const uint4 *>(a.tab) + i);
    __syncthreads();
    const uint32_t segs = (a.n + kSegment - 1) / kSegment, Q = a.Q, S = a.S;
    // unit u: state u % Q at the start of segment 1 + u / Q
    for (uint32_t u = (blockIdx.x - a.start_ctas) * blockDim.x + threadIdx.x; u < (segs - 1) * Q;
         u += (gridDim.x - a.start_ctas) * blockDim.x) {
        const uint32_t g = 1 + u / Q, q = u % Q;
        const uint32_t b = g * kSegment, len = min(kSegment, a.n - b);
        WalkNfa<W> inst;
#pragma unroll
        for (int w = 0; w < W; ++w) inst.s[w] = (q >> 5) == static_cast<uint32_t>(w) ? 1u << (q & 31) : 0u;
        uint32_t *h = a.met + (static_cast<size_t>(g) * Q + q) * (kSegment * W);
        for (uint32_t p = 0; p < len; p += kRound) {
#pragma unroll
            for (int j = 0; j < kRound; ++j) {
                const uint32_t c = p + j < len ? min(static_cast<uint32_t>(__ldg(a.text + b + p + j)), S - 1) : 0u;
                inst.step(a, smem, c, j);
            }
            inst.count(len - p);
#pragma unroll
            for (int j = 0; j < kRound; ++j)
#pragma unroll
                for (int w = 0; w < W; ++w) h[(p + j) * W + w] = inst.seen[j][w];
        }
#pragma unroll
        for (int w = 0; w < W; ++w) a.exit[(static_cast<size_t>(g) * Q + q) * W + w] = inst.s[w];
    }
}

template <int W>
__global__ void __launch_bounds__(256) long_finish(const WalkArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    WalkOut<3, kWalkStage> out{reinterpret_cast<uint32_t *>(smem) + wid * (2 * 3 * kWalkStage), 0u, 0u, 0u, 0ull};
    const uint32_t segs = (a.n + kSegment - 1) / kSegment, Q = a.Q;
    constexpr int PER = kSegment / 32;   // positions per lane
    for (uint32_t i = blockIdx.x * nw + wid; i < a.n; i += gridDim.x * nw) {
        uint32_t s[W];
        uint32_t any = 0;
#pragma unroll
        for (int w = 0; w < W; ++w) any |= s[w] = a.entry[static_cast<size_t>(i) * W + w];
        for (uint32_t g = i / kSegment + 1; g < segs && any; ++g) {
            uint32_t to[W], met[PER][W];
#pragma unroll
            for (int w = 0; w < W; ++w) {
                to[w] = 0;
#pragma unroll
                for (int x = 0; x < PER; ++x) met[x][w] = 0;
            }
#pragma unroll
            for (int v = 0; v < W; ++v) {
                for (uint32_t m = s[v]; m; m &= m - 1) {   // (the same in every lane)
                    const size_t u = static_cast<size_t>(g) * Q + 32 * v + __ffs(m) - 1;
#pragma unroll
                    for (int w = 0; w < W; ++w) {
                        to[w] |= a.exit[u * W + w];
#pragma unroll
                        for (int x = 0; x < PER; ++x) met[x][w] |= a.met[(u * kSegment + 32 * x + lane) * W + w];
                    }
                }
            }
#pragma unroll
            for (int x = 0; x < PER; ++x)
#pragma unroll
                for (int w = 0; w < W; ++w) {
                    // (positions past the end of the text hold no final state)
                    uint32_t f = g * kSegment + 32 * x + lane < a.n ? met[x][w] : 0u;
                    uint32_t m;
                    while ((m = __ballot_sync(FULLMASK, f != 0)) != 0) {
                        const uint32_t c = __popc(m);
                        out.room(a, c, lane);
                        if (f) {
                            uint32_t *p = out.row(__popc(m & lanemask_lt()));
                            p[0] = i;
                            p[1] = g * kSegment + 32 * x + lane;
                            p[2] = 32 * w + __ffs(f) - 1;
                            f &= f - 1;
                        }
                        out.n += c;
                    }
                }
            any = 0;
#pragma unroll
            for (int w = 0; w < W; ++w) any |= s[w] = to[w];
        }
    }
    out.finish(a, lane);
    scan_status_out(a.status, a.status_out, a.done, nullptr);
}

// ------------------------------------------------------------ host helpers
uint32_t walk_nfa_words(int Q) { return Q <= 32 ? 1u : 2u; }

template <class K>
static cudaError_t launch_walk_t(K k, const WalkArgs &a, int grid, int threads, uint32_t smem, int which,
                                 std::atomic<uint32_t> &smem_set, cudaStream_t s) {
    if (smem > 48 * 1024 && !(smem_set.load(std::memory_order_relaxed) >> which & 1u)) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
        if (e != cudaSuccess) return e;
        smem_set.fetch_or(1u << which, std::memory_order_relaxed);
    }
    k<<<grid, threads, smem, s>>>(a);
    return cudaGetLastError();
}

// Ranges and CTAs for the starts: one start per lane while there are fewer
// than the GPU holds (two CTAs of 16 warps per SM), in CTAs small enough to
// use every SM; then longer ranges. Returns the CTAs, `nw` their warps.
static uint32_t start_shape(WalkArgs &a, int nsm, uint32_t &nw) {
    const uint64_t lanes = static_cast<uint64_t>(2 * nsm) * kWalkThreads;
    a.range = static_cast<uint32_t>((a.n + lanes - 1) / lanes) * 32;
    const uint64_t warps = (static_cast<uint64_t>(a.n) + a.range - 1) / a.range;
    const uint64_t per = (warps + nsm - 1) / nsm;
    nw = static_cast<uint32_t>(per < kWalkThreads / 32 ? per : kWalkThreads / 32);
    return static_cast<uint32_t>((warps + nw - 1) / nw);
}

cudaError_t launch_walk(WalkArgs a, int kind, int nsm, std::atomic<uint32_t> &smem_set, cudaStream_t s) {
    const bool sm = kind == 1 || a.tab_bytes <= kWalkTabSmem;
    a.sm_stage = sm ? (a.tab_bytes + 15u) & ~15u : 0u;
    uint32_t nw;
    const int grid = static_cast<int>(start_shape(a, nsm, nw));
    const uint32_t smem = a.sm_stage + nw * 2 * kWalkStage * 12;
    const int threads = static_cast<int>(32 * nw);
    if (kind == 0) {
        if (sm) return launch_walk_t(walk<WalkDfa<true>, true>, a, grid, threads, smem, 3, smem_set, s);
        return launch_walk_t(walk<WalkDfa<false>, false>, a, grid, threads, smem, 4, smem_set, s);
    }
    if (walk_nfa_words(a.Q) == 1) return launch_walk_t(walk<WalkNfa<1>, true>, a, grid, threads, smem, 5, smem_set, s);
    return launch_walk_t(walk<WalkNfa<2>, true>, a, grid, threads, smem, 6, smem_set, s);
}

size_t long_scratch_words(uint32_t n, int Q) {
    const size_t W = walk_nfa_words(Q), segs = (n + kSegment - 1) / kSegment;
    return W * (n + segs * Q + segs * Q * kSegment);
}

cudaError_t launch_long(WalkArgs a, uint32_t *scratch, int nsm, std::atomic<uint32_t> &smem_set, cudaStream_t s) {
    const size_t W = walk_nfa_words(a.Q), segs = (a.n + kSegment - 1) / kSegment;
    a.entry = scratch;
    a.exit = a.entry + W * a.n;
    a.met = a.exit + W * segs * a.Q;
    a.sm_stage = (a.tab_bytes + 15u) & ~15u;
    uint32_t nw;
    a.start_ctas = start_shape(a, nsm, nw);
    const uint32_t units = static_cast<uint32_t>(segs - 1) * a.Q, threads = 32 * nw;
    const uint32_t unit_ctas = units == 0 ? 0u : std::min<uint32_t>((units + threads - 1) / threads, 2u * nsm);
    const uint32_t smem = a.sm_stage + nw * 2 * kWalkStage * 12;
    const int grid = static_cast<int>(a.start_ctas + unit_ctas);
    cudaError_t e = W == 1 ? launch_walk_t(long_walk<1>, a, grid, threads, smem, 7, smem_set, s)
                           : launch_walk_t(long_walk<2>, a, grid, threads, smem, 8, smem_set, s);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(std::min<uint64_t>((a.n + 7) / 8, 4ull * nsm)));
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = 8 * 2 * kWalkStage * 12;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return W == 1 ? cudaLaunchKernelEx(&cfg, long_finish<1>, a) : cudaLaunchKernelEx(&cfg, long_finish<2>, a);
}

}  // namespace pfsm
