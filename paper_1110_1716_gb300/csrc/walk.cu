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
// those of parts of the set it was entered with, so `long_walk` runs every
// segment from small sets of states (a lane each) beside every start to the
// end of its own segment, and `long_finish` finds the set that each start
// enters each later segment with and reports what those results hold for it.
// A DFA is run as the NFA of single successors.
//
// Measured, whole scans: 6-state DFA without a dead state, 6001 symbols (3.4 M
// matches, 41 MB) 3.5 ms -> 45 us, 8-state NFA with a live core 101 ms -> 44 us;
// 20,011 symbols 288 and 273 us. long_walk 13 us: a chain of 64 steps;
// long_finish 33 us: instruction issue, about one row of 32 lanes per 35. With
// a warp per start that went from segment to segment, a lane per position,
// the scans took 83 and 160 us; with starts and chunks of segments side by
// side but still a lane per position (12 of 64 report) 74 and 113; with rows
// for sets of four states 78 and 74.
//
// The results are kept for every set of up to B neighbouring states (B = 4: 15
// rows per four states, so that a set costs one read per four states; B = 1,
// the states alone, where those would not fit the scratch).
template <int B>
__host__ __device__ constexpr uint32_t long_rows(uint32_t Q) {
    return (Q + B - 1) / B * ((1u << B) - 1);
}
// Row r as a set of states (states from Q on lead nowhere).
template <int W, int B>
__device__ __forceinline__ void long_row_set(uint32_t r, uint32_t (&s)[W]) {
    const uint32_t at = r / ((1u << B) - 1) * B;
#pragma unroll
    for (int w = 0; w < W; ++w) s[w] = at / 32 == static_cast<uint32_t>(w) ? (r % ((1u << B) - 1) + 1) << (at % 32) : 0u;
}
// f(row) for the rows whose union is `s`.
template <int W, int B, class F>
__device__ __forceinline__ void long_each(const uint32_t (&s)[W], F &&f) {
    constexpr uint32_t SUB = (1u << B) - 1;
#pragma unroll
    for (int w = 0; w < W; ++w) {
        uint32_t r = w * (32 / B) * SUB;
        for (uint32_t m = s[w]; m; m >>= B, r += SUB) {
            if (B == 1) {
                const uint32_t skip = __ffs(m) - 1;
                m >>= skip;
                r += skip;
            }
            if (m & SUB) f(r + (m & SUB) - 1);
        }
    }
}

template <int W, int B>
__global__ void __launch_bounds__(kWalkThreads, 2) long_walk(const WalkArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    if (blockIdx.x < a.start_ctas) {
        walk_starts<WalkNfa<W>, true, true>(a, smem);
        return;
    }
    for (uint32_t i = threadIdx.x; i < (a.tab_bytes + 15) / 16; i += blockDim.x)
        reinterpret_cast<uint4 *>(smem)[i] = __ldg(reinterpret_cast<const uint4 *>(a.tab) + i);
    __syncthreads();
    const uint32_t segs = (a.n + kSegment - 1) / kSegment, S = a.S, rows = long_rows<B>(a.Q);
    // unit u: row u % rows at the start of segment 1 + u / rows
    for (uint32_t u = (blockIdx.x - a.start_ctas) * blockDim.x + threadIdx.x; u < (segs - 1) * rows;
         u += (gridDim.x - a.start_ctas) * blockDim.x) {
        const uint32_t g = 1 + u / rows, r = u % rows;
        const uint32_t b = g * kSegment, len = min(kSegment, a.n - b);
        WalkNfa<W> inst;
        long_row_set<W, B>(r, inst.s);
        uint32_t *h = a.met + (static_cast<size_t>(g) * rows + r) * (kSegment * W);
        uint64_t hits = 0;
        for (uint32_t p = 0; p < len; p += kRound) {
#pragma unroll
            for (int j = 0; j < kRound; ++j) {
                const uint32_t c = p + j < len ? min(static_cast<uint32_t>(__ldg(a.text + b + p + j)), S - 1) : 0u;
                inst.step(a, smem, c, j);
            }
            inst.count(len - p);
#pragma unroll
            for (int j = 0; j < kRound; ++j) {
#pragma unroll
                for (int w = 0; w < W; ++w) h[(p + j) * W + w] = inst.seen[j][w];
                hits |= static_cast<uint64_t>((inst.seen[j][0] | inst.seen[j][W - 1]) != 0) << (p + j);
            }
        }
        a.hits[static_cast<size_t>(g) * rows + r] = hits;
#pragma unroll
        for (int w = 0; w < W; ++w) a.exit[(static_cast<size_t>(g) * rows + r) * W + w] = inst.s[w];
    }
}

constexpr uint32_t kChunk = 8;   // segments per chunk (long_finish)

// Groups of starts with anything to report in chunk c: those whose next
// segment is one of the chunk's or comes before it.
__host__ __device__ __forceinline__ uint32_t long_groups(uint32_t n, uint32_t c) {
    const uint32_t last = (n - 1) / kSegment;   // the text's last segment
    const uint32_t upto = c * kChunk + kChunk - 1 < last ? c * kChunk + kChunk - 1 : last;
    return (upto * kSegment + 32 / kChunk - 1) / (32 / kChunk);
}

// The set that segment (or chunk) g is left with when it is entered with `s`.
template <int W, int B>
__device__ __forceinline__ void long_step(uint32_t (&s)[W], const uint32_t *exit, uint32_t g, uint32_t rows) {
    uint32_t to[W] = {};
    long_each<W, B>(s, [&](uint32_t r) {
        const uint32_t *e = exit + (static_cast<size_t>(g) * rows + r) * W;
#pragma unroll
        for (int w = 0; w < W; ++w) to[w] |= e[w];
    });
#pragma unroll
    for (int w = 0; w < W; ++w) s[w] = to[w];
}

// A warp takes four starts and the eight segments of one chunk at a time: each
// lane finds the set that one of the starts enters one of the segments with
// (by whole chunks as far as it can: every CTA first composes the exits of
// each chunk) and reports that pair's matches.
template <int W, int B>
__global__ void __launch_bounds__(256) long_finish(const WalkArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const uint32_t segs = (a.n + kSegment - 1) / kSegment, rows = long_rows<B>(a.Q);
    const uint32_t chunks = (segs + kChunk - 1) / kChunk;
    WalkOut<3, kWalkStage> out{reinterpret_cast<uint32_t *>(smem) + wid * (2 * 3 * kWalkStage), 0u, 0u, 0u, 0ull};
    uint32_t *over = reinterpret_cast<uint32_t *>(smem + a.sm_stage);   // exits of whole chunks
    const uint32_t *exit = a.exit;
    if (a.seg_smem) {
        uint32_t *e = over + chunks * rows * W;
        for (uint32_t x = rows * W + threadIdx.x; x < segs * rows * W; x += blockDim.x) e[x] = a.exit[x];
        exit = e;
        __syncthreads();
    }
    // (nothing enters the first chunk whole, nothing leaves the last one)
    for (uint32_t u = rows + threadIdx.x; u + rows < chunks * rows; u += blockDim.x) {
        uint32_t s[W];
        long_row_set<W, B>(u % rows, s);
        for (uint32_t y = 0; y < kChunk; ++y) long_step<W, B>(s, exit, u / rows * kChunk + y, rows);
#pragma unroll
        for (int w = 0; w < W; ++w) over[u * W + w] = s[w];
    }
    __syncthreads();
    constexpr uint32_t STARTS = 32 / kChunk;
    uint32_t c = 0, t = blockIdx.x * nw + wid;
    while (true) {
        // the t-th group of chunk c, counted over the starts that begin before its last segment
        uint32_t groups = 0;
        while (c < chunks && t >= (groups = long_groups(a.n, c))) {
            t -= groups;
            ++c;
        }
        if (c == chunks) break;
        uint32_t s[W] = {};
        {
            const uint32_t i = t * STARTS + lane / kChunk, g = c * kChunk + lane % kChunk;
            uint32_t h = i / kSegment + 1;
            if (i < a.n && g < segs && h <= g) {
#pragma unroll
                for (int w = 0; w < W; ++w) s[w] = a.entry[static_cast<size_t>(i) * W + w];
                while (h < g) {
                    const bool whole = h % kChunk == 0 && h + kChunk <= g;
                    long_step<W, B>(s, whole ? over : exit, whole ? h / kChunk : h, rows);
                    h += whole ? kChunk : 1u;
                }
            }
        }
        // every lane reports its own pair, position after position, a row of
        // all lanes at a time
        const uint32_t i = t * STARTS + lane / kChunk, g = c * kChunk + lane % kChunk;
        const size_t u = static_cast<size_t>(g) * rows;
        uint64_t at = 0;   // positions with final states
        long_each<W, B>(s, [&](uint32_t r) { at |= __ldg(a.hits + u + r); });
        uint32_t f[W] = {}, pos = 0;
        auto next = [&]() {
            pos = __ffsll(static_cast<long long>(at)) - 1;
            at &= at - 1;
            long_each<W, B>(s, [&](uint32_t r) {
                const uint32_t *h = a.met + ((u + r) * kSegment + pos) * W;
#pragma unroll
                for (int w = 0; w < W; ++w) f[w] |= __ldg(h + w);
            });
        };
        if (at) next();
        uint32_t m;
        while ((m = __ballot_sync(FULLMASK, (f[0] | f[W - 1]) != 0)) != 0) {
            const uint32_t n = __popc(m);
            out.room(a, n, lane);
            if ((m >> lane) & 1u) {
                const int w = W == 2 && f[0] == 0 ? 1 : 0;
                uint32_t *p = out.row(__popc(m & lanemask_lt()));
                p[0] = i;
                p[1] = g * kSegment + pos;
                if (w == 0) {
                    p[2] = __ffs(f[0]) - 1;
                    f[0] &= f[0] - 1;
                } else {
                    p[2] = 32 + __ffs(f[W - 1]) - 1;
                    f[W - 1] &= f[W - 1] - 1;
                }
                if ((f[0] | f[W - 1]) == 0 && at) next();
            }
            out.n += n;
        }
        t += gridDim.x * nw;
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

static size_t long_words(uint32_t n, int Q, uint32_t rows) {
    const size_t W = walk_nfa_words(Q), segs = (n + kSegment - 1) / kSegment;
    return W * (n + segs * rows + segs * rows * kSegment) + 2 * segs * rows;
}
bool long_fits(uint32_t n, int Q, size_t words) { return long_words(n, Q, long_rows<1>(Q)) <= words; }

template <int W, int B>
static cudaError_t launch_long_t(WalkArgs a, uint32_t *scratch, int nsm, std::atomic<uint32_t> &smem_set, cudaStream_t s) {
    const uint32_t segs = (a.n + kSegment - 1) / kSegment, rows = long_rows<B>(a.Q);
    constexpr int which = 10 + 4 * (W - 1) + (B == 1 ? 2 : 0);
    a.hits = reinterpret_cast<unsigned long long *>(scratch);
    a.entry = scratch + static_cast<size_t>(2) * segs * rows;
    a.exit = a.entry + static_cast<size_t>(W) * a.n;
    a.met = a.exit + static_cast<size_t>(W) * segs * rows;
    a.sm_stage = (a.tab_bytes + 15u) & ~15u;
    uint32_t nw;
    a.start_ctas = start_shape(a, nsm, nw);
    const uint32_t units = (segs - 1) * rows, threads = 32 * nw;
    const uint32_t unit_ctas = units == 0 ? 0u : std::min<uint32_t>((units + threads - 1) / threads, 2u * nsm);
    const uint32_t smem = a.sm_stage + nw * 2 * kWalkStage * 12;
    const int grid = static_cast<int>(a.start_ctas + unit_ctas);
    cudaError_t e = launch_walk_t(long_walk<W, B>, a, grid, threads, smem, which, smem_set, s);
    if (e != cudaSuccess) return e;
    const uint32_t chunks = (segs + kChunk - 1) / kChunk;
    uint64_t groups = 0;
    for (uint32_t c = 0; c < chunks; ++c) groups += long_groups(a.n, c);
    a.sm_stage = 8 * 2 * kWalkStage * 12;
    // the segments' exits too while four CTAs still fit an SM
    const uint32_t exits = segs * rows * W * 4;
    a.seg_smem = exits <= 16384 ? 1u : 0u;
    const uint32_t fsmem = a.sm_stage + chunks * rows * W * 4 + (a.seg_smem ? exits : 0u);
    if (fsmem > 48 * 1024 && !(smem_set.load(std::memory_order_relaxed) >> (which + 1) & 1u)) {
        e = cudaFuncSetAttribute(long_finish<W, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
        if (e != cudaSuccess) return e;
        smem_set.fetch_or(2u << which, std::memory_order_relaxed);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(std::max<uint64_t>(1, std::min<uint64_t>((groups + 7) / 8, 4ull * nsm))));
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = fsmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, long_finish<W, B>, a);
}

cudaError_t launch_long(const WalkArgs &a, uint32_t *scratch, size_t words, int nsm, std::atomic<uint32_t> &smem_set,
                        cudaStream_t s) {
    const bool four = long_words(a.n, a.Q, long_rows<4>(a.Q)) <= words;
    if (walk_nfa_words(a.Q) == 1)
        return four ? launch_long_t<1, 4>(a, scratch, nsm, smem_set, s) : launch_long_t<1, 1>(a, scratch, nsm, smem_set, s);
    return four ? launch_long_t<2, 4>(a, scratch, nsm, smem_set, s) : launch_long_t<2, 1>(a, scratch, nsm, smem_set, s);
}

}  // namespace pfsm
