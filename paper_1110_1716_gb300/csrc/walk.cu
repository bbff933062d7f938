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

#include "scan_device.cuh"

namespace pfsm {

constexpr int kWalkThreads = 512;
constexpr uint32_t kWalkStage = 192;       // staged matches per warp and half (two halves)
constexpr uint32_t kWalkTabSmem = 32768;   // tables up to this size are copied to shared memory
constexpr int kRound = 8;                  // symbols per round
constexpr uint32_t kSegment = 64;          // symbols per segment (long_walk)

// The eight text bytes from position pos (those past the end of the text are
// unspecified).
__device__ __forceinline__ uint64_t window8(uintptr_t text, uintptr_t end, uint32_t pos) {
    const uintptr_t at = text + pos, lo = at & ~static_cast<uintptr_t>(7);
    const uint32_t sh = static_cast<uint32_t>(at & 7) * 8;
    const uint64_t a = __ldg(reinterpret_cast<const unsigned long long *>(lo));
    const uint64_t b = lo + 8 < end ? __ldg(reinterpret_cast<const unsigned long long *>(lo + 8)) : 0ull;
    return sh ? (a >> sh) | (b << (64 - sh)) : a;
}

// A warp's match buffer: one half fills while the place of the other's
// matches in the output is being reserved, so that no round waits for the
// atomic's round trip.
struct WalkOut {
    uint32_t *buf;              // two halves of kWalkStage matches
    uint32_t half;              // the one that fills
    uint32_t n;                 // its matches
    uint32_t leaving;           // matches of the other half, not yet copied
    unsigned long long base;    //   (lane 0) their place

    // copies what is leaving
    __device__ __forceinline__ void copy(const WalkArgs &a, int lane) {
        if (leaving == 0) return;
        const unsigned long long b = __shfl_sync(FULLMASK, base, 0);
        const uint32_t words =
            b >= a.cap ? 0u : 3 * static_cast<uint32_t>(min(static_cast<unsigned long long>(leaving), a.cap - b));
        uint32_t *o = a.out + b * 3;
        const uint32_t *from = buf + (half ^ 1) * (3 * kWalkStage);
        __syncwarp();
        for (uint32_t w = lane; w < words; w += 32) o[w] = from[w];
        __syncwarp();
        leaving = 0;
    }
    // the filling half leaves; the other must have been copied
    __device__ __forceinline__ void turn(const WalkArgs &a, int lane) {
        if (lane == 0) base = atomicAdd(&a.status[0], static_cast<unsigned long long>(n));
        leaving = n;
        n = 0;
        half ^= 1;
    }
};

// A DFA instance: its state; the table has the dead state as its last row.
template <bool TAB_SMEM>
struct WalkDfa {
    uint32_t s;
    uint32_t seen[kRound];   // the round's table entries
    uint32_t hits;           // bit j: the j-th of them is final
    __device__ __forceinline__ void begin(const WalkArgs &a) { s = a.q0; }
    __device__ __forceinline__ void step(const WalkArgs &a, const uint8_t *tab, uint32_t c, int j) {
        const uint32_t ix = s * a.S + c;
        const uint32_t e = TAB_SMEM ? reinterpret_cast<const uint16_t *>(tab)[ix]
                                    : __ldg(reinterpret_cast<const uint16_t *>(a.tab) + ix);
        s = e & 0x7FFFu;
        seen[j] = s;
        if (j == 0) hits = 0;
        hits |= (e >> 15) << j;
    }
    __device__ __forceinline__ bool alive(const WalkArgs &a) const { return s != static_cast<uint32_t>(a.Q); }
    // matches of the round's first `lim` symbols
    __device__ __forceinline__ uint32_t count(uint32_t lim) {
        if (lim < kRound) hits &= (1u << lim) - 1;
        return __popc(hits);
    }
    __device__ __forceinline__ void put_out(const WalkArgs &a, uint32_t start, uint32_t pos, unsigned long long at) const {
#pragma unroll
        for (int j = 0; j < kRound; ++j) {
            if ((hits >> j) & 1u) {
                if (at < a.cap) {
                    uint32_t *o = a.out + at * 3;
                    o[0] = start;
                    o[1] = pos + j;
                    o[2] = seen[j];
                }
                ++at;
            }
        }
    }
    __device__ __forceinline__ void put(const WalkArgs &a, uint32_t start, uint32_t pos, uint32_t *p) const {
#pragma unroll
        for (int j = 0; j < kRound; ++j) {
            if ((hits >> j) & 1u) {
                p[0] = start;
                p[1] = pos + j;
                p[2] = seen[j];
                p += 3;
            }
        }
    }
};

// An NFA instance: its states as a bitset of W words of 32. The table holds,
// per eight states and symbol, the targets of each of their 256 subsets.
template <int W>
struct WalkNfa {
    uint32_t s[W];
    uint32_t seen[kRound][W];   // the round's final states
    uint32_t sets[kRound][W];   // and sets
    __device__ __forceinline__ void begin(const WalkArgs &a) {
#pragma unroll
        for (int w = 0; w < W; ++w) s[w] = a.first[w];
    }
    __device__ __forceinline__ void step(const WalkArgs &a, const uint8_t *tab, uint32_t c, int j) {
        const uint32_t *t = reinterpret_cast<const uint32_t *>(tab) + c * (256 * W);
        const uint32_t row = a.S * 256 * W;
        uint32_t n[W];
#pragma unroll
        for (int w = 0; w < W; ++w) n[w] = 0;
#pragma unroll
        for (int g = 0; g < 4 * W; ++g) {
            if (g * 8 < a.Q) {
                const uint32_t *e = t + g * row + ((s[g >> 2] >> (8 * (g & 3))) & 0xFFu) * W;
#pragma unroll
                for (int w = 0; w < W; ++w) n[w] |= e[w];
            }
        }
#pragma unroll
        for (int w = 0; w < W; ++w) {
            s[w] = n[w];
            sets[j][w] = n[w];
            seen[j][w] = n[w] & a.finals[w];
        }
    }
    __device__ __forceinline__ bool alive(const WalkArgs &) const { return (s[0] | s[W - 1]) != 0; }
    // the segment ended `lim` symbols into the round, or the instance died:
    // the set it enters the next segment with (segments are whole rounds, but
    // a start's first round is not aligned to them)
    __device__ __forceinline__ void leave(const WalkArgs &a, uint32_t start, uint32_t lim) const {
#pragma unroll
        for (int w = 0; w < W; ++w) {
            uint32_t v = s[w];
#pragma unroll
            for (int j = 0; j < kRound - 1; ++j) v = lim == static_cast<uint32_t>(j) + 1 ? sets[j][w] : v;
            a.entry[static_cast<size_t>(start) * W + w] = v;
        }
    }
    __device__ __forceinline__ uint32_t count(uint32_t lim) {
        uint32_t c = 0;
#pragma unroll
        for (int j = 0; j < kRound; ++j)
#pragma unroll
            for (int w = 0; w < W; ++w) {
                if (static_cast<uint32_t>(j) >= lim) seen[j][w] = 0;
                c += __popc(seen[j][w]);
            }
        return c;
    }
    __device__ __forceinline__ void put_out(const WalkArgs &a, uint32_t start, uint32_t pos, unsigned long long at) const {
#pragma unroll
        for (int j = 0; j < kRound; ++j)
#pragma unroll
            for (int w = 0; w < W; ++w)
                for (uint32_t f = seen[j][w]; f; f &= f - 1, ++at) {
                    if (at >= a.cap) continue;
                    uint32_t *o = a.out + at * 3;
                    o[0] = start;
                    o[1] = pos + j;
                    o[2] = 32 * w + __ffs(f) - 1;
                }
    }
    __device__ __forceinline__ void put(const WalkArgs &, uint32_t start, uint32_t pos, uint32_t *p) const {
#pragma unroll
        for (int j = 0; j < kRound; ++j)
#pragma unroll
            for (int w = 0; w < W; ++w)
                for (uint32_t f = seen[j][w]; f; f &= f - 1) {
                    p[0] = start;
                    p[1] = pos + j;
                    p[2] = 32 * w + __ffs(f) - 1;
                    p += 3;
                }
    }
};

// Walks the warp's range of starts; with SEG (long_walk below) only to the end
// of the start's own segment of the text, leaving the sets held there in
// a.entry.
template <class I, bool TAB_SMEM, bool SEG>
__device__ __forceinline__ void walk_starts(const WalkArgs &a, uint8_t *smem) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
    if (TAB_SMEM) {
        uint4 *d = reinterpret_cast<uint4 *>(smem);
        const uint4 *g = reinterpret_cast<const uint4 *>(a.tab);
        for (uint32_t i = tid; i < (a.tab_bytes + 15) / 16; i += blockDim.x) d[i] = __ldg(g + i);
        __syncthreads();
    }
    WalkOut out{reinterpret_cast<uint32_t *>(smem + a.sm_stage) + wid * (2 * 3 * kWalkStage), 0u, 0u, 0u, 0ull};
    const uint32_t n = a.n, S = a.S;
    const uintptr_t text = reinterpret_cast<uintptr_t>(a.text), end = text + n;
    const uint64_t lo = (static_cast<uint64_t>(blockIdx.x) * nw + wid) * a.range;
    uint32_t head = lo < n ? static_cast<uint32_t>(lo) : n;              // the range's next start
    const uint32_t stop = lo + a.range < n ? static_cast<uint32_t>(lo + a.range) : n;
    bool bad = false, act = false;
    I inst;
    inst.begin(a);
    uint32_t start = 0, pos = 0;
    while (true) {
        const uint32_t idle = __ballot_sync(FULLMASK, !act);
        bool fresh = false;
        if (idle && head < stop) {
            const uint32_t mine = head + __popc(idle & lanemask_lt());
            fresh = !act && mine < stop;
            if (fresh) {
                start = pos = mine;
                inst.begin(a);
                act = true;
            }
            head = min(stop, head + __popc(idle));
        } else if (idle == FULLMASK) {
            break;
        }
        const uint64_t w = act ? window8(text, end, pos) : 0ull;
        // every symbol is some start's first; one out of range fails the scan,
        // whatever is stepped in its place
        bad |= fresh && (static_cast<uint32_t>(w) & 0xFFu) >= S;
#pragma unroll
        for (int j = 0; j < kRound; ++j) inst.step(a, smem, min(static_cast<uint32_t>(w >> (8 * j)) & 0xFFu, S - 1), j);
        // symbols left (of the segment)
        const uint32_t lim = !act ? 0u : SEG ? min(n, (start / kSegment + 1) * kSegment) - pos : n - pos;
        const uint32_t c = inst.count(lim);
        if (__any_sync(FULLMASK, c != 0)) {
            uint32_t incl = c;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t t = __shfl_up_sync(FULLMASK, incl, d);
                if (lane >= d) incl += t;
            }
            const uint32_t total = __shfl_sync(FULLMASK, incl, 31);
            if (out.n + total > kWalkStage) {
                out.copy(a, lane);
                out.turn(a, lane);
            }
            if (total <= kWalkStage) {
                inst.put(a, start, pos, out.buf + out.half * (3 * kWalkStage) + 3 * (out.n + incl - c));
                out.n += total;
            } else {   // a round of very many matches: straight to the output
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(&a.status[0], static_cast<unsigned long long>(total));
                base = __shfl_sync(FULLMASK, base, 0) + (incl - c);
                inst.put_out(a, start, pos, base);
            }
        }
        pos += kRound;
        const bool on = act && lim > kRound && inst.alive(a);
        if constexpr (SEG) {
            if (act && !on) inst.leave(a, start, lim);
        }
        act = on;
    }
    out.copy(a, lane);
    out.turn(a, lane);
    out.copy(a, lane);
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
    WalkOut out{reinterpret_cast<uint32_t *>(smem) + wid * (2 * 3 * kWalkStage), 0u, 0u, 0u, 0ull};
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
                        if (out.n + c > kWalkStage) {
                            out.copy(a, lane);
                            out.turn(a, lane);
                        }
                        if (f) {
                            uint32_t *p = out.buf + out.half * (3 * kWalkStage) + 3 * (out.n + __popc(m & lanemask_lt()));
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
    out.copy(a, lane);
    out.turn(a, lane);
    out.copy(a, lane);
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
