// Device building blocks of the direct scan, shared by the single-text kernels
// (walk.cu) and the batch kernels (flat_batch.cu).
#pragma once

#include "scan_device.cuh"

namespace pfsm {

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

// A warp's match buffer: two halves of STAGE rows of OUTW words ([job,] start,
// end, state); one half fills while the place of the other's
// matches in the output is being reserved, so that no round waits for the
// atomic's round trip.
template <int OUTW, uint32_t STAGE>
struct WalkOut {
    uint32_t *buf;
    uint32_t half;              // the one that fills
    uint32_t n;                 // its matches
    uint32_t leaving;           // matches of the other half, not yet copied
    unsigned long long base;    //   (lane 0) their place

    // copies what is leaving
    __device__ __forceinline__ void copy(const WalkArgs &a, int lane) {
        if (leaving == 0) return;
        const unsigned long long b = __shfl_sync(FULLMASK, base, 0);
        const uint32_t words =
            b >= a.cap ? 0u : OUTW * static_cast<uint32_t>(min(static_cast<unsigned long long>(leaving), a.cap - b));
        uint32_t *o = a.out + b * OUTW;
        const uint32_t *from = buf + (half ^ 1) * (OUTW * STAGE);
        __syncwarp();
        for (uint32_t w = lane; w < words; w += 32) o[w] = from[w];
        __syncwarp();
        leaving = 0;
    }
    // room for `c` (<= STAGE) more rows, and where row r of them goes
    __device__ __forceinline__ void room(const WalkArgs &a, uint32_t c, int lane) {
        if (n + c > STAGE) {
            copy(a, lane);
            turn(a, lane);
        }
    }
    __device__ __forceinline__ uint32_t *row(uint32_t r) const { return buf + half * (OUTW * STAGE) + OUTW * (n + r); }
    // everything leaves (before the job changes, and at the end)
    __device__ __forceinline__ void finish(const WalkArgs &a, int lane) {
        copy(a, lane);
        turn(a, lane);
        copy(a, lane);
    }
    // the filling half leaves; the other must have been copied
    __device__ __forceinline__ void turn(const WalkArgs &a, int lane) {
        if (lane == 0 && n) {
            base = atomicAdd(&a.status[0], static_cast<unsigned long long>(n));
            if (OUTW == 4) atomicAdd(&a.job_counts[a.orig], static_cast<unsigned long long>(n));
        }
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
    template <int OUTW>
    __device__ __forceinline__ void put_out(const WalkArgs &a, uint32_t start, uint32_t pos, unsigned long long at) const {
#pragma unroll
        for (int j = 0; j < kRound; ++j) {
            if ((hits >> j) & 1u) {
                if (at < a.cap) {
                    uint32_t *o = a.out + at * OUTW;
                    if (OUTW == 4) *o++ = a.orig;
                    o[0] = start;
                    o[1] = pos + j;
                    o[2] = seen[j];
                }
                ++at;
            }
        }
    }
    template <int OUTW>
    __device__ __forceinline__ void put(const WalkArgs &a, uint32_t start, uint32_t pos, uint32_t *p) const {
#pragma unroll
        for (int j = 0; j < kRound; ++j) {
            if ((hits >> j) & 1u) {
                if (OUTW == 4) *p++ = a.orig;
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
    template <int OUTW>
    __device__ __forceinline__ void put_out(const WalkArgs &a, uint32_t start, uint32_t pos, unsigned long long at) const {
#pragma unroll
        for (int j = 0; j < kRound; ++j)
#pragma unroll
            for (int w = 0; w < W; ++w)
                for (uint32_t f = seen[j][w]; f; f &= f - 1, ++at) {
                    if (at >= a.cap) continue;
                    uint32_t *o = a.out + at * OUTW;
                    if (OUTW == 4) *o++ = a.orig;
                    o[0] = start;
                    o[1] = pos + j;
                    o[2] = 32 * w + __ffs(f) - 1;
                }
    }
    template <int OUTW>
    __device__ __forceinline__ void put(const WalkArgs &a, uint32_t start, uint32_t pos, uint32_t *p) const {
#pragma unroll
        for (int j = 0; j < kRound; ++j)
#pragma unroll
            for (int w = 0; w < W; ++w)
                for (uint32_t f = seen[j][w]; f; f &= f - 1) {
                    if (OUTW == 4) *p++ = a.orig;
                    p[0] = start;
                    p[1] = pos + j;
                    p[2] = 32 * w + __ffs(f) - 1;
                    p += 3;
                }
    }
};

// Walks the starts [head, stop) of the text, one per lane at a time; with SEG
// (long_walk) only to the end of the start's own segment of the text, leaving
// the sets held there in a.entry. `tab`: the table's shared copy, if it has one.
template <class I, bool SEG, int OUTW, uint32_t STAGE>
__device__ __forceinline__ void walk_range(const WalkArgs &a, const uint8_t *tab, uint32_t head, uint32_t stop,
                                           WalkOut<OUTW, STAGE> &out, bool &bad, int lane) {
    const uint32_t n = a.n, S = a.S;
    const uintptr_t text = reinterpret_cast<uintptr_t>(a.text), end = text + n;
    bool act = false;
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
        for (int j = 0; j < kRound; ++j) inst.step(a, tab, min(static_cast<uint32_t>(w >> (8 * j)) & 0xFFu, S - 1), j);
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
            if (total <= STAGE) {
                out.room(a, total, lane);
                inst.template put<OUTW>(a, start, pos, out.row(incl - c));
                out.n += total;
            } else {   // a round of very many matches: straight to the output
                unsigned long long base = 0;
                if (lane == 0) {
                    base = atomicAdd(&a.status[0], static_cast<unsigned long long>(total));
                    if (OUTW == 4) atomicAdd(&a.job_counts[a.orig], static_cast<unsigned long long>(total));
                }
                base = __shfl_sync(FULLMASK, base, 0) + (incl - c);
                inst.template put_out<OUTW>(a, start, pos, base);
            }
        }
        pos += kRound;
        const bool on = act && lim > kRound && inst.alive(a);
        if constexpr (SEG) {
            if (act && !on) inst.leave(a, start, lim);
        }
        act = on;
    }
}

}  // namespace pfsm
