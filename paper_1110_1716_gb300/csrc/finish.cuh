// Device building blocks of the kernels that finish the sieve's candidates,
// shared by the single-text kernels (sieve.cu) and the batch kernels
// (flat_batch.cu).
#pragma once

#include "sieve.cuh"

namespace pfsm {

// The eight text bytes from position pos (those past the end of the text are
// unspecified).
__device__ __forceinline__ uint64_t bytes8_at(uintptr_t text, uintptr_t end, uint32_t pos) {
    const uintptr_t at = text + pos, lo = at & ~static_cast<uintptr_t>(7);
    const uint32_t sh = static_cast<uint32_t>(at & 7) * 8;
    uint64_t w = __ldg(reinterpret_cast<const unsigned long long *>(lo)) >> sh;
    if (sh && lo + 8 < end) w |= __ldg(reinterpret_cast<const unsigned long long *>(lo + 8)) << (64 - sh);
    return w;
}

// A warp's matches on their way out: rows of OUTW words ([text,] start, end,
// state) in shared memory, which leave with one atomic on the count per few
// dozen and, in a batch, one per text among them. (With one atomic per row of
// lanes, texts dense in matches waited for it: a batch of one text of 64 MiB
// and 1.08 M matches 694 us, now 326; 4 MiB and 0.23 M 283 us, now 186.) Rows
// are written word by word: the caller's buffer may begin at any multiple of
// four bytes.
constexpr uint32_t kOutRows = 64;
template <int OUTW, class Args>
struct RowOut {
    const Args &a;    // out, cap, status and, in a batch, job_counts
    uint32_t *rows;   // kOutRows * OUTW words of the warp's own
    uint32_t n;

    __device__ __forceinline__ void flush(int lane) {
        if (n == 0) return;
        __syncwarp();
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(&a.status[0], static_cast<unsigned long long>(n));
        base = __shfl_sync(FULLMASK, base, 0);
        if constexpr (OUTW == 4) {
            for (uint32_t r = lane; r < (n + 31) / 32 * 32; r += 32) {
                const uint32_t m = __ballot_sync(FULLMASK, r < n);
                if (r < n) {
                    const uint32_t orig = rows[r * OUTW], peers = __match_any_sync(m, orig);
                    if (lane == __ffs(peers) - 1)
                        atomicAdd(&a.job_counts[orig], static_cast<unsigned long long>(__popc(peers)));
                }
            }
        }
        const uint32_t words =
            base >= a.cap ? 0u : OUTW * static_cast<uint32_t>(min(static_cast<unsigned long long>(n), a.cap - base));
        uint32_t *o = a.out + base * OUTW;
        for (uint32_t w = lane; w < words; w += 32) o[w] = rows[w];
        __syncwarp();
        n = 0;
    }
    // The match (start, end, st) of every lane with `has`, in text `orig`.
    __device__ __forceinline__ void emit(bool has, uint32_t orig, uint32_t start, uint32_t end, uint32_t st, int lane) {
        const uint32_t m = __ballot_sync(FULLMASK, has);
        if (m == 0) return;
        if (n + __popc(m) > kOutRows) flush(lane);
        if (has) {
            uint32_t *p = rows + OUTW * (n + __popc(m & lanemask_lt()));
            if (OUTW == 4) *p++ = orig;
            p[0] = start;
            p[1] = end;
            p[2] = st;
        }
        n += __popc(m);
    }
};

// One start of a DFA per lane with `act`, to its end: the first k symbols by
// the prefix table, then by chains (the only way on from a state, up to eight
// symbols, compared at once) and single steps where the automaton branches.
// What bounds a start is its chain of dependent reads; a planted 32-byte
// signature takes some six instead of 32.
// The text is T.text, T.n symbols of it, reported as text `orig`; the machine's
// fields are M's (a kernel's arguments or a DevMachine, read where they are
// needed).
template <class Out, class Text, class Mach>
__device__ __forceinline__ void run_dfa(const Text &T, const Mach &M, uint32_t orig, bool act, uint32_t start, Out &out, int lane,
                                        uint64_t pol_keep) {
    const uint32_t n = T.n, S = static_cast<uint32_t>(M.S), k = static_cast<uint32_t>(M.k);
    const uintptr_t text = reinterpret_cast<uintptr_t>(T.text), end = text + n;
    uint32_t pos = start, s = static_cast<uint32_t>(M.q0);
    if (act && k && n - start >= k) {
        const uint64_t w = bytes8_at(text, end, pos);
        uint32_t gi = 0;
        bool in = true;
        for (uint32_t j = 0; j < k; ++j) {
            const uint32_t c = static_cast<uint32_t>(w >> (8 * j)) & 0xFFu;
            in &= c < S;
            gi |= c << (j * M.sbits);
        }
        if (in) {
            const uint32_t e = ldg_u16_keep(M.memo + gi, pol_keep);
            if (e == PT_SKIP) {
                act = false;
            } else if (!(e & PT_REC)) {   // a state; records and walks step from q0
                s = e;
                pos += k;
                if (pos >= n) act = false;
            }
        }
    }
    while (__any_sync(FULLMASK, act)) {
        bool hit = false;
        if (act) {
            if (!PFSM_OK_IDX(s < static_cast<uint32_t>(M.Q), out.a.status)) s = 0;
            const uint4 ch = __ldg(M.chain + s);
            const uint64_t w = bytes8_at(text, end, pos);
            const uint32_t len = ch.z & 0xFFu;
            if (len) {
                const uint64_t want = ch.x | (static_cast<uint64_t>(ch.y) << 32);
                // (no final state before the end of a chain: one that
                // passes the end of the text reports nothing)
                if (n - pos < len || ((w ^ want) << (64 - 8 * len)) != 0) {
                    act = false;
                } else {
                    s = ch.w;
                    pos += len;
                    hit = (ch.z >> 8) & 1u;
                }
            } else {
                const uint32_t c = static_cast<uint32_t>(w) & 0xFFu;
                const uint32_t e = c < S ? ldg_u16_keep(M.dtab + s * S + c, pol_keep) : DEAD16;
                if (e == DEAD16) {
                    act = false;
                } else {
                    s = e & 0x7FFFu;
                    hit = (e & FINAL_BIT) != 0;
                    ++pos;
                }
            }
            if (pos >= n) act = false;
        }
        out.emit(hit, orig, start, pos - 1, s, lane);
    }
}

// Where a candidate list overflowed, every start of the text is looked at.
// `starts_left`: those of the lane's four starts [first, first + 4), below
// `to`, that the survival bitmap of m-grams leaves (bit r: first + r; fewer
// than m symbols before the end: left). They are run when a warp is full of
// them; 32 neighbouring starts at a time idled most lanes (256 MiB of planted
// patterns, tiles / neighbours / full warps, ms: 1000-signature trie 4.4, 11.2,
// 1.8; DNA trie 2.3, 11.5, 1.6).
__device__ __forceinline__ uint32_t starts_left(const uint8_t *text, uint32_t n, uint64_t first, uint64_t to,
                                                const uint32_t *surv2, int m, int sbits, uint64_t pol_keep) {
    uint32_t w[4] = {0, 0, 0, 0};
    if (first < to) {
        const uintptr_t at = reinterpret_cast<uintptr_t>(text);
        const uint32_t i0 = static_cast<uint32_t>(first);
        uint32_t lo = 0, hi = 0;
        uint64_t b = 0;
        if (sbits == 2) pack32_at(text, n, i0, lo, hi);
        else b = bytes8_at(at, at + n, i0);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            if (first + r >= to) continue;
            w[r] = 1u;
            if (m == 0 || first + r + m > n) continue;
            uint32_t g = 0;
            if (sbits == 2) {
                g = __funnelshift_r(lo, hi, 2 * r);
            } else {
                // (eight bytes hold m symbols, and those of all four starts up to m = 5)
                const uint64_t v = m <= 5 ? b >> (8 * r) : bytes8_at(at, at + n, i0 + r);
                for (int j = 0; j < m; ++j)
                    g |= (static_cast<uint32_t>(v >> (8 * j)) & ((1u << sbits) - 1)) << (j * sbits);
            }
            g &= (1u << (m * sbits)) - 1;
            w[r] = ldg_u32_keep(surv2 + (g >> 5), pol_keep) >> (g & 31);
        }
    }
    uint32_t keep = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) keep |= (w[r] & 1u) << r;
    return keep;
}

}  // namespace pfsm
