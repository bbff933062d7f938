// Device building blocks of the sieve, shared by the single-text kernels
// (sieve.cu) and the batch kernels (flat_batch.cu).
#pragma once

#include "scan_device.cuh"

namespace pfsm {

constexpr uint32_t kSpan = 2048;   // bytes a warp tests per step: 4 x 16 per lane

__device__ __forceinline__ uint4 ldg_stream(const uint8_t *p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

// Symbols i .. i + 31 of the text as 2-bit symbols (from the 16-byte blocks
// that hold them; symbols past the end of the text are unspecified).
__device__ __forceinline__ void pack32_at(const uint8_t *text, uint32_t n, uint32_t i, uint32_t &g0,
                                          uint32_t &g1) {
    const uintptr_t at = reinterpret_cast<uintptr_t>(text) + i;
    const uintptr_t end = reinterpret_cast<uintptr_t>(text) + n;
    const uintptr_t a = at & ~static_cast<uintptr_t>(15);
    uint32_t p[3] = {0u, 0u, 0u};
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        if (a + 16 * b < end) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(a + 16 * b));
            p[b] = pack16(v.x, v.y, v.z, v.w);
        }
    }
    const uint32_t sh = static_cast<uint32_t>(at & 15) * 2;
    g0 = __funnelshift_r(p[0], p[1], sh);
    g1 = __funnelshift_r(p[1], p[2], sh);
}

// Copies a near bitmap to shared memory (NT threads, their loads all in
// flight at once).
template <uint32_t BYTES, int NT>
__device__ __forceinline__ void stage_near(uint8_t *to, const uint32_t *from, int tid) {
    uint4 *d = reinterpret_cast<uint4 *>(to);
    const uint4 *g = reinterpret_cast<const uint4 *>(from);
    uint4 v[BYTES / 16 / NT];
#pragma unroll
    for (uint32_t i = 0; i < BYTES / 16 / NT; ++i) v[i] = __ldg(g + i * NT + tid);
#pragma unroll
    for (uint32_t i = 0; i < BYTES / 16 / NT; ++i) d[i * NT + tid] = v[i];
}

// Appends the lanes' kept starts (bit r of `keep`: start first + r) to the
// candidates, one atomic per call. `tag` goes with them, and in a batch the
// job.
template <bool BATCH>
__device__ __forceinline__ void sieve_append(const SieveArgs &a, uint32_t keep, uint32_t first, uint32_t tag,
                                             int lane) {
    uint32_t incl = __popc(keep);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(FULLMASK, incl, d);
        if (lane >= d) incl += t;
    }
    const uint32_t total = __shfl_sync(FULLMASK, incl, 31);
    if (total == 0) return;
    uint32_t at = 0;
    if (lane == 0) {
        if (BATCH) {
            const unsigned long long n = atomicAdd(a.cand_sum, static_cast<unsigned long long>(total));
            at = n < a.cand_cap ? static_cast<uint32_t>(n) : a.cand_cap;   // (and at most 128 more)
        } else {
            at = atomicAdd(a.cand_n, total);
        }
    }
    at = __shfl_sync(FULLMASK, at, 0) + incl - __popc(keep);
    while (keep) {
        const uint32_t r = __ffs(keep) - 1;
        keep &= keep - 1;
        if (at < a.cand_cap) {
            if (BATCH) reinterpret_cast<uint4 *>(a.cand)[at] = make_uint4(a.job, first + r, tag, 0u);
            else a.cand[at] = make_uint2(first + r, tag);
        }
        ++at;
    }
}

// Symbols i .. i + 7 as 16 bits; i + 7 < n.
__device__ __forceinline__ uint32_t pack8_at(const uint8_t *text, uint32_t i) {
    const uintptr_t at = reinterpret_cast<uintptr_t>(text) + i;
    const uintptr_t lo = at & ~static_cast<uintptr_t>(7);
    const uint32_t sh = static_cast<uint32_t>(at & 7) * 8;
    uint64_t w = __ldg(reinterpret_cast<const unsigned long long *>(lo)) >> sh;
    if (sh) w |= __ldg(reinterpret_cast<const unsigned long long *>(lo + 8)) << (64 - sh);
    return pack2(w);
}

// The second and third level for `k` starts {start, its first 16 symbols} of
// an NFA (NfaMemoBuilder): the record of its first k + L2_SYMS symbols, then
// whether that record's set can still report given the next L3_SYMS. What
// is left becomes a candidate with its record. In a batch (whose NFAs are
// all `lean`) every candidate has one: a start with fewer symbols left than
// the record takes the record of its symbols and zeros, whose matches past
// the end of the text are dropped when they are reported.
template <bool BATCH>
__device__ __forceinline__ void sieve_levels(const SieveArgs &a, const uint2 *list2, uint32_t k, int lane,
                                             uint64_t pol_keep) {
    bool keep = false;
    uint2 e = make_uint2(0u, 0u);
    uint32_t tag = SIEVE_NO_RECORD;
    if (static_cast<uint32_t>(lane) < k) {
        e = list2[lane];
        keep = true;
        const uint32_t kk = static_cast<uint32_t>(a.k), at = kk + L2_SYMS;
        const uint32_t rest = a.n - e.x;
        if (BATCH && rest < at + 8) {
            if (rest < 16) e.y &= (1u << (2 * rest)) - 1;
            keep = false;
            if (rest >= a.min_match) {
                const uint32_t x = ldg_u16_keep(a.memox + (e.y & ((1u << (2 * kk)) - 1)), pol_keep);
                if (x != L2_NONE)
                    tag = ldg_u16_keep(a.l2tab + x * L2_GRAMS + ((e.y >> (2 * kk)) & (L2_GRAMS - 1)), pol_keep);
                keep = x != L2_NONE && tag != L2_EMPTY;
            }
        } else if (rest >= at + 8) {
            const uint32_t x = ldg_u16_keep(a.memox + (e.y & ((1u << (2 * kk)) - 1)), pol_keep);
            const uint32_t h = pack8_at(a.text, e.x + at) & (L3_GRAMS - 1);
            if (x != L2_NONE) {
                const uint32_t o2 = ldg_u16_keep(a.l2tab + x * L2_GRAMS + ((e.y >> (2 * kk)) & (L2_GRAMS - 1)), pol_keep);
                keep = o2 != L2_EMPTY &&
                       ((ldg_u32_keep(a.l3 + o2 * (L3_GRAMS / 32) + (h >> 5), pol_keep) >> (h & 31)) & 1u);
                tag = o2;
            } else if (BATCH) {
                keep = false;   // (lean: no start lives without a record)
            }
        }
    }
    sieve_append<BATCH>(a, keep ? 1u : 0u, e.x, tag, lane);
}

// Tests the starts of the warp's first `k` list entries one by one. DNA: the
// deep bitmap of single starts; those that pass go on to the next levels (an
// NFA with such tables: by list2, 32 at a time) or become candidates.
template <int KIND, bool BATCH>
__device__ __forceinline__ void sieve_refine(const SieveArgs &a, const uint32_t *list, uint32_t k, uint2 *list2,
                                             uint32_t &cnt2, int lane, uint64_t pol_keep) {
    uint32_t keep = 0, first = 0, win = 0;   // bit r: start first + r stays
    if (static_cast<uint32_t>(lane) < k) {
        if (KIND == SIEVE_DNA) {
            first = list[2 * lane];
            win = list[2 * lane + 1];
            uint32_t w[SIEVE_DNA_STEP];
#pragma unroll
            for (int r = 0; r < SIEVE_DNA_STEP; ++r) {
                const uint32_t i = first + r;
                w[r] = i < a.n ? 1u : 0u;
                if (i < a.n && a.n - i >= SIEVE_DEEP_M) {
                    const uint32_t g = (win >> (2 * r)) & ((1u << (2 * SIEVE_DEEP_M)) - 1);
                    w[r] = ldg_u32_keep(a.surv2 + (g >> 5), pol_keep) >> (g & 31);
                }
            }
#pragma unroll
            for (int r = 0; r < SIEVE_DNA_STEP; ++r) keep |= (w[r] & 1u) << r;
        } else {
            // the gram began at list[lane], the last of the SIEVE_BYTE_STEP starts
            const uint32_t p = list[lane];
            first = p - (SIEVE_BYTE_STEP - 1);
#pragma unroll
            for (int r = 0; r < SIEVE_BYTE_STEP; ++r) keep |= (first + r < a.n ? 1u : 0u) << r;
            if (a.surv2 && p + 4 <= a.n && p >= SIEVE_BYTE_STEP) {
                // three bytes from each start: bytes p - 3 .. p + 2, in the
                // aligned words before and at p
                const uint32_t *q = reinterpret_cast<const uint32_t *>(a.text + p);
                const uint32_t w0 = __ldg(q - 1), w1 = __ldg(q);
                uint32_t w[SIEVE_BYTE_STEP];
#pragma unroll
                for (int r = 0; r < SIEVE_BYTE_STEP; ++r) {
                    const uint32_t g =
                        (r == SIEVE_BYTE_STEP - 1 ? w1 : __funnelshift_r(w0, w1, 8 * (r + 1))) & 0xFFFFFFu;
                    w[r] = ldg_u32_keep(a.surv2 + (g >> 5), pol_keep) >> (g & 31);
                }
                keep = 0;
#pragma unroll
                for (int r = 0; r < SIEVE_BYTE_STEP; ++r) keep |= (w[r] & 1u) << r;
            }
        }
    }
    if (KIND != SIEVE_DNA || !a.l3) {
        sieve_append<BATCH>(a, keep, first, SIEVE_NO_RECORD, lane);
        return;
    }
#pragma unroll
    for (int r = 0; r < SIEVE_DNA_STEP; ++r) {
        const uint32_t m = __ballot_sync(FULLMASK, (keep >> r) & 1u);
        if ((keep >> r) & 1u) list2[cnt2 + __popc(m & lanemask_lt())] = make_uint2(first + r, win >> (2 * r));
        cnt2 += __popc(m);
        if (cnt2 >= 32) {
            cnt2 -= 32;
            __syncwarp();
            sieve_levels<BATCH>(a, list2 + cnt2, 32, lane, pol_keep);
            __syncwarp();
        }
    }
}

// Lists the grams of one step whose bit is set in `hit`, one per lane at a
// time, and refines full warps of them. The grams lie P symbols apart: bit k
// belongs to the lane's 16 bytes in the step's (k / (16 / P))-th 512 bytes;
// `first` is the step's first position.
template <int KIND, bool BATCH, class Win>
__device__ __forceinline__ void sieve_collect(const SieveArgs &a, uint32_t hit, uint32_t first, uint32_t *list,
                                              uint32_t &cnt, uint2 *list2, uint32_t &cnt2, int lane, uint64_t pol_keep,
                                              Win &&win) {
    constexpr int W = KIND == SIEVE_DNA ? 2 : 1;   // words per list entry
    constexpr uint32_t P = KIND == SIEVE_DNA ? SIEVE_DNA_STEP : SIEVE_BYTE_STEP;
    while (true) {
        uint32_t m = 0;
        while (cnt < 32 && (m = __ballot_sync(FULLMASK, hit != 0)) != 0) {
            if (hit) {
                const uint32_t k = __ffs(hit) - 1;
                hit &= hit - 1;
                uint32_t *e = list + W * (cnt + __popc(m & lanemask_lt()));
                e[0] = first + 512 * (k / (16 / P)) + 16 * lane + P * (k % (16 / P));
                if (KIND == SIEVE_DNA) e[1] = win(k);
            }
            cnt += __popc(m);
        }
        if (cnt < 32) break;
        cnt -= 32;
        __syncwarp();
        sieve_refine<KIND, BATCH>(a, list + W * cnt, 32, list2, cnt2, lane, pol_keep);
        __syncwarp();
    }
}

// Any byte >= S among the text's bytes of a step that starts at position
// `first` (only called when one of the 2 KB is).
static __device__ __noinline__ bool bad_step(const uint8_t *text, uint32_t n, uint32_t S, int64_t first, uint32_t span,
                                      int lane) {
    bool bad = false;
    for (uint32_t o = lane; o < span; o += 32) {
        const int64_t p = first + o;
        if (p >= 0 && p < static_cast<int64_t>(n) && __ldg(text + p) >= S) bad = true;
    }
    return bad;
}

// One warp takes steps of 2 KB, from 16-byte boundaries of the address space
// so that no text needs realigning; the four loads of a lane are in flight
// together. A step wholly inside the text needs no bounds.
//
// DNA: the near bitmap (NEAR_SM: in shared memory, long texts) drops 4 in 5
// pairs of starts of the 256-motif NFA, the deep one (L2) leaves 1 in 46.
// Pairs: quads of starts would need half the shared-memory reads, but more
// L2 reads (0.66 per quad against 0.50), and those bound the kernel (66
// against 57 us per 64 MiB). 32 warps per SM, the most that fit beside the
// bitmap, measured best (24: 62 us, 16: 75 us).
// C: 512-byte pieces per step.
// Steps b0, b0 + stride .. below b1 of the text; what is left in the lists is
// taken by sieve_rest.
template <bool NEAR_SM, int C, bool BATCH>
__device__ __forceinline__ void dna_steps(const SieveArgs &a, const uint8_t *near, uint32_t *list, uint2 *list2,
                                          uint32_t b0, uint32_t b1, uint32_t stride, uint32_t &cnt, uint32_t &cnt2,
                                          bool &bad, int lane, uint64_t pol_keep) {
    constexpr uint32_t NEAR_WORDS = (1u << (2 * SIEVE_NEAR_M)) / 32;
    constexpr int P = SIEVE_DNA_STEP, G = 16 / P;   // grams per lane and 16 bytes
    constexpr int SH = 2 * (P - 1);   // a gram begins P - 1 symbols past the first of its starts
    constexpr uint32_t SPAN = 512 * C;
    const uint32_t n = a.n, S = a.S;
    const uint32_t *deep = a.deep;
    const uint32_t shift = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(a.text) & 15);
    const uint32_t span = n + shift;   // (n is below 2^32 - 256)
    // the step's 16 bytes per lane and piece, and the 16 after it (lane 0)
    const uint8_t *src = a.text - shift + static_cast<uint64_t>(b0) * SPAN + 16 * lane;
    uint32_t left = b1 > b0 ? span - b0 * SPAN : 0;   // bytes from the step fetched next to the end
    uint4 v[C + 1];
    auto fetch = [&]() {
#pragma unroll
        for (int c = 0; c <= C; ++c)
            v[c] = (c < C || lane == 0) && 512 * c + 16 * static_cast<uint32_t>(lane) < left ? ldg_stream(src + 512 * c)
                                                                                         : make_uint4(0u, 0u, 0u, 0u);
    };
    fetch();
    for (uint32_t b = b0; b < b1; b += stride) {
        const uint32_t first = b * SPAN - shift;   // the step's first position (may wrap below 0: past n)
        // inside: every symbol of the step and of the next 16 bytes belongs to the text
        const bool inside = first < n && left >= SPAN + 16;
        uint32_t x = 0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            if (S == 4) x |= (v[c].x | v[c].y | v[c].z | v[c].w) & 0xFCFCFCFCu;
            else x |= bytes_ge32(v[c].x, S) | bytes_ge32(v[c].y, S) | bytes_ge32(v[c].z, S) | bytes_ge32(v[c].w, S);
        }
        if (__any_sync(FULLMASK, x != 0))
            bad |= bad_step(a.text, n, S, static_cast<int64_t>(b) * SPAN - shift, SPAN, lane);
        if (!inside) {   // bytes around the text would spill into its packed symbols
#pragma unroll
            for (int c = 0; c <= C; ++c) {
                v[c].x &= 0x03030303u;
                v[c].y &= 0x03030303u;
                v[c].z &= 0x03030303u;
                v[c].w &= 0x03030303u;
            }
        }
        uint32_t pk[C + 1], nx[C];
#pragma unroll
        for (int c = 0; c <= C; ++c) pk[c] = pack16_sym(v[c].x, v[c].y, v[c].z, v[c].w);
        // the next step's loads are in flight while this one is tested
        src += static_cast<uint64_t>(stride) * SPAN;
        left = b + stride < b1 ? left - stride * SPAN : 0;
        fetch();
        // the 16 symbols after the lane's own: the next lane's, the last
        // lane's from the first lane's next block
#pragma unroll
        for (int c = 0; c < C; ++c) nx[c] = __shfl_sync(FULLMASK, lane == 0 ? pk[c + 1] : pk[c], lane + 1);
        uint32_t hit = 0xFFFFFFFFu >> (32 - C * G);
        if (NEAR_SM) {
            hit = 0;
#pragma unroll
            for (int c = C - 1; c >= 0; --c) {
                uint32_t w[G];
#pragma unroll
                for (int q = 0; q < G; ++q) {
                    const uint32_t t = __funnelshift_r(pk[c], nx[c], 2 * P * q + SH);
                    w[q] = *reinterpret_cast<const uint32_t *>(near + ((t >> 3) & (NEAR_WORDS * 4 - 4)));
                }
                // bitmap bits are stored from the top of a word down, so that
                // a left shift by the gram brings its bit to the top
#pragma unroll
                for (int q = G - 1; q >= 0; --q) {
                    const uint32_t t = __funnelshift_r(pk[c], nx[c], 2 * P * q + SH);
                    hit = __funnelshift_l(w[q] << (t & 31), hit, 1);
                }
            }
        }
#pragma unroll
        for (int c = 0; c < C; ++c) {
            uint32_t w[G];
#pragma unroll
            for (int q = 0; q < G; ++q) {
                w[q] = 0u;
                const uint32_t t = __funnelshift_r(pk[c], nx[c], 2 * P * q + SH);
                if ((hit >> (G * c + q)) & 1u)
                    w[q] = ldg_u32_keep(deep + ((t & ((1u << (2 * SIEVE_DEEP_M)) - 1)) >> 5), pol_keep) << (t & 31);
            }
            uint32_t d = 0;
#pragma unroll
            for (int q = G - 1; q >= 0; --q) d = __funnelshift_l(w[q], d, 1);
            hit &= ~(((1u << G) - 1) << (G * c)) | (d << (G * c));
        }
        if (!inside) {
            // starts whose 16 symbols pass the end of the text stay; those
            // wholly past it or before it go
            for (int k = 0; k < C * G; ++k) {
                const int64_t p = static_cast<int64_t>(b) * SPAN - shift + 512 * (k / G) + 16 * lane + P * (k % G);
                if (p >= static_cast<int64_t>(n) || p + P <= 0) hit &= ~(1u << k);
                else if (p + 16 > static_cast<int64_t>(n)) hit |= 1u << k;
            }
        }
        sieve_collect<SIEVE_DNA, BATCH>(a, hit, first, list, cnt, list2, cnt2, lane, pol_keep, [&](uint32_t k) {
            const uint32_t c = k / G;
            uint32_t lo = pk[0], hi = nx[0];
#pragma unroll
            for (int y = 1; y < C; ++y) {
                lo = c == static_cast<uint32_t>(y) ? pk[y] : lo;
                hi = c == static_cast<uint32_t>(y) ? nx[y] : hi;
            }
            return __funnelshift_r(lo, hi, 2 * P * (k % G));
        });
    }
}

// Bytes: the aligned words of the text, looked up by hash. With the next
// step's loads in flight 32 warps per SM read 5.3 TB/s; 48 warps without them
// 3.7 TB/s.
template <bool NEAR_SM, bool BATCH>
__device__ __forceinline__ void byte_steps(const SieveArgs &a, const uint8_t *near, uint32_t *list, uint32_t b0,
                                           uint32_t b1, uint32_t stride, uint32_t &cnt, bool &bad, int lane,
                                           uint64_t pol_keep) {
    const uint32_t n = a.n;
    const uint32_t shift = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(a.text) & 15);
    const uint32_t span = n + shift;   // (n is below 2^32 - 256)
    const uint8_t *src = a.text - shift + static_cast<uint64_t>(b0) * kSpan + 16 * lane;
    uint32_t left = b1 > b0 ? span - b0 * kSpan : 0;   // bytes from the step fetched next to the end
    auto fetch = [&](uint4 *v) {
        if (left >= kSpan) {
#pragma unroll
            for (int c = 0; c < 4; ++c) v[c] = ldg_stream(src + 512 * c);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                v[c] = 512 * c + 16 * static_cast<uint32_t>(lane) < left ? ldg_stream(src + 512 * c)
                                                                       : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    uint4 v[4];
    uint32_t none = 0;
    fetch(v);
    for (uint32_t b = b0; b < b1; b += stride) {
        const uint32_t first = b * kSpan - shift;   // the step's first position (may wrap below 0: past n)
        const bool inside = first < n && left >= kSpan;
        // the next step's loads are in flight while this one is tested
        uint4 ahead[4];
        src += static_cast<uint64_t>(stride) * kSpan;
        left = b + stride < b1 ? left - stride * kSpan : 0;
        fetch(ahead);
        // the bit of word i lands at bit i of `hit`
        uint32_t hit = 0;
#pragma unroll
        for (int c = 3; c >= 0; --c) {
            const uint32_t x[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
            uint32_t w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t h = sieve_hash_word(x[q]) * 4;
                w[q] = NEAR_SM ? *reinterpret_cast<const uint32_t *>(near + h) : __ldg(a.near + h / 4);
            }
#pragma unroll
            for (int q = 3; q >= 0; --q) hit = __funnelshift_l(w[q] << (x[q] & 31), hit, 1);
        }
        if (a.S < 256) {
            uint64_t y = 0;
#pragma unroll
            for (int c = 0; c < 4; ++c)
                y |= bytes_ge(v[c].x | (static_cast<uint64_t>(v[c].y) << 32), a.S) |
                     bytes_ge(v[c].z | (static_cast<uint64_t>(v[c].w) << 32), a.S);
            if (__any_sync(FULLMASK, y != 0))
                bad |= bad_step(a.text, n, a.S, static_cast<int64_t>(b) * kSpan - shift, kSpan, lane);
        }
        if (!inside) {
            // a gram before the text or past it is none (a start with less
            // than SIEVE_BYTE_STEP symbols left reports nothing); one that passes
            // the end keeps its starts
            for (int k = 0; k < 16; ++k) {
                const int64_t p = static_cast<int64_t>(b) * kSpan - shift + 512 * (k >> 2) + 16 * lane + 4 * (k & 3);
                if (p < 0 || p >= static_cast<int64_t>(n)) hit &= ~(1u << k);
                else if (p + 4 > static_cast<int64_t>(n)) hit |= 1u << k;
            }
        }
        sieve_collect<SIEVE_BYTES, BATCH>(a, hit, first, list, cnt, nullptr, none, lane, pol_keep, [](uint32_t) { return 0u; });
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = ahead[c];
    }
}

// What the steps left in the lists.
template <int KIND, bool BATCH>
__device__ __forceinline__ void sieve_rest(const SieveArgs &a, const uint32_t *list, uint2 *list2, uint32_t &cnt,
                                           uint32_t &cnt2, int lane, uint64_t pol_keep) {
    __syncwarp();
    if (cnt) sieve_refine<KIND, BATCH>(a, list, cnt, list2, cnt2, lane, pol_keep);
    __syncwarp();
    if (cnt2) sieve_levels<BATCH>(a, list2, cnt2, lane, pol_keep);
    __syncwarp();
    cnt = cnt2 = 0;
}

}  // namespace pfsm
