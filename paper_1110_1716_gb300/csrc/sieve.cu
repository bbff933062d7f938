// The sieve: single-text scans in two kernels, for machines with sieve tables
// (sieve_tables.cu).
//
// `sieve` streams the text once, straight from global memory into registers
// (16 bytes per lane, the next loads in flight), and tests one gram per
// SIEVE_BYTE_STEP starts. Where the bit is set, the starts are tested one by one
// against the deep survival bitmap, and those that pass are appended to a
// list of candidates. It holds no instance and reports no match, so it needs
// few registers and runs at full occupancy; `finish_dfa` / `finish_nfa` then
// run the few candidates (1 in 100 for the 256-motif NFA, 1 in 10,000 for
// the 1000-signature trie), spread evenly over the SMs.
//
// Measured on GB300 against the tile kernel that such scans took before
// (device time per scan): 1000-signature trie, 1 GiB: 752 -> 203 us (5.3
// TB/s of text; bound by shared-memory wavefronts of the random bitmap reads,
// 85 % of peak, and DRAM, 72 %); 4 MB: 40 -> 17 us; 256-motif NFA, 64 MiB:
// 213 -> 72 us (bound by the random 32-byte reads of the bitmaps in L2, one
// request per cycle and SM at 70 % of peak); 100 KB: 18 -> 17 us.
//
// Should the candidates outgrow their list, the finishing kernel takes every
// start of the text instead (the list is then ignored): slower, same result.
#include <atomic>

#include "scan_device.cuh"

namespace pfsm {

constexpr int kSmemLimit = 232448;   // opt-in shared memory per CTA

constexpr uint32_t kSpan = 2048;              // bytes a warp tests per step: 4 x 16 per lane
constexpr int kSieveList = 64;                // a warp's list: refined by 32, up to 32 more at a time

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

// Appends the lanes' kept starts (bit r of `keep`: start first + r) to the
// candidates, one atomic per call. `tag` goes with them.
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
    if (lane == 0) at = atomicAdd(a.cand_n, total);
    at = __shfl_sync(FULLMASK, at, 0) + incl - __popc(keep);
    while (keep) {
        const uint32_t r = __ffs(keep) - 1;
        keep &= keep - 1;
        if (at < a.cand_cap) a.cand[at] = make_uint2(first + r, tag);
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
// is left becomes a candidate with its record.
__device__ __forceinline__ void sieve_levels(const SieveArgs &a, const uint2 *list2, uint32_t k, int lane,
                                             uint64_t pol_keep) {
    bool keep = false;
    uint2 e = make_uint2(0u, 0u);
    uint32_t tag = SIEVE_NO_RECORD;
    if (static_cast<uint32_t>(lane) < k) {
        e = list2[lane];
        keep = true;
        const uint32_t kk = static_cast<uint32_t>(a.k), at = kk + L2_SYMS;
        if (a.n - e.x >= at + 8) {
            const uint32_t x = ldg_u16_keep(a.memox + (e.y & ((1u << (2 * kk)) - 1)), pol_keep);
            const uint32_t h = pack8_at(a.text, e.x + at) & (L3_GRAMS - 1);
            if (x != L2_NONE) {
                const uint32_t o2 = ldg_u16_keep(a.l2tab + x * L2_GRAMS + ((e.y >> (2 * kk)) & (L2_GRAMS - 1)), pol_keep);
                keep = o2 != L2_EMPTY &&
                       ((ldg_u32_keep(a.l3 + o2 * (L3_GRAMS / 32) + (h >> 5), pol_keep) >> (h & 31)) & 1u);
                tag = o2;
            }
        }
    }
    sieve_append(a, keep ? 1u : 0u, e.x, tag, lane);
}

// Tests the starts of the warp's first `k` list entries one by one. DNA: the
// deep bitmap of single starts; those that pass go on to the next levels (an
// NFA with such tables: by list2, 32 at a time) or become candidates.
template <int KIND>
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
        sieve_append(a, keep, first, SIEVE_NO_RECORD, lane);
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
            sieve_levels(a, list2 + cnt2, 32, lane, pol_keep);
            __syncwarp();
        }
    }
}

// Lists the grams of one step whose bit is set in `hit`, one per lane at a
// time, and refines full warps of them. The grams lie P symbols apart: bit k
// belongs to the lane's 16 bytes in the step's (k / (16 / P))-th 512 bytes;
// `first` is the step's first position.
template <int KIND, class Win>
__device__ __forceinline__ void sieve_collect(const SieveArgs &a, uint32_t hit, uint32_t first, uint32_t *list,
                                              uint32_t &cnt, uint2 *list2, uint32_t &cnt2, int lane, uint64_t pol_keep,
                                              Win &&win) {
    constexpr int W = KIND == SIEVE_DNA ? 2 : 1;   // words per list entry
    constexpr uint32_t P = KIND == SIEVE_DNA ? SIEVE_DNA_STEP : SIEVE_BYTE_STEP;
    uint32_t m;
    while ((m = __ballot_sync(FULLMASK, hit != 0)) != 0) {
        if (hit) {
            const uint32_t k = __ffs(hit) - 1;
            hit &= hit - 1;
            uint32_t *e = list + W * (cnt + __popc(m & lanemask_lt()));
            e[0] = first + 512 * (k / (16 / P)) + 16 * lane + P * (k % (16 / P));
            if (KIND == SIEVE_DNA) e[1] = win(k);
        }
        cnt += __popc(m);
        if (cnt >= 32) {
            cnt -= 32;
            __syncwarp();
            sieve_refine<KIND>(a, list + W * cnt, 32, list2, cnt2, lane, pol_keep);
            __syncwarp();
        }
    }
}

// Any byte >= S among the text's bytes of a step that starts at position
// `first` (only called when one of the 2 KB is).
__device__ __noinline__ bool bad_step(const uint8_t *text, uint32_t n, uint32_t S, int64_t first, uint32_t span,
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
template <bool NEAR_SM, int C>
__global__ void __launch_bounds__(NEAR_SM ? 1024 : 256, 1) sieve_dna(const SieveArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    constexpr uint32_t NEAR_WORDS = (1u << (2 * SIEVE_NEAR_M)) / 32;
    constexpr int P = SIEVE_DNA_STEP, G = 16 / P;   // grams per lane and 16 bytes
    constexpr int SH = 2 * (P - 1);   // a gram begins P - 1 symbols past the first of its starts
    constexpr uint32_t SPAN = 512 * C;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
    const uint64_t pol_keep = policy_evict_last();
    const uint32_t n = a.n;
    const uint32_t shift = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(a.text) & 15);
    const uint64_t span = static_cast<uint64_t>(n) + shift;
    const uint32_t steps = static_cast<uint32_t>((span + SPAN - 1) / SPAN);
    // the step's 16 bytes per lane and piece, and the 16 after it (lane 0)
    auto fetch = [&](uint64_t b, uint4 *v) {
        const uint64_t o0 = b * SPAN;
        const uint8_t *src = a.text - shift + o0 + 16 * lane;
#pragma unroll
        for (int c = 0; c <= C; ++c)
            v[c] = (c < C || lane == 0) && o0 + 512 * c + 16 * lane < span ? ldg_stream(src + 512 * c)
                                                                           : make_uint4(0u, 0u, 0u, 0u);
    };
    uint4 v[C + 1];
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * nw;
    fetch(blockIdx.x * nw + wid, v);
    if (NEAR_SM) {
        uint4 *d = reinterpret_cast<uint4 *>(smem);
        const uint4 *g = reinterpret_cast<const uint4 *>(a.near);
        for (uint32_t i = tid; i < NEAR_WORDS / 4; i += blockDim.x) d[i] = __ldg(g + i);
        __syncthreads();
    }
    // per warp: the list of grams {first start, 16 symbols}, the list of starts
    uint32_t *list = reinterpret_cast<uint32_t *>(smem + (NEAR_SM ? NEAR_WORDS * 4 : 0)) + wid * (kSieveList * 4);
    uint2 *list2 = reinterpret_cast<uint2 *>(list + kSieveList * 2);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    uint32_t cnt = 0, cnt2 = 0;   // list entries (warp-uniform)
    bool bad = false;
    for (uint64_t b = blockIdx.x * nw + wid; b < steps; b += stride) {
        const uint64_t o0 = b * SPAN;
        const uint32_t first = static_cast<uint32_t>(o0) - shift;   // the step's first position (may wrap below 0)
        // inside: every symbol of the step and of the next 16 bytes belongs to the text
        const bool inside = o0 >= shift && o0 + SPAN + 16 <= span;
        uint32_t x = 0;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            if (a.S == 4) x |= (v[c].x | v[c].y | v[c].z | v[c].w) & 0xFCFCFCFCu;
            else x |= bytes_ge32(v[c].x, a.S) | bytes_ge32(v[c].y, a.S) | bytes_ge32(v[c].z, a.S) | bytes_ge32(v[c].w, a.S);
        }
        if (__any_sync(FULLMASK, x != 0))
            bad |= bad_step(a.text, n, a.S, static_cast<int64_t>(o0) - shift, SPAN, lane);
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
        fetch(b + stride, v);
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
                    w[q] = *reinterpret_cast<const uint32_t *>(smem + ((t >> 3) & (NEAR_WORDS * 4 - 4)));
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
                    w[q] = ldg_u32_keep(a.deep + ((t & ((1u << (2 * SIEVE_DEEP_M)) - 1)) >> 5), pol_keep) << (t & 31);
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
                const int64_t p = static_cast<int64_t>(o0) - shift + 512 * (k / G) + 16 * lane + P * (k % G);
                if (p >= static_cast<int64_t>(n) || p + P <= 0) hit &= ~(1u << k);
                else if (p + 16 > static_cast<int64_t>(n)) hit |= 1u << k;
            }
        }
        sieve_collect<SIEVE_DNA>(a, hit, first, list, cnt, list2, cnt2, lane, pol_keep, [&](uint32_t k) {
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
    __syncwarp();
    if (cnt) sieve_refine<SIEVE_DNA>(a, list, cnt, list2, cnt2, lane, pol_keep);
    __syncwarp();
    if (cnt2) sieve_levels(a, list2, cnt2, lane, pol_keep);
    if (bad) atomicOr(&a.status[1], ERR_SYMBOL);
}

// Bytes: the aligned words of the text, looked up by hash. With the next
// step's loads in flight 32 warps per SM read 5.3 TB/s; 48 warps without them
// 3.7 TB/s.
template <bool NEAR_SM>
__global__ void __launch_bounds__(512, NEAR_SM ? 2 : 1) sieve_bytes(const SieveArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    constexpr uint32_t NEAR_WORDS = (1u << SIEVE_HASH_BITS) / 32;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
    const uint64_t pol_keep = policy_evict_last();
    if (NEAR_SM) {
        uint4 *d = reinterpret_cast<uint4 *>(smem);
        const uint4 *g = reinterpret_cast<const uint4 *>(a.near);
        for (uint32_t i = tid; i < NEAR_WORDS / 4; i += blockDim.x) d[i] = __ldg(g + i);
        __syncthreads();
    }
    uint32_t *list = reinterpret_cast<uint32_t *>(smem + (NEAR_SM ? NEAR_WORDS * 4 : 0)) + wid * kSieveList;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t n = a.n;
    const uint32_t shift = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(a.text) & 15);
    const uint64_t span = static_cast<uint64_t>(n) + shift;
    const uint32_t steps = static_cast<uint32_t>((span + kSpan - 1) / kSpan);
    uint32_t cnt = 0, cnt2 = 0;   // list entries (warp-uniform)
    bool bad = false;
    auto fetch = [&](uint64_t b, uint4 *v) {
        const uint64_t o0 = b * kSpan;
        const uint8_t *src = a.text - shift + o0 + 16 * lane;
        if (o0 + kSpan <= span) {
#pragma unroll
            for (int c = 0; c < 4; ++c) v[c] = ldg_stream(src + 512 * c);
        } else {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                v[c] = o0 + 512 * c + 16 * lane < span ? ldg_stream(src + 512 * c) : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    uint4 v[4];
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * nw;
    fetch(blockIdx.x * nw + wid, v);
    for (uint64_t b = blockIdx.x * nw + wid; b < steps; b += stride) {
        // the next step's loads are in flight while this one is tested
        uint4 ahead[4];
        fetch(b + stride, ahead);
        const uint64_t o0 = b * kSpan;
        const uint32_t first = static_cast<uint32_t>(o0) - shift;   // the step's first position (may wrap below 0)
        const bool inside = o0 >= shift && o0 + kSpan <= span;
        // the bit of word i lands at bit i of `hit`
        uint32_t hit = 0;
#pragma unroll
        for (int c = 3; c >= 0; --c) {
            const uint32_t x[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
            uint32_t w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t h = sieve_hash_word(x[q]) * 4;
                w[q] = NEAR_SM ? *reinterpret_cast<const uint32_t *>(smem + h) : __ldg(a.near + h / 4);
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
                bad |= bad_step(a.text, n, a.S, static_cast<int64_t>(o0) - shift, kSpan, lane);
        }
        if (!inside) {
            // a gram before the text or past it is none (a start with less
            // than SIEVE_BYTE_STEP symbols left reports nothing); one that passes
            // the end keeps its starts
            for (int k = 0; k < 16; ++k) {
                const int64_t p = static_cast<int64_t>(o0) - shift + 512 * (k >> 2) + 16 * lane + 4 * (k & 3);
                if (p < 0 || p >= static_cast<int64_t>(n)) hit &= ~(1u << k);
                else if (p + 4 > static_cast<int64_t>(n)) hit |= 1u << k;
            }
        }
        sieve_collect<SIEVE_BYTES>(a, hit, first, list, cnt, nullptr, cnt2, lane, pol_keep, [](uint32_t) { return 0u; });
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = ahead[c];
    }
    __syncwarp();
    if (cnt) sieve_refine<SIEVE_BYTES>(a, list, cnt, nullptr, cnt2, lane, pol_keep);
    if (bad) atomicOr(&a.status[1], ERR_SYMBOL);
}

__device__ __forceinline__ void finish_status_out(const SieveArgs &a) {
    scan_status_out(a.status, a.status_out, a.done, a.cand_n);
}

// ------------------------------------------------------------ candidates: DFA
// The eight text bytes from position pos (those past the end of the text are
// unspecified).
__device__ __forceinline__ uint64_t bytes8_at(uintptr_t text, uintptr_t end, uint32_t pos) {
    const uintptr_t at = text + pos, lo = at & ~static_cast<uintptr_t>(7);
    const uint32_t sh = static_cast<uint32_t>(at & 7) * 8;
    uint64_t w = __ldg(reinterpret_cast<const unsigned long long *>(lo)) >> sh;
    if (sh && lo + 8 < end) w |= __ldg(reinterpret_cast<const unsigned long long *>(lo + 8)) << (64 - sh);
    return w;
}

// One thread per candidate, over the text in global memory: the first k
// symbols by the prefix table, then by chains (the only way on from
// a state, up to eight symbols, compared at once) and single steps where the
// automaton branches. What bounds a candidate is its chain of dependent
// reads; a planted 32-byte signature takes some six instead of 32.
__global__ void __launch_bounds__(256) finish_dfa(const SieveArgs a) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t found = *a.cand_n;
    const bool every = found > a.cand_cap;   // the list is incomplete: every start
    const uint32_t total = every ? a.n : found;
    const uint64_t pol_keep = policy_evict_last();
    const int lane = threadIdx.x & 31;
    const uint32_t n = a.n, S = a.S, kk = static_cast<uint32_t>(a.k);
    const uintptr_t text = reinterpret_cast<uintptr_t>(a.text), end = text + n;
    // neighbouring candidates go to different CTAs, so that few of them still
    // use every SM
    const uint64_t warps = static_cast<uint64_t>(gridDim.x) * (blockDim.x >> 5);
    const uint64_t gw = static_cast<uint64_t>(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    for (uint64_t x0 = gw * 32; x0 < total; x0 += warps * 32) {
        const uint64_t x = x0 + lane;
        bool act = x < total;
        const uint32_t start = !act ? 0u : every ? static_cast<uint32_t>(x) : a.cand[x].x;
        uint32_t pos = start, s = a.q0;
        if (act && kk && n - start >= kk) {
            const uint64_t w = bytes8_at(text, end, pos);
            uint32_t gi = 0;
            bool in = true;
            for (uint32_t j = 0; j < kk; ++j) {
                const uint32_t c = static_cast<uint32_t>(w >> (8 * j)) & 0xFFu;
                in &= c < S;
                gi |= c << (j * a.sbits);
            }
            if (in) {
                const uint32_t e = ldg_u16_keep(a.memo + gi, pol_keep);
                if (e == PT_SKIP) {
                    act = false;
                } else if (!(e & PT_REC)) {   // a state; records and walks step from q0
                    s = e;
                    pos += kk;
                    if (pos >= n) act = false;
                }
            }
        }
        while (__any_sync(FULLMASK, act)) {
            bool hit = false;
            if (act) {
                if (!PFSM_OK_IDX(s < static_cast<uint32_t>(a.Q), a.status)) s = a.q0;
                const uint4 ch = __ldg(a.chain + s);
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
                    const uint32_t e = c < S ? ldg_u16_keep(a.dtab + s * S + c, pol_keep) : DEAD16;
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
            // the lanes that report on this symbol: one atomic
            const uint32_t m = __ballot_sync(FULLMASK, hit);
            if (m) {
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(&a.status[0], static_cast<unsigned long long>(__popc(m)));
                base = __shfl_sync(FULLMASK, base, 0) + __popc(m & lanemask_lt());
                if (hit && base < a.cap) {
                    uint32_t *o = a.out + base * 3;
                    o[0] = start;
                    o[1] = pos - 1;
                    o[2] = s;
                }
            }
        }
    }
    finish_status_out(a);
}

// ------------------------------------------------------------ candidates: NFA
// What a lane runs: the states of one strand (sv_strand) of one instance's
// set, base + j for the bits j of mask. Strands never meet, so the parts of a
// set run on their own and report nothing twice.
constexpr int RUN_PARTS = 3;
constexpr int kRunItems = 32 * RUN_PARTS;   // per warp
struct RunItem {
    uint32_t start, pos, base, mask;
};

// Runs the items of the lanes with `act` to their end, reporting final states.
// A symbol moves every state up by 1 .. 8 (its band row's byte), so the set
// after it is the OR of the bytes, shifted, over base + 1. A set that spreads
// over more than 32 states goes to the whole warp as a bitset over Q.
static __device__ __forceinline__ void run_items(const OView &ov, const MView &mv, const TileView &tv, const Smem &sm,
                                                 bool act, RunItem it, uint32_t &sn, int lane, uint64_t pol_keep) {
    const uint32_t n = tv.n;
    const uint32_t *band = sm.band, *fin = sm.band + mv.Q;
    uint32_t g0 = 0, g1 = 0, left = 0;
    while (__any_sync(FULLMASK, act)) {
        if (act && left == 0) {
            if (it.pos < n) pack32_at(tv.text, n, it.pos, g0, g1);
            left = 32;
        }
        uint64_t next = 0;
        bool wide = false;
        if (act && it.pos < n) {
            const uint32_t c8 = (g0 & 3u) * 8;
            uint32_t m = it.mask;
            while (m) {
                const uint32_t j = __ffs(m) - 1;
                m &= m - 1;
                if (!PFSM_OK_IDX(it.base + j < static_cast<uint32_t>(mv.Q), ov.status)) break;
                next |= static_cast<uint64_t>((band[it.base + j] >> c8) & 0xFFu) << j;
            }
        }
        act = act && next != 0;
        uint32_t hits = 0, base = 0;
        if (act) {
            const uint32_t sh = __ffsll(static_cast<long long>(next)) - 1;
            next >>= sh;
            base = it.base + 1 + sh;
            wide = (next >> 32) != 0;
            if (!wide) hits = static_cast<uint32_t>(next) & __funnelshift_r(fin[base >> 5], fin[(base >> 5) + 1], base & 31);
        }
        uint32_t wm = __ballot_sync(FULLMASK, wide);
        while (wm) {
            const int src = __ffs(wm) - 1;
            wm &= wm - 1;
            const uint32_t b = __shfl_sync(FULLMASK, it.base, src), k = __shfl_sync(FULLMASK, it.mask, src);
            uint32_t *b0 = sm.coop, *b1 = sm.coop + mv.Wq;
            for (uint32_t w = lane; w < static_cast<uint32_t>(mv.Wq); w += 32) {
                b0[w] = 0;
                b1[w] = 0;
            }
            __syncwarp();
            if ((k >> lane) & 1u) atomicOr(&b0[(b + lane) >> 5], 1u << ((b + lane) & 31));
            __syncwarp();
            coop_run_body<3>(ov, mv, band, tv, b0, b1, __shfl_sync(FULLMASK, it.start, src),
                             __shfl_sync(FULLMASK, it.pos, src), 0xFFFFFFFFu, lane, pol_keep);
            if (lane == src) act = false;
        }
        while (__any_sync(FULLMASK, hits != 0)) {
            const uint32_t f = base + (hits ? __ffs(hits) - 1 : 0u);
            warp_emit<3>(hits != 0, it.start, it.pos, f, sm.stage, sn, ov, tv, lane);
            hits &= hits - 1;
        }
        it.base = base;
        it.mask = static_cast<uint32_t>(next);
        ++it.pos;
        g0 = __funnelshift_r(g0, g1, 2);
        g1 >>= 2;
        --left;
    }
}

// The candidates of an NFA, a warp's 32 at a time: those that come with a
// second-level record report its matches and run on from its set, split into
// strands (run_items); the others (near the end of the text, machines without
// such tables, records of many states) take the general exact path.
__global__ void __launch_bounds__(kFinishThreads, 2) finish_nfa(const ScanArgs a, const SieveArgs sv) {
    extern __shared__ __align__(128) uint8_t smem[];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
    const Smem sm = smem_regions(smem, a, wid, nw);
    const OView ov{a.out, a.cap, a.status, nullptr, a.carry, a.carry_n, 0u, a.stage_n};
    const MView mv{a.Q, a.S, a.q0, a.k, a.sbits, a.Wq, a.surv_m, a.surv2_m, a.surv2, a.dtab, a.off, a.tgt,
                   a.tail, a.ecl_off, a.ecl_tgt, a.l2tab, a.pool2, a.memox, a.status, a.pool_n,
                   a.memo_n};
    const TileView tv{nullptr, a.text, 0u, 0u, a.n, 0u, 0u};
    const uint64_t pol_keep = policy_evict_last();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t found = *sv.cand_n, n = a.n;
    const bool every = found > sv.cand_cap;   // the list is incomplete: every start
    const uint32_t total = every ? n : found;
    // few candidates spread over every warp: `per` of them at a time; CTAs
    // without one leave before they copy the tables
    const uint64_t warps = static_cast<uint64_t>(gridDim.x) * nw;
    const uint32_t per = static_cast<uint32_t>(min(static_cast<uint64_t>(32), (total + warps - 1) / warps));
    if (static_cast<uint64_t>(blockIdx.x) * per >= total) {
        finish_status_out(sv);
        return;
    }
    stage_nfa(smem, a.sm_band, a.sm_pool, a.band_smem ? a.band : nullptr, a.Q, nullptr, 0u, tid, blockDim.x);
    __syncthreads();
    const uint32_t kk = static_cast<uint32_t>(a.k);
    const uint32_t mask = (1u << (2 * kk)) - 1;
    uint2 *items = reinterpret_cast<uint2 *>(smem + a.sm_list) + wid * kRunItems;   // {lane << 16 | base, mask}
    uint32_t sn = 0, wq_n = 0;
    for (uint64_t x0 = (static_cast<uint64_t>(wid) * gridDim.x + blockIdx.x) * per; x0 < total;) {
        const uint64_t x = x0 + lane;
        bool have = static_cast<uint32_t>(lane) < per && x < total;
        uint2 c = make_uint2(static_cast<uint32_t>(x), SIEVE_NO_RECORD);
        if (have && !every) c = sv.cand[x];
        uint32_t e = PT_SKIP;      // entry for the exact path
        bool from_l2 = false;
        uint32_t parts = 0, matches = 0;
        uint32_t pb[RUN_PARTS], pm[RUN_PARTS];
        if (have && c.y != SIEVE_NO_RECORD) {
            // the header and the words after it in one round trip (16 bytes of
            // slack follow the records)
            const uint32_t *r = a.pool2 + c.y;
            const uint32_t hdr = __ldg(r), w1 = __ldg(r + 1), w2 = __ldg(r + 2), w3 = __ldg(r + 3);
            matches = hdr & 0xFFFFu;
            uint32_t strand = 0xFFFFFFFFu;
            bool fits = sv.strand != nullptr;
#pragma unroll
            for (int p = 0; p < RUN_PARTS; ++p) pb[p] = pm[p] = 0u;
            for (uint32_t x = 0; x < (hdr >> 16) && fits; ++x) {
                const uint32_t at = matches + x;
                const uint32_t q = at == 0 ? w1 : at == 1 ? w2 : at == 2 ? w3 : __ldg(r + 1 + at);
                const uint32_t st = __ldg(sv.strand + q);   // (states ascend, so a strand's follow one another)
                if (st != strand) {
                    strand = st;
                    fits = parts < static_cast<uint32_t>(RUN_PARTS);
#pragma unroll
                    for (int p = 0; p < RUN_PARTS; ++p)
                        if (static_cast<uint32_t>(p) == parts) pb[p] = q;
                    ++parts;
                }
#pragma unroll
                for (int p = 0; p < RUN_PARTS; ++p)
                    if (static_cast<uint32_t>(p) + 1 == parts) {
                        fits = fits && q - pb[p] < 32;
                        pm[p] |= 1u << ((q - pb[p]) & 31);
                    }
            }
            if (!fits) {
                e = c.y;
                from_l2 = true;
                parts = matches = 0;
            }
        } else if (have) {
            uint32_t g0, g1;
            pack32_at(a.text, n, c.x, g0, g1);
            if (every && n - c.x >= SIEVE_DEEP_M) {
                const uint32_t d = g0 & ((1u << (2 * SIEVE_DEEP_M)) - 1);
                have = (ldg_u32_keep(sv.surv2 + (d >> 5), pol_keep) >> (d & 31)) & 1u;
            }
            if (have) {
                if (n - c.x >= kk) {
                    e = a.memo[g0 & mask];
                } else if (a.tail) {
                    const int jl = static_cast<int>(n - c.x);
                    e = __ldg(a.tail + tail_base(jl, 2) + (g0 & ((1u << (2 * jl)) - 1)));
                } else {
                    e = PT_WALK;
                }
            }
        }
        const uint32_t qm = __ballot_sync(FULLMASK, e != PT_SKIP);
        if (e != PT_SKIP) {
            const uint32_t at = wq_n + __popc(qm & lanemask_lt());
            sm.wq_start[at] = c.x;
            sm.wq_info[at] = static_cast<uint16_t>(e);
            queue_flag(sm.wq_flag, at, from_l2);
        }
        wq_n += __popc(qm);
        __syncwarp();
        if (__any_sync(FULLMASK, matches != 0))
            emit_record_matches<3>(matches, a.pool2, c.y + 1, c.x, sm.stage, sn, ov, tv, lane);
        uint32_t incl = parts;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(FULLMASK, incl, d);
            if (lane >= d) incl += t;
        }
        const uint32_t runs = __shfl_sync(FULLMASK, incl, 31);
#pragma unroll
        for (int p = 0; p < RUN_PARTS; ++p)
            if (static_cast<uint32_t>(p) < parts)
                items[incl - parts + p] = make_uint2(static_cast<uint32_t>(lane) << 16 | pb[p], pm[p]);
        __syncwarp();
        for (uint32_t r0 = 0; r0 < runs; r0 += 32) {
            const bool act = r0 + lane < runs;
            const uint2 v = act ? items[r0 + lane] : make_uint2(0u, 0u);
            RunItem it;
            it.start = __shfl_sync(FULLMASK, c.x, v.x >> 16);
            it.pos = it.start + kk + L2_SYMS;
            it.base = v.x & 0xFFFFu;
            it.mask = v.y;
            run_items(ov, mv, tv, sm, act, it, sn, lane, pol_keep);
        }
        __syncwarp();
        x0 += warps * per;
        // the queue is drained when another 32 would not fit and at the end
        if (wq_n && (wq_n + 32 > static_cast<uint32_t>(WARP_QUEUE) || x0 >= total)) {
            drain_nfa<3>(ov, mv, tv, sm, wq_n, sn, lane, pol_keep);
            wq_n = 0;
            __syncwarp();
        }
    }
    stage_flush<3>(sm.stage, sn, ov, 0u, lane);
    finish_status_out(sv);
}

// ------------------------------------------------------------ host helpers
// Sets a kernel's shared-memory limit once per context (bit `which` of
// *done; setting it twice from two threads is harmless).
template <class K>
static cudaError_t allow_smem(K k, int which, std::atomic<uint32_t> &done) {
    if (done.load(std::memory_order_relaxed) >> which & 1u) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
    if (e == cudaSuccess) done.fetch_or(1u << which, std::memory_order_relaxed);
    return e;
}

template <class K>
static cudaError_t launch_steps(K k, const SieveArgs &a, uint32_t span, int threads, int per_sm, uint32_t smem, int nsm,
                                cudaStream_t s) {
    const uint64_t warps = (static_cast<uint64_t>(a.n) + 15 + span - 1) / span;
    const uint64_t ctas = (warps + threads / 32 - 1) / (threads / 32);
    const int grid = static_cast<int>(ctas < static_cast<uint64_t>(nsm) * per_sm ? ctas : nsm * per_sm);
    k<<<grid, threads, smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_sieve(const SieveArgs &a, int kind, int nsm, std::atomic<uint32_t> &smem_set, cudaStream_t s) {
    // the shared copy of the near bitmap (128 KB, or 2 x 64 KB per SM) pays
    // once every warp has several steps to test with it
    const bool near_sm = a.n >= (8u << 20);
    if (kind == SIEVE_DNA) {
        const uint32_t lists = kSieveList * 16;
        if (!near_sm) return launch_steps(sieve_dna<false, 1>, a, 512, 64, 16, 2 * lists, nsm, s);
        cudaError_t e = allow_smem(sieve_dna<true, 2>, 0, smem_set);
        if (e != cudaSuccess) return e;
        return launch_steps(sieve_dna<true, 2>, a, 1024, 1024, 1, (1u << (2 * SIEVE_NEAR_M)) / 8 + 32 * lists, nsm, s);
    }
    const uint32_t lists = kSieveList * 4;
    if (!near_sm) return launch_steps(sieve_bytes<false>, a, kSpan, 64, 16, 2 * lists, nsm, s);
    cudaError_t e = allow_smem(sieve_bytes<true>, 1, smem_set);
    if (e != cudaSuccess) return e;
    return launch_steps(sieve_bytes<true>, a, kSpan, 512, 2, (1u << SIEVE_HASH_BITS) / 8 + 16 * lists, nsm, s);
}

template <class K, class... A>
static cudaError_t launch_dependent(K kernel, int grid, int threads, uint32_t smem, cudaStream_t s, const A &...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(static_cast<unsigned>(threads));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// CTAs of a finishing kernel: candidates are few per symbol, and a short text
// has few of them whatever it holds.
static int finish_grid(uint32_t n, uint32_t symbols, int most) {
    const uint32_t want = n / symbols + 8;
    return static_cast<int>(want < static_cast<uint32_t>(most) ? want : static_cast<uint32_t>(most));
}

cudaError_t launch_finish_dfa(const SieveArgs &a, int nsm, cudaStream_t s) {
    return launch_dependent(finish_dfa, finish_grid(a.n, 8192, 4 * nsm), 256, 0u, s, a);
}

uint32_t layout_finish_nfa(ScanArgs &a, uint32_t band_bytes, uint32_t coop_bytes) {
    constexpr uint32_t nw = kFinishThreads / 32;
    uint32_t o = 0;
    auto take = [&](uint32_t bytes) {
        const uint32_t r = o;
        o += (bytes + 15u) & ~15u;
        return r;
    };
    a.sm_misc = take(sizeof(Misc));
    a.sm_band = take(band_bytes);
    a.band_smem = band_bytes > 0;
    a.sm_list = take(nw * kRunItems * sizeof(uint2));
    a.sm_queue = take(nw * WARP_QUEUE * 6 + nw * (WARP_QUEUE / 8));
    a.sm_stage = take(nw * a.stage_n * 16);
    a.sm_slots = take(nw * 2 * NFA_SLOT * 32 * 2);
    a.sm_coop = take(coop_bytes);
    a.coop_smem = coop_bytes > 0;
    return (o + 127) & ~127u;
}

cudaError_t launch_finish_nfa(const ScanArgs &a, const SieveArgs &sv, uint32_t smem, int nsm,
                              std::atomic<uint32_t> &smem_set, cudaStream_t s) {
    if (smem > 48 * 1024) {
        cudaError_t e = allow_smem(finish_nfa, 2, smem_set);
        if (e != cudaSuccess) return e;
    }
    return launch_dependent(finish_nfa, finish_grid(sv.n, 2048, 2 * nsm), kFinishThreads, smem, s, a, sv);
}

}  // namespace pfsm
