// Flat batches: the texts of a batch whose machines the sieve (sieve.cuh) or
// the direct scan (walk.cuh) takes, in two launches whatever the number of
// texts and machines.
//
// `flat_front` runs over the steps of all texts, sorted by class (2-bit
// sieve, byte sieve, direct scan) and machine: every CTA takes an equal share
// of their cost and every warp consecutive steps of it, so no step is claimed
// and nobody waits. `flat_finish` runs the sieves' candidates of all texts,
// each lane with its own text and machine.
//
// Measured, whole calls, against one tile kernel per class and shape plus the
// carry kernel in a graph: 64 requests over 24 machines 450 -> 69 us, of which
// flat_front takes 25 and flat_finish 12 (chains of dependent loads: a request
// is a few steps long); 10,000 texts over 16 machines, 1.1 GB, 4.7 -> 1.25 ms;
// 8 machines over 8 MiB each 350 -> 105 us. With full warps of steps flat_front
// is bound like the single-text kernels: 64 MiB of DNA 72 us against 60,
// 256 MiB of bytes 61 us against 50; the rest is the start of a share (its
// job, arguments and first loads) and arguments read from shared memory
// instead of the constant bank. Steps of 512 bytes of DNA (1 KB, as the
// single-text kernel takes: spills beside the arguments, 80 us); the text loop
// as a call of its own 87 us.
#include <algorithm>
#include <atomic>

#include "finish.cuh"
#include "walk.cuh"

namespace pfsm {

// Last job of [lo, hi) whose first step is <= x (every lane calls it).
__device__ __forceinline__ uint32_t flat_job(const BatchJob *jobs, uint32_t lo, uint32_t hi, uint32_t x, int lane) {
    while (hi - lo > 1) {
        const uint32_t each = (hi - lo + 31) / 32, at = lo + lane * each;
        const uint32_t m = __ballot_sync(FULLMASK, at < hi && jobs[at].unit_begin <= x);
        const uint32_t r = 31 - __clz(m);   // lane 0 always holds (lo's first step is <= x)
        lo += r * each;
        hi = min(hi, lo + each);
    }
    return lo;
}

// A warp's arguments for one text: the building blocks take them by reference.
union FlatWarp {
    SieveArgs sieve;
    WalkArgs walk;
};

// Steps [s0, s1) of class CLS by the calling warp.
template <int CLS, bool BIG>
__device__ __forceinline__ void flat_steps(const FlatArgs &A, FlatWarp &wa, uint32_t s0, uint32_t s1, int wid, int lane,
                                           uint64_t pol_keep) {
    if (s0 >= s1) return;
    const uint8_t *near = pfsm_dyn_smem;   // BIG: the near bitmap
    uint8_t *own = pfsm_dyn_smem + flat_own(CLS, BIG, wid);
    uint32_t *list = reinterpret_cast<uint32_t *>(own);
    uint2 *list2 = reinterpret_cast<uint2 *>(list + kSieveList * 2);
    uint32_t cnt = 0, cnt2 = 0;
    bool bad = false;
    WalkOut<4, kFlatStage> out{reinterpret_cast<uint32_t *>(own), 0u, 0u, 0u, 0ull};
    for (uint32_t j = flat_job(A.jobs, A.job_lo[CLS], A.job_hi[CLS], s0, lane); s0 < s1; ++j) {
        const BatchJob &J = A.jobs[j];
        const DevMachine &M = A.machs[J.mach];
        uint32_t b0, b1;
        flat_take(J, BIG, s0, s1, b0, b1);
        if (b0 >= b1) continue;   // the padding after a text
        __syncwarp();
        if (lane == 0) {
            if (CLS == FLAT_WALK) {
                WalkArgs &a = wa.walk;
                a.text = J.text;
                a.n = J.n;
                a.Q = M.Q;
                a.S = M.S;
                a.q0 = M.q0;
                a.tab = M.walk;
                for (int w = 0; w < 2; ++w) {
                    a.first[w] = M.walk_first[w];
                    a.finals[w] = M.walk_finals[w];
                }
                a.out = A.out;
                a.cap = A.cap;
                a.status = A.status;
                a.job_counts = A.job_counts;
                a.orig = J.orig;
            } else {
                SieveArgs &a = wa.sieve;
                a.text = J.text;
                a.n = J.n;
                a.S = M.S;
                a.near = M.sv_near;
                a.deep = M.sv_deep;
                a.surv2 = CLS == FLAT_DNA || (M.sbits == 8 && M.surv2_m == 3) ? M.surv2 : nullptr;
                a.memox = M.memox;
                a.l2tab = M.l2tab;
                a.l3 = M.kind == 1 ? M.sv_l3 : nullptr;
                a.k = M.k;
                a.min_match = M.min_match;
                a.job = j;
                a.cand = reinterpret_cast<uint2 *>(A.cand[M.kind]);
                a.cand_sum = A.cand_n + M.kind;
                a.cand_cap = A.cand_cap;
            }
        }
        __syncwarp();
        if (CLS == FLAT_DNA) {
            dna_steps<BIG, 1, true>(wa.sieve, near, list, list2, b0, b1, 1, cnt, cnt2, bad, lane, pol_keep);
            sieve_rest<SIEVE_DNA, true>(wa.sieve, list, list2, cnt, cnt2, lane, pol_keep);
        } else if (CLS == FLAT_BYTES) {
            byte_steps<BIG, true>(wa.sieve, near, list, b0, b1, 1, cnt, bad, lane, pol_keep);
            sieve_rest<SIEVE_BYTES, true>(wa.sieve, list, list2, cnt, cnt2, lane, pol_keep);
        } else {
            constexpr uint32_t R = flat_step(FLAT_WALK, BIG);
            const uint32_t head = b0 * R;
            const uint32_t stop = b1 == J.ntiles ? J.n : b1 * R;
            const uint8_t *tab = reinterpret_cast<const uint8_t *>(wa.walk.tab);
            const int words = M.walk_words;
            if (words == 0) walk_range<WalkDfa<false>, false>(wa.walk, tab, head, stop, out, bad, lane);
            else if (words == 1) walk_range<WalkNfa<1>, false>(wa.walk, tab, head, stop, out, bad, lane);
            else walk_range<WalkNfa<2>, false>(wa.walk, tab, head, stop, out, bad, lane);
            out.finish(wa.walk, lane);
        }
    }
    if (bad) atomicOr(&A.status[1], ERR_SYMBOL);
}

// BIG: one CTA of 32 warps per SM with the machine's near bitmap in shared
// memory (copied again where the CTA's share passes to the next machine);
// otherwise small CTAs that read the bitmaps through L1 and L2.
//
// The CTAs share the steps group by group: the deep bitmaps of the machines
// they test with at one time have to stay in L2 (8 MB each, read at random).
// 10,000 texts over 8 motif and 8 signature sets: all machines at once 1.63 ms
// for the kernel, 1.16 ms with two sets to a group, 0.90 ms with one.
template <bool BIG>
__global__ void __launch_bounds__(BIG ? 1024 : 128, 1) flat_front(const __grid_constant__ FlatArgs A) {
    __shared__ FlatWarp warps[BIG ? 32 : 4];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const uint32_t nw = blockDim.x >> 5;
    const uint64_t pol_keep = policy_evict_last();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    uint64_t from = 0;
    for (uint32_t g = 0; g < A.groups; ++g) {
        // this CTA's share of the group's cost, as steps of each class
        const uint64_t part = A.group_end[g] - from;
        const uint64_t x0 = from + part * blockIdx.x / gridDim.x, x1 = from + part * (blockIdx.x + 1) / gridDim.x;
        from += part;
        uint64_t base = 0;
#pragma unroll
        for (int c = 0; c < FLAT_CLASSES; ++c) {
            const uint32_t cost = flat_cost(c, BIG);
            auto step_at = [&](uint64_t x) -> uint32_t {
                return static_cast<uint32_t>(x <= base ? 0 : min(A.steps[c], (x - base + cost - 1) / cost));
            };
            uint32_t s0 = step_at(x0);
            const uint32_t s1 = step_at(x1);
            base += A.steps[c] * cost;
            while (s0 < s1) {
                uint32_t e = s1;
                if (BIG && c != FLAT_WALK) {
                    // one machine at a time: its near bitmap, then its steps
                    const BatchJob &J = A.jobs[flat_job(A.jobs, A.job_lo[c], A.job_hi[c], s0, lane)];
                    const DevMachine &M = A.machs[J.mach];
                    e = min(s1, M.flat_end);
                    __syncthreads();   // every warp is done with the bitmap before
                    if (c == FLAT_DNA) stage_near<(1u << (2 * SIEVE_NEAR_M)) / 8, 1024>(pfsm_dyn_smem, M.sv_near, tid);
                    else stage_near<(1u << SIEVE_HASH_BITS) / 8, 1024>(pfsm_dyn_smem, M.sv_near, tid);
                    __syncthreads();
                } else if (BIG) {
                    __syncthreads();   // the match buffers lie where the bitmap was
                }
                const uint32_t per = (e - s0 + nw - 1) / nw;
                const uint32_t w0 = min(e, s0 + wid * per), w1 = min(e, w0 + per);
                if (c == FLAT_DNA) flat_steps<FLAT_DNA, BIG>(A, warps[wid], w0, w1, wid, lane, pol_keep);
                else if (c == FLAT_BYTES) flat_steps<FLAT_BYTES, BIG>(A, warps[wid], w0, w1, wid, lane, pol_keep);
                else flat_steps<FLAT_WALK, BIG>(A, warps[wid], w0, w1, wid, lane, pol_keep);
                s0 = e;
            }
        }
    }
}

// ------------------------------------------------------------ candidates
using FlatOut = RowOut<4, FlatArgs>;

// One DFA candidate per lane, each with its own text and machine.
__device__ __forceinline__ void flat_dfa(const FlatArgs &A, FlatOut &out, bool act, uint32_t job, uint32_t start, int lane,
                                         uint64_t pol_keep) {
    const BatchJob &J = A.jobs[job];
    run_dfa(J, A.machs[J.mach], J.orig, act, start, out, lane, pol_keep);
}

// One NFA candidate per lane with its second-level record: the record's
// matches, then its set by strands (see run_items; a strand of at most 64
// states always fits its mask).
__device__ __forceinline__ void flat_nfa(const FlatArgs &A, FlatOut &out, bool act, uint32_t job, uint32_t start, uint32_t rec,
                                         uint4 *items, int lane) {
    const BatchJob &J = A.jobs[job];
    const DevMachine &M = A.machs[J.mach];
    const uint32_t n = J.n, orig = J.orig;
    uint32_t matches = 0, parts = 0;
    uint32_t pb[SIEVE_PARTS];
    uint64_t pm[SIEVE_PARTS];
    const uint32_t *r = M.pool2 + (act ? rec : 0u);
    if (act) {
        // the header and the words after it in one round trip (16 bytes of
        // slack follow the records)
        const uint32_t hdr = __ldg(r), w1 = __ldg(r + 1), w2 = __ldg(r + 2), w3 = __ldg(r + 3);
        matches = hdr & 0xFFFFu;
        uint32_t strand = 0xFFFFFFFFu;
        for (uint32_t x = 0; x < (hdr >> 16); ++x) {
            const uint32_t at = matches + x;
            const uint32_t q = at == 0 ? w1 : at == 1 ? w2 : at == 2 ? w3 : __ldg(r + 1 + at);
            const uint32_t st = __ldg(M.sv_strand + q);
            const bool first = st != strand;
            strand = st;
            parts += first;
#pragma unroll
            for (int p = 0; p < SIEVE_PARTS; ++p)
                if (static_cast<uint32_t>(p) + 1 == parts) {
                    if (first) {
                        pb[p] = q;
                        pm[p] = 0;
                    }
                    pm[p] |= 1ull << ((q - pb[p]) & 63);
                }
        }
    }
    // the record's matches (a record of a start near the end of its text may
    // hold some past it)
    for (uint32_t x = 0; __any_sync(FULLMASK, x < matches); ++x) {
        const uint32_t w = x < matches ? __ldg(r + 1 + x) : 0u;
        const uint32_t step = w >> 16;
        out.emit(x < matches && step < n - start, orig, start, start + step, w & 0xFFFFu, lane);
    }
    uint32_t incl = parts;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(FULLMASK, incl, d);
        if (lane >= d) incl += t;
    }
    const uint32_t runs = __shfl_sync(FULLMASK, incl, 31);
#pragma unroll
    for (int p = 0; p < SIEVE_PARTS; ++p)
        if (static_cast<uint32_t>(p) < parts)
            items[incl - parts + p] = make_uint4(lane, pb[p], static_cast<uint32_t>(pm[p]), static_cast<uint32_t>(pm[p] >> 32));
    __syncwarp();
    for (uint32_t r0 = 0; r0 < runs; r0 += 32) {
        bool on = r0 + lane < runs;
        const uint4 v = on ? items[r0 + lane] : make_uint4(lane, 0u, 0u, 0u);
        // the item's candidate: its text and machine
        const uint32_t ijob = __shfl_sync(FULLMASK, job, v.x), istart = __shfl_sync(FULLMASK, start, v.x);
        const BatchJob &IJ = A.jobs[ijob];
        const DevMachine &IM = A.machs[IJ.mach];
        const uint32_t in = IJ.n, iorig = IJ.orig;
        const uint8_t *text = IJ.text;
        const uint32_t *band = IM.band, *fin = band + IM.Q;
        uint32_t base = v.y, pos = istart + static_cast<uint32_t>(IM.k) + L2_SYMS;
        uint64_t mask = v.z | (static_cast<uint64_t>(v.w) << 32);
        uint32_t g0 = 0, g1 = 0, left = 0;
        on = on && pos < in;
        while (__any_sync(FULLMASK, on)) {
            if (on && left == 0) {
                pack32_at(text, in, pos, g0, g1);
                left = 32;
            }
            uint64_t next = 0, hits = 0;
            if (on) {
                const uint32_t c8 = (g0 & 3u) * 8;
                for (uint64_t m = mask; m; m &= m - 1) {
                    const uint32_t j = __ffsll(static_cast<long long>(m)) - 1;
                    if (!PFSM_OK_IDX(base + j < static_cast<uint32_t>(IM.Q), A.status)) break;
                    next |= static_cast<uint64_t>((__ldg(band + base + j) >> c8) & 0xFFu) << j;
                }
                on = next != 0;
            }
            if (on) {
                const uint32_t sh = __ffsll(static_cast<long long>(next)) - 1;
                mask = next >> sh;
                base += 1 + sh;
                // finality of states base .. base + 63 (words past the bitmap
                // hold no state of the mask)
                const uint32_t b = base >> 5, o = base & 31;
                const uint32_t f0 = __ldg(fin + b), f1 = __ldg(fin + b + 1), f2 = __ldg(fin + b + 2);
                hits = mask & (__funnelshift_r(f0, f1, o) | (static_cast<uint64_t>(__funnelshift_r(f1, f2, o)) << 32));
            }
            while (__any_sync(FULLMASK, hits != 0)) {
                out.emit(hits != 0, iorig, istart, pos, base + (hits ? __ffsll(static_cast<long long>(hits)) - 1 : 0), lane);
                hits &= hits - 1;
            }
            ++pos;
            on = on && pos < in;
            g0 = __funnelshift_r(g0, g1, 2);
            g1 >>= 2;
            --left;
        }
    }
    __syncwarp();
}

// The fallback's candidates, collected per warp in a part of the place of the
// list that overflowed: starts that the bitmap of single starts leaves
// (kEveryLeft), then (NFA) those with a record (kEveryFound). Each warp's runs
// are called from one place: with one for every way to fill a warp the code
// outgrew the instruction cache, and warps waited for instructions half of the
// time (256 MiB, 48 motifs: 7.0 ms, now 3.6).
constexpr uint32_t kEveryLeft = 160, kEveryFound = 64;
constexpr uint32_t kEveryPlace = kEveryLeft / 2 + kEveryFound;   // entries of 16 bytes

// The starts [from, to) of one NFA's text, as the front kernel and the list
// would have brought them: four starts per lane through the bitmap, then the
// records and the runs of full warps of what is left.
__device__ __forceinline__ void flat_every_nfa(const FlatArgs &A, uint32_t j, uint64_t from, uint64_t to, uint4 *place,
                                               unsigned long long *ready_n, uint4 *items, FlatOut &out, int lane,
                                               uint64_t pol_keep) {
    const BatchJob &J = A.jobs[j];
    const DevMachine &M = A.machs[J.mach];
    uint2 *left = reinterpret_cast<uint2 *>(place);   // {start, its first 16 symbols}
    uint4 *found = place + kEveryLeft / 2;            // as the list of the front kernel has them
    SieveArgs a{};
    a.text = J.text;
    a.n = J.n;
    a.k = M.k;
    a.min_match = M.min_match;
    a.memox = M.memox;
    a.l2tab = M.l2tab;
    a.l3 = M.sv_l3;
    a.job = j;
    a.cand = reinterpret_cast<uint2 *>(found);
    a.cand_sum = ready_n;
    a.cand_cap = kEveryFound;
    const uint32_t *surv2 = M.surv2;
    uint32_t cnt = 0, ready = 0;   // entries of both
    while (true) {
        while (ready < 32 && (cnt || from < to)) {
            if (cnt < 32 && from < to) {
                const uint64_t first = from + 4 * lane;
                const uint32_t keep = starts_left(a.text, a.n, first, to, surv2, SIEVE_DEEP_M, 2, pol_keep);
                uint32_t g0 = 0, g1 = 0;
                if (keep) pack32_at(a.text, a.n, static_cast<uint32_t>(first), g0, g1);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint32_t m = __ballot_sync(FULLMASK, (keep >> r) & 1u);
                    if ((keep >> r) & 1u)
                        left[cnt + __popc(m & lanemask_lt())] =
                            make_uint2(static_cast<uint32_t>(first) + r, __funnelshift_r(g0, g1, 2 * r));
                    cnt += __popc(m);
                }
                from += 128;
                continue;
            }
            const uint32_t k = min(cnt, 32u);
            cnt -= k;
            __syncwarp();
            sieve_levels<true>(a, left + cnt, k, lane, pol_keep);
            __syncwarp();
            ready = static_cast<uint32_t>(*static_cast<volatile unsigned long long *>(ready_n));
            __syncwarp();
        }
        if (ready == 0) break;
        const uint32_t k = min(ready, 32u);
        ready -= k;
        const uint4 c = found[ready + min(static_cast<uint32_t>(lane), k - 1)];
        __syncwarp();
        if (lane == 0) *ready_n = ready;
        __syncwarp();
        flat_nfa(A, out, static_cast<uint32_t>(lane) < k, c.x, c.y, c.z, items, lane);
    }
}

// The same for a DFA.
__device__ __forceinline__ void flat_every_dfa(const FlatArgs &A, uint32_t j, uint64_t from, uint64_t to, uint4 *place,
                                               FlatOut &out, int lane, uint64_t pol_keep) {
    const BatchJob &J = A.jobs[j];
    const DevMachine &M = A.machs[J.mach];
    uint32_t *left = reinterpret_cast<uint32_t *>(place), cnt = 0;
    while (from < to || cnt) {
        for (; cnt < 32 && from < to; from += 128) {
            const uint64_t first = from + 4 * lane;
            const uint32_t keep = starts_left(J.text, J.n, first, to, M.surv2, M.surv2 ? M.surv2_m : 0, M.sbits, pol_keep);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint32_t m = __ballot_sync(FULLMASK, (keep >> r) & 1u);
                if ((keep >> r) & 1u) left[cnt + __popc(m & lanemask_lt())] = static_cast<uint32_t>(first) + r;
                cnt += __popc(m);
            }
        }
        const uint32_t k = min(cnt, 32u);
        cnt -= k;
        __syncwarp();
        const bool act = static_cast<uint32_t>(lane) < k;
        const uint32_t start = act ? left[cnt + lane] : 0u;
        __syncwarp();
        if (k) flat_dfa(A, out, act, j, start, lane, pol_keep);
    }
}

// Every start of the texts of one kind, a few steps at a time, dealt out in
// turn to `warps` warps (this one is the me-th): texts may be long, and what a
// start costs differs from place to place. A function of its own, so that the
// kernel needs no more registers than the candidates do.
static __device__ __noinline__ void flat_every(const FlatArgs &A, uint32_t kind, uint64_t me, uint64_t warps,
                                               unsigned long long *ready_n, uint4 *items, uint32_t *rows, int lane) {
    const uint64_t pol_keep = policy_evict_last();
    uint4 *place = A.cand[kind] + me * kEveryPlace;
    if (lane == 0) *ready_n = 0;
    FlatOut out{A, rows, 0u};
    for (int c = 0; c < FLAT_WALK; ++c) {
        const uint64_t span = flat_step(c, false);   // (the same in both forms)
        const uint32_t steps = static_cast<uint32_t>(A.steps[c]), each = c == FLAT_DNA ? 8u : 2u;
        for (uint64_t x = me * each; x < steps; x += warps * each) {
            uint32_t s0 = static_cast<uint32_t>(x);
            const uint32_t s1 = static_cast<uint32_t>(min(static_cast<uint64_t>(steps), x + each));
            for (uint32_t j = flat_job(A.jobs, A.job_lo[c], A.job_hi[c], s0, lane); s0 < s1; ++j) {
                const BatchJob &J = A.jobs[j];
                const uint32_t b0 = s0 - J.unit_begin, b1 = min(J.ntiles, b0 + (s1 - s0));
                s0 = j + 1 < A.job_hi[c] ? min(s1, A.jobs[j + 1].unit_begin) : s1;
                if (b0 >= b1 || static_cast<uint32_t>(A.machs[J.mach].kind) != kind) continue;
                const uint64_t to = min(static_cast<uint64_t>(J.n), b1 * span);
                if (kind == 1) flat_every_nfa(A, j, b0 * span, to, place, ready_n, items, out, lane, pol_keep);
                else flat_every_dfa(A, j, b0 * span, to, place, out, lane, pol_keep);
            }
        }
    }
    out.flush(lane);
}

// Even CTAs run the DFA candidates, odd ones the NFA candidates. A list that
// overflowed (2 M) is replaced by every start of the texts of its kind: 256 MiB
// dense in matches, class kernels and these, ms: 1000-signature trie 4.1, 2.3;
// DNA trie 4.5, 2.2; 256 motifs 3.9, 2.7 and 6.4, 4.1; 48 motifs 5.7, 3.6. All
// CTAs for one kind where the other has no candidates: unions of motif sets
// 593 -> 625 us.
__global__ void __launch_bounds__(256, 4) flat_finish(const __grid_constant__ FlatArgs A) {
    __shared__ uint4 items_sm[8][32 * SIEVE_PARTS];
    __shared__ unsigned long long ready_sm[8];   // flat_every
    __shared__ uint32_t rows_sm[8][kOutRows * 4];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t pol_keep = policy_evict_last();
    const uint32_t kind = blockIdx.x & 1, ctas = gridDim.x / 2;
    const unsigned long long found = A.cand_n[kind];
    const uint64_t warps = static_cast<uint64_t>(ctas) * 8, me = static_cast<uint64_t>(wid) * ctas + blockIdx.x / 2;
    uint4 *items = items_sm[wid];
    if (found > A.cand_cap) {
        flat_every(A, kind, me, warps, ready_sm + wid, items, rows_sm[wid], lane);
        return;
    }
    FlatOut out{A, rows_sm[wid], 0u};
    const uint32_t per = static_cast<uint32_t>(min(32ull, (found + warps - 1) / warps));
    for (uint64_t x0 = me * per; x0 < found; x0 += warps * per) {
        const bool act = static_cast<uint32_t>(lane) < per && x0 + lane < found;
        const uint4 c = act ? A.cand[kind][x0 + lane] : A.cand[kind][x0];
        if (kind == 0) flat_dfa(A, out, act, c.x, c.y, lane, pol_keep);
        else flat_nfa(A, out, act, c.x, c.y, c.z, items, lane);
    }
    out.flush(lane);
}

// ------------------------------------------------------------ host helpers
cudaError_t launch_flat(const FlatArgs &a, bool big, int nsm, std::atomic<uint32_t> &smem_set, cudaStream_t s) {
    uint64_t steps = 0;
    for (int c = 0; c < FLAT_CLASSES; ++c) steps += a.steps[c];
    if (steps == 0) return cudaSuccess;
    if (big) {
        constexpr uint32_t smem = flat_own(FLAT_DNA, true, 32);
        static_assert(smem >= flat_own(FLAT_WALK, true, 32), "the match buffers fit the sieve's regions");
        if (!(smem_set.load(std::memory_order_relaxed) >> 9 & 1u)) {
            const cudaError_t e = cudaFuncSetAttribute(flat_front<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e != cudaSuccess) return e;
            smem_set.fetch_or(1u << 9, std::memory_order_relaxed);
        }
        flat_front<true><<<nsm, 1024, smem, s>>>(a);
    } else {
        constexpr uint32_t smem = flat_own(FLAT_WALK, false, 4);
        const int grid = static_cast<int>(std::min<uint64_t>((steps + 3) / 4, 8ull * nsm));
        flat_front<false><<<grid, 128, smem, s>>>(a);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (a.steps[FLAT_DNA] + a.steps[FLAT_BYTES] == 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(big ? 8 * nsm : 2 * nsm));
    cfg.blockDim = dim3(256);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, flat_finish, a);
}

}  // namespace pfsm
