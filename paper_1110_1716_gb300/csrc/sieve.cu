// The sieve: single-text scans in two kernels, for machines with sieve tables
// (sieve_tables.cu).
//
// `sieve` streams the text once, straight from global memory into registers
// (16 bytes per lane, the next loads in flight), and tests one gram per
// SIEVE_BYTE_STEP starts. Where the bit is set, the starts are tested one by one
// against the deep survival bitmap, and those that pass are appended to a
// list of candidates. It holds no instance and reports no match: in its form for
// long texts 61 - 63 registers and 32 warps per SM, as many as fit beside the
// bitmap; for short ones 72 (DNA) and 104 (bytes) in CTAs of two warps.
// `finish_dfa` / `finish_nfa` then run the few candidates (1 in 100 for the
// 256-motif NFA, 1 in 10,000 for the 1000-signature trie), spread evenly over
// the SMs.
//
// Measured on GB300 against the tile kernel that such scans took before
// (device time per scan): 1000-signature trie, 1 GiB: 752 -> 203 us (5.3
// TB/s of text; bound by shared-memory wavefronts of the random bitmap reads,
// 85 % of peak, and DRAM, 72 %); 4 MB: 40 -> 17 us; 256-motif NFA, 64 MiB:
// 213 -> 69 us (bound by the random 32-byte reads of the bitmaps in L2, one
// request per cycle and SM at 70 % of peak); 100 KB: 18 -> 17 us.
//
// Should the candidates outgrow their list (4 M), the finishing kernel takes
// every start of the text that the bitmap of single starts leaves instead: same
// result, in 0.4 - 0.75 of the tile kernel's time (finish.cuh).
#include <atomic>

#include "finish.cuh"

namespace pfsm {

constexpr int kSmemLimit = 232448;   // opt-in shared memory per CTA

template <bool NEAR_SM, int C>
__global__ void __launch_bounds__(NEAR_SM ? 1024 : 256, 1) sieve_dna(const SieveArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    constexpr uint32_t NEAR_BYTES = (1u << (2 * SIEVE_NEAR_M)) / 8;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const uint64_t pol_keep = policy_evict_last();
    if (NEAR_SM) {
        stage_near<NEAR_BYTES, 1024>(smem, a.near, threadIdx.x);
        __syncthreads();
    }
    // per warp: the list of grams {first start, 16 symbols}, the list of starts
    uint32_t *list = reinterpret_cast<uint32_t *>(smem + (NEAR_SM ? NEAR_BYTES : 0)) + wid * (kSieveList * 4);
    uint2 *list2 = reinterpret_cast<uint2 *>(list + kSieveList * 2);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    uint32_t cnt = 0, cnt2 = 0;
    bool bad = false;
    const uint32_t steps = (a.n - 1 + static_cast<uint32_t>(reinterpret_cast<uintptr_t>(a.text) & 15)) / (512 * C) + 1;
    dna_steps<NEAR_SM, C, false>(a, smem, list, list2, blockIdx.x * nw + wid, steps,
                                 gridDim.x * nw, cnt, cnt2, bad, lane, pol_keep);
    sieve_rest<SIEVE_DNA, false>(a, list, list2, cnt, cnt2, lane, pol_keep);
    if (bad) atomicOr(&a.status[1], ERR_SYMBOL);
}

template <bool NEAR_SM>
__global__ void __launch_bounds__(512, NEAR_SM ? 2 : 1) sieve_bytes(const SieveArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    constexpr uint32_t NEAR_BYTES = (1u << SIEVE_HASH_BITS) / 8;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const uint64_t pol_keep = policy_evict_last();
    if (NEAR_SM) {
        stage_near<NEAR_BYTES, 512>(smem, a.near, threadIdx.x);
        __syncthreads();
    }
    uint32_t *list = reinterpret_cast<uint32_t *>(smem + (NEAR_SM ? NEAR_BYTES : 0)) + wid * kSieveList;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    uint32_t cnt = 0, none = 0;
    bool bad = false;
    const uint32_t steps = (a.n - 1 + static_cast<uint32_t>(reinterpret_cast<uintptr_t>(a.text) & 15)) / kSpan + 1;
    byte_steps<NEAR_SM, false>(a, smem, list, blockIdx.x * nw + wid, steps, gridDim.x * nw, cnt,
                               bad, lane, pol_keep);
    sieve_rest<SIEVE_BYTES, false>(a, list, nullptr, cnt, none, lane, pol_keep);
    if (bad) atomicOr(&a.status[1], ERR_SYMBOL);
}

__device__ __forceinline__ void finish_status_out(const SieveArgs &a) {
    scan_status_out(a.status, a.status_out, a.done, a.cand_n);
}

// ------------------------------------------------------------ candidates: DFA
// One thread per candidate (run_dfa), over the text in global memory.
// Neighbouring candidates go to different CTAs, so that few of them still use
// every SM. Where the list is incomplete, every start is looked at, 128 of a
// warp at a time, and those left are run when a warp is full of them.
__global__ void __launch_bounds__(256) finish_dfa(const SieveArgs a) {
    __shared__ uint32_t rows_sm[8][kOutRows * 3];
    __shared__ uint32_t left_sm[8][160];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t found = *a.cand_n;
    const bool every = found > a.cand_cap;
    const uint32_t total = every ? a.n : found, each = every ? 128u : 32u;
    const uint64_t pol_keep = policy_evict_last();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t warps = static_cast<uint64_t>(gridDim.x) * (blockDim.x >> 5);
    RowOut<3, SieveArgs> out{a, rows_sm[wid], 0u};
    uint32_t *left = left_sm[wid], cnt = 0;   // every: starts to run
    uint64_t x0 = (static_cast<uint64_t>(wid) * gridDim.x + blockIdx.x) * each;
    while (true) {
        bool act;
        uint32_t start = 0;
        if (!every) {
            if (x0 >= total) break;
            act = x0 + lane < total;
            if (act) start = a.cand[x0 + lane].x;
            x0 += warps * each;
        } else {
            for (; cnt < 32 && x0 < total; x0 += warps * each) {
                const uint64_t first = x0 + 4 * lane;
                const uint32_t keep = starts_left(a.text, a.n, first, total, a.all2, a.all_m, a.sbits, pol_keep);
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const uint32_t m = __ballot_sync(FULLMASK, (keep >> r) & 1u);
                    if ((keep >> r) & 1u) left[cnt + __popc(m & lanemask_lt())] = static_cast<uint32_t>(first) + r;
                    cnt += __popc(m);
                }
            }
            if (cnt == 0) break;
            const uint32_t k = min(cnt, 32u);
            cnt -= k;
            __syncwarp();
            act = static_cast<uint32_t>(lane) < k;
            if (act) start = left[cnt + lane];
            __syncwarp();
        }
        run_dfa(a, a, 0u, act, start, out, lane, pol_keep);
    }
    out.flush(lane);
    finish_status_out(a);
}

// ------------------------------------------------------------ candidates: NFA
// What a lane runs: the states of one strand (sv_strand) of one instance's
// set, base + j for the bits j of mask. Strands never meet, so the parts of a
// set run on their own and report nothing twice.
constexpr int kRunItems = 32 * SIEVE_PARTS;   // per warp
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

// Where the list is incomplete, each warp uses a part of its place for starts
// that the bitmap leaves (kEveryLeft) and those with a record (kEveryFound).
constexpr uint32_t kEveryLeft = 160, kEveryFound = 64;
struct EveryState {
    uint2 *left;           // the warp's part
    uint64_t x0;           // the next start to look at
    uint32_t cnt, ready;   // entries of both
};
// Collects candidates until a warp is full of them or the text ends, and takes
// up to 32 from the end: their number is returned, `ready` is where they lie. A
// function of its own, for the kernel's sake where lists are complete.
static __device__ __noinline__ uint32_t every_fill(const SieveArgs &sv, EveryState &ev, uint32_t *ready_n, uint64_t warps,
                                                   int lane) {
    const uint64_t pol_keep = policy_evict_last();
    const uint32_t n = sv.n;
    uint2 *left = ev.left, *found = left + kEveryLeft;
    uint64_t x0 = ev.x0;
    uint32_t cnt = ev.cnt, ready = ev.ready;
    SieveArgs lv = sv;
    lv.cand = found;
    lv.cand_n = ready_n;
    lv.cand_cap = kEveryFound;
    while (ready < 32 && (cnt || x0 < n)) {
        if (cnt < 32 && x0 < n) {
            const uint64_t first = x0 + 4 * lane;
            const uint32_t keep = starts_left(sv.text, n, first, n, sv.surv2, SIEVE_DEEP_M, 2, pol_keep);
            uint32_t g0 = 0, g1 = 0;
            if (keep) pack32_at(sv.text, n, static_cast<uint32_t>(first), g0, g1);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint32_t m = __ballot_sync(FULLMASK, (keep >> r) & 1u);
                if ((keep >> r) & 1u)
                    left[cnt + __popc(m & lanemask_lt())] =
                        make_uint2(static_cast<uint32_t>(first) + r, __funnelshift_r(g0, g1, 2 * r));
                cnt += __popc(m);
            }
            x0 += warps * 128;
            continue;
        }
        const uint32_t k = min(cnt, 32u);
        cnt -= k;
        __syncwarp();
        if (sv.l3) {
            sieve_levels<false>(lv, left + cnt, k, lane, pol_keep);
            __syncwarp();
            ready = *static_cast<volatile uint32_t *>(ready_n);
        } else {
            if (static_cast<uint32_t>(lane) < k) found[ready + lane] = make_uint2(left[cnt + lane].x, SIEVE_NO_RECORD);
            ready += k;
        }
        __syncwarp();
    }
    const uint32_t k = min(ready, 32u);
    ready -= k;
    __syncwarp();
    if (lane == 0) *ready_n = ready;
    __syncwarp();
    ev.x0 = x0;
    ev.cnt = cnt;
    ev.ready = ready;
    return k;
}

// The candidates of an NFA, a warp's 32 at a time: those that come with a
// second-level record report its matches and run on from its set, split into
// strands (run_items); the others (near the end of the text, machines without
// such tables, records of many states) take the general exact path.
constexpr uint32_t kQueueBytes = WARP_QUEUE * 6 + WARP_QUEUE / 8;   // of a warp (smem_regions)
static_assert(kQueueBytes % 4 == 0, "the counters behind the queues are aligned");
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
    const uint64_t warp = static_cast<uint64_t>(wid) * gridDim.x + blockIdx.x;
    uint32_t *ready_n = reinterpret_cast<uint32_t *>(smem + a.sm_queue + nw * kQueueBytes) + wid;
    EveryState ev;
    if (every) {
        ev.left = sv.cand + warp * (kEveryLeft + kEveryFound);
        ev.x0 = warp * 128;
        ev.cnt = ev.ready = 0;
        if (lane == 0) *ready_n = 0;
    }
    bool done = false;
    for (uint64_t x0 = warp * per; !done && (every || x0 < total);) {
        bool have;
        uint2 c = make_uint2(0u, SIEVE_NO_RECORD);
        if (!every) {
            have = static_cast<uint32_t>(lane) < per && x0 + lane < total;
            if (have) c = sv.cand[x0 + lane];
            x0 += warps * per;
            done = x0 >= total;
        } else {
            const uint32_t k = every_fill(sv, ev, ready_n, warps, lane);
            have = static_cast<uint32_t>(lane) < k;
            if (have) c = ev.left[kEveryLeft + ev.ready + lane];
            __syncwarp();
            done = ev.ready == 0 && ev.cnt == 0 && ev.x0 >= total;
        }
        uint32_t e = PT_SKIP;      // entry for the exact path
        bool from_l2 = false;
        uint32_t parts = 0, matches = 0;
        uint32_t pb[SIEVE_PARTS], pm[SIEVE_PARTS];
        if (have && c.y != SIEVE_NO_RECORD) {
            // the header and the words after it in one round trip (16 bytes of
            // slack follow the records)
            const uint32_t *r = a.pool2 + c.y;
            const uint32_t hdr = __ldg(r), w1 = __ldg(r + 1), w2 = __ldg(r + 2), w3 = __ldg(r + 3);
            matches = hdr & 0xFFFFu;
            uint32_t strand = 0xFFFFFFFFu;
            bool fits = sv.strand != nullptr;
#pragma unroll
            for (int p = 0; p < SIEVE_PARTS; ++p) pb[p] = pm[p] = 0u;
            for (uint32_t x = 0; x < (hdr >> 16) && fits; ++x) {
                const uint32_t at = matches + x;
                const uint32_t q = at == 0 ? w1 : at == 1 ? w2 : at == 2 ? w3 : __ldg(r + 1 + at);
                const uint32_t st = __ldg(sv.strand + q);   // (states ascend, so a strand's follow one another)
                if (st != strand) {
                    strand = st;
                    fits = parts < static_cast<uint32_t>(SIEVE_PARTS);
#pragma unroll
                    for (int p = 0; p < SIEVE_PARTS; ++p)
                        if (static_cast<uint32_t>(p) == parts) pb[p] = q;
                    ++parts;
                }
#pragma unroll
                for (int p = 0; p < SIEVE_PARTS; ++p)
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
            if (n - c.x >= kk) {
                e = a.memo[g0 & mask];
            } else if (a.tail) {
                const int jl = static_cast<int>(n - c.x);
                e = __ldg(a.tail + tail_base(jl, 2) + (g0 & ((1u << (2 * jl)) - 1)));
            } else {
                e = PT_WALK;
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
        for (int p = 0; p < SIEVE_PARTS; ++p)
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
        // the queue is drained when another 32 would not fit and at the end
        if (wq_n && (wq_n + 32 > static_cast<uint32_t>(WARP_QUEUE) || done)) {
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
    // once the steps tested with it outweigh the copying (whole scans, with
    // it and without: DNA 1 MiB 22.6 and 20.5 us, 2 MiB 22.2 and 21.8, 3 MiB
    // 23.1 and 26.1, 8 MiB 26.8 and 39.8; bytes 1 MiB 12.3 and 12.3, 4 MiB
    // 14.3 and 16.4, 8 MiB 14.4 and 18.6; between 2 and 8 MiB both are right: 16
    // files of 4 MB with their matches sorted took 337 and 329 us, which is
    // within what runs differ by)
    const bool near_sm = a.n >= (kind == SIEVE_DNA ? 3u : 8u) << 20;
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
    // (eight CTAs fit an SM; four do but for long texts dense in candidates)
    return launch_dependent(finish_dfa, finish_grid(a.n, 8192, (a.n >= 64u << 20 ? 8 : 4) * nsm), 256, 0u, s, a);
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
    a.sm_queue = take(nw * (kQueueBytes + 4));   // the warps' queues, then their counters (ready_n)
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
