// The host side of batches (csrc/batch.cu) without a GPU: the CUDA runtime and
// the rest of the library are replaced by stand-ins (host_cuda.h and below),
// and the launch of a flat batch is replayed step by step as its warps take
// them. Compiled by g++ (test_batch_host_cpu.py).
#include <mutex>

#include "batch.cu"
#include "host_cuda.h"

using namespace pfsm;

// What the launches of the last call did.
static struct Seen {
    int flat, graph;          // launches of the flat kernels, of the class graph
    int big, groups;
    int64_t steps, missed;    // flat steps of the texts; those not taken exactly once
    int64_t bounds;           // group bounds that do not ascend to the total
    int null_lists;           // a sieved flat launch without candidate lists
    int64_t used;             // machines whose use was recorded
} seen;
static uint32_t chunk = 5;    // steps a warp takes

void host_graph_launched() { seen.graph++; }

namespace pfsm {
uint32_t layout_smem(ScanArgs &, int, int, const SmemNeed &) { return 4096; }
int max_units_ctas_per_sm(int, int, uint32_t) { return 1; }
int batch_class(int kind, int, int, bool) { return kind ? 6 : 0; }
cudaError_t launch_units(int, const BatchArgs *, int, int, uint32_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_carry_batch(const BatchArgs *, int, cudaStream_t) { return cudaSuccess; }
bool default_params(const Machine &) { return true; }
bool walk_takes_batch(const Machine &, uint64_t) { return true; }
size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
int ensure_words(uint32_t **, size_t *, size_t) { return PFSM_OK; }
int make_resident(pfsm_ctx *, int, Machine &m, cudaStream_t, bool) { return m.full = true, PFSM_OK; }
int mark_use(pfsm_ctx *, cudaStream_t, Machine *const *, size_t k) { return seen.used = static_cast<int64_t>(k), PFSM_OK; }
Slot *get_slot(pfsm_ctx *, cudaStream_t, int) { return nullptr; }
void collect_timing(pfsm_ctx *, Slot *, int) {}
int finish_status(const unsigned long long *hs, uint64_t, uint64_t *n) { return *n = hs[0], PFSM_OK; }

// Every chunk of a class's steps as a warp of flat_front takes it.
cudaError_t launch_flat(const FlatArgs &a, bool big, int, std::atomic<uint32_t> &, cudaStream_t) {
    seen.flat++;
    seen.big = big;
    seen.groups = static_cast<int>(a.groups);
    if (a.steps[FLAT_DNA] + a.steps[FLAT_BYTES] && (!a.cand[0] || !a.cand[1])) seen.null_lists++;
    uint64_t total = 0, from = 0;
    for (int c = 0; c < FLAT_CLASSES; ++c) {
        total += a.steps[c] * flat_cost(c, big);
        std::vector<std::vector<int>> took(a.job_hi[c] - a.job_lo[c]);
        for (uint32_t j = a.job_lo[c]; j < a.job_hi[c]; ++j) took[j - a.job_lo[c]].assign(a.jobs[j].ntiles, 0);
        for (uint64_t x = 0; x < a.steps[c]; x += chunk) {
            uint32_t s0 = static_cast<uint32_t>(x);
            const uint32_t s1 = static_cast<uint32_t>(std::min<uint64_t>(a.steps[c], x + chunk));
            uint32_t j = a.job_lo[c];
            while (j + 1 < a.job_hi[c] && a.jobs[j + 1].unit_begin <= s0) ++j;   // as flat_job
            for (; s0 < s1; ++j) {
                if (j >= a.job_hi[c]) {
                    seen.missed++;
                    break;
                }
                uint32_t b0, b1;
                flat_take(a.jobs[j], big, s0, s1, b0, b1);
                for (uint32_t b = b0; b < b1; ++b) took[j - a.job_lo[c]][b]++;
            }
        }
        for (auto &t : took)
            for (int n : t) {
                seen.steps++;
                seen.missed += n != 1;
            }
    }
    if (a.groups < 1 || a.groups > static_cast<uint32_t>(kFlatGroups)) return seen.bounds++, cudaSuccess;
    for (uint32_t g = 0; g < a.groups; ++g) {
        seen.bounds += a.group_end[g] < from;
        from = a.group_end[g];
    }
    seen.bounds += from != total;
    return cudaSuccess;
}
}  // namespace pfsm

// ------------------------------------------------------------ entry points
extern "C" {
// A context whose machine i + 1 has flat class cls[i] (-1: none).
pfsm_ctx *hb_ctx(const int32_t *cls, int32_t k) {
    pfsm_ctx *c = new pfsm_ctx();
    c->nsm = 152;
    for (int32_t i = 0; i < k; ++i) {
        Machine &m = c->machines[i + 1];
        m.Q = 8;
        m.S = cls[i] == FLAT_BYTES ? 256 : 4;
        m.sbits = cls[i] == FLAT_BYTES ? 8 : 2;
        m.k = 2;
        m.sv_kind = cls[i] == FLAT_DNA ? SIEVE_DNA : cls[i] == FLAT_BYTES ? SIEVE_BYTES : SIEVE_NONE;
        m.walks = cls[i] == FLAT_WALK;
    }
    return c;
}
void hb_free(pfsm_ctx *c) {
    batch_free(c);
    delete c;
}
// The shared memory of a warp of flat_front for class c: {from, to}.
void hb_own(int32_t c, int32_t big, uint32_t warp, uint32_t *range) {
    range[0] = flat_own(c, big != 0, warp);
    range[1] = range[0] + flat_own_bytes(c);
}
void hb_fail(int n) { host_fail_in = n; }
void hb_chunk(uint32_t n) { chunk = n; }
// One batch of texts of n[i] symbols at address text[i] for machine aut[i].
int hb_scan(pfsm_ctx *c, const int32_t *aut, const uint64_t *text, const uint64_t *n, int32_t k, int64_t *out) {
    std::vector<pfsm_job> jobs(k);
    std::vector<uint64_t> counts(k);
    for (int32_t i = 0; i < k; ++i) jobs[i] = pfsm_job{aut[i], 0u, reinterpret_cast<const uint8_t *>(text[i]), n[i]};
    seen = Seen{};
    uint64_t total = 0;
    const int st = pfsm_scan_batch(c, jobs.data(), k, nullptr, 0, counts.data(), &total, nullptr);
    const int64_t v[] = {seen.flat, seen.graph, seen.big, seen.groups, seen.steps, seen.missed, seen.bounds, seen.null_lists, seen.used};
    memcpy(out, v, sizeof(v));
    return st;
}
}
