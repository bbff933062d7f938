// The library's host side without a GPU (csrc/pfsm_api.cu, sieve_tables.cu,
// batch.cu over the stand-ins of host_cuda.h): loading, residency and the
// choice of a scan's kernels, which are recorded instead of launched. Exports
// the C ABI as far as those files define it, and the hl_* functions below.
// Compiled by g++ (test_residency_host_cpu.py).
#include <mutex>
#include <string>

#include "pfsm_api.cu"
#include "sieve_tables.cu"
#include "batch.cu"
#include "host_cuda.h"

static std::string launched;   // since the last hl_launched()
void host_graph_launched() { launched += "classes "; }

namespace pfsm {
static cudaError_t note(const char *what) { return launched += what, launched += " ", cudaSuccess; }
uint32_t layout_smem(ScanArgs &a, int, int, const SmemNeed &need) {
    a.coop_smem = need.coop_bytes > 0;
    return 4096;
}
uint32_t layout_finish_nfa(ScanArgs &a, uint32_t, uint32_t coop) { return a.coop_smem = coop > 0, 4096; }
int max_ctas_per_sm(int, int, int, uint32_t, bool, int) { return 1; }
int max_units_ctas_per_sm(int, int, uint32_t) { return 1; }
int batch_class(int kind, int, int, bool) { return kind ? 6 : 0; }
cudaError_t launch_units(int, const BatchArgs *, int, int, uint32_t, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_carry_batch(const BatchArgs *, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_scan(const ScanArgs &, int, int, int, uint32_t, cudaStream_t) { return note("tiles"); }
cudaError_t launch_carry(const ScanArgs &, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_carry_nfa(const ScanArgs &, int, int, cudaStream_t) { return cudaSuccess; }
static const char *sieve_name(const SieveArgs &a) { return a.near && a.cand ? "sieve" : "sieve-without-tables"; }
cudaError_t launch_sieve(const SieveArgs &a, int, int, std::atomic<uint32_t> &, cudaStream_t) { return note(sieve_name(a)); }
cudaError_t launch_finish_dfa(const SieveArgs &, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_finish_nfa(const ScanArgs &, const SieveArgs &, uint32_t, int, std::atomic<uint32_t> &, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t launch_walk(WalkArgs a, int, int, std::atomic<uint32_t> &, cudaStream_t) {
    return note(a.tab ? "walk" : "walk-without-table");
}
cudaError_t launch_long(const WalkArgs &a, uint32_t *scratch, size_t, int, std::atomic<uint32_t> &, cudaStream_t) {
    return note(a.tab && scratch ? "long" : "long-without-tables");
}
uint32_t walk_nfa_words(int Q) { return Q <= 32 ? 1u : 2u; }
bool long_fits(uint32_t, int, size_t) { return true; }
cudaError_t launch_flat(const FlatArgs &a, bool, int, std::atomic<uint32_t> &, cudaStream_t) {
    for (int c = 0; c < FLAT_CLASSES; ++c)
        for (uint32_t j = a.job_lo[c]; j < a.job_hi[c]; ++j) {
            const DevMachine &m = a.machs[a.jobs[j].mach];
            if (c == FLAT_WALK ? !m.walk : !m.sv_near || !a.cand[0]) return note("flat-without-tables");
        }
    return note("flat");
}
}  // namespace pfsm

extern "C" {
void hl_fail(int n) { host_fail_in = n; }
void hl_largest(uint64_t n) { host_largest = n ? n : ~size_t(0); }
// What was launched since the last call, by name.
const char *hl_launched() {
    static std::string s;
    s = launched;
    launched.clear();
    return s.c_str();
}
}
