// Load-time tables of the sieve (sieve.cu): which grams can occur a few
// symbols into an instance that still matters.
//
// A start i is dead when its instance meets no final state and holds no state
// any more after some symbols; only the others can report. One lookup at a
// sampled position answers for `step` starts at once: for the gram w read at
// position p, the bit of w is set when, for some offset o < step and some o
// symbols before p, an instance started at p - o is still alive after w or
// meets a final state inside w. A clear bit settles all `step` starts. This
// needs every final state to lie at least `step` symbols from q0 (a shorter
// match would end before the gram); other machines have no sieve.
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <thread>
#include <vector>

#include "pfsm_host.h"

namespace pfsm {

namespace {

// delta as edges, in the order of their states and symbols; targets as
// state | FINAL_BIT, epsilon closures among them.
struct Delta {
    int Q = 0, S = 0;
    std::vector<uint32_t> row;     // first edge of every state
    std::vector<uint8_t> sym;      // per edge
    std::vector<uint16_t> tgt;
    std::vector<uint32_t> off;     // alphabets of at most 4: first edge of every (state, symbol)
    std::vector<uint16_t> start;   // the states an instance starts with
    void add(int a, uint16_t t) {
        sym.push_back(static_cast<uint8_t>(a));
        tgt.push_back(t);
    }
};

void flatten(const Machine &m, Delta &d) {
    d.Q = m.Q;
    d.S = m.S;
    d.row.assign(static_cast<size_t>(m.Q) + 1, 0);
    d.start.assign(1, static_cast<uint16_t>(m.q0));
    const bool small = m.S <= 4;
    if (small) d.off.assign(static_cast<size_t>(m.Q) * m.S + 1, 0);
    std::vector<uint16_t> ts;
    constexpr uint64_t DEAD4 = 0x0001000100010001ull * DEAD16;
    for (int q = 0; q < m.Q; ++q) {
        d.row[q] = static_cast<uint32_t>(d.tgt.size());
        const size_t r = static_cast<size_t>(q) * m.S;
        for (int a = 0; a < m.S; ++a) {
            if (small) d.off[r + a] = static_cast<uint32_t>(d.tgt.size());
            if (m.kind == 0) {
                const uint16_t *e = m.dtab.data() + r + a;
                if (!small && (a & 3) == 0 && a + 4 <= m.S) {   // wide rows are mostly dead
                    uint64_t four;
                    memcpy(&four, e, sizeof(four));
                    if (four == DEAD4) {
                        a += 3;
                        continue;
                    }
                }
                if (*e != DEAD16) d.add(a, *e);
                continue;
            }
            const uint32_t lo = m.off[r + a], hi = m.off[r + a + 1];
            if (m.ecl_off.empty()) {
                for (uint32_t e = lo; e < hi; ++e) d.add(a, m.tgt[e]);
                continue;
            }
            ts.clear();
            for (uint32_t e = lo; e < hi; ++e) {
                const uint32_t t = m.tgt[e] & 0x7FFF;
                ts.push_back(m.tgt[e]);
                ts.insert(ts.end(), m.ecl_tgt.begin() + m.ecl_off[t], m.ecl_tgt.begin() + m.ecl_off[t + 1]);
            }
            std::sort(ts.begin(), ts.end());
            ts.erase(std::unique(ts.begin(), ts.end()), ts.end());
            for (uint16_t t : ts) d.add(a, t);
        }
    }
    d.row[m.Q] = static_cast<uint32_t>(d.tgt.size());
    if (small) d.off[static_cast<size_t>(m.Q) * m.S] = static_cast<uint32_t>(d.tgt.size());
    if (!m.ecl_off.empty())
        for (uint32_t x = m.ecl_off[m.q0]; x < m.ecl_off[m.q0 + 1]; ++x)
            d.start.push_back(static_cast<uint16_t>(m.ecl_tgt[x] & 0x7FFF));
}

// The states an instance can hold after 0 .. step - 1 symbols; false when one
// of them, past the start, is final.
bool sampled_states(const Delta &d, int step, std::vector<uint16_t> &u) {
    std::vector<uint8_t> in(d.Q, 0);
    std::vector<uint16_t> cur = d.start;
    u = cur;
    for (uint16_t q : cur) in[q] = 1;
    for (int o = 1; o < step; ++o) {
        std::vector<uint8_t> seen(d.Q, 0);
        std::vector<uint16_t> nxt;
        for (uint16_t q : cur)
            for (uint32_t e = d.row[q]; e < d.row[q + 1]; ++e) {
                const uint16_t t = d.tgt[e];
                if (t & FINAL_BIT) return false;
                if (!seen[t]) {
                    seen[t] = 1;
                    nxt.push_back(t);
                }
            }
        for (uint16_t q : nxt)
            if (!in[q]) {
                in[q] = 1;
                u.push_back(q);
            }
        cur.swap(nxt);
    }
    return true;
}

// ---- 2-bit symbols: one bit per m-gram (symbol j at bits 2j of the index) ----
// Depth-first over the grams. The subtrees are split by symbol 5 and the
// high bit of symbol 4 (index bits 9 .. 11) into 8 parts, one per thread:
// those bits choose the cache line, so no two threads write one line.
constexpr int kParts = 8;

struct GramWalk {
    const Delta &d;
    const std::vector<uint8_t> &next;   // per state: the symbols it has successors on
    int mm;
    uint32_t *bits;
    uint64_t limit;      // give up past this many set bits
    int part;            // -1: the whole tree
    uint32_t flip;       // 31: bits stored from the top of a word down
    uint64_t ones = 0;
    std::vector<uint32_t> mark;
    uint32_t stamp = 0;
    std::vector<std::vector<uint16_t>> lv;

    GramWalk(const Delta &dd, const std::vector<uint8_t> &nx, int m, uint32_t *b, uint64_t lim, int p, uint32_t f)
        : d(dd), next(nx), mm(m), bits(b), limit(lim), part(p), flip(f), mark(dd.Q, 0), lv(m + 1) {}

    bool mine(int depth, uint32_t prefix) const {
        if (part < 0) return true;
        if (depth > 5) return ((prefix >> 9) & 7u) == static_cast<uint32_t>(part);
        if (depth == 5) return ((prefix >> 9) & 1u) == static_cast<uint32_t>(part & 1);
        return true;
    }
    void set_range(uint32_t p, int depth) {   // every extension of a depth-long prefix
        const uint32_t rest = static_cast<uint32_t>(mm - depth) * 2;
        for (uint32_t hw = 0; hw < (1u << rest); ++hw) {
            const uint32_t w = p | (hw << (2 * depth));
            if (depth < 6 && !mine(6, w)) continue;
            bits[w >> 5] |= 1u << ((w & 31) ^ flip);
            ++ones;
        }
    }
    void run(int depth, uint32_t prefix) {
        const std::vector<uint16_t> &s = lv[depth];
        if (ones > limit) return;
        if (depth + 1 == mm) {   // the last symbol: alive when any state has a successor
            uint32_t any = 0;
            for (uint16_t q : s) any |= next[q];
            for (int a = 0; a < 4; ++a)
                if ((any >> a) & 1u) {
                    const uint32_t w = prefix | (static_cast<uint32_t>(a) << (2 * depth));
                    bits[w >> 5] |= 1u << ((w & 31) ^ flip);
                    ++ones;
                }
            return;
        }
        for (int a = 0; a < d.S; ++a) {
            const uint32_t p = prefix | (static_cast<uint32_t>(a) << (2 * depth));
            if (!mine(depth + 1, p)) continue;
            std::vector<uint16_t> &n = lv[depth + 1];
            n.clear();
            bool hit = false;
            ++stamp;
            for (uint16_t q : s) {
                const size_t r = static_cast<size_t>(q) * d.S + a;
                for (uint32_t e = d.off[r]; e < d.off[r + 1]; ++e) {
                    const uint16_t t = d.tgt[e], ts = t & 0x7FFF;
                    hit |= (t & FINAL_BIT) != 0;
                    if (mark[ts] == stamp) continue;
                    mark[ts] = stamp;
                    n.push_back(ts);
                }
            }
            if (hit) set_range(p, depth + 1);
            else if (!n.empty()) run(depth + 1, p);
        }
    }
};

// Per state: the symbols it has successors on.
std::vector<uint8_t> successor_symbols(const Delta &d) {
    std::vector<uint8_t> next(d.Q, 0);
    for (int q = 0; q < d.Q; ++q)
        for (int a = 0; a < d.S; ++a)
            if (d.off[static_cast<size_t>(q) * d.S + a] != d.off[static_cast<size_t>(q) * d.S + a + 1])
                next[q] |= static_cast<uint8_t>(1u << a);
    return next;
}

// The m-gram bitmap of instances that hold `from`; false (and no bitmap)
// when more than `limit` grams are set. `flip` 31: stored from the top of a
// word down, as the sieve reads them. `grams`: on entry those set in the
// bitmap of shorter grams that was built before (0: none), afterwards those
// set in this one. Fewer than kFewGrams walk on faster alone than threads start
// (a set of 4 motifs, 296 9-grams: 0.25 against 0.75 ms; of 16, 2284: 1.0
// against 0.75).
constexpr uint64_t kFewGrams = 1024;
bool gram_bits(const Delta &d, const std::vector<uint16_t> &from, int mm, uint64_t limit, uint32_t flip,
               std::vector<uint32_t> &bits, uint64_t &grams) {
    const std::vector<uint8_t> next = successor_symbols(d);
    bits.assign((size_t(1) << (2 * mm)) / 32, 0);
    const bool split = mm >= 10;
    const int parts = split ? kParts : 1;
    // (a part may hold four times its share before it gives up on its own)
    const uint64_t part_limit = split ? limit / kParts * 4 : limit;
    std::vector<uint64_t> ones(parts, 0);
    auto work = [&](int p) {
        GramWalk w(d, next, mm, bits.data(), part_limit, split ? p : -1, flip);
        w.lv[0] = from;
        w.run(0, 0);
        ones[p] = w.ones;
    };
    const int threads = grams && grams < kFewGrams
                            ? 1
                            : std::min<int>(parts, std::max(1u, std::thread::hardware_concurrency()));
    if (threads <= 1) {
        for (int p = 0; p < parts; ++p) work(p);
    } else {
        std::atomic<int> at{0};
        std::vector<std::thread> pool;
        auto loop = [&]() {
            for (int p; (p = at.fetch_add(1)) < parts;) work(p);
        };
        for (int t = 1; t < threads; ++t) {
            try {
                pool.emplace_back(loop);
            } catch (...) {
                break;   // no more threads: the others share the parts
            }
        }
        loop();
        for (std::thread &t : pool) t.join();
    }
    uint64_t total = 0;
    bool over = false;
    for (uint64_t o : ones) {
        total += o;
        over |= o > part_limit;
    }
    grams = total;
    if (over || total > limit) {
        bits.clear();
        return false;
    }
    return true;
}

// ---- wider symbols: the 4-grams as bytes, hashed to SIEVE_HASH_BITS bits ----
struct ByteWalk {
    const Delta &d;
    std::vector<uint32_t> &bits;
    uint32_t ones = 0;
    uint64_t steps = 0;
    bool over = false;

    void add(uint32_t gram) {
        uint32_t &w = bits[sieve_hash_word(gram)];
        const uint32_t bit = 0x80000000u >> (gram & 31);
        ones += (w & bit) ? 0u : 1u;
        w |= bit;
        if (++steps > (1u << 21) || ones > SIEVE_HASH_MAX) over = true;
    }
    void all(int depth, uint32_t gram) {   // every extension
        if (over) return;
        if (depth == 4) {
            add(gram);
            return;
        }
        for (int a = 0; a < d.S && !over; ++a) all(depth + 1, gram | (static_cast<uint32_t>(a) << (8 * depth)));
    }
    void run(uint16_t q, int depth, uint32_t gram) {
        if (over) return;
        if (depth == 4) {
            add(gram);
            return;
        }
        for (uint32_t e = d.row[q]; e < d.row[q + 1] && !over; ++e) {
            const uint16_t t = d.tgt[e];
            const uint32_t g = gram | (static_cast<uint32_t>(d.sym[e]) << (8 * depth));
            if (t & FINAL_BIT) all(depth + 1, g);
            else run(t, depth + 1, g);
        }
    }
};

}  // namespace

// The chains of a sieved DFA (see pfsm_internal.h).
static void build_chains(Machine &m, const Delta &d) {
    constexpr uint32_t NONE = 0xFFFFFFFFu;
    std::vector<uint32_t> only(d.Q, NONE);   // symbol << 16 | target of a state with one way on
    for (int q = 0; q < d.Q; ++q) {
        if (d.row[q + 1] - d.row[q] == 1) only[q] = (static_cast<uint32_t>(d.sym[d.row[q]]) << 16) | d.tgt[d.row[q]];
    }
    m.chain.assign(static_cast<size_t>(d.Q) * 4, 0u);
    for (int q = 0; q < d.Q; ++q) {
        uint32_t *c = m.chain.data() + static_cast<size_t>(q) * 4;
        uint32_t s = static_cast<uint32_t>(q), len = 0;
        bool fin = false;
        while (len < 8 && !fin && only[s] != NONE) {
            c[len >> 2] |= (only[s] >> 16) << (8 * (len & 3));
            fin = (only[s] & FINAL_BIT) != 0;
            s = only[s] & 0x7FFFu;
            ++len;
        }
        c[2] = len | (fin ? 256u : 0u);
        c[3] = s;
    }
}

// The strands of a sieved NFA (see sv_strand): parts of the machine that no
// edge joins once q0 is left.
static void build_strands(Machine &m) {
    m.sv_strand.clear();
    if (m.kind != 1 || m.band.empty()) return;
    std::vector<int> up(m.Q);
    for (int q = 0; q < m.Q; ++q) up[q] = q;
    auto root = [&](int q) {
        while (up[q] != q) q = up[q] = up[up[q]];
        return q;
    };
    for (int q = 0; q < m.Q; ++q) {
        if (q != m.q0 && m.band[q] == BAND_CSR) return;
        for (uint32_t e = m.off[static_cast<size_t>(q) * m.S]; e < m.off[static_cast<size_t>(q + 1) * m.S]; ++e) {
            const int t = m.tgt[e] & 0x7FFF;
            if (t == m.q0) return;
            if (q != m.q0) up[root(q)] = root(t);
        }
    }
    // numbered so that equal neighbours are one strand: a strand's states need
    // not be consecutive, but those of a set must not alternate
    m.sv_strand.resize(m.Q);
    for (int q = 0; q < m.Q; ++q) m.sv_strand[q] = static_cast<uint16_t>(root(q));
    int last = -1;
    std::vector<uint8_t> closed(m.Q, 0);
    for (int q = 0; q < m.Q; ++q) {
        if (q == m.q0) continue;
        const int r = m.sv_strand[q];
        if (r == last) continue;
        if (closed[r]) {   // two strands alternate: their sets would split wrongly
            m.sv_strand.clear();
            return;
        }
        if (last >= 0) closed[last] = 1;
        last = r;
    }
}

// Fills m.sv_kind and the sieve's tables. The limits only keep out machines
// whose bitmaps drop next to nothing: with 1 start in 25 left by the deep
// bitmap (760 motifs) the sieve still takes 1.74 against the tile kernel's
// 2.74 ms per 16 MiB, with 1 in 98 (256 motifs) 33 against 66 us.
void build_sieve(Machine &m) {
    m.sv_kind = SIEVE_NONE;
    m.sv_near.clear();
    m.sv_deep.clear();
    m.chain.clear();
    m.sv_strand.clear();
    const bool dna = m.sbits == 2 && m.sm_m2 == SIEVE_DEEP_M;
    const bool bytes = m.kind == 0 && m.sbits > 2;
    if (!dna && !bytes) return;
    const uint64_t direct = m.sm_ones2;
    if (dna && direct * 8 > (1ull << (2 * SIEVE_DEEP_M))) return;
    Delta d;
    flatten(m, d);
    std::vector<uint16_t> u;
    if (!sampled_states(d, dna ? SIEVE_DNA_STEP : SIEVE_BYTE_STEP, u)) return;
    if (dna) {
        uint64_t grams = m.sm_ones;
        if (!gram_bits(d, u, SIEVE_NEAR_M, (1ull << (2 * SIEVE_NEAR_M)) * 3 / 4, 31, m.sv_near, grams)) return;
        // What is left of the near grams three symbols on, by how the direct
        // ones thin out from 9 symbols to 13: instances that live on as those
        // of random DFAs do would fill the deep bitmap past its limit, and
        // finding that out takes several times as long as the other tables.
        auto share = [](const std::vector<uint32_t> &v) {
            uint64_t n = 0;
            for (uint32_t w : v) n += static_cast<uint64_t>(__builtin_popcount(w));
            return static_cast<double>(n) / (32.0 * static_cast<double>(v.size()));
        };
        const double at9 = m.sm_m == 9 ? share(m.surv) : 0.0;
        const double at13 = static_cast<double>(direct) / static_cast<double>(1ull << (2 * SIEVE_DEEP_M));
        if (at9 > 0.0 && share(m.sv_near) * std::pow(at13 / at9, 0.75) > 1.25 / 8) {
            m.sv_near.clear();
            return;
        }
        if (!gram_bits(d, u, SIEVE_DEEP_M, (1ull << (2 * SIEVE_DEEP_M)) / 8, 31, m.sv_deep, grams)) {
            m.sv_near.clear();
            return;
        }
        m.sv_kind = SIEVE_DNA;
        if (m.kind == 0) build_chains(m, d);
        else build_strands(m);
        return;
    }
    m.sv_near.assign((1u << SIEVE_HASH_BITS) / 32, 0);
    ByteWalk w{d, m.sv_near};
    for (uint16_t q : u) w.run(q, 0, 0);
    if (w.over) {
        m.sv_near.clear();
        return;
    }
    m.sv_kind = SIEVE_BYTES;
    build_chains(m, d);
}

// Whether every start of a sieved NFA that can report has a second-level
// record whose set a lane can run (see Machine::sv_lean); sets the length of
// the shortest match.
static bool lean(Machine &m, const Delta &d) {
    if (m.sv_strand.empty() || m.memox.empty() || m.k + L2_SYMS > SIEVE_DEEP_M) return false;
    std::vector<int> dist(m.Q, -1);
    std::vector<uint16_t> cur = d.start;
    for (uint16_t q : cur) dist[q] = 0;
    m.min_match = 0;
    for (uint32_t len = 1; !cur.empty() && !m.min_match; ++len) {
        std::vector<uint16_t> nxt;
        for (uint16_t q : cur)
            for (uint32_t e = d.row[q]; e < d.row[q + 1]; ++e) {
                if (d.tgt[e] & FINAL_BIT) m.min_match = len;
                const uint16_t t = d.tgt[e] & 0x7FFF;
                if (dist[t] >= 0) continue;
                dist[t] = static_cast<int>(len);
                nxt.push_back(t);
            }
        cur.swap(nxt);
    }
    if (m.min_match < static_cast<uint32_t>(m.k)) return false;   // (or nothing is ever reported)
    for (size_t g = 0; g < m.memox.size(); ++g)
        if (m.memo[g] != PT_SKIP && m.memox[g] == L2_NONE) return false;
    std::vector<int> lo(m.Q, m.Q), hi(m.Q, -1);
    for (int q = 0; q < m.Q; ++q) {
        const int r = m.sv_strand[q];
        if (q == m.q0) continue;
        lo[r] = std::min(lo[r], q);
        hi[r] = std::max(hi[r], q);
        if (hi[r] - lo[r] >= 64) return false;
    }
    for (size_t at = 0; at < m.pool2.size();) {
        const uint32_t nm = m.pool2[at] & 0xFFFFu, ns = m.pool2[at] >> 16;
        int parts = 0, last = -1;
        for (uint32_t x = 0; x < ns; ++x) {
            const int r = m.sv_strand[m.pool2[at + 1 + nm + x]];
            parts += r != last;
            last = r;
        }
        if (parts > SIEVE_PARTS) return false;
        at += 1 + nm + ns;
    }
    return true;
}

// The third level of a sieved NFA (see L3_SYMS); rebuilt with the records.
void build_level3(Machine &m) {
    m.sv_l3.clear();
    m.sv_lean = false;
    if (m.kind != 1 || m.sv_kind != SIEVE_DNA || m.l2tab.empty() || m.pool2.empty() ||
        m.pool2.size() > L3_MAX_ROWS)
        return;
    Delta d;
    flatten(m, d);
    m.sv_l3.assign(m.pool2.size() * (L3_GRAMS / 32), 0u);
    const std::vector<uint8_t> next = successor_symbols(d);
    GramWalk w(d, next, L3_SYMS, nullptr, ~0ull, -1, 0);
    for (size_t at = 0; at < m.pool2.size();) {
        const uint32_t nm = m.pool2[at] & 0xFFFFu, ns = m.pool2[at] >> 16;
        uint32_t *to = m.sv_l3.data() + at * (L3_GRAMS / 32);
        if (nm) {
            std::fill(to, to + L3_GRAMS / 32, 0xFFFFFFFFu);
        } else {
            w.lv[0].assign(m.pool2.begin() + at + 1, m.pool2.begin() + at + 1 + ns);
            w.bits = to;
            w.run(0, 0);
        }
        at += 1 + nm + ns;
    }
    m.sv_lean = lean(m, d);
}

// The bitset form of a machine of at most 64 states (see WalkArgs::tab).
static bool bitset_table(Machine &m, const Delta &d) {
    const uint32_t W = walk_nfa_words(m.Q), groups = (m.Q + 7) / 8;
    const size_t words = static_cast<size_t>(groups) * m.S * 256 * W;
    if (m.Q > 64 || words * 4 > 64 * 1024) return false;
    m.walk_tab.assign(words, 0u);
    std::vector<uint64_t> to(static_cast<size_t>(m.Q) * m.S, 0);
    for (int q = 0; q < m.Q; ++q)
        for (uint32_t e = d.row[q]; e < d.row[q + 1]; ++e)
            to[static_cast<size_t>(q) * m.S + d.sym[e]] |= 1ull << (d.tgt[e] & 0x7FFF);
    for (uint32_t g = 0; g < groups; ++g)
        for (int a = 0; a < m.S; ++a)
            for (uint32_t sub = 0; sub < 256; ++sub) {
                uint64_t t = 0;
                for (int b = 0; b < 8; ++b)
                    if ((sub >> b & 1u) && static_cast<int>(8 * g) + b < m.Q)
                        t |= to[static_cast<size_t>(8 * g + b) * m.S + a];
                for (uint32_t w = 0; w < W; ++w)
                    m.walk_tab[((static_cast<size_t>(g) * m.S + a) * 256 + sub) * W + w] =
                        static_cast<uint32_t>(t >> (32 * w));
            }
    uint64_t first = 0, fin = 0;
    for (uint16_t q : d.start) first |= 1ull << q;
    for (int q = 0; q < m.Q; ++q)
        if (m.fin[q]) fin |= 1ull << q;
    for (int w = 0; w < 2; ++w) {
        m.walk_first[w] = static_cast<uint32_t>(first >> (32 * w));
        m.walk_finals[w] = static_cast<uint32_t>(fin >> (32 * w));
    }
    return true;
}

// Instances of a machine of at most 64 states on uniform symbols.
namespace {
struct Tries {
    int S;
    std::vector<uint64_t> to;   // per state and symbol
    uint64_t first = 0, x = 0x9E3779B97F4A7C15ull;
    Tries(const Machine &m, const Delta &d) : S(m.S), to(static_cast<size_t>(m.Q) * m.S, 0) {
        for (int q = 0; q < m.Q; ++q)
            for (uint32_t e = d.row[q]; e < d.row[q + 1]; ++e)
                to[static_cast<size_t>(q) * S + d.sym[e]] |= 1ull << (d.tgt[e] & 0x7FFF);
        for (uint16_t q : d.start) first |= 1ull << q;
    }
    uint64_t step(uint64_t s) {
        x = x * 6364136223846793005ull + 1442695040888963407ull;
        const uint32_t a = static_cast<uint32_t>(((x >> 32) * static_cast<uint64_t>(S)) >> 32);
        uint64_t n = 0;
        for (; s; s &= s - 1) n |= to[static_cast<size_t>(__builtin_ctzll(s)) * S + a];
        return n;
    }
};
}  // namespace

// Whether 1 in 16 or more of the instances live for 256 uniform symbols
// (tried on 256 fixed texts).
static bool lives_long(const Machine &m, const Delta &d) {
    Tries t(m, d);
    int alive = 0;
    for (int i = 0; i < 256; ++i) {
        uint64_t s = t.first;
        for (int j = 0; j < 256 && s; ++j) s = t.step(s);
        alive += s != 0;
    }
    return alive >= 16;
}

// Machine::walk_states (of 2048 instances).
static double states_held(const Machine &m, const Delta &d) {
    Tries t(m, d);
    constexpr int runs = 2048;
    uint64_t sum = 0;
    for (int i = 0; i < runs && sum <= 3 * runs; ++i)
        for (uint64_t s = t.step(t.first); s && sum <= 3 * runs; s = t.step(s))
            sum += static_cast<uint64_t>(__builtin_popcountll(s));
    return static_cast<double>(sum) / runs;
}

// From how many symbols on the tile kernel, which drops most starts by the
// shallow bitmap before it steps them, beats the direct scan, which steps every
// one. It costs more to begin with (10 - 40 us a scan) and less per symbol
// where few starts are left. us per 2^20 symbols, of long texts:
//   DFAs: the direct scan 7, the tile kernel by the share of starts left and
//   the width of a symbol: 0.04 - 0.07 of DNA 5 - 6, 0.13 9; bytes 0.02 1.7,
//   0.16 6.5, 0.27 11; 0.09 of 20 symbols 12
//   NFAs: the direct scan by the words read per symbol, 8.5 + 2.4 per eight
//   states of a one-word set, 8 per eight of a two-word set; the tile kernel
//   5 where few starts are left, and where a quarter is, 8 and 8 more for every
//   state that a start holds over its life (32 states 12 and 15, 64 states
//   11 - 44; sets that grow 600)
// Whole scans, direct and tiles: 64-state DNA DFA 4 MiB 42, 56, 8 MiB 71, 60,
// 64 MiB 501, 410; 64 states over bytes 2 MiB 26, 28, 4 MiB 41, 29, 64 MiB
// 461, 116; NFAs of 64 states 1 MiB 87, 37 and 104, 137, 2 MiB 150, 47 and
// 177, 153; of 32, 4 MiB 88, 122, 8 MiB 161, 129.
static uint64_t walk_limit(const Machine &m) {
    constexpr uint64_t MiB = 1ull << 20, none = ~0ull;
    if (m.sm_m == 0 || m.lives) return none;
    const double left = static_cast<double>(m.sm_ones) / static_cast<double>(1ull << (m.sm_m * m.sbits));
    if (m.kind == 0) {
        if (m.sbits == 8) return left <= 1 / 32.0 ? 4 * MiB : left <= 1 / 6.0 ? 8 * MiB : none;
        return left <= (m.sbits == 2 ? 1 / 8.0 : m.sbits == 7 ? 1 / 16.0 : 1 / 24.0) ? 8 * MiB : none;
    }
    if (m.sbits > 3 || m.walk_states > 2.5) return none;
    const int words = (m.Q + 7) / 8;
    const double walk = m.Q > 32 ? 8.0 * words : 8.5 + 2.4 * words;
    const double gain = walk - (5 + (3 + 8 * m.walk_states) * std::min(1.0, 4 * left));
    return gain < 1.5 ? none : std::max(MiB / 2, static_cast<uint64_t>(20 / gain * MiB));
}

// In a batch the class kernels come with a graph launch (one machine's texts,
// direct and class kernels: 64 states over bytes, 64 of 64 KiB 66, 56, 16 of
// 1 MiB 187, 81; 64-state DNA DFA, 16 of 1 MiB 228, 269, 64 of 1 MiB 912, 858;
// NFA of 32 states, 64 of 64 KiB 121, 139, 16 of 1 MiB 411, 337).
bool walk_takes_batch(const Machine &m, uint64_t n) {
    return m.walks && (m.walk_limit == ~0ull || n < (m.kind == 1 ? 2 : m.sbits == 8 ? 1 : 8) * m.walk_limit);
}

// Whether the machine's scans walk every start (walk.cu), and the tables for
// it. DFAs: tables that L1 can hold, where the shallow survival bitmap would
// pass at least 1 start in 256 (1 MiB, whole calls: 16384 states and 1 start
// in 12 left, 22 us against the tiles' 30; 706 states and 1 in 21, 18 against
// 25; 3000 states and 1 in 174, 29 against 29). NFAs: at most 64 states, tables of at most 64 KB.
void build_walk(Machine &m) {
    m.walks = m.lives = false;
    m.walk_tab.clear();
    m.walk_limit = ~0ull;
    if (m.sv_kind != SIEVE_NONE) return;
    if (m.kind == 0) {
        if (static_cast<size_t>(m.Q) * m.S * 2 > 160 * 1024) return;
        uint64_t ones = 0;
        for (uint32_t w : m.surv) ones += static_cast<uint64_t>(__builtin_popcount(w));
        if (!m.surv.empty() && ones * 256 < (1ull << (m.sm_m * m.sbits))) return;
    } else if (m.Q > 64) {
        return;
    }
    Delta d;
    if (m.Q <= 64) {
        flatten(m, d);
        m.lives = lives_long(m, d);
        if ((m.kind == 1 || m.lives) && bitset_table(m, d)) {
            m.walks = true;
            if (!m.lives) m.walk_states = states_held(m, d);
            m.walk_limit = walk_limit(m);
            return;
        }
        m.lives = false;
        if (m.kind == 1) return;
    }
    // a DFA's table with the dead state as state Q, a row that leads to itself
    const size_t cells = static_cast<size_t>(m.Q) * m.S;
    std::vector<uint16_t> t(cells + m.S + 1, static_cast<uint16_t>(m.Q));
    for (size_t i = 0; i < cells; ++i)
        if (m.dtab[i] != DEAD16) t[i] = m.dtab[i];
    m.walk_tab.assign((cells + m.S + 1) / 2, 0u);
    memcpy(m.walk_tab.data(), t.data(), m.walk_tab.size() * 4);
    m.walks = true;
    m.walk_limit = walk_limit(m);
}

// The survival bitmap of an NFA over 2-bit symbols (bit set: an instance
// started at q0 meets a final state within the m symbols or still holds a
// state after them); false when fewer than half of the m-grams are clear.
// `grams` as for gram_bits.
bool survival_bits_dna(const Machine &m, int mm, std::vector<uint32_t> &bits, uint64_t &grams) {
    Delta d;
    flatten(m, d);
    return gram_bits(d, d.start, mm, (1ull << (2 * mm)) / 2, 0, bits, grams);
}

}  // namespace pfsm
