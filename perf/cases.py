"""What the scan library is used for, as cases that can be timed.

A case names a machine family, an entry point, sizes, and how many texts one
pass scans. ``prepare`` makes what a program holds before the calls (a context
with the machines loaded, the texts on the GPU, output buffers with room for
the matches), ``run`` is one pass through the public entry points, ``work``
counts the bytes that the pass cannot do without. The machines of a case are
the generators' machines for ``machine_seed``; the texts come from the seed of
``prepare``.

A scan returns its matches in no particular order, so ``run`` brings the
matches of its texts into one that does not change, as a program that reads
them does. Many dense matches of a DNA automaton go to a chart (the final state
by start and length, or by start and end). Others are sorted in text order,
each match packed into one 64-bit key (text, start, length, final state:
nothing is lost); unused places of the buffer hold a key of -1 rows. All
outputs are whole numbers.
"""
import functools
import math

import numpy as np
import torch

import paper_1110_1716_gb300 as P
import workloads as W

DEV = "cuda:0"


def listed():
    return [
        # The smallest call: single requests of the serving mix (its median
        # text is 4 KiB), each waited for; launches and host time count.
        dict(name="dfa_4kib_requests", entry="scan", machine="dfa", states=64, machine_seed=1,
             n=4096, shift=0, calls=32, wait=True),
        # A dense scan: 64-state DNA automaton, about one match per symbol.
        dict(name="dfa_1mib", entry="scan", machine="dfa", states=64, machine_seed=1,
             n=1 << 20, shift=0, calls=2, wait=False),
        # The largest automaton of the serving fleet (its table does not fit
        # shared memory), ragged texts in the middle of a larger buffer.
        dict(name="dfa_16k_states_odd", entry="scan", machine="dfa", states=16384, machine_seed=11,
             n=1_000_037, shift=3, calls=2, wait=False),
        # Gene-sized records of a file: odd length and address.
        dict(name="motif_100kb_records", entry="scan", machine="motif", patterns=256, machine_seed=1,
             n=100_003, shift=5, calls=32, wait=False),
        # The headline scan: chromosome-sized texts against 256 motifs.
        dict(name="motif_64mib", entry="scan", machine="motif", patterns=256, machine_seed=0,
             n=64 << 20, shift=0, calls=4, wait=False),
        # Files of a few MB against the byte signatures, odd length and address.
        dict(name="trie_4mb_files", entry="scan", machine="trie", patterns=1000, machine_seed=2,
             n=4_194_301, shift=9, calls=16, wait=False),
        # Disk images or traffic captures against 1000 byte signatures.
        dict(name="trie_1gib", entry="scan", machine="trie", patterns=1000, machine_seed=0,
             n=1 << 30, shift=0, calls=2, wait=False),
        # What the server packs into one batch: some tens of short requests
        # over a fleet of machines of all three kinds.
        dict(name="batch_64_requests", entry="batch", mix="fleet", machines=24, machine_seed=3,
             texts=64, calls=4),
        # Offline scan of a collection: 10,000 texts of 100 B - 1 MiB, 16 machines.
        dict(name="batch_10k_texts", entry="batch", mix="half", machines=16, machine_seed=0,
             texts=10_000, hi=1 << 20, calls=1),
        # Texts against several motif sets that come and go on their own.
        dict(name="union_8_motif_sets", entry="union", machine="motif", patterns=48, machines=8,
             machine_seed=4, n=8_388_593, shift=0, calls=4, wait=True),
        # The quadratic case of the method: every instance lives to the end
        # of the text (a DFA without a dead state).
        dict(name="long_lived_dfa", entry="scan", machine="live_dfa", states=6, machine_seed=8,
             n=6001, shift=0, calls=1, wait=True),
        # The same for an NFA whose state sets never empty.
        dict(name="long_lived_nfa", entry="scan", machine="live_nfa", states=8, machine_seed=7,
             n=6001, shift=0, calls=1, wait=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dfa", "dfa", "motif", "motif", "motif", "trie", "trie", "trie", "batch",
                       "batch", "batch", "union", "live_dfa", "live_nfa"])
    ms = rng.randrange(1, 1000)
    one = dict(entry="scan", machine=kind, machine_seed=ms,
               shift=rng.choice([0, 0, rng.randrange(1, 16)]), wait=rng.random() < 0.4)
    if kind == "dfa":
        n = _log_int(rng, 1000, 2 << 20)
        return dict(one, states=_log_int(rng, 64, 16384), n=n, calls=_calls(rng, 64, 4 << 20, n))
    if kind == "motif":
        n = _log_int(rng, 4000, 64 << 20)
        return dict(one, patterns=_log_int(rng, 32, 256), n=n, calls=_calls(rng, 64, 256 << 20, n))
    if kind == "trie":
        n = _log_int(rng, 4000, 1 << 30)
        return dict(one, patterns=_log_int(rng, 100, 1000), n=n, calls=_calls(rng, 64, 1 << 30, n))
    if kind == "batch":
        texts = _log_int(rng, 16, 10_000)
        if texts < 400:
            return dict(entry="batch", mix="fleet", machines=rng.randrange(4, 33), machine_seed=ms,
                        texts=texts, calls=rng.randrange(1, 5))
        return dict(entry="batch", mix="half", machines=2 * rng.randrange(2, 9), machine_seed=ms,
                    texts=texts, hi=_log_int(rng, 1 << 16, 1 << 20), calls=1)
    if kind == "union":
        n = _log_int(rng, 100_000, 16 << 20)
        return dict(one, entry="union", machine="motif", patterns=_log_int(rng, 16, 96),
                    machines=rng.randrange(2, 13), n=n, calls=_calls(rng, 8, 32 << 20, n), wait=True)
    if kind == "live_dfa":
        return dict(one, states=rng.randrange(5, 13), machine_seed=rng.choice([8, 18]),
                    n=rng.randrange(2000, 6002), shift=0, calls=1, wait=True)
    return dict(one, states=rng.randrange(6, 10), n=rng.randrange(2000, 5000), shift=0, calls=1,
                wait=True)


def _calls(rng, most, symbols, n):
    """Texts of one pass: at most `most`, and at most `symbols` in all."""
    return max(1, min(rng.randrange(1, most + 1), symbols // n))


# ---------------------------------------------------------------- machines and patterns
@functools.lru_cache(maxsize=128)
def _machine(kind, size, seed):
    """(machine, alphabet, patterns as (rows, lengths) or None): patterns are
    texts that the machine matches, for planting."""
    if kind == "dfa":
        # the first machine from this seed on that gets anywhere from q0
        while True:
            d = W.dfa_random(seed, Q=size)
            if _reached(d) > size // 2:
                return d, 4, None
            seed += 1000
    if kind == "live_dfa":
        return W.dfa_random(seed, Q=size, S=4, dead=-1, finals=[1], p_dead=0.0), 4, None
    if kind == "live_nfa":
        return W.live_core_nfa(size - 3, seed), 4, None
    if kind == "motif":
        motifs = W.motif_set(seed, n_motifs=size)
        rng = np.random.default_rng(seed + 1)
        pats = [W.motif_instance(m, rng) for m in motifs for _ in range(4)]
        return W.motif_nfa(motifs)[0], 4, _padded(pats)
    sigs = W.signature_set(seed, n_sigs=size)
    return W.trie_dfa(sigs)[0], 256, _padded([np.frombuffer(s, dtype=np.uint8) for s in sigs])


def _reached(d):
    seen, new = {d.q0}, [d.q0]
    while new:
        new = list({int(t) for q in new for t in d.delta[q]} - seen - {d.dead})
        seen.update(new)
    return len(seen)


def _padded(pats):
    lens = np.array([len(p) for p in pats], dtype=np.int64)
    rows = np.zeros((len(pats), int(lens.max())), dtype=np.uint8)
    for i, p in enumerate(pats):
        rows[i, :len(p)] = p
    return rows, lens


def _symbols(n, alphabet, dna, g):
    """n symbols on the GPU: bytes, uniform DNA, or DNA with 40 % C and G."""
    if alphabet == 256:
        return torch.randint(0, 256, (n,), dtype=torch.uint8, device=DEV, generator=g)
    if not dna:
        return torch.randint(0, 4, (n,), dtype=torch.uint8, device=DEV, generator=g)
    # ten tenths: 3 A, 2 C, 2 G, 3 T
    x = torch.randint(0, 10, (n,), dtype=torch.uint8, device=DEV, generator=g)
    return (x >= 3).to(torch.uint8) + (x >= 5).to(torch.uint8) + (x >= 7).to(torch.uint8)


def _plant(text, pos, pats, which):
    """Writes pattern which[i] at pos[i] (GPU index writes, host-made lists;
    the positions are far enough apart not to overlap)."""
    rows, lens = pats
    col = np.arange(rows.shape[1])
    keep = col[None, :] < lens[which][:, None]
    at = (pos[:, None] + col[None, :])[keep]
    text[torch.from_numpy(at).to(DEV)] = torch.from_numpy(rows[which][keep]).to(DEV)


def _plants(rng, n, every, width):
    """About one position in `every` symbols, at least `width` apart."""
    k = max(1, n // every)
    pos = np.arange(k, dtype=np.int64) * every + rng.integers(0, max(1, every - width), size=k)
    return pos[pos + width <= n]


_EVERY = {"motif": 10_000, "trie": 1 << 16}   # one planted pattern per so many symbols


# ---------------------------------------------------------------- what a program holds
class State:
    pass


LENGTHS = 64   # columns of a DNA automaton's chart: its matches are shorter


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    rng = np.random.default_rng(seed)
    s = State()
    s.entry, s.calls = case["entry"], case["calls"]
    s.pf = P.Pfsm(0)
    if s.entry == "batch":
        return _prepare_batch(s, case, g, rng)
    s.wait = case["wait"]
    kind, n, ms, shift = case["machine"], case["n"], case["machine_seed"], case["shift"]
    count = case.get("machines", 1)
    made = [_machine(kind, case.get("patterns", case.get("states")), ms + i) for i in range(count)]
    s.auts = [s.pf.load(m[0]) for m in made]
    s.n, s.texts = n, []
    # the texts lie one behind the other, `shift` bytes past a 64-byte line
    step = (n + shift + 63) // 64 * 64
    data = _symbols(step * s.calls, made[0][1], kind == "motif", g)
    for c in range(s.calls):
        text = data[c * step + shift:c * step + shift + n]
        s.texts.append(text)
        if kind in _EVERY:
            for m in made:
                pos = _plants(rng, n, _EVERY[kind] * count, m[2][0].shape[1])
                _plant(text, pos, m[2], rng.integers(0, len(m[2][1]), size=len(pos)))
    # room for the matches: some tens of thousands of symbols per match of a
    # pattern set, a few matches per symbol of a DNA automaton, one per so
    # many symbols of the rest of the text for an instance that never dies
    charted = kind.startswith("live") or kind == "dfa" and n * s.calls > 1 << 18
    cap = {"dfa": 8 * n + 4096 if charted else 3 * n, "live_dfa": n * n // 2 + 64, "live_nfa": n * n // 16 + 65_536,
           "motif": n // 3600 + 96, "trie": n // 45_000 + 64}[kind]
    if s.entry == "union":
        cap = n // 2400 + 256
    s.cols = 3 if s.entry == "scan" else 4
    s.out = torch.full((s.calls, cap, s.cols), -1, dtype=torch.int32, device=DEV)
    s.status = torch.zeros((s.calls, 2), dtype=torch.int64, device=DEV)
    s.chart = None
    if charted:
        # final state (0: no match) by start and length, or by start and end
        s.width = LENGTHS if kind == "dfa" else n
        s.alpha = s.width - 1 if kind == "dfa" else s.width
        s.chart = torch.zeros((s.calls, n * s.width), dtype=torch.int32, device=DEV)
    else:
        s.key = _key_weights(s.cols, n.bit_length(), 13)
        # texts of a pass are told apart by a term of their own
        s.text_term = torch.arange(s.calls, dtype=torch.int64, device=DEV)[:, None] << (
            15 + 13 + n.bit_length() + (4 if s.cols == 4 else 0))
    return s


def _prepare_batch(s, case, g, rng):
    count, ms = case["machines"], case["machine_seed"]
    mrng = np.random.default_rng(ms)
    if case["mix"] == "half":
        # motif sets and signature sets of the full size, half and half
        what = [("motif", 256) if i < count // 2 else ("trie", 1000) for i in range(count)]
    else:
        # the serving fleet: three kinds, 64 - 16,384 states, log-uniform
        what = []
        for _ in range(count):
            size = int(W.loguniform_lengths(mrng, 1, 64, 16384)[0])
            k = ("dfa", "motif", "trie")[int(mrng.integers(0, 3))]
            what.append((k, size if k == "dfa" else max(1, size // (19 if k == "motif" else 20))))
    made = [_machine(k, size, 1000 * ms + 100 + i) for i, (k, size) in enumerate(what)]
    s.auts = np.array([s.pf.load(m[0]) for m in made], dtype=np.int32)
    k = case["texts"]
    s.jobs, s.bufs = [], []
    for _ in range(s.calls):
        if case["mix"] == "half":
            lens = W.loguniform_lengths(rng, k, 100, case["hi"])
            job = rng.integers(0, count, size=k)
        else:
            # request sizes: lognormal, median 4 KiB, sigma 1.5; popular machines first
            lens = np.clip(np.exp(rng.normal(math.log(4096), 1.5, size=k)), 64, 262_144).astype(np.int64)
            p = np.arange(1, count + 1, dtype=np.float64) ** -1.1
            job = rng.choice(count, size=k, p=p / p.sum())
        ptrs = np.zeros(k, dtype=np.uint64)
        for alphabet in (4, 256):
            mine = np.nonzero(np.array([made[j][1] == alphabet for j in job]))[0]
            if not len(mine):
                continue
            off = np.concatenate([[0], np.cumsum(lens[mine])])
            buf = _symbols(int(off[-1]), alphabet, True, g)
            kind = "motif" if alphabet == 4 else "trie"
            for x, m in enumerate(made):
                if m[1] != alphabet or m[2] is None:
                    continue
                width = m[2][0].shape[1]
                own = np.nonzero(job[mine] == x)[0]
                at = [off[t] + _plants(rng, int(lens[mine[t]]), _EVERY[kind], width) for t in own]
                at = np.concatenate(at) if at else np.zeros(0, dtype=np.int64)
                if len(at):
                    _plant(buf, at, m[2], rng.integers(0, len(m[2][1]), size=len(at)))
            ptrs[mine] = buf.data_ptr() + off[:-1].astype(np.uint64)
            s.bufs.append(buf)
        s.jobs.append(P.job_table(s.auts[job], ptrs, lens))
    s.cols = 4
    cap = int(k * _mean_length(case)) // 4000 + 16_384 if case["mix"] == "half" else k * 32_768
    s.out = torch.empty((cap, 4), dtype=torch.int32, device=DEV)
    s.keys = torch.full((s.calls, cap), -1, dtype=torch.int64, device=DEV)
    s.key = _key_weights(4, 21, 13)
    return s


def _mean_length(case):
    if case["mix"] == "half":
        return (case["hi"] - 100) / math.log(case["hi"] / 100)
    return 4096 * math.exp(1.5 ** 2 / 2) * 0.95


def _key_weights(cols, start_bits, len_bits):
    """Weights w with row . w = [text,] start, end - start, state packed into
    one non-negative integer (15 bits of state)."""
    w_start = 1 << (15 + len_bits)
    w = [w_start - (1 << 15), 1 << 15, 1]
    if cols == 4:
        w = [w_start << start_bits] + w
    return torch.tensor(w, dtype=torch.int64, device=DEV)


# ---------------------------------------------------------------- one pass
def run(s):
    if s.entry == "batch":
        return _run_batch(s)
    totals = []
    for c in range(s.calls):
        if s.entry == "union":
            st, _, total = P.pfsm_scan_union(s.pf.ctx, s.auts, s.texts[c], s.n, s.out[c])
        elif s.wait:
            st, total = P.pfsm_scan(s.pf.ctx, s.auts[0], s.texts[c], s.n, s.out[c])
        else:
            st, total = P.PFSM_OK, 0
            P.pfsm_scan_async(s.pf.ctx, s.auts[0], s.texts[c], s.n, s.out[c], s.status[c])
        if st != P.PFSM_OK:
            raise RuntimeError(P.strerror(st))
        totals.append(total)
    if s.chart is None:
        # every row of the buffers at once: the unused ones hold -1
        matches = torch.sort(((s.out * s.key).sum(2) + s.text_term).view(-1))[0]
        return {"counts": totals, "status": s.status, "matches": matches}
    if not s.wait:
        totals = s.status[:, 0].tolist()
    for c in range(s.calls):
        rows = s.out[c, :totals[c]]
        at = torch.add(rows[:, 1], rows[:, 0], alpha=s.alpha)
        s.chart[c].index_put_((at,), rows[:, 2])
    return {"counts": totals, "chart": s.chart}


def _run_batch(s):
    counts = []
    for c in range(s.calls):
        st, per_text, total = P.pfsm_scan_batch(s.pf.ctx, s.jobs[c], s.out)
        if st != P.PFSM_OK:
            raise RuntimeError(P.strerror(st))
        counts.append(per_text.astype(np.int64))
        s.keys[c, :total] = torch.sort((s.out[:total] * s.key).sum(1))[0]
    return {"counts": counts, "matches": s.keys}


def work(case):
    """Every text symbol read once, every match row (12 or 16 bytes) written
    once. The number of matches is the generators' average."""
    calls = case["calls"]
    if case["entry"] == "batch":
        n = case["texts"] * _mean_length(case)
        rows = n / 8000 if case["mix"] == "half" else 0.1 * n
        return {"bytes": calls * (n + 16 * rows), "flops": 0}
    n, kind = case["n"], case["machine"]
    if case["entry"] == "union":
        return {"bytes": calls * (n + 16 * n / 4000), "flops": 0}
    rows = {"dfa": 0.3 * n if case.get("states") != 64 else 1.0 * n, "motif": n / 5000, "trie": n / 57_000,
            "live_dfa": n * n / 9.5, "live_nfa": n * n / 122}[kind]
    return {"bytes": calls * (n + 12 * rows), "flops": 0}


def exact(case, seed):
    """Every output is a whole number, so there is nothing to round."""
    return None
