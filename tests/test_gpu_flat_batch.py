"""Batches whose texts run flat (sieve and direct scan, default parameters)
against the oracle: mixed machines, texts around the steps' and grams' edges,
both front kernels, lists that overflow, beside machines that keep to the
class kernels."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_1716_gb300 as P  # noqa: E402


def fleet():
    motifs = [W.motif_set(20 + i, n_motifs=n) for i, n in enumerate((3, 40, 120))]
    sigs = [W.signature_set(30 + i, n_sigs=n) for i, n in enumerate((20, 300))]
    ms = [(W.motif_nfa(m)[0], 4, [W.motif_instance(x, np.random.default_rng(i)) for x in m]) for i, m in enumerate(motifs)]
    ms += [(W.trie_dfa(s)[0], 256, [np.frombuffer(x, np.uint8) for x in s]) for s in sigs]
    ms += [(W.dfa_random(1), 4, None), (W.dfa_random(7, Q=3000), 4, None), (W.eps_free(W.fig1_union()), 3, None),
           (W.live_core_nfa(5, 3), 4, None), (W.dfa_random(9, Q=40, S=20), 20, None)]
    # short signatures: no sieve, the class kernels run them
    short = [b"\x01\x02", b"\x07\x08\x09\x0a", b"\x01\x02\x03"]
    ms.append((W.trie_dfa(short)[0], 256, [np.frombuffer(x, np.uint8) for x in short]))
    return ms


def make_text(m, n, seed):
    aut, S, pats = m
    rng = np.random.default_rng(seed)
    t = W.text_dna(n, seed) if S == 4 else rng.integers(0, S, n).astype(np.uint8)
    if pats:
        for at in range(0, n, 150):
            p = pats[int(rng.integers(len(pats)))]
            t[at:at + len(p)] = p[:n - at]
        p = pats[seed % len(pats)]
        if n >= len(p):
            t[n - len(p):] = p
    return t


def check(pf, auts, jobs, texts, want, machines):
    """One packed buffer, so that texts begin at odd addresses."""
    off = np.concatenate([[0], np.cumsum([len(t) for t in texts])])
    data = pf.to_device(np.concatenate(texts + [np.zeros(64, np.uint8)]))
    table = P.job_table([auts[j] for j in jobs], [data.data_ptr() + int(o) for o in off[:-1]], [len(t) for t in texts])
    total = sum(len(w) for w in want)
    out = torch.empty((total + 8, 4), dtype=torch.int32, device="cuda")
    st, counts, got_total = P.pfsm_scan_batch(pf.ctx, table, out)
    assert st == P.PFSM_OK and got_total == total
    assert counts.tolist() == [len(w) for w in want]
    rows = out[:total].cpu().numpy().view(np.uint32)
    rows = rows[np.lexsort(rows.T[::-1])]
    at = 0
    for i, w in enumerate(want):
        mine = rows[at:at + len(w)]
        assert (mine[:, 0] == i).all() and np.array_equal(mine[:, 1:], w), (i, jobs[i], len(texts[i]))
        at += len(w)


@pytest.fixture(scope="module")
def world():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ms = fleet()
    pf = P.Pfsm(0)
    auts = [pf.load(m[0]) for m in ms]
    lens = [0, 1, 2, 5, 7, 11, 12, 13, 15, 16, 20, 21, 31, 33, 100, 255, 256, 257, 511, 512, 513, 1023, 1025, 2049, 5003]
    jobs, texts, want = [], [], []
    for i, n in enumerate(lens * 4):
        j = (i * 7 + i // len(lens)) % len(ms)
        if ms[j][0] is ms[8][0]:
            n = min(n, 600)   # the live core reports a quadratic number
        t = make_text(ms[j], n, 1000 + i)
        jobs.append(j)
        texts.append(t)
        want.append(oracle.scan(ms[j][0], t))
    yield pf, ms, auts, jobs, texts, want
    pf.close()


def test_small_batch(world):
    pf, ms, auts, jobs, texts, want = world
    check(pf, auts, jobs, texts, want, ms)


def test_without_class_kernels(world):
    pf, ms, auts, jobs, texts, want = world
    keep = [i for i in range(len(jobs)) if jobs[i] != len(ms) - 1]
    check(pf, auts, [jobs[i] for i in keep], [texts[i] for i in keep], [want[i] for i in keep], ms)


def test_large_batch(world):
    """Past the size from which the near bitmaps are copied to shared memory,
    several machines per CTA's share."""
    pf, ms, auts, jobs, texts, want = world
    big = [(0, 3_000_001), (1, 2_000_003), (2, 4_500_007), (3, 4_000_001), (4, 5_000_011), (5, 100_003)]
    jobs, texts, want = list(jobs), list(texts), list(want)
    for k, (j, n) in enumerate(big):
        t = make_text(ms[j], n, 77 + k)
        jobs.insert(5 * k, j)
        texts.insert(5 * k, t)
        want.insert(5 * k, oracle.scan(ms[j][0], t))
    check(pf, auts, jobs, texts, want, ms)


def test_candidate_lists_overflow(world):
    pf, ms, auts, jobs, texts, want = world
    P.pfsm_test_carry_cap(pf.ctx, 16, 0)
    try:
        check(pf, auts, jobs, texts, want, ms)
    finally:
        P.pfsm_test_carry_cap(pf.ctx, 0, 0)


def test_bad_symbol_and_capacity(world):
    pf, ms, auts, jobs, texts, want = world
    data = [pf.to_device(t) for t in texts]
    table = [(auts[j], d, d.numel()) for j, d in zip(jobs, data)]
    total = sum(len(w) for w in want)
    out = torch.empty((100, 4), dtype=torch.int32, device="cuda")
    st, counts, got = P.pfsm_scan_batch(pf.ctx, table, out)
    assert st == P.PFSM_E_OVERFLOW and got == total and counts.tolist() == [len(w) for w in want]
    for kind in (1, 5):   # a motif set's and a DFA's text
        i = next(i for i in range(len(jobs)) if jobs[i] == kind and len(texts[i]) > 300)
        u = texts[i].copy()
        u[299] = 4
        bad = list(table)
        bad[i] = (auts[kind], pf.to_device(u), len(u))
        with pytest.raises(P.PfsmError) as e:
            P.pfsm_scan_batch(pf.ctx, bad, torch.empty((total + 100, 4), dtype=torch.int32, device="cuda"))
        assert e.value.status == P.PFSM_E_INVAL


def test_union_over_one_text(world):
    pf, ms, auts, _, _, _ = world
    t = make_text(ms[1], 200_001, 5)
    picks = [0, 1, 2, 5, 6]
    want = [oracle.scan(ms[j][0], t) for j in picks]
    total = sum(len(w) for w in want)
    out = torch.empty((total + 1, 4), dtype=torch.int32, device="cuda")
    st, counts, got = P.pfsm_scan_union(pf.ctx, [auts[j] for j in picks], pf.to_device(t), None, out)
    assert st == P.PFSM_OK and got == total and counts.tolist() == [len(w) for w in want]
    rows = out[:total].cpu().numpy().view(np.uint32)
    rows = rows[np.lexsort(rows.T[::-1])]
    assert np.array_equal(rows[:, 1:], np.concatenate(want))


def late_start(m, n, seed):
    """A text whose matches all begin in its first symbols (machines of plain
    random tables: random symbols throughout)."""
    aut, S, pats = m
    if not pats:
        return make_text(m, n, seed)
    t = W.text_dna(n, seed) if S == 4 else np.random.default_rng(seed).integers(0, S, n).astype(np.uint8)
    at, step = seed % 5, 512 if S == 4 else 2048
    for i in range(3):
        p = pats[(seed + i) % len(pats)]
        t[at + i * step:at + i * step + len(p)] = p
    return t


def test_empty_texts_between_texts_of_a_large_batch(world):
    """Past the size of the large form, an empty text before every text of
    several steps, for machines of every class: matches in the first steps."""
    pf, ms, auts, _, _, _ = world
    jobs, texts, want = [], [], []
    for i in range(1500):
        j = (0, 3, 2, 5, 1, 4, 9)[i % 7]
        t = late_start(ms[j], 5000 + 37 * (i % 211) + (8192 if ms[j][1] == 256 else 0), 3000 + i)
        for u in (np.zeros(0, np.uint8), t):
            jobs.append(j)
            texts.append(u)
            want.append(oracle.scan(ms[j][0], u))
    assert sum(len(t) for j, t in zip(jobs, texts) if ms[j][2]) > 8 << 20
    check(pf, auts, jobs, texts, want, ms)


@pytest.mark.parametrize("words", [1, 2, 3])
def test_rows_at_any_word(world, words):
    """Output rows that begin 4, 8 and 12 bytes past a 16-byte boundary, for a
    batch and for a union, with nothing written around them."""
    pf, ms, auts, jobs, texts, want = world
    data = [pf.to_device(t) for t in texts]
    u = make_text(ms[1], 50_001, 5)
    ud = pf.to_device(u)
    picks = [0, 1, 2, 5]
    parts = [oracle.scan(ms[j][0], u) for j in picks]
    for rows in (want, parts):
        total = sum(len(w) for w in rows)
        buf = torch.full((4 * total + 8,), -7, dtype=torch.int32, device="cuda")
        assert buf.data_ptr() % 16 == 0
        out = buf[words:words + 4 * total].view(total, 4)
        if rows is want:
            st, counts, got = P.pfsm_scan_batch(pf.ctx, [(auts[j], d, d.numel()) for j, d in zip(jobs, data)], out)
        else:
            st, counts, got = P.pfsm_scan_union(pf.ctx, [auts[j] for j in picks], ud, None, out)
        assert st == P.PFSM_OK and got == total and counts.tolist() == [len(w) for w in rows]
        m = out.cpu().numpy().view(np.uint32)
        m = m[np.lexsort(m.T[::-1])]
        assert np.array_equal(m[:, 0], np.repeat(np.arange(len(rows)), [len(w) for w in rows]))
        assert np.array_equal(m[:, 1:], np.concatenate(rows))
        assert (buf[:words] == -7).all() and (buf[words + 4 * total:] == -7).all()


@pytest.mark.parametrize("n", [300_001, 9_500_003])
def test_candidate_lists_overflow_in_long_texts(world, n):
    """Lists that overflow in texts of many steps, beside texts of few: every
    start is run, step by step, in both forms of the front kernel."""
    pf, ms, auts, jobs, texts, want = world
    jobs, texts, want = list(jobs[:40]), list(texts[:40]), list(want[:40])
    for k, (j, m) in enumerate([(1, n), (4, n - 7), (2, n // 3), (3, 4097), (0, 513)]):
        t = make_text(ms[j], m, 91 + k)
        jobs.insert(7 * k, j)
        texts.insert(7 * k, t)
        want.insert(7 * k, oracle.scan(ms[j][0], t))
    P.pfsm_test_carry_cap(pf.ctx, 1000, 0)
    try:
        check(pf, auts, jobs, texts, want, ms)
    finally:
        P.pfsm_test_carry_cap(pf.ctx, 0, 0)


def test_more_candidates_than_32_bits_count(world):
    """Four texts of 1 GiB and one of 1 MiB whose starts are nearly all
    candidates: more than 2^32 of them, a list's length more than a multiple of
    it."""
    pf = world[0]
    trie, _ = W.trie_dfa([bytes(7) + b"\x01"])
    a = pf.load(trie)
    n, m = 1 << 30, 1 << 20
    text = torch.zeros(n, dtype=torch.uint8, device="cuda")
    ends = np.array([7, 4099, 12_345_678, 500_000_003, n - 1])
    text[torch.from_numpy(ends).cuda()] = 1
    jobs = [(a, text, n)] * 4 + [(a, text[4096:4096 + m], m)]
    want = [[(int(e) - 7, int(e)) for e in ends]] * 4 + [[]]   # (a match begins before the last text)
    total = sum(len(w) for w in want)
    out = torch.empty((total + 8, 4), dtype=torch.int32, device="cuda")
    st, counts, got = P.pfsm_scan_batch(pf.ctx, jobs, out)
    P.pfsm_unload(pf.ctx, a)
    assert st == P.PFSM_OK and got == total and counts.tolist() == [len(w) for w in want]
    rows = sorted(map(tuple, out[:total, :3].tolist()))
    assert rows == [(i, s, e) for i, w in enumerate(want) for s, e in w]
