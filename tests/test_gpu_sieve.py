"""The sieve (scans with default parameters) against the oracle, at the sizes
and addresses where its blocks, its grams and its candidate list end."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_1716_gb300 as P  # noqa: E402


@pytest.fixture(scope="module")
def pf():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = P.Pfsm(0)
    yield p
    p.close()


def motif(seed=3, n_motifs=40):
    motifs = W.motif_set(seed, n_motifs=n_motifs)
    return W.motif_nfa(motifs)[0], motifs


def motif_text(motifs, n, every, seed):
    t = W.text_dna(n, seed)
    if n > 64:
        W.plant_motifs(t, motifs, every, seed + 1)
        inst = W.motif_instance(motifs[seed % len(motifs)], np.random.default_rng(seed))
        t[n - len(inst):] = inst   # a match that ends with the text
        t[:len(inst)] = inst       # and one that begins with it
    return t


def trie_text(sigs, n, every, seed):
    t = W.text_uniform(n, 256, seed)
    for i, at in enumerate(range(0, n, every)):
        s = np.frombuffer(sigs[(seed + i) % len(sigs)], dtype=np.uint8)
        t[at:at + len(s)] = s[:max(0, n - at)]
    s = np.frombuffer(sigs[seed % len(sigs)], dtype=np.uint8)
    if n >= len(s):
        t[n - len(s):] = s
    return t


def scan_at(pf, a, t, shift, cap=200_000):
    big = pf.to_device(np.concatenate([np.full(shift, 255, np.uint8), t, np.full(40, 255, np.uint8)]))
    out = torch.empty((cap, 3), dtype=torch.int32, device="cuda")
    st, cnt = P.pfsm_scan(pf.ctx, a, big[shift:shift + len(t)], None, out)
    assert st == P.PFSM_OK
    return oracle.sort_matches(out[:cnt].cpu().numpy().view(np.uint32))


SIZES = [1, 3, 4, 5, 13, 15, 16, 17, 31, 32, 495, 496, 497, 511, 512, 513, 527, 992, 4096, 20_011]


@pytest.mark.parametrize("shift", [0, 1, 2, 3, 7, 12, 15])
def test_sieve_edges(pf, shift):
    nfa, motifs = motif()
    sigs = W.signature_set(5, n_sigs=60, len_lo=4, len_hi=12)
    trie, _ = W.trie_dfa(sigs)
    an, at = pf.load(nfa), pf.load(trie)
    for n in SIZES:
        t = motif_text(motifs, n, 90, 100 * shift + n)
        assert np.array_equal(scan_at(pf, an, t, shift), oracle.scan(nfa, t)), ("motif", n)
        t = trie_text(sigs, n, 61, 100 * shift + n)
        assert np.array_equal(scan_at(pf, at, t, shift), oracle.scan(trie, t)), ("trie", n)


@pytest.mark.parametrize("n", [(8 << 20) - 1, (8 << 20) + 1234])
def test_sieve_long_texts(pf, n):
    """Both sides of the length from which the near bitmap is in shared memory."""
    nfa, motifs = motif(4, 200)
    t = motif_text(motifs, n, 5000, 9)
    assert np.array_equal(scan_at(pf, pf.load(nfa), t, 5), oracle.scan(nfa, t))
    sigs = W.signature_set(6, n_sigs=1000)
    trie, _ = W.trie_dfa(sigs)
    t = trie_text(sigs, n, 9001, 10)
    assert np.array_equal(scan_at(pf, pf.load(trie), t, 6), oracle.scan(trie, t))


def test_sieve_candidate_list_overflows(pf):
    """More candidates than the list holds: every start is run instead."""
    nfa, motifs = motif(7, 64)
    t = motif_text(motifs, 60_001, 60, 1)
    sigs = W.signature_set(8, n_sigs=100, len_lo=4, len_hi=9)
    trie, _ = W.trie_dfa(sigs)
    u = trie_text(sigs, 50_003, 40, 2)
    an, at = pf.load(nfa), pf.load(trie)
    P.pfsm_test_carry_cap(pf.ctx, 64, 0)
    try:
        assert np.array_equal(scan_at(pf, an, t, 3), oracle.scan(nfa, t))
        assert np.array_equal(scan_at(pf, at, u, 3), oracle.scan(trie, u))
    finally:
        P.pfsm_test_carry_cap(pf.ctx, 0, 0)


@pytest.mark.parametrize("S", [3, 20, 130, 200])
def test_sieve_other_alphabets(pf, S):
    """Alphabets of other widths; a symbol out of range inside the text is
    refused, the bytes around the text are not looked at."""
    sigs = [bytes(x % S for x in s) for s in W.signature_set(9 + S, n_sigs=50, len_lo=6, len_hi=14)]
    trie, _ = W.trie_dfa(sigs, S=S)
    a = pf.load(trie)
    t = np.random.default_rng(S).integers(0, S, 30_011).astype(np.uint8)
    for i in range(0, len(t) - 20, 300):
        s = np.frombuffer(sigs[i % len(sigs)], dtype=np.uint8)
        t[i:i + len(s)] = s
    assert np.array_equal(scan_at(pf, a, t, 5), oracle.scan(trie, t))
    for bad in (0, 17, 30_010):
        u = t.copy()
        u[bad] = S
        with pytest.raises(P.PfsmError) as e:
            scan_at(pf, a, u, 5)
        assert e.value.status == P.PFSM_E_INVAL


def test_sieve_needs_finals_past_its_step(pf):
    """Matches shorter than the sieve's step: the machine has no sieve."""
    for sigs in ([b"\x01\x02", b"\x05\x06\x07\x08\x09"], [b"\x07\x08\x09", b"\x01\x02\x03\x04\x05\x06"]):
        trie, _ = W.trie_dfa(sigs)
        t = np.random.default_rng(1).integers(0, 10, 20_001).astype(np.uint8)
        assert np.array_equal(scan_at(pf, pf.load(trie), t, 2), oracle.scan(trie, t))


@pytest.mark.parametrize("n", [(3 << 20) - 1, (3 << 20) + 77])
def test_dna_sieve_on_both_sides_of_3_mib(pf, n):
    """2-bit symbols have the near bitmap in shared memory from 3 MiB on."""
    nfa, motifs = motif(11, 90)
    t = motif_text(motifs, n, 4000, 12)
    assert np.array_equal(scan_at(pf, pf.load(nfa), t, 9), oracle.scan(nfa, t))
    trie, _ = W.trie_dfa([bytes(x & 3 for x in s) for s in W.signature_set(13, n_sigs=60, len_lo=12, len_hi=20)], S=4)
    assert np.array_equal(scan_at(pf, pf.load(trie), t, 2), oracle.scan(trie, t))
