"""Asynchronous scans captured in a CUDA graph (after one scan on the stream,
which makes the automaton resident): every replay scans the text as it then
is. Machines of all routes, among them one whose warp-wide bitsets do not fit
shared memory."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_1716_gb300 as P  # noqa: E402

MACHINES = {
    "dfa": lambda: W.dfa_random(1),
    "long_lived_dfa": lambda: W.dfa_random(18, Q=6, S=4, dead=-1, finals=[1, 4], p_dead=0.0),
    "long_lived_nfa": lambda: W.live_core_nfa(5, 7),
    "trie": lambda: W.trie_dfa(W.signature_set(5, n_sigs=100, len_lo=4, len_hi=9))[0],
    "motifs": lambda: W.motif_nfa(W.motif_set(3, n_motifs=40))[0],
    "motifs_16k_states": lambda: W.motif_nfa(W.motif_set(9, n_motifs=800))[0],
    "eps": lambda: W.fig1_union(),
}


@pytest.mark.parametrize("name", sorted(MACHINES))
@pytest.mark.parametrize("n", [1500, 200_003])
def test_captured_scans(name, n):
    m = MACHINES[name]()
    if name.startswith("long"):
        n = min(n, 1500)
    texts = [W.text_uniform(n, m.S, 10 + i) for i in range(3)]
    plain = W.eps_free(m) if name == "eps" else m
    want = [oracle.scan(plain, t) for t in texts]
    with P.Pfsm(0) as pf:
        a = pf.load(m)
        text = torch.from_numpy(texts[0]).cuda()
        out = torch.empty((max(len(w) for w in want) + 8, 3), dtype=torch.int32, device="cuda")
        status = torch.zeros(2, dtype=torch.int64, device="cuda")
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        P.pfsm_scan_async(pf.ctx, a, text, n, out, status, stream=s)
        s.synchronize()
        assert status.tolist() == [len(want[0]), 0]
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            P.pfsm_scan_async(pf.ctx, a, text, n, out, status, stream=s)
        for t, w in list(zip(texts, want)) + [(texts[1], want[1])]:
            text.copy_(torch.from_numpy(t))
            out.fill_(-1)
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            assert status.tolist() == [len(w), 0]
            assert np.array_equal(oracle.sort_matches(out[:len(w)].cpu().numpy().view(np.uint32)), w)
        # scans outside the graph, between replays, on the same stream
        P.pfsm_scan_async(pf.ctx, a, text, n, out, status, stream=s)
        s.synchronize()
        assert status.tolist() == [len(want[1]), 0]
        del g
        P.pfsm_evict(pf.ctx, a)
        assert P.pfsm_scan(pf.ctx, a, text, n, out)[0] == P.PFSM_OK
        P.pfsm_unload(pf.ctx, a)
    # nothing of the capture is left for the next context's calls
    with P.Pfsm(0) as pf:
        got = oracle.sort_matches(pf.scan_numpy(pf.load(m), texts[0]))
        assert np.array_equal(got, want[0])


@pytest.mark.parametrize("n_motifs", [256, 450, 700])
def test_captured_scan_with_bitsets_in_global_memory(n_motifs):
    """A text long enough for the tile kernel's full CTAs, which leave no
    shared memory for the bitsets: the scratch that the captured kernel needs
    is there after a scan on the stream, whatever kernel that took. (Compared
    with the scan outside the graph.)"""
    m = W.motif_nfa(W.motif_set(9, n_motifs=n_motifs))[0]
    n = 6_000_011
    text = torch.from_numpy(W.text_dna(n, 5)).cuda()
    with P.Pfsm(0) as pf:
        a = pf.load(m)
        out = torch.empty((2, 1 << 16, 3), dtype=torch.int32, device="cuda")
        status = torch.zeros((2, 2), dtype=torch.int64, device="cuda")
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        P.pfsm_scan_async(pf.ctx, a, text, n, out[0], status[0], stream=s)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            P.pfsm_scan_async(pf.ctx, a, text, n, out[1], status[1], stream=s)
        g.replay()
        torch.cuda.synchronize()
        (k, e), (k1, e1) = status.tolist()
        assert 100 < k <= 1 << 16 and (k1, e, e1) == (k, 0, 0)
        x, y = (oracle.sort_matches(o[:k].cpu().numpy().view(np.uint32)) for o in out)
        assert np.array_equal(x, y)
        del g
