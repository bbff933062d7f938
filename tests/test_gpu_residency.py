"""Budgets that hold only the core of an automaton's image (the tables of the
tile and class kernels): scans and batches against the oracle, and back to the
whole image when there is room."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_1716_gb300 as P  # noqa: E402


def automata(kind):
    if kind == "motifs":
        sets = [W.motif_set(40 + i, n_motifs=30) for i in range(3)]
        return [W.motif_nfa(s)[0] for s in sets], sets
    if kind == "tries":
        sets = [W.signature_set(50 + i, n_sigs=80) for i in range(3)]
        return [W.trie_dfa(s)[0] for s in sets], sets
    return [W.dfa_random(1, finals=[1 + i, 9 + 2 * i, 30]) for i in range(3)], None


def text(kind, sets, n, seed):
    if kind == "motifs":
        t = W.text_dna(n, seed)
        for s in sets:
            W.plant_motifs(t, s, 700, seed)
    elif kind == "tries":
        t = W.text_uniform(n, 256, seed)
        for i, at in enumerate(range(0, n - 40, 90)):
            s = np.frombuffer(sets[i % 3][(seed + i) % 80], np.uint8)
            t[at:at + len(s)] = s
    else:
        t = W.text_uniform(n, 4, seed)
    return t


@pytest.mark.parametrize("kind", ["motifs", "tries", "dense"])
@pytest.mark.parametrize("share", [0.99, 1.6, 2.2, 3.0])
def test_core_images(kind, share):
    autos, sets = automata(kind)
    with P.Pfsm(0) as pf:
        whole = max(P.pfsm_aut_bytes(pf.ctx, pf.load(x))[0] for x in autos)
    budget = int(share * whole)
    with P.Pfsm(0, budget_bytes=budget) as pf:
        ids = [pf.load(x) for x in autos]
        texts = [text(kind, sets, 30_000 + 7 * i, i) for i in range(3)]
        want = [[oracle.scan(x, t) for t in texts] for x in autos]
        s2 = torch.cuda.Stream()
        for rnd in range(2):
            for i in range(3):
                got = oracle.sort_matches(pf.scan_numpy(ids[i], texts[rnd]))
                assert np.array_equal(got, want[i][rnd]), (rnd, i)
            for pair in ([0, 1], [1, 2], [2, 0], [0, 1, 2]):
                try:
                    out, counts = pf.scan_batch([(ids[j], texts[k]) for k, j in enumerate(pair)])
                except P.PfsmError as e:
                    # refused only where not even the cores fit (of motif
                    # sets a good half of the image)
                    assert e.status == P.PFSM_E_NOMEM and share < len(pair) * (0.6 if kind == "motifs" else 1)
                    continue
                rows = out.cpu().numpy().view(np.uint32)
                rows = rows[np.lexsort(rows.T[::-1])]
                assert counts.tolist() == [len(want[j][k]) for k, j in enumerate(pair)]
                assert np.array_equal(rows[:, 1:], np.concatenate([want[j][k] for k, j in enumerate(pair)]))
                # a scan on another stream while the batch's images change
                st = torch.zeros(2, dtype=torch.int64, device="cuda")
                o = torch.empty((len(want[pair[0]][1]) + 8, 3), dtype=torch.int32, device="cuda")
                d = pf.to_device(texts[1])
                s2.wait_stream(torch.cuda.current_stream())
                P.pfsm_scan_async(pf.ctx, ids[pair[0]], d, None, o, st, stream=s2)
                torch.cuda.synchronize()
                w = want[pair[0]][1]
                assert st.tolist() == [len(w), 0]
                assert np.array_equal(oracle.sort_matches(o[:len(w)].cpu().numpy().view(np.uint32)), w)
            assert P.pfsm_get_stats(pf.ctx)["resident_bytes"] <= budget
