"""The direct scan and the tile kernel on both sides of the text length where
the one gives way to the other, alone and in batches, against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W
from conftest import oracle_parallel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_1716_gb300 as P  # noqa: E402

MIB = 1 << 20


def random_nfa(Q, S, seed, p):
    rng = np.random.default_rng(seed)
    edges = [(q, x, t) for q in range(Q) for x in range(S) for t in range(Q) if rng.random() < p / Q]
    return W.nfa_from_edges(Q, S, 0, edges, [q for q in range(Q) if rng.random() < 0.2] or [Q - 1])


@pytest.mark.parametrize("make,limit", [
    (lambda: W.dfa_random(12, Q=64, S=256, p_dead=0.9), 4 * MIB),
    (lambda: W.dfa_random(11), 8 * MIB),
    (lambda: random_nfa(64, 4, 3, 0.5), MIB // 2),
])
def test_both_sides_of_the_limit(make, limit):
    m = make()
    t = W.text_uniform(limit + 5, m.S, 3)
    want = oracle_parallel(m, t[:limit])
    with P.Pfsm(0) as pf:
        a = pf.load(m)
        data = pf.to_device(np.concatenate([np.full(3, 255, np.uint8), t]))
        out = torch.empty((len(want) + 64, 3), dtype=torch.int32, device="cuda")
        for n in (limit - 1, limit):
            st, k = P.pfsm_scan(pf.ctx, a, data[3:], n, out)
            assert st == P.PFSM_OK
            got = oracle.sort_matches(out[:k].cpu().numpy().view(np.uint32))
            assert np.array_equal(got, want[want[:, 1] < n]), n


def test_batches_of_direct_scans_and_class_kernels():
    """One machine's texts past the limit together, another's below it."""
    ms = [W.dfa_random(12, Q=64, S=256, p_dead=0.9), random_nfa(40, 4, 9, 0.5), W.dfa_random(1), random_nfa(8, 4, 8, 0.3)]
    lens = [700_001, 90_000, 0, 30_011, 1_500_000, 300_007, 17, 70_000, 2_100_003, 600_001, 5_003, 64]
    jobs = [(i % 4) for i in range(len(lens))]
    texts = [W.text_uniform(n, ms[j].S, 60 + i) if n else np.zeros(0, np.uint8) for i, (j, n) in enumerate(zip(jobs, lens))]
    want = [oracle_parallel(ms[j], t) if len(t) else np.zeros((0, 3), np.uint32) for j, t in zip(jobs, texts)]
    with P.Pfsm(0) as pf:
        ids = [pf.load(m) for m in ms]
        out, counts = pf.scan_batch([(ids[j], t) for j, t in zip(jobs, texts)])
        assert counts.tolist() == [len(w) for w in want]
        rows = out.cpu().numpy().view(np.uint32)
        rows = rows[np.lexsort(rows.T[::-1])]
        assert np.array_equal(rows[:, 1:], np.concatenate(want))
