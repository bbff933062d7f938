"""Long-lived instances (segments, chunks of eight segments, sets of up to four
states at a time or single states) against the oracle: text lengths around the
segments' and chunks' edges, one and two words per set, and scratch that holds
the rows of four states, only those of single states, or neither."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_1716_gb300 as P  # noqa: E402

MACHINES = {
    "dfa6": lambda: W.dfa_random(18, Q=6, S=4, dead=-1, finals=[1, 4], p_dead=0.0),
    "dfa33": lambda: W.dfa_random(19, Q=33, S=3, dead=-1, finals=[1, 2, 3], p_dead=0.0),
    "nfa8": lambda: W.live_core_nfa(5, 7),
    "nfa43": lambda: W.live_core_nfa(40, 9, p=0.05),
}


def scratch(n, Q, per):
    """Words of scratch with rows for every set of `per` neighbouring states."""
    words, segs = (1 if Q <= 32 else 2), -(-n // 64)
    rows = -(-Q // per) * (2 ** per - 1)
    return words * (n + 65 * segs * rows) + 2 * segs * rows


@pytest.fixture(scope="module")
def pf():
    f = P.Pfsm(0)
    yield f
    f.close()


@pytest.mark.parametrize("name", sorted(MACHINES))
@pytest.mark.parametrize("n", [512, 513, 576, 577, 1023, 1024, 1025, 1087, 1089, 2500])
def test_long_lived(pf, name, n):
    m = MACHINES[name]()
    a = pf.load(m)
    t = W.text_uniform(n, m.S, n)
    want = oracle.scan(m, t)
    data = pf.to_device(np.concatenate([np.zeros(n % 16, np.uint8), t, np.zeros(64, np.uint8)]))
    out = torch.empty((len(want) + 8, 3), dtype=torch.int32, device="cuda")
    for entries in (0, -(-scratch(n, m.Q, 1) // 2), 1):
        P.pfsm_test_carry_cap(pf.ctx, entries, 0)
        try:
            st, total = P.pfsm_scan(pf.ctx, a, data[n % 16:], n, out)
        finally:
            P.pfsm_test_carry_cap(pf.ctx, 0, 0)
        rows = out[:total].cpu().numpy().view(np.uint32)
        assert st == P.PFSM_OK and np.array_equal(oracle.sort_matches(rows), want), entries
    P.pfsm_unload(pf.ctx, a)
