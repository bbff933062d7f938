"""The direct scan (dense DFAs and NFAs of at most 64 states, default
parameters) against the oracle: text lengths around a lane's window, a warp's
range and several ranges, unaligned texts, set sizes around the bitset words."""
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


def scan_at(pf, a, t, shift, cap):
    big = pf.to_device(np.concatenate([np.full(shift, 255, np.uint8), t, np.full(40, 255, np.uint8)]))
    out = torch.empty((max(1, cap), 3), dtype=torch.int32, device="cuda")
    st, cnt = P.pfsm_scan(pf.ctx, a, big[shift:shift + len(t)], None, out, cap)
    return st, cnt, oracle.sort_matches(out[:min(cnt, cap)].cpu().numpy().view(np.uint32))


def same(pf, a, m, t, shift=0):
    want = oracle.scan(m, t)
    st, cnt, got = scan_at(pf, a, t, shift, len(want))
    assert st == P.PFSM_OK and cnt == len(want)
    assert np.array_equal(got, want)


SIZES = [1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 1023, 1024, 1025, 20_011]


@pytest.mark.parametrize("shift", [0, 1, 5, 8, 15])
def test_dfa_sizes(pf, shift):
    d = W.dfa_random(5, Q=40, S=4, p_dead=0.3)
    a = pf.load(d)
    for n in SIZES:
        same(pf, a, d, W.text_uniform(n, 4, 50 + n), shift)


@pytest.mark.parametrize("S,Q", [(1, 3), (2, 9), (3, 300), (5, 100), (17, 600), (200, 30), (256, 60), (4, 5000), (4, 16384)])
def test_dfa_tables(pf, S, Q):
    """Tables in shared memory and in global memory, other alphabets."""
    d = W.dfa_random(100 + S + Q, Q=Q, S=S, p_dead=0.35)
    same(pf, pf.load(d), d, W.text_uniform(12_345, S, S), 3)


@pytest.mark.parametrize("n", [155_648, 155_649, 400_003])
def test_dfa_ranges_of_several_starts_per_lane(pf, n):
    d = W.dfa_random(1)
    same(pf, pf.load(d), d, W.text_uniform(n, 4, n), 2)


def random_nfa(Q, S, seed, p):
    rng = np.random.default_rng(seed)
    edges = [(q, x, t) for q in range(Q) for x in range(S) for t in range(Q) if rng.random() < p / Q]
    fins = [q for q in range(Q) if rng.random() < 0.2] or [Q - 1]
    return W.nfa_from_edges(Q, S, 0, edges, fins)


@pytest.mark.parametrize("Q,S", [(2, 2), (7, 4), (8, 4), (9, 4), (31, 3), (32, 4), (33, 4), (40, 5), (63, 4), (64, 4), (16, 16)])
def test_nfa_sets(pf, Q, S):
    m = random_nfa(Q, S, Q * 31 + S, 0.9)
    a = pf.load(m)
    for n in (1, 9, 33, 3001):
        same(pf, a, m, W.text_uniform(n, S, n + Q), 1)


def test_nfa_with_epsilon_edges(pf):
    m = W.fig1_union()
    a = pf.load(m)
    t = W.text_uniform(5000, 3, 4)
    want = oracle.scan(W.eps_free(m), t)
    st, cnt, got = scan_at(pf, a, t, 7, len(want))
    assert st == P.PFSM_OK and np.array_equal(got, want)


@pytest.mark.parametrize("n", [511, 512, 513, 575, 576, 577, 1999])
def test_long_lived_instances(pf, n):
    """Instances that never die, segment by segment: DFAs without a dead state
    and NFAs with a live core, one and two words per set."""
    for m in (W.dfa_random(18, Q=6, S=4, dead=-1, finals=[1, 4], p_dead=0.0),
              W.dfa_random(19, Q=33, S=3, dead=-1, finals=[1, 2, 3], p_dead=0.0),
              W.live_core_nfa(5, 7), W.live_core_nfa(24, 8), W.live_core_nfa(40, 9, p=0.05)):
        same(pf, pf.load(m), m, W.text_uniform(n, m.S, n), n % 16)


def test_capacity_and_symbols(pf):
    d = W.dfa_random(1)
    a = pf.load(d)
    t = W.text_uniform(30_000, 4, 9)
    want = oracle.scan(d, t)
    st, cnt, got = scan_at(pf, a, t, 0, 1000)
    assert st == P.PFSM_E_OVERFLOW and cnt == len(want)
    assert len(np.unique(got, axis=0)) == 1000 and set(map(tuple, got)) <= set(map(tuple, want))
    assert scan_at(pf, a, t, 0, 0)[1] == len(want)
    for at in (0, 12_345, 29_999):
        u = t.copy()
        u[at] = 4
        with pytest.raises(P.PfsmError) as e:
            scan_at(pf, a, u, 0, 60_000)
        assert e.value.status == P.PFSM_E_INVAL
    same(pf, a, d, t, 0)   # the counters are clear again
