"""Byte tries whose matches lie in the last few bytes of a text: starts whose
8-byte filter window is not wholly clear of the end."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1110_1716_gb300 as P  # noqa: E402


@pytest.mark.parametrize("spt", [8, 32])
@pytest.mark.parametrize("n", [5, 8, 13, 24, 4099, 20_013])
def test_trie_matches_that_end_with_the_text(n, spt):
    trie, _ = W.trie_dfa([b"\x01\x02\x03\x04\x05", b"\x03\x04\x05", b"\x09\x08\x07\x06"])
    t = np.full(n, 0x20, dtype=np.uint8)
    t[n - 5:] = [1, 2, 3, 4, 5]
    t[:5] = [1, 2, 3, 4, 5]
    want = oracle.scan(trie, t)
    assert len(want) >= 2
    with P.Pfsm(0) as pf:
        a = pf.load(trie)
        P.pfsm_set_params(pf.ctx, a, {"spt": spt})
        assert np.array_equal(oracle.sort_matches(pf.scan_numpy(a, t)), want)
