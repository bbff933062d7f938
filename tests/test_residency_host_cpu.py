"""Loading, residency and the choice of kernels without a GPU
(host_library.cpp: the library's host files over stand-ins for the CUDA
runtime)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
OK, E_NOMEM = 0, 2
P = ctypes.c_void_p


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "libhost_library.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-pthread",
                    "-I" + os.path.join(cuda, "include"), "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_1110_1716_gb300", "csrc"),
                    os.path.join(HERE, "host_library.cpp"), "-o", so, "-ldl"], check=True)
    lib = ctypes.CDLL(so)
    lib.hl_launched.restype = ctypes.c_char_p
    return lib


MACHINES = {
    "trie": (lambda: W.trie_dfa(W.signature_set(5, n_sigs=50))[0], "sieve"),
    "motifs": (lambda: W.motif_nfa(W.motif_set(3, n_motifs=12))[0], "sieve"),
    "dense_dfa": (lambda: W.dfa_random(1), "walk"),
    "live_dfa": (lambda: W.dfa_random(18, Q=6, S=4, dead=-1, finals=[1], p_dead=0.0), "long"),
    "live_nfa": (lambda: W.live_core_nfa(5, 7), "long"),
}


class Host:
    def __init__(self, lib, budget=0):
        self.lib = lib
        self.ctx = P()
        assert lib.pfsm_ctx_create(0, ctypes.c_uint64(budget), ctypes.byref(self.ctx)) == OK

    def load(self, m):
        a = ctypes.c_int32()
        f = np.ascontiguousarray(m.final, dtype=np.uint8)
        if hasattr(m, "delta"):
            d = np.ascontiguousarray(m.delta, dtype=np.int16)
            st = self.lib.pfsm_load_dfa(self.ctx, P(d.ctypes.data), m.Q, m.S, m.q0, m.dead, P(f.ctypes.data), ctypes.byref(a))
        else:
            d = np.ascontiguousarray(m.bits, dtype=np.uint32)
            st = self.lib.pfsm_load_nfa(self.ctx, P(d.ctypes.data), m.Q, m.S, m.q0, P(f.ctypes.data), ctypes.byref(a))
        return st, a.value

    def launched(self):
        return self.lib.hl_launched().decode().split()

    def scan(self, a, n=2000):
        text = np.zeros(n, dtype=np.uint8)
        k = ctypes.c_uint64()
        st = self.lib.pfsm_scan(self.ctx, a, P(text.ctypes.data), ctypes.c_uint64(n), P(), ctypes.c_uint64(0), ctypes.byref(k), P())
        return st, self.launched()

    def __enter__(self):
        return self

    def __exit__(self, *e):
        self.lib.pfsm_ctx_destroy(self.ctx)


@pytest.mark.parametrize("name", sorted(MACHINES))
def test_no_room_for_the_scratch_of_the_newer_kernels(lib, name):
    """A scan that finds no room for the sieve's candidates (also the scratch
    of long-lived instances) takes the kernel that needs none; the next one
    tries again."""
    make, route = MACHINES[name]
    with Host(lib) as h:
        st, a = h.load(make())
        assert st == OK
        lib.hl_largest(24 << 20)
        try:
            assert h.scan(a) == (OK, [route if route == "walk" else "tiles"])
        finally:
            lib.hl_largest(0)
        assert h.scan(a) == (OK, [route])


def stats(h):
    v = np.zeros(6, dtype=np.uint64)   # resident_bytes, budget_bytes, loads, evictions, reloads, (counts)
    h.lib.pfsm_get_stats(h.ctx, P(v.ctypes.data))
    return int(v[0])


def aut_bytes(h, a):
    n = ctypes.c_uint64()
    assert h.lib.pfsm_aut_bytes(h.ctx, a, ctypes.byref(n), None) == OK
    return n.value


def batch(h, auts, n=3000):
    text = np.zeros(n, dtype=np.uint8)
    jobs = np.zeros(len(auts), dtype=[("aut", "<i4"), ("reserved", "<u4"), ("text", "<u8"), ("n", "<u8")])
    jobs["aut"], jobs["text"], jobs["n"] = auts, text.ctypes.data, n
    total = ctypes.c_uint64()
    st = h.lib.pfsm_scan_batch(h.ctx, P(jobs.ctypes.data), len(auts), P(), ctypes.c_uint64(0), P(), ctypes.byref(total), P())
    return st, h.launched()


# bytes of the tables that the tile kernel reads (what an automaton held before
# there were tables of the sieve and of direct scans)
def core(lib, make):
    with Host(lib) as h:
        st, a = h.load(make())
        whole = aut_bytes(h, a)
        lo, hi = 0, whole
    while hi - lo > 256:      # the smallest budget that loads it
        mid = (lo + hi) // 2 // 256 * 256
        with Host(lib, mid) as h:
            st, a = h.load(make())
            lo, hi = (lo, mid) if st == OK else (mid, hi)
    return hi, whole


@pytest.mark.parametrize("name", ["trie", "motifs", "dense_dfa"])
def test_budgets_that_hold_the_core_alone(lib, name):
    make, route = MACHINES[name]
    small, whole = core(lib, make)
    assert small < whole
    if name == "motifs":      # 8 MB of deep bitmap and the third level in the rest
        assert small < 0.6 * whole
    with Host(lib, whole - 256) as h:
        st, a = h.load(make())
        assert st == OK and h.scan(a) == (OK, ["tiles"]) and batch(h, [a, a]) == (OK, ["classes"])
        assert stats(h) == small <= whole - 256
    with Host(lib, whole) as h:
        st, a = h.load(make())
        assert st == OK and h.scan(a) == (OK, [route]) and batch(h, [a]) == (OK, ["flat"])
    # two automata: both cores, and one whole image beside a core
    for budget, want in ((2 * small, ["classes"]), (small + whole, ["classes", "flat"]), (2 * whole, ["flat"])):
        with Host(lib, budget) as h:
            a, b = h.load(make())[1], h.load(make())[1]
            for _ in range(3):
                assert batch(h, [a, b]) == (OK, want), budget
                assert stats(h) <= budget
            # each alone: the other makes room for the whole image, or leaves the core in place
            for x in (a, b, a):
                st, got = h.scan(x)
                assert st == OK and got in ([route], ["tiles"])
                assert stats(h) <= budget
    # one whole image is never the last: with room again, a core is completed
    with Host(lib, 2 * small) as h:
        a, b = h.load(make())[1], h.load(make())[1]
        assert batch(h, [a, b]) == (OK, ["classes"])
        h.lib.pfsm_unload(h.ctx, b)
        if 2 * small >= whole:
            assert h.scan(a) == (OK, [route]) and stats(h) == whole
    with Host(lib, small - 256) as h:
        assert h.load(make())[0] == E_NOMEM


def test_a_batch_that_does_not_fit_is_still_refused(lib):
    make, _ = MACHINES["motifs"]
    small, whole = core(lib, make)
    with Host(lib, 2 * small - 256) as h:
        a, b = h.load(make())[1], h.load(make())[1]
        assert batch(h, [a, b])[0] == E_NOMEM
        assert h.scan(a)[0] == OK and h.scan(b)[0] == OK and batch(h, [a])[0] == OK


def random_nfa(Q, S, seed, p):
    rng = np.random.default_rng(seed)
    edges = [(q, x, t) for q in range(Q) for x in range(S) for t in range(Q) if rng.random() < p / Q]
    return W.nfa_from_edges(Q, S, 0, edges, [q for q in range(Q) if rng.random() < 0.2] or [Q - 1])


MIB = 1 << 20


@pytest.mark.parametrize("make,below,above", [
    (lambda: W.dfa_random(11), 8 * MIB - 1, 8 * MIB),                        # 0.07 of the starts left by the bitmap
    (lambda: W.dfa_random(1), 99 * MIB, None),                               # 0.75
    (lambda: W.dfa_random(12, Q=64, S=256, p_dead=0.9), 4 * MIB - 1, 4 * MIB),   # 0.02
    (lambda: W.dfa_random(12, Q=64, S=256, p_dead=0.3), 99 * MIB, None),
    (lambda: random_nfa(64, 4, 3, 0.5), MIB // 2 - 1, MIB // 2),             # 0.8 states held
    (lambda: random_nfa(64, 4, 64, 0.9), 99 * MIB, None),                    # 6.6
    (lambda: random_nfa(32, 4, 32, 0.9), 99 * MIB, None),                    # no bitmap
    (lambda: random_nfa(8, 4, 8, 0.3), 99 * MIB, None),
    (lambda: random_nfa(32, 4, 32, 0.3), 4 * MIB, 9 * MIB),
    (lambda: random_nfa(40, 2, 47, 0.6), MIB // 2 - 1, MIB),                 # hardly any start left
])
def test_texts_too_long_for_the_direct_scan(lib, make, below, above):
    with Host(lib) as h:
        st, a = h.load(make())
        assert h.scan(a, below) == (OK, ["walk"])
        if above:
            assert h.scan(a, above) == (OK, ["tiles"])


def test_long_lived_instances_keep_to_their_segments(lib):
    with Host(lib) as h:
        st, a = h.load(W.live_core_nfa(5, 7))
        assert h.scan(a, 99 * MIB) == (OK, ["long"])
