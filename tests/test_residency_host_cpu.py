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
