"""The host side of batches without a GPU (host_batch.cpp: csrc/batch.cu over
stand-ins for the CUDA runtime, where launching the flat kernels replays how
their warps take the steps of the texts)."""
import ctypes
import os
import subprocess
import traceback

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
DNA, BYTES, WALK = 0, 1, 2
E_NOMEM = 2
FIELDS = ("flat", "graph", "big", "groups", "steps", "missed", "bounds", "null_lists", "used")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "libhost_batch.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    # (an array index out of bounds traps)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic",
                    "-fsanitize=bounds", "-fsanitize-undefined-trap-on-error",
                    "-I" + os.path.join(cuda, "include"), "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_1110_1716_gb300", "csrc"),
                    os.path.join(HERE, "host_batch.cpp"), "-o", so, "-ldl"], check=True)
    lib = ctypes.CDLL(so)
    lib.hb_ctx.restype = ctypes.c_void_p
    lib.hb_free.argtypes = [ctypes.c_void_p]
    return lib


class Host:
    """A context over machines of the given flat classes."""

    def __init__(self, lib, classes):
        self.lib = lib
        c = np.array(classes, dtype=np.int32)
        self.ctx = ctypes.c_void_p(lib.hb_ctx(c.ctypes.data_as(ctypes.c_void_p), len(c)))

    def scan(self, auts, lens, addrs=None):
        a = np.array(auts, dtype=np.int32) + 1
        n = np.array(lens, dtype=np.uint64)
        t = np.array(addrs if addrs is not None else np.full(len(n), 1 << 20), dtype=np.uint64)
        out = np.zeros(len(FIELDS), dtype=np.int64)
        p = [x.ctypes.data_as(ctypes.c_void_p) for x in (a, t, n, out)]
        st = self.lib.hb_scan(self.ctx, p[0], p[1], p[2], len(n), p[3])
        return st, dict(zip(FIELDS, out.tolist()))

    def __enter__(self):
        return self

    def __exit__(self, *e):
        self.lib.hb_free(self.ctx)


@pytest.mark.parametrize("big", [False, True])
@pytest.mark.parametrize("chunk", [1, 2, 5, 16, 1 << 20])
def test_every_step_is_taken_once(lib, big, chunk):
    """Texts of no, few and many steps in any order, whatever share of the
    steps a warp is dealt."""
    rng = np.random.default_rng(chunk + big)
    lens = np.where(rng.random(600) < 0.4, 0, np.exp(rng.uniform(0, np.log(20_000), 600))).astype(np.int64)
    auts = rng.integers(0, 9, 600)
    if big:
        lens = np.concatenate([lens, [5 << 20, 0, 4 << 20, 0]])
        auts = np.concatenate([auts, [0, 0, 1, 1]])
    lib.hb_chunk(chunk)
    with Host(lib, [DNA, BYTES, WALK] * 3) as h:
        st, got = h.scan(auts, lens, (1 << 20) + rng.integers(0, 64, len(lens)))
    assert st == 0 and got["flat"] == 1 and got["graph"] == 0 and got["big"] == big
    assert got["steps"] > 600 and got["missed"] == 0 and got["bounds"] == 0


@pytest.mark.parametrize("machines", [1, 31, 32, 40, 200])
@pytest.mark.parametrize("cls", [DNA, BYTES, WALK])
def test_groups_of_machines_without_symbols(lib, machines, cls):
    """More machines than groups, all or all but one of them with empty texts
    only (in a child process: a trap ends it)."""
    def run():
        lib.hb_chunk(3)
        with Host(lib, [cls] * machines) as h:
            st, got = h.scan(list(range(machines)) * 2, [0] * (2 * machines))
            assert st == 0 and got["flat"] == 0 and got["graph"] == 0 and got["used"] == machines
            for n in (1, 777, 9 << 20):
                st, got = h.scan(list(range(machines)) * 2, [0] * machines + [n] + [0] * (machines - 1))
                assert st == 0 and got["flat"] == 1 and got["missed"] == 0 and got["bounds"] == 0
                assert got["groups"] == 1
            # as many bytes for every machine as the large form takes
            st, got = h.scan(range(machines), [9 << 20] * machines)
            assert st == 0 and got["missed"] == 0 and got["bounds"] == 0 and got["groups"] <= 32

    pid = os.fork()
    if pid == 0:
        try:
            run()
            os._exit(0)
        except BaseException:
            traceback.print_exc()
            os._exit(1)
    assert os.waitpid(pid, 0)[1] == 0


@pytest.mark.parametrize("nth", range(1, 9))
@pytest.mark.parametrize("cls", [DNA, BYTES, WALK])
def test_a_call_after_one_that_found_no_memory(lib, nth, cls):
    """The nth device allocation of a batch fails, on a new stream and where
    its buffers grow: the next call allocates what is missing."""
    with Host(lib, [cls]) as h:
        for jobs in (3, 700, 3000):
            lib.hb_fail(nth)
            st, got = h.scan([0] * jobs, [5000] * jobs)
            lib.hb_fail(0)
            assert st in (0, E_NOMEM) and got["flat"] + got["graph"] == (st == 0) and got["null_lists"] == 0
            st, got = h.scan([0] * jobs, [5000] * jobs)
            assert st == 0 and got["flat"] == 1 and got["null_lists"] == 0 and got["missed"] == 0


def own(lib, cls, big, warp):
    r = np.zeros(2, dtype=np.uint32)
    lib.hb_own(cls, int(big), warp, r.ctypes.data_as(ctypes.c_void_p))
    return r


def apart(x, y):
    return x[1] <= y[0] or y[1] <= x[0]


def test_warps_of_the_front_kernel_do_not_share_memory(lib):
    """Small form: nothing keeps the warps of a CTA in the same class, so one
    warp's region for any class lies apart from another's for any class. Large
    form: the warps meet where the class changes; the sieves' lists lie past
    the 128 KB of the near bitmap."""
    classes = (DNA, BYTES, WALK)
    for w in range(4):
        for v in range(4):
            for c in classes:
                for d in classes:
                    assert v == w or apart(own(lib, c, False, w), own(lib, d, False, v)), (w, c, v, d)
    for c in classes:
        regions = [own(lib, c, True, w) for w in range(32)]
        assert all(apart(regions[w], regions[v]) for w in range(32) for v in range(w))
        assert c == WALK or min(r[0] for r in regions) >= 128 << 10
        assert max(r[1] for r in regions) <= (128 << 10) + 32 * 1024


@pytest.mark.parametrize("cls", [DNA, BYTES, WALK])
def test_no_room_for_the_candidate_lists(lib, cls):
    """The class kernels take sieved texts where the lists find no room; the
    next call tries again."""
    with Host(lib, [cls, WALK]) as h:
        if cls != WALK:
            lib.hb_fail(1)
            st, got = h.scan([0, 1], [5000, 5000])
            lib.hb_fail(0)
            assert st == 0 and got["graph"] == 1 and got["flat"] == 1 and got["used"] == 2
            assert got["null_lists"] == 0 and got["missed"] == 0
        st, got = h.scan([0, 1], [5000, 5000])
        assert st == 0 and got["graph"] == 0 and got["flat"] == 1 and got["missed"] == 0
