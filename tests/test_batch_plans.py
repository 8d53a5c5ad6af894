"""Which work items the launches of a batch read, on a host stand-in for the
CUDA runtime (fake_runtime.cpp) linked with the library's api.cu: calls with
other buffers while earlier ones still run, and an autotune that fails."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

import synth
from paper_2410_10447_gb300 import adgb
from paper_2410_10447_gb300.adgb import _build as B

HERE = os.path.dirname(os.path.abspath(__file__))
MAXG = adgb.MAX_GENES


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cmd = [nvcc, *B.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-I", B.INCLUDE, "-I", B.CSRC, "-shared",
           "-cudart", "none", "-Xlinker", "-Bsymbolic", "-o", out, os.path.join(HERE, "fake_runtime.cpp"),
           os.path.join(B.CSRC, "api.cu")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = C.CDLL(out)
    L.adgb_last_error.restype = C.c_char_p
    return L


class Batch:
    """One batch of a 20- and a 40-atom ligand on the fake device."""

    N_POSES = [7, 5]

    def __init__(self, lib):
        self.lib, self.h = lib, C.c_void_p()
        assert lib.adgb_create(C.byref(self.h), 0, C.byref(adgb._Options(0, 0, 0, 0, 0))) == 0
        rec = synth.make_receptor(3, 8, 4)
        g = adgb._Grid(8, 8, 8, rec["spacing"], (C.c_float * 3)(*rec["origin"]), 4)
        maps, i = np.ascontiguousarray(rec["maps"], np.float32), C.c_int()
        assert lib.upload_receptor_grids(self.h, C.byref(g), C.c_void_p(maps.ctypes.data), C.byref(i)) == 0
        rid, lids = i.value, []
        for n in (20, 40):
            d, _keep = adgb._ligand_desc(synth.make_ligand(5 + n, n, 4, 4))
            assert lib.upload_ligand_torsion_tree(self.h, C.byref(d), C.byref(i)) == 0
            lids.append(i.value)
        a = [np.asarray(x, np.int32) for x in ([rid, rid], lids, self.N_POSES)]
        assert lib.batch_create(self.h, 2, *[C.c_void_p(x.ctypes.data) for x in a], C.byref(i)) == 0, self.error()
        self.bid = i.value

    def error(self):
        return self.lib.adgb_last_error(self.h)

    def buffers(self):
        n = sum(self.N_POSES)
        return np.zeros((n, MAXG), np.float32), np.zeros(n, np.float32)

    def search(self, genes, energy, iters=5):
        p = adgb._LSParams(iters, 0.8, 0.01, -1, 0)
        rc = self.lib.batch_local_search_dev(self.h, self.bid, C.c_void_p(genes.ctypes.data), C.byref(p),
                                             C.c_void_p(energy.ctypes.data), None)
        assert rc == 0, self.error()

    def autotune(self, genes):
        return self.lib.batch_autotune(self.h, self.bid, C.c_void_p(genes.ctypes.data), 5, None)

    def close(self):
        assert self.lib.batch_release(self.h, self.bid) == 0
        assert self.lib.adgb_destroy(self.h) == 0


def test_calls_with_other_buffers_while_earlier_launches_run(lib):
    b = Batch(lib)
    bufs = [b.buffers() for _ in range(5)]
    for genes, energy in bufs:      # nothing has run when the next call comes
        b.search(genes, energy)
    assert lib.fake_queued() > 0
    lib.fake_run()
    for genes, energy in bufs:      # every genotype of every call was searched once
        assert np.array_equal(energy, np.ones_like(energy))
    b.search(*bufs[4])              # and again by the present graph
    lib.fake_run()
    assert np.all(bufs[4][1] == 2)
    b.close()


def test_autotune_while_a_launch_runs(lib):
    b = Batch(lib)
    genes, energy = b.buffers()
    b.search(genes, energy)
    assert b.autotune(genes) == 0
    lib.fake_run()
    assert np.array_equal(energy, np.ones_like(energy)) and lib.fake_freed_reads() == 0
    b.close()


@pytest.mark.parametrize("nth", [0, 1, 3, 5])
def test_failed_autotune_leaves_the_batch_as_it_was(lib, nth):
    b = Batch(lib)
    genes, energy = b.buffers()
    b.search(genes, energy)
    lib.fake_run()
    lib.fake_fail_elapsed(nth)
    assert b.autotune(genes) == -4    # EDEVICE
    lib.fake_fail_elapsed(-1)
    b.search(genes, energy)
    lib.fake_run()
    assert np.all(energy == 2) and lib.fake_freed_reads() == 0
    b.close()
