"""Tensor memory of CTA pairs, checked on the host over the whole tile space: pairs
that fit on an SM together by their shared memory also fit by their columns, so no
two of them ever wait for columns that the other holds."""
import ctypes
import itertools
import os
import subprocess

import numpy as np
import pytest

import oracle as O

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_04178_gb300", "csrc")
SHIM = """
#include "pm_footprint.cuh"
extern "C" void footprint(int elem, int halves, int cg, int BK, int stages, int tmem_a, int G, const int16_t* BM,
                          const int16_t* BN, long* out) {
  const pm::GemmFootprint f = pm::gemm_footprint(elem, halves, cg, BK, stages, tmem_a, G, BM, BN);
  out[0] = (long)f.smem; out[1] = f.alloc_cols; out[2] = f.staged; out[3] = f.stage_bytes;
}
extern "C" long pair_smem(long bytes, int cols) { return (long)pm::pair_smem((size_t)bytes, cols); }
extern "C" long smem_per_sm() { return (long)pm::kSmemPerSm; }
extern "C" long smem_dynamic() { return (long)pm::kSmemDynamic; }
"""


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    d = tmp_path_factory.mktemp("footprint")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "shim.so"),
                    str(d / "shim.cpp")], check=True)
    lib = ctypes.CDLL(str(d / "shim.so"))
    for f in (lib.pair_smem, lib.smem_per_sm, lib.smem_dynamic):
        f.restype = ctypes.c_long
    return lib


def footprint(shim, dt, cg, BK, stages, tmem_a, BMs, BNs):
    out = (ctypes.c_long * 4)()
    bm, bn = np.array(BMs, np.int16), np.array(BNs, np.int16)
    shim.footprint((4, 2, 1)[dt], 2 if dt == 0 else 1, cg, BK, stages, tmem_a, len(BMs),
                   bm.ctypes.data_as(ctypes.c_void_p), bn.ctypes.data_as(ctypes.c_void_p), out)
    return list(out)


def tiles(dt, cg, BK, stages, tmem_a):
    return [(a, b) for a in (64, 128, 256) for b in (64, 128, 256) if O.cfg_valid(a, b, BK, stages, cg, dt, tmem_a)]


def all_launches():
    for dt, cg, stages, tmem_a in itertools.product((0, 1, 2), (1, 2), range(2, 7), (0, 1)):
        for BK in ((32, 64), (64, 128), (64, 128))[dt]:
            ts = tiles(dt, cg, BK, stages, tmem_a)
            for t in ts:
                yield dt, cg, BK, stages, tmem_a, [t[0]], [t[1]]
            if dt == 1 and tmem_a == 0:                        # grouped launches mix tiles
                for t, u in itertools.combinations(ts, 2):
                    yield dt, cg, BK, stages, tmem_a, [t[0], u[0]], [t[1], u[1]]


def test_every_launch_fits_an_sm(shim):
    n = 0
    for dt, cg, BK, stages, tmem_a, bm, bn in all_launches():
        smem, cols, staged, stage = footprint(shim, dt, cg, BK, stages, tmem_a, bm, bn)
        assert stages * stage + 1024 + 16384 * staged <= smem <= shim.smem_dynamic()
        assert cols in (32, 64, 128, 256, 512)
        if cg == 1:                                            # only pairs hold more than they use
            assert smem == stages * stage + 1024 + 16384 * staged
        n += 1
    assert n > 600


def test_resident_pairs_have_their_columns(shim):
    least = {256: shim.pair_smem(49 * 1024, 256)}              # the pair form of the MMA rate probe
    for dt, cg, BK, stages, tmem_a, bm, bn in all_launches():
        if cg == 2:
            smem, cols, _, _ = footprint(shim, dt, cg, BK, stages, tmem_a, bm, bn)
            least[cols] = min(smem, least.get(cols, smem))
    assert set(least) == {64, 128, 256, 512}
    # any number of CTAs of each width that the shared memory of an SM admits
    budget = shim.smem_per_sm()
    counts = [range(budget // least[c] + 1) for c in sorted(least)]
    for k in itertools.product(*counts):
        if sum(i * least[c] for i, c in zip(k, sorted(least))) <= budget:
            assert sum(i * c for i, c in zip(k, sorted(least))) <= 512, k
