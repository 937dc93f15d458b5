"""How 3D sweeps are cut into blocks: the rule (compiled for the host) against every possible cut, and
thin grids, whose few tiles want many segments, against the oracle."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "lbch3_plan.h"
extern "C" int plan(int tiles, int nz, int warm, int sms, int* len) { return lbch3::plan_segments(tiles, nz, warm, sms, len); }
"""
SMS = 152


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SRC)
    lib = str(d / "libplan.so")
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2501_03759_gb300", "csrc"),
                    str(d / "plan.cpp"), "-o", lib], check=True)
    fn = ctypes.CDLL(lib).plan

    def call(tiles, nz, warm):
        length = ctypes.c_int(0)
        return fn(tiles, nz, warm, SMS, ctypes.byref(length)), length.value

    return call


def predicted(tiles, nz, warm, length):
    q = -(-tiles * -(-nz // length) // SMS)
    return (length + warm) * (1.1 * (q // 2) + q % 2)


@pytest.mark.parametrize("tiles,nz", [(1, 1), (1, 4096), (2, 2000), (4, 1000), (2, 200), (12, 200), (32, 100), (171, 256),
                                      (666, 512), (40141, 128)])
@pytest.mark.parametrize("warm", [4, 5])
def test_plan_covers_the_grid_and_is_the_best_cut(plan, tiles, nz, warm):
    blocks, length = plan(tiles, nz, warm)
    assert 1 <= length <= nz and blocks == tiles * -(-nz // length)
    best = min(predicted(tiles, nz, warm, k) for k in range(1, nz + 1))
    assert predicted(tiles, nz, warm, length) <= best * (1 + 1e-12)


@pytest.mark.parametrize("tiles,nz", [(1, 4096), (2, 2000), (4, 1000)])
def test_thin_grids_fill_the_gpu(plan, tiles, nz):
    blocks, _ = plan(tiles, nz, 4)
    assert blocks >= 0.9 * 2 * SMS  # two blocks per SM


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(16, 14, 700), (31, 14, 401), (8, 30, 130)])
def test_thin_grid_matches_the_oracle(shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2501_03759_gb300 import lbch

    nx, ny, nz = shape
    phi0 = np.random.default_rng(9).uniform(-0.5, 0.5, (nz, ny, nx))
    got = []
    for chunks in ([5], [1] * 5):
        s = lbch.Solver3(lbch.make_params3(nx, ny, nz, alpha=0.4))
        s.init_field(phi0)
        for n in chunks:
            s.step(n)
        got.append(s.field())
        s.close()
    assert np.array_equal(got[0], got[1])
    p = oracle.Params3(nx, ny, nz, alpha=0.4)
    ref = oracle.phi3(p, oracle.step3(p, oracle.init3(p, phi0), 5))
    assert np.abs(got[0] - ref).max() <= 2e-6
