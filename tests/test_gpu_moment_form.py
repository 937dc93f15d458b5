"""Runs of steps in moment form (the sums a collision needs in place of the populations): a run
gives bit for bit what its steps give one by one (single steps go from populations to
populations), at the widths where strips, padded rows and lanes end and at the fewest rows; large
FP32 fields of that form match the FP64 oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2501_03759_gb300 import lbch  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    lbch.load()


def field(nx, ny, seed):
    """Noise with flat regions at -1 and +1 (the guard at grad phi = 0, tails of 1e-10)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    phi = torch.rand((ny, nx), generator=g, device="cuda") - 0.5
    phi[:, : nx // 3] = -1.0
    phi[: ny // 3] = 1.0
    return phi.contiguous()


def run(nx, ny, storage, chunks):
    s = lbch.Solver(lbch.make_params(nx, ny, alpha=0.4, storage=storage))
    s.init_field_device(field(nx, ny, 5))
    for n in chunks:
        s.step(n)
    image = s.save_state_device()
    s.close()
    return image


def populations_equal(a, b, nx, ny, storage):
    """The population planes of two saved states (their row padding is not part of the state)."""
    n, ps = nx * ny, (nx * ny + 63) // 64 * 64
    planes = [(4 * k * ps, 4 * n) for k in range(9 if storage == lbch.STORE_F32 else 2)]
    if storage != lbch.STORE_F32:
        base = (8 * ps + 255) // 256 * 256
        planes += [(base + 2 * k * ps, 2 * n) for k in range(8)]
    return all(torch.equal(a[o:o + m], b[o:o + m]) for o, m in planes)


DEV = [(4, 4), (8, 1), (60, 2), (120, 3), (124, 9), (128, 7), (132, 16), (244, 33), (512, 40)]
BIG = [(1348, 1360), (1349, 1360), (1361, 1347), (1366, 1343), (128, 16000), (27, 65536)]


# FP32 fields that fit in L2: those with an edge that is no multiple of 32 (and at least 8 columns).
SMALL = [(8, 5), (9, 7), (33, 1), (61, 90), (100, 100), (121, 33), (128, 40), (130, 4), (241, 31), (500, 37)]


@pytest.mark.parametrize("nx,ny,storage", [(nx, ny, st) for st in (lbch.STORE_BF16_DEV, lbch.STORE_F16_DEV) for nx, ny in DEV]
                         + [(nx, ny, lbch.STORE_F32) for nx, ny in BIG + [(1366, 1)] + SMALL])
@pytest.mark.parametrize("n", [4, 5, 23])
def test_run_equals_its_steps_bitwise(nx, ny, storage, n):
    a = run(nx, ny, storage, [n])
    b = run(nx, ny, storage, [1] * n)
    assert populations_equal(a, b, nx, ny, storage)
    c = run(nx, ny, storage, [1, n - 1])  # entered from the other buffer
    assert populations_equal(c, b, nx, ny, storage)


@pytest.mark.parametrize("nx,ny", [(1348, 1360), (1361, 1347)])
def test_large_fp32_field_matches_oracle_windows(nx, ny):
    """Bound: 1e-6 after 10 steps, as for every FP32 field (oracle windows padded by the steps'
    footprint are exact), at the seams and at strip and segment ends."""
    phi0 = W.noise(nx, ny, 0.5, 3)
    s = lbch.Solver(lbch.make_params(nx, ny, alpha=0.3))
    s.init_field(phi0)
    m0 = s.mass()
    s.step(10)
    g = s.field()
    w = 16
    p = oracle.Params(nx, ny, alpha=0.3)
    for x0, y0 in [(0, 0), (nx - w, ny - w), (nx - w, 0), (112, 5), (600, ny // 2)]:
        ref = oracle.run_window(p, phi0, x0, y0, w, w, 10)
        assert np.abs(g[y0:y0 + w, x0:x0 + w] - ref).max() <= 1e-6, (x0, y0)
    # each node's sum is kept to rounding at the scale of mu_alpha: far below an ulp of phi per step
    assert abs(s.mass() - m0) <= 1e-9 * nx * ny
    s.close()


def test_batch_of_large_and_small_fields_bitwise():
    """Large FP32 fields step in moment form in a batch as alone, small ones in populations;
    fields can be initialised again after an even number of steps."""
    sizes, alpha = [(1360, 1348), (64, 64), (1352, 1360), (250, 33)], [0.3, 0.1, 0.2, 0.4]
    b = lbch.Batch(lbch.make_params(8, 8), [s[0] for s in sizes], [s[1] for s in sizes], alpha)
    phi0 = [W.noise(nx, ny, 0.3, 7 + i) for i, (nx, ny) in enumerate(sizes)]
    for i in range(4):
        b.init_field(i, phi0[i])
    b.step(6)
    b.init_field(0, phi0[0])
    b.init_field(1, phi0[1])
    b.step(71)
    for i, (nx, ny) in enumerate(sizes):
        s = lbch.Solver(lbch.make_params(nx, ny, alpha=alpha[i]))
        s.init_field(phi0[i])
        s.step(71 if i < 2 else 77)
        assert np.array_equal(b.field(i), s.field()), i
        s.close()
    b.close()


@pytest.mark.parametrize("shape", [(4, 3, 2), (30, 14, 5), (31, 15, 4), (33, 17, 9), (61, 29, 1), (100, 3, 40), (7, 64, 33), (62, 15, 6),
                                   (63, 14, 70), (94, 5, 7), (125, 29, 3)])
def test_3d_run_equals_its_steps_and_matches_the_oracle(shape):
    """D3Q15 at the edges of the 30 x 14 and 62 x 14 tiles and of the planes' runs: a run's phi equals its
    steps' bit for bit, and both match the oracle within the bound of the 3D parity tests."""
    nx, ny, nz = shape
    phi0 = np.random.default_rng(8).uniform(-0.5, 0.5, (nz, ny, nx))
    phi0[:, :, : nx // 3] = -1.0
    got = []
    for chunks in ([6], [1] * 6, [2, 4]):
        s = lbch.Solver3(lbch.make_params3(nx, ny, nz, alpha=0.4))
        s.init_field(phi0)
        m0 = s.mass()
        for n in chunks:
            s.step(n)
        got.append(s.field())
        assert abs(s.mass() - m0) <= 1e-8 * phi0.size
        s.close()
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])
    p = oracle.Params3(nx, ny, nz, alpha=0.4)
    ref = oracle.phi3(p, oracle.step3(p, oracle.init3(p, phi0), 6))
    assert np.abs(got[0] - ref).max() <= 2e-6
