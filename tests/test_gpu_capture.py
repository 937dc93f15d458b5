"""Steps and readings enqueued while the caller captures the stream: replayed, the captured graph
gives bit for bit what the same calls give when they run directly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2501_03759_gb300 import lbch  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    lbch.load()


def noise(shape, seed):
    return np.random.default_rng(seed).uniform(-0.1, 0.1, shape)


# Populations and moment form, rows of 16 bytes and ragged ones, the scalar 16-bit kernels; `warm`:
# the same calls ran before the capture, so the context already holds its own graph of steps.
@pytest.mark.parametrize("nx,ny,storage", [(64, 64, 0), (101, 97, 0), (1400, 1400, 0), (256, 256, 1), (66, 50, 2)])
@pytest.mark.parametrize("warm", [False, True])
def test_captured_steps_of_one_field(nx, ny, storage, warm):
    side = torch.cuda.Stream()
    s = lbch.Solver(lbch.make_params(nx, ny, alpha=0.3, storage=storage), stream=side)
    s.init_field(noise((ny, nx), 1))
    image = s.save_state_device()
    log = torch.zeros(2, dtype=torch.float64, device="cuda")
    phi = torch.empty((ny, nx), device="cuda")
    torch.cuda.synchronize()

    def work():
        s.restore_state_device(image)  # a copy before the first step
        for n in (1, 5, 40, 3):
            s.step(n)
        s.mass_device(log[0:1])
        s.free_energy_device(log[1:2])
        s.phi_device(phi)
        s.step(20)

    def result():
        torch.cuda.synchronize()
        return log.cpu().numpy().copy(), phi.cpu().numpy().copy(), s.field()

    if warm:
        with torch.cuda.stream(side):
            work()
        torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        work()
    for _ in range(2):
        graph.replay()
    got = result()
    with torch.cuda.stream(side):
        work()
    for a, b in zip(got, result()):
        assert np.array_equal(a, b)
    s.close()


# One group of fields or both, runs with and without the batch's graph of 64 steps.
@pytest.mark.parametrize("sizes", [[64, 128], [100, 33], [64, 100, 33, 128]])
def test_captured_steps_of_a_batch(sizes):
    side = torch.cuda.Stream()
    b = lbch.Batch(lbch.make_params(8, 8), sizes, sizes, [0.1] * len(sizes), stream=side)
    out = [torch.empty((n, n), device="cuda") for n in sizes]

    def init():
        for i, n in enumerate(sizes):
            b.init_field(i, noise((n, n), i))
        torch.cuda.synchronize()

    def work():
        b.step(2)
        b.step(70)
        for i, o in enumerate(out):
            b.phi_device(i, o)

    init()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        work()
    graph.replay()
    torch.cuda.synchronize()
    got = [o.cpu().numpy().copy() for o in out]
    init()
    with torch.cuda.stream(side):
        work()
    torch.cuda.synchronize()
    for a, o in zip(got, out):
        assert np.array_equal(a, o.cpu().numpy())
    b.close()


@pytest.mark.parametrize("rates", [{}, {"s": [1.0, 1.2] + [1.0] * 13}])
def test_captured_steps_in_3d(rates):
    side = torch.cuda.Stream()
    s = lbch.Solver3(lbch.make_params3(40, 33, 20, alpha=0.3, **rates), stream=side)
    phi0 = noise((20, 33, 40), 2)
    s.init_field(phi0)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        s.step(7)
        s.step(1)
    graph.replay()
    torch.cuda.synchronize()
    got = s.field()
    s.init_field(phi0)
    s.step(7)
    s.step(1)
    assert np.array_equal(got, s.field())
    s.close()
