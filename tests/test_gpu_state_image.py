"""Saved states: equal states give equal images, whatever the buffers and the target held before."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2501_03759_gb300 import lbch  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    lbch.load()


# Node counts that are no multiple of 64 (planes end in padding), by one node and by almost 64, and
# one that is; rows of 16 bytes and ragged ones.
@pytest.mark.parametrize("nx,ny", [(65, 1), (21, 3), (100, 33), (101, 97), (64, 64), (1001, 517)])
@pytest.mark.parametrize("storage", [lbch.STORE_F32, lbch.STORE_BF16_DEV, lbch.STORE_F16_DEV])
def test_equal_states_give_equal_images(nx, ny, storage):
    images = []
    for fill, chunks in ((0x00, [12]), (0xFF, [1] * 12), (0x5A, [5, 7])):
        s = lbch.Solver(lbch.make_params(nx, ny, alpha=0.3, storage=storage))
        s.workspace.fill_(fill)
        s.init_field(W.noise(nx, ny, 0.2, 4))
        for n in chunks:
            s.step(n)
        image = torch.full((lbch.lbch_state_bytes(s.params),), fill, dtype=torch.uint8, device="cuda")
        images.append(s.save_state_device(image))
        s.restore_state_device(image)
        assert torch.equal(s.save_state_device(), image)
        s.close()
    assert torch.equal(images[0], images[1]) and torch.equal(images[0], images[2])
