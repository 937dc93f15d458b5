"""Which kernel a weight gradient runs on: tcgen05 where rows are a multiple of 16 pixels and the
tensors 16-byte aligned, mma.sync elsewhere."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2501_03759_gb300 import lbnop  # noqa: E402


@pytest.mark.parametrize("width,tc", [(16, 1), (32, 1), (48, 1), (112, 1), (128, 1), (208, 1), (8, 0), (24, 0), (130, 0)])
@pytest.mark.parametrize("ci,co", [(96, 96), (16, 16)])
def test_weight_gradient_path(width, tc, ci, co):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    x, dy = (torch.from_numpy(W.bf16_exact((2, 3, width, c), 5 + c, 1.0).astype(np.float32)).cuda().to(torch.bfloat16)
             for c in (ci, co))
    dw = torch.empty((9, co, ci), dtype=torch.float32, device="cuda")
    before, rows128 = lbnop.lbnop_tc_wgrad_launches(), lbnop.lbnop_tc_launches()
    lbnop.lbnop_conv3x3_bwd_weight(x.data_ptr(), dy.data_ptr(), 2, 3, width, ci, co, dw.data_ptr(),
                                   torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert lbnop.lbnop_tc_fault() == 0
    assert lbnop.lbnop_tc_wgrad_launches() - before == tc
    assert lbnop.lbnop_tc_launches() - rows128 == (1 if width % 128 == 0 else 0)
    assert torch.isfinite(dw).all()
