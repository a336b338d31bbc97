"""The gradients of lv_price are tensors of their own (needs a GB300)."""
import pytest

import workloads as W
from paper_2002_02481_gb300 import build, lv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["float32", "float64"])
def test_gradients_do_not_share_storage(dtype):
    import torch

    from paper_2002_02481_gb300.autograd import lv_price
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    surf, opt = W.config_small()
    s = lv.Surface.from_workload(surf, lv.load())
    S0 = torch.tensor(opt.S0, dtype=torch.float64, device="cuda", requires_grad=True)
    sigma = torch.tensor(surf.sigma, dtype=getattr(torch, dtype), device="cuda", requires_grad=True)
    lv_price(S0, sigma, s, opt.r, opt.K, opt.T, opt.n_steps, 1024, 3).backward()
    s.close()
    a, b = S0.grad.untyped_storage(), sigma.grad.untyped_storage()
    assert a.data_ptr() != b.data_ptr()
    assert b.nbytes() == sigma.numel() * sigma.element_size() and sigma.grad.storage_offset() == 0
    assert sigma.grad.data_ptr() % 16 == 0
