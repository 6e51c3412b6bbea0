"""frlap_learn_grad across its launches' boundaries: pairs go through the transforms eight at a time, and the
network's backward pass takes tiles of 64 entries on at most 304 CTAs.  A batch equals the mean of its parts."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _grad(fl, plan, params, r, e):
    work = torch.empty(fl.frlap_learn_workspace_bytes(plan, r.shape[0]) + 256, dtype=torch.uint8, device="cuda")
    work = work[(-work.data_ptr()) % 256:]
    grad, loss = torch.empty_like(params), torch.empty(1, dtype=torch.float64, device="cuda")
    fl.frlap_learn_grad(plan, params, r, e, grad, loss, work)
    return grad.double(), loss.item()


# octants of 17 x 17 (five tiles, the last of 33 entries), 257 x 17 (69) and 129 x 257 (518, more than the CTAs)
@pytest.mark.parametrize("Ns,B", [((16, 9), 1), ((16, 9), 9), ((250, 12), 8), ((128, 256), 17), ((9, 16, 7), 9)])
def test_batch_is_the_mean_of_its_parts(frlap, Ns, B):
    d = len(Ns)
    plan = frlap.Plan(d, 1.3, 2.0 / max(Ns), Ns)
    g = torch.Generator(device="cuda")
    g.manual_seed(4)
    e = torch.randn((B,) + plan.shape, dtype=torch.float64, device="cuda", generator=g)
    r = torch.stack([frlap.frlap_apply(plan, v) for v in e])
    params = 0.1 * torch.randn(frlap.MLP_NPARAM, dtype=torch.float32, device="cuda", generator=g)
    grad, loss = _grad(frlap, plan, params, r, e)
    parts = [_grad(frlap, plan, params, r[i:i + 1].contiguous(), e[i:i + 1].contiguous()) for i in range(B)]
    mean = sum(p[0] for p in parts) / B
    # FP32 tile sums on both sides: 64 products of relative rounding 2^-24 each, over random signs
    assert torch.linalg.norm(grad - mean).item() <= 1e-5 * torch.linalg.norm(mean).item()
    assert loss == pytest.approx(float(np.mean([p[1] for p in parts])), rel=1e-12)
