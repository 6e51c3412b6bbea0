"""The fixed-point engines: a vector with a non-finite entry is NaN throughout and leaves the others of its batch as they
are, in F64 and DF64 (rows above and below the length at which DF64 sets its scale once, four, eight and sixteen
entries a thread, 2D, 3D and the split stage); and the training spectra are the F64 engine's on every plan.
"""
import numpy as np
import pytest

import frlap_inputs as inp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["F64", "DF64"])
@pytest.mark.parametrize("Ns", [(40, 33), (300, 257), (1100, 300), (12, 40, 9), (6, 4200)])
def test_a_non_finite_vector_stays_alone(frlap, Ns, prec):
    import torch

    plan = frlap.Plan(len(Ns), 1.2, 2.0 / max(Ns), Ns, prec=getattr(frlap, "FRLAP_" + prec))
    us = torch.from_numpy(np.stack([inp.normal_field(Ns, seed=s) for s in range(4)])).cuda()
    ys = frlap.frlap_apply_batch(plan, us)
    flat = us.view(4, -1)
    for where, bad in ((0, float("nan")), (plan.M // 2, float("inf")), (plan.M - 1, -float("inf"))):
        keep = flat[2, where].item()
        flat[2, where] = bad
        zs = frlap.frlap_apply_batch(plan, us)
        flat[2, where] = keep
        assert bool(torch.isnan(zs[2]).all())
        for b in (0, 1, 3):
            assert torch.equal(zs[b], ys[b])
    assert torch.equal(frlap.frlap_apply_batch(plan, us), ys)  # nothing is left behind


@pytest.mark.parametrize("Ns", [(100, 70), (20, 24, 17)])
def test_training_gradients_are_the_same_on_df64_plans(frlap, Ns):
    import torch

    e = torch.from_numpy(np.stack([inp.normal_field(Ns, seed=s) for s in range(3)])).cuda()
    out = []
    for prec in (frlap.FRLAP_F64, frlap.FRLAP_DF64):
        plan = frlap.Plan(len(Ns), 1.2, 2.0 / max(Ns), Ns, prec=prec)
        check = frlap.Plan(len(Ns), 1.2, 2.0 / max(Ns), Ns, prec=frlap.FRLAP_F64)
        r = frlap.frlap_apply_batch(check, e)
        rng = np.random.default_rng(1)
        params = torch.from_numpy((0.1 * rng.standard_normal(frlap.MLP_NPARAM)).astype(np.float32)).cuda()
        grad, loss = torch.empty_like(params), torch.empty(1, dtype=torch.float64, device="cuda")
        work = torch.empty(frlap.frlap_learn_workspace_bytes(plan, 3) + 256, dtype=torch.uint8, device="cuda")
        frlap.frlap_learn_grad(plan, params, r, e, grad, loss, work[(-work.data_ptr()) % 256:])
        out.append((grad, loss))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert bool(torch.isfinite(out[0][0]).all()) and bool(out[0][0].any())
