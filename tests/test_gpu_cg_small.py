"""CG on short vectors, whose iterations run their vector part in one kernel (at most 32768 entries), and on the
first ones above.  The solution's residual is formed with a separate FP64 apply.  Tolerance: the solve stops at
rtol = 1e-12 by its own residual; the two residuals differ by the applies' rounding, at most 1e-15 lambda_max ||x||
<= 1e-15 kappa ||f||, kappa below 200 at alpha = 0.8 on these grids: 2e-13, so 1.2e-12 in all.
"""
import pytest

import frlap_inputs as inp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "df64"])
@pytest.mark.parametrize("precond", ["none", "strang"])
@pytest.mark.parametrize("Ns", [(2, 2), (4, 3), (40, 33), (65, 64), (182, 182), (183, 182), (33, 33, 32), (33, 33, 34)])
def test_residual_of_short_solves(frlap, Ns, precond, prec):
    import torch

    d, h = len(Ns), 2.0 / max(Ns)
    plan = frlap.Plan(d, 0.8, h, Ns, prec=getattr(frlap, "FRLAP_" + prec.upper()))
    check = frlap.Plan(d, 0.8, h, Ns, prec=frlap.FRLAP_F64)
    f = torch.from_numpy(inp.normal_field(Ns, seed=3)).cuda()
    pre = getattr(frlap, "FRLAP_PRECOND_" + precond.upper())
    if precond == "strang":
        frlap.frlap_precond_strang(plan)
    x, it, rel, code = frlap.frlap_pcg_solve(plan, f, rtol=1e-12, precond=pre)
    assert code == 0 and it >= 1
    res = torch.linalg.norm(f - frlap.frlap_apply(check, x)) / torch.linalg.norm(f)
    assert float(res) <= 1.2e-12
    again, it2, _, _ = frlap.frlap_pcg_solve(plan, f, rtol=1e-12, precond=pre)
    assert it2 == it and torch.equal(x, again)  # sums in a fixed order
