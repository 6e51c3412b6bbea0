"""The fixed-point symbol product where the symbol leaves the range of normal doubles.  A = h^-alpha A_1, so a huge h makes
it subnormal and a tiny one overflow."""
import numpy as np
import pytest

import frlap_inputs as inp

pytestmark = pytest.mark.gpu

SHAPES = [(33, 33), (33, 200), (12, 7, 9), (6, 4200)]


@pytest.mark.parametrize("prec", ["F64", "DF64"])
@pytest.mark.parametrize("Ns", SHAPES)
def test_subnormal_symbol(frlap, Ns, prec):
    """lambda / prod P between about 1e-313 and 1e-309: its entries are multiples of 2^-1074 = 5e-324, each rounded
    some log2(prod P) < 20 times on the way, 1e-13 of the largest; with the engine's own rounding far below, 1e-11
    lambda_max ||u|| holds amply, while a leading bit too many would be 2.2e-308, a hundred times the largest."""
    import torch

    d, alpha, prec = len(Ns), 1.8, getattr(frlap, "FRLAP_" + prec)
    one = frlap.Plan(d, alpha, 1.0, Ns, prec=frlap.FRLAP_F64)
    sym = one.symbol()
    target = 1e-309 / float(sym.max())  # h^-alpha
    h = target ** (-1.0 / alpha)
    scale = np.longdouble(h) ** np.longdouble(-alpha) * np.longdouble(1e300)
    u = torch.from_numpy(inp.normal_field(Ns, seed=21)).cuda()
    plan = frlap.Plan(d, alpha, h, Ns, prec=prec)
    assert 0.0 < float(plan.symbol().max()) < 2.2e-308
    y = frlap.frlap_apply(plan, u * 1e300)
    ref = frlap.frlap_apply(one, u) * float(scale)
    lam_max = float(sym.max()) * float(np.prod([float(p) for p in one.P])) * float(scale)
    assert float(torch.linalg.norm(y - ref)) <= 1e-11 * lam_max * float(torch.linalg.norm(u))


@pytest.mark.parametrize("prec", ["F64", "DF64"])
@pytest.mark.parametrize("Ns", SHAPES)
def test_overflown_symbol(frlap, Ns, prec):
    """h^-alpha = 1e313: no entry of the product may come out finite, for a vector of zeros either (0 times infinity)."""
    import torch

    plan = frlap.Plan(len(Ns), 1.9, 10.0 ** (-313 / 1.9), Ns, prec=getattr(frlap, "FRLAP_" + prec))
    assert not bool(torch.isfinite(plan.symbol()).any())
    u = torch.from_numpy(inp.normal_field(Ns, seed=22)).cuda()
    assert not bool(torch.isfinite(frlap.frlap_apply(plan, u * 1e-200)).any())
    assert bool(torch.isnan(frlap.frlap_apply(plan, u * 0.0)).all())


@pytest.mark.parametrize("prec", ["F64", "DF64"])
def test_zero_symbol(frlap, prec):
    """h^-alpha below the subnormal range: A is zero."""
    import torch

    plan = frlap.Plan(2, 1.9, 1e200, (40, 40), prec=getattr(frlap, "FRLAP_" + prec))
    assert not bool(plan.symbol().any())
    u = torch.from_numpy(inp.normal_field((40, 40), seed=23)).cuda()
    assert not bool(frlap.frlap_apply(plan, u * 1e300).any())
