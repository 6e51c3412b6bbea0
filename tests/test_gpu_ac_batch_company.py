"""An instance of the batched Allen-Cahn launch gives the same bits and iteration counts whatever other instances the
call holds: as many of its own shape, and more shapes than the launch has parallel branches.
"""
import pytest
import torch

import frlap_inputs as inp

pytestmark = pytest.mark.gpu


def _run(frlap, specs, plans):
    us = [torch.from_numpy(inp.uniform_field((N, N), seed=5 + k)).cuda() for k, N, _ in specs]
    iters, status, code = frlap.frlap_allen_cahn_batch(plans, us, 1e-3, 0.05, 3, rtol=1e-10)
    assert code == 0 and all(s == 0 for s in status)
    return us, iters


@pytest.mark.parametrize("prec", ["F64", "DF64"])
@pytest.mark.parametrize("Ns", [(400,) * 8, (300, 64, 257, 96, 200, 33, 64, 300)])
def test_bits_do_not_depend_on_the_company(frlap, Ns, prec):
    alphas = (1.5, 1.2, 1.9, 1.35, 1.7, 1.6, 1.45, 1.8)
    specs = [(k, N, a) for k, (N, a) in enumerate(zip(Ns, alphas))]
    plans = [frlap.Plan(2, a, 2.0 / N, (N, N), prec=getattr(frlap, "FRLAP_" + prec)) for _, N, a in specs]
    us, iters = _run(frlap, specs, plans)
    for k in (0, 2, 7):
        alone, it = _run(frlap, specs[k:k + 1], plans[k:k + 1])
        assert it[0] == iters[k] and torch.equal(alone[0], us[k])
