"""DF64 applies of rows that one spike dominates, where a scale set once per row costs most: against the F64 engine at
every first-stage length (the F64 engine is checked against the defining sum in test_gpu_fixed_point.py).

Bound, over lambda_max ||u||: with L <= 512 points in a transformed row the fixed unit is 2^-60 L of the row's largest
value, entered by the conversion, two twiddled stages and the real-data split, so at most 4 * 2^-51 of a spike's row;
F64's own rounding is below 2^-52: 2.0e-15.  Longer rows follow the data in both engines: the same bits.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [32, 64, 128, 256, 512, 1024, 2048, 4096, 8192])
@pytest.mark.parametrize("rows", [2, 40])
def test_spikes_over_noise(frlap, N, rows):
    import torch

    h, alpha = 2.0 / N, 0.5
    plans = [frlap.Plan(2, alpha, h, (N, rows), prec=p) for p in (frlap.FRLAP_DF64, frlap.FRLAP_F64)]
    lam_max = float(plans[1].symbol().abs().max()) * float(np.prod([float(p) for p in plans[1].P]))
    g = torch.Generator("cuda").manual_seed(N + rows)
    for noise in (0.0, 1e-6, 1e-3, 0.1):
        for pos in (0, 1, N // 3, N - 2):
            u = noise * torch.randn(plans[0].shape, dtype=torch.float64, device="cuda", generator=g)
            u[:, pos] += 1.0
            yd, yf = (frlap.frlap_apply(p, u) for p in plans)
            err = float(torch.linalg.norm(yd - yf)) / (lam_max * float(torch.linalg.norm(u)))
            assert err <= 4 * 2.0 ** -51 + 2.0 ** -52, (noise, pos, err)
            if N > 512:
                assert torch.equal(yd, yf)
