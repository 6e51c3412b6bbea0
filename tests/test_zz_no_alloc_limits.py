"""frlap_apply_noalloc at the edge of its limit, which is one on the spectra alone: rectangular grids whose spectra
just fit 32 MiB are taken, with the line exponents of the FP64-class engines beside them, and the next ones refused.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _spectra(frlap, Ns, c):
    n = [v - 1 for v in Ns]
    P = [max(32, 1 << (2 * v - 2).bit_length()) for v in n]
    up = lambda b: -(-b // 256) * 256
    H = P[0] // 2 + 1
    if len(Ns) == 2:
        return up(c * H * n[1]) * (2 if P[1] > 8192 else 1)
    return up(c * H * n[2] * n[1]) + up(c * H * P[1] * n[2])


@pytest.mark.parametrize("prec", [0, 3])
@pytest.mark.parametrize("Ns", [(1025, 2047), (513, 4087), (513, 4089), (17, 513, 81), (513, 513, 3)])
def test_spectra_that_just_fit(frlap, Ns, prec):
    assert _spectra(frlap, Ns, 16) <= frlap.NOALLOC_MAX_BYTES
    plan = frlap.Plan(len(Ns), 1.3, 2.0 / max(Ns), Ns, prec=prec)
    u = torch.randn(plan.shape, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    y = torch.full_like(u, float("nan"))
    frlap.frlap_apply_noalloc(plan, u, y)
    assert torch.equal(y, frlap.frlap_apply(plan, u))  # the same kernels on the same data


@pytest.mark.parametrize("Ns", [(1025, 2048), (513, 4090), (17, 513, 82), (513, 513, 4)])
def test_the_next_grids_are_refused(frlap, Ns):
    assert _spectra(frlap, Ns, 16) > frlap.NOALLOC_MAX_BYTES
    plan = frlap.Plan(len(Ns), 1.3, 2.0 / max(Ns), Ns, prec=0)
    u = torch.zeros(plan.shape, dtype=torch.float64, device="cuda")
    with pytest.raises(frlap.FrlapError) as exc:
        frlap.frlap_apply_noalloc(plan, u)
    assert exc.value.code == 1
