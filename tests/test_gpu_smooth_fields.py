"""F64 applies of smooth fields, whose spectra spread over many decades: the symbol weighs the smallest values most, so what
counts is the rounding unit relative to a line's largest value.  (N(0,1) vectors do not show it.)

Reference: the same product in long double, from the plan's own symbol, so only the transforms are compared.  Bound,
normwise over lambda_max ||u||: a forward transform's values carry a unit of 2^-61.5 of the row's largest one, in about four
places, and that largest value is at most sqrt(L) <= 2^6 times the rms of the row's spectrum: 4 * 2^6 * 2^-61.5 = 2^-53.5;
columns and inverse transforms stay below that.  2^-53 (an FP64 FFT product has 0.6 to 0.9 times that).
"""
import numpy as np
import pytest

import frlap_inputs as inp

pytestmark = pytest.mark.gpu


def _exact(plan, u):
    import scipy.fft as sf

    P = [int(p) for p in plan.P][:u.ndim][::-1]  # slowest axis first, as u
    lam = plan.symbol().cpu().numpy().astype(np.longdouble)
    for ax in range(u.ndim - 1):  # the octant to the half spectrum
        lam = np.concatenate([lam, np.flip(np.take(lam, range(1, lam.shape[ax] - 1), axis=ax), axis=ax)], axis=ax)
    U = np.zeros(P, dtype=np.longdouble)
    box = tuple(slice(0, n) for n in u.shape)
    U[box] = u
    scale = np.longdouble(1)
    for p in P:
        scale *= p
    return sf.irfftn(sf.rfftn(U, workers=8) * lam * scale, s=P, workers=8)[box]


def _fields(Ns):
    h = 2.0 / max(Ns)
    x = [h * np.arange(1, N) for N in Ns]
    L = [h * N for N in Ns]
    d = len(Ns)

    def prod(parts):
        out = np.ones((1,) * d)
        for r, p in enumerate(parts):
            shape = [1] * d
            shape[d - 1 - r] = -1
            out = out * p.reshape(shape)
        return np.ascontiguousarray(out)

    yield "boundary layer", prod([np.sin(np.pi * a / b) ** 0.9 for a, b in zip(x, L)])
    yield "sine", prod([np.sin(np.pi * a / b) for a, b in zip(x, L)])
    yield "cut gaussian", prod([np.exp(-4.0 * (a - 0.1 * b) ** 2) for a, b in zip(x, L)])
    yield "constant", prod([np.ones_like(a) for a in x])


@pytest.mark.parametrize("Ns", [(64, 64), (250, 300), (512, 40), (1024, 64), (2048, 60), (4096, 32), (32, 4096), (8192, 6),
                                (20, 4200), (40, 33, 50), (256, 12, 9)])
def test_normwise_error_of_smooth_fields(frlap, Ns):
    import torch

    plan = frlap.Plan(len(Ns), 1.8, 2.0 / max(Ns), Ns, prec=frlap.FRLAP_F64)
    lam_max = float(plan.symbol().abs().max()) * float(np.prod([float(p) for p in plan.P]))
    for name, u in _fields(Ns):
        y = frlap.frlap_apply(plan, torch.from_numpy(u).cuda()).cpu().numpy()
        err = np.linalg.norm((y - _exact(plan, u)).astype(float)) / (lam_max * np.linalg.norm(u))
        print(f"{Ns} {name}: {err:.2e}")
        assert err <= 2.0 ** -53, (name, err)


def test_largest_poisson_problem_reaches_its_tolerance(frlap):
    """4095^2, alpha = 1.8, to 1e-10: the true residual's floor is the rounding of A x for the smooth solution, times
    up to lambda_max.  Native FP64 transforms reach 7.2e-11."""
    import torch

    N, alpha = 4096, 1.8
    Ns, h = (N, N), 2.0 / N
    f = torch.from_numpy(inp.gaussian_sum_field(Ns, h, seed=1)).cuda()
    plan = frlap.Plan(2, alpha, h, Ns, prec=frlap.FRLAP_DF64)
    frlap.frlap_precond_tau(plan)
    x, it, rel, code = frlap.frlap_pcg_solve(plan, f, rtol=1e-10, precond=frlap.FRLAP_PRECOND_TAU)
    assert code == 0 and rel <= 1e-10 and it <= 14
