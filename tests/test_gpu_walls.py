"""F64 applies of vectors that one grid line, or one point, dominates: lines across it have exponents far above the
values of the others, which must not cost the others their bits.

Reference: the same product in long double from the plan's own symbol.  Bound, normwise over lambda_max ||u||: a line's
rounding unit is 2^-58 of its largest value; 0.6 of it in each of at most five stages, over the sqrt(L) <= 2^6 bins of a
line with a single peak: 5 * 0.6 * 2^6 * 2^-58 = 3 * 2^-52.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _exact(plan, u):
    import scipy.fft as sf

    P = [int(p) for p in plan.P][:u.ndim][::-1]
    lam = plan.symbol().cpu().numpy().astype(np.longdouble)
    for ax in range(u.ndim - 1):
        lam = np.concatenate([lam, np.flip(np.take(lam, range(1, lam.shape[ax] - 1), axis=ax), axis=ax)], axis=ax)
    U = np.zeros(P, dtype=np.longdouble)
    box = tuple(slice(0, n) for n in u.shape)
    U[box] = u
    scale = np.longdouble(1)
    for p in P:
        scale *= p
    return sf.irfftn(sf.rfftn(U, workers=8) * lam * scale, s=P, workers=8)[box]


@pytest.mark.parametrize("alpha", [0.5, 1.8])
@pytest.mark.parametrize("Ns", [(64, 40), (300, 500), (512, 100), (1024, 64), (2048, 300), (60, 2048), (33, 20, 17),
                                (20, 130, 40)])
def test_walls_and_spikes(frlap, Ns, alpha):
    import torch

    plan = frlap.Plan(len(Ns), alpha, 2.0 / max(Ns), Ns, prec=frlap.FRLAP_F64)
    lam_max = float(plan.symbol().abs().max()) * float(np.prod([float(p) for p in plan.P]))
    rng = np.random.default_rng(8)
    shape = plan.shape
    for noise in (0.0, 1e-3):
        for where in (["axis", ax] for ax in range(len(shape))), (["point", 0], ["point", 3]):
            for kind, at in where:
                u = noise * rng.standard_normal(shape)
                if kind == "axis":
                    index = [slice(None)] * len(shape)
                    index[at] = shape[at] // 3
                else:
                    index = [n * at // 10 for n in shape]
                u[tuple(index)] += 1.0
                y = frlap.frlap_apply(plan, torch.from_numpy(u).cuda()).cpu().numpy()
                err = np.linalg.norm((y - _exact(plan, u)).astype(float)) / (lam_max * np.linalg.norm(u))
                assert err <= 3 * 2.0 ** -52, (noise, kind, at, err)
