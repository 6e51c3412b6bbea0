"""The FP64 engine's block fixed-point transforms: accuracy, exact scaling, zeros and non-finite values.

The reference is the defining sum y_i = -c sum_j a_|i-j| u_j (eqs. A-2D / A-3D) in extended precision, at
sampled rows, so it shares no transform with the library.  Tolerance, per entry, for i.i.d. N(0,1) input:
2^-49 lambda_max.  An FP64 FFT product of such a vector (rms 1) has an entrywise error of about
2^-53 sqrt(2 log2(prod P)) <= 2^-50.5 lambda_max in the mean square; the fixed-point unit is 2^-58 of a
line's largest value, below that, and the factor 2^1.5 covers the largest of 40 samples.
"""
import numpy as np
import pytest

import frlap_inputs as inp

pytestmark = pytest.mark.gpu

# every transform length the plans admit, on rows and on columns, with ragged ends; 3D with its y and z lines
SHAPES = [(32, 32), (17, 40), (40, 17), (100, 70), (130, 9), (9, 130), (300, 257), (256, 513), (600, 12), (12, 600),
          (1025, 5), (5, 1025), (2049, 6), (6, 2049), (4097, 3), (3, 4097), (2, 2),
          (12, 7, 9), (33, 9, 17), (5, 70, 6), (6, 5, 130), (40, 40, 40), (3, 300, 4)]


def _operator(fl, Ns, alpha, prec):
    from oracle import scheme

    d, N = len(Ns), max(Ns)
    h = 2.0 / N
    coef = fl.frlap_coeffs(d, alpha, 2.0, h, Ns).cpu().numpy()
    plan = fl.Plan(d, alpha, h, Ns, prec=prec)
    lam_max = float(plan.symbol().abs().max()) * float(np.prod([float(p) for p in plan.P]))
    return plan, coef, scheme.c_d_alpha(d, alpha), lam_max


@pytest.mark.parametrize("Ns", SHAPES)
def test_entries_against_the_defining_sum(frlap, Ns):
    import torch

    plan, coef, c, lam_max = _operator(frlap, Ns, 1.3, frlap.FRLAP_F64)
    u = inp.normal_field(Ns, seed=11)
    y = frlap.frlap_apply(plan, torch.from_numpy(u).cuda()).cpu().numpy()
    rng = np.random.default_rng(3)
    ul = u.astype(np.longdouble)
    grids = [np.arange(n) for n in u.shape]
    worst = 0.0
    for _ in range(40):
        i = [int(rng.integers(n)) for n in u.shape]
        a = coef[np.ix_(*[np.abs(g - k) for g, k in zip(grids, i)])]
        ref = -np.longdouble(c) * np.sum(a.astype(np.longdouble) * ul)
        worst = max(worst, abs(float(y[tuple(i)] - ref)))
    assert worst < 2.0 ** -49 * lam_max, (worst / lam_max)


@pytest.mark.parametrize("Ns", [(100, 70), (600, 40), (12, 40, 9)])
@pytest.mark.parametrize("e", [-960, -40, 900])
def test_scaling_by_a_power_of_two_is_exact(frlap, Ns, e):
    """Fixed point with an exponent per line: 2^e u gives the same integers, so 2^e y exactly."""
    import torch

    plan, _, _, _ = _operator(frlap, Ns, 1.3, frlap.FRLAP_F64)
    u = torch.from_numpy(inp.normal_field(Ns, seed=5)).cuda()
    y = frlap.frlap_apply(plan, u)
    ys = frlap.frlap_apply(plan, u * 2.0 ** e)  # (torch.ldexp on the GPU takes an inexact power)
    assert torch.equal(ys, y * 2.0 ** e)


def test_rows_of_very_different_scales(frlap):
    """Rows between 1e-120 and 1: every row's error stays relative to the whole vector, and the product is
    that of the sum of the parts."""
    import torch

    Ns = (70, 100)
    plan, coef, c, lam_max = _operator(frlap, Ns, 0.8, frlap.FRLAP_F64)
    u = inp.normal_field(Ns, seed=7)
    u *= 10.0 ** -np.linspace(0, 120, u.shape[0])[:, None]
    u[10] = 0.0
    y = frlap.frlap_apply(plan, torch.from_numpy(u).cuda()).cpu().numpy()
    ul = u.astype(np.longdouble)
    grids = [np.arange(n) for n in u.shape]
    for i in [(0, 0), (1, 40), (10, 3), (50, 68), (98, 20)]:
        a = coef[np.ix_(*[np.abs(g - k) for g, k in zip(grids, i)])]
        ref = -np.longdouble(c) * np.sum(a.astype(np.longdouble) * ul)
        assert abs(float(y[i] - ref)) < 2.0 ** -49 * lam_max


@pytest.mark.parametrize("Ns", [(100, 70), (12, 40, 9)])
def test_zero_and_non_finite_inputs(frlap, Ns):
    import torch

    plan, _, _, _ = _operator(frlap, Ns, 1.1, frlap.FRLAP_F64)
    u = torch.zeros(plan.shape, dtype=torch.float64, device="cuda")
    assert torch.equal(frlap.frlap_apply(plan, u), u)
    for bad in (float("nan"), float("inf"), -float("inf")):
        v = u.clone()
        v.view(-1)[plan.M // 2] = bad
        assert bool(torch.isnan(frlap.frlap_apply(plan, v)).all())
    tiny = torch.full(plan.shape, 5e-324, dtype=torch.float64, device="cuda")
    assert bool(torch.isfinite(frlap.frlap_apply(plan, tiny)).all())


def test_split_middle_stage(frlap):
    """A 16384-point y embedding (two half-length transforms), against the defining sum at sampled rows."""
    import torch

    Ns = (6, 4200)
    plan, coef, c, lam_max = _operator(frlap, Ns, 1.3, frlap.FRLAP_F64)
    assert plan.P[1] == 16384
    u = inp.normal_field(Ns, seed=2)
    y = frlap.frlap_apply(plan, torch.from_numpy(u).cuda()).cpu().numpy()
    ul = u.astype(np.longdouble)
    grids = [np.arange(n) for n in u.shape]
    for i in [(0, 0), (17, 4), (2100, 2), (4095, 0), (4096, 1), (4198, 4)]:
        a = coef[np.ix_(*[np.abs(g - k) for g, k in zip(grids, i)])]
        ref = -np.longdouble(c) * np.sum(a.astype(np.longdouble) * ul)
        assert abs(float(y[i] - ref)) < 2.0 ** -49 * lam_max


@pytest.mark.parametrize("Ns", SHAPES)
def test_df64_first_stage_entries(frlap, Ns):
    """The DF64 engine's first stage, whose scale is set once per row.  With L points in a row (P <= 8192) its
    unit after the last butterfly is 2^-60 L max|u|, and back on the grid that is sqrt(L) 2^-60 max|u| lambda_max
    in the mean square: 2^-51.2 lambda_max at L = 8192 and max|u| = 5, three times that for the largest of 40
    samples.  Beside the other stages' 2^-49 the bound is 2^-48 lambda_max."""
    import torch

    plan, coef, c, lam_max = _operator(frlap, Ns, 1.3, frlap.FRLAP_DF64)
    u = inp.normal_field(Ns, seed=13)
    B = 3  # a batch: its last CTA's rows are ragged
    us = torch.stack([torch.from_numpy(u).cuda() * s for s in (1.0, 0.0, 2.0 ** -70)])
    ys = frlap.frlap_apply_batch(plan, us).cpu().numpy()
    assert ys.shape[0] == B and not ys[1].any()
    assert np.array_equal(ys[2], ys[0] * 2.0 ** -70)
    rng = np.random.default_rng(4)
    ul = u.astype(np.longdouble)
    grids = [np.arange(n) for n in u.shape]
    for _ in range(40):
        i = [int(rng.integers(n)) for n in u.shape]
        a = coef[np.ix_(*[np.abs(g - k) for g, k in zip(grids, i)])]
        ref = -np.longdouble(c) * np.sum(a.astype(np.longdouble) * ul)
        assert abs(float(ys[0][tuple(i)] - ref)) < 2.0 ** -48 * lam_max


@pytest.mark.parametrize("prec,bound", [("f64", 2.0 ** -49), ("df64", 2.0 ** -48)])
@pytest.mark.parametrize("Ns", [(16, 52, 52), (32, 52, 52), (64, 40, 40), (128, 40, 40), (256, 300), (64, 609),
                                (64, 610), (40, 16, 40), (40, 40, 16), (16, 40, 130), (9, 600), (100, 512),
                                (30, 512), (100, 200), (250, 250), (12, 40, 40)])
def test_four_eight_and_sixteen_entries_a_thread(frlap, Ns, prec, bound):
    """Plans of few lines give a thread four or eight entries, others sixteen (the first edge, 2432 threads at
    sixteen: 608 and 609 rows of 64 points): against the defining sum at the bounds above, and a batch of 9 bit for
    bit its vectors' applies."""
    import torch

    plan, coef, c, lam_max = _operator(frlap, Ns, 1.3, getattr(frlap, "FRLAP_" + prec.upper()))
    us = torch.from_numpy(np.stack([inp.normal_field(Ns, seed=s) for s in range(9)])).cuda()
    ys = frlap.frlap_apply_batch(plan, us)
    for u, y in zip(us, ys):
        assert torch.equal(y, frlap.frlap_apply(plan, u.clone()))
    ul, y = us[0].cpu().numpy().astype(np.longdouble), ys[0].cpu().numpy()
    rng = np.random.default_rng(5)
    grids = [np.arange(k) for k in ul.shape]
    for _ in range(40):
        i = [int(rng.integers(k)) for k in ul.shape]
        a = coef[np.ix_(*[np.abs(g - k) for g, k in zip(grids, i)])]
        ref = -np.longdouble(c) * np.sum(a.astype(np.longdouble) * ul)
        assert abs(float(y[tuple(i)] - ref)) < bound * lam_max
