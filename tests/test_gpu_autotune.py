"""The autotuner of the fixed-point stages times what later calls run: vectors that are not zero (a line of zeros takes
other branches), each launch shape once, and it reports the lines per CTA that are launched.
"""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,dt", [("F64", torch.float64), ("DF64", torch.float64), ("F32", torch.float32)])
def test_timed_on_vectors_that_are_not_zero(frlap, prec, dt):
    plan = frlap.Plan(2, 1.4, 2.0 / 100, (100, 70), prec=getattr(frlap, "FRLAP_" + prec))
    lib = frlap.lib()
    n = int(lib.frlap_autotune_workspace_bytes(plan.handle, 3))
    work = torch.zeros(n + 256, dtype=torch.uint8, device="cuda")
    work = work[(-work.data_ptr()) % 256:][:n]
    assert lib.frlap_plan_autotune(plan.handle, 3, ctypes.c_void_p(work.data_ptr()), None, None) == 0
    M = 99 * 69
    u = work.view(dt)[:3 * M].double()  # the vectors stand first in the workspace
    assert bool((u != 0).all()) and float(u.abs().max()) <= 1.0
    assert float(u.abs().mean()) > 0.4 and abs(float(u.mean())) < 0.02  # uniform: 0.5, 0 +- 0.004


@pytest.mark.parametrize("prec", ["F64", "DF64"])
def test_few_lines_report_the_fixed_choice(frlap, prec):
    """Two 99 x 69 vectors: all stages run four entries a thread, with the built-in lines per CTA: as many as 256
    threads hold, halved while the launch has fewer than 304 CTAs, in whole warps.  Row lines of 128 points take 32
    threads (138 of them: one a CTA), column lines of 256 points 64 (258: one)."""
    plan = frlap.Plan(2, 1.4, 2.0 / 100, (100, 70), prec=getattr(frlap, "FRLAP_" + prec))
    assert plan.P[0] == 256 and plan.P[1] == 256
    for _ in range(3):
        assert frlap.frlap_plan_autotune(plan, 2)[0][:3] == [1, 1, 1]
    # rows of 16 points (N = 12: 4 threads a line) need 8 lines for a warp
    plan = frlap.Plan(2, 1.4, 2.0 / 12, (12, 12), prec=getattr(frlap, "FRLAP_" + prec))
    assert plan.P[0] == 32
    for _ in range(3):
        assert frlap.frlap_plan_autotune(plan, 2)[0][:3] == [8, 4, 8]


def test_reported_choices_reproduce_themselves(frlap):
    """Eight entries a thread: the reported lines keep a CTA within 512 threads (a line of L points: L / 8)."""
    plan = frlap.Plan(2, 1.4, 2.0 / 250, (250, 250), prec=frlap.FRLAP_F64)
    c, _ = frlap.frlap_plan_autotune(plan, 8)
    for tl, L in zip(c[:3], (256, 512, 256)):
        assert 1 <= tl <= 512 // (L // 8)
