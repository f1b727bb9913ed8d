"""The early Newton iterates of a stage stay in double-float arithmetic while
the pseudo-time ramp reduces ||F|| slowly, and a floor of the double-float
residual below the tolerance still hands over to FP64."""
import math

import numpy as np
import pytest
import torch

import cases
import helpers as Hp

pytestmark = pytest.mark.gpu


def _stage(ctx, q, tol, low_above, dt=0.01, **kw):
    from paper_1910_03693_gb300.api import esdirk_tableau
    A, b = esdirk_tableau(3)
    qn = ctx.pack(torch.from_numpy(q).cuda())
    qi = qn.clone()
    st = ctx.esdirk_stage(A, 2, dt, qn, [ctx.residual(qn), torch.empty_like(qn), None, None], qi, tol=tol,
                          dtau_init=dt / 10, dtau_max=dt, m=60, rtol=0.1, max_it=100, low_above=low_above, **kw)
    return qi, qn, st


def _flow():
    """Taylor-Green at Ma 0.1 with acoustic waves: the first iterates are slow."""
    m, q, phys = cases.workload_tgv(6, 3)
    X = np.concatenate(cases.solution_point_positions(m))
    Q = q.reshape(-1, 5).copy()
    wave = 0.002 * sum(math.cos(0.3 * k) * np.cos(X @ np.array(d) + k) for k, d in
                       enumerate([(3, 2, -1), (-4, 1, 5), (2, -5, 3), (5, 4, 2)]))
    Q[:, 4] *= 1 + wave
    Q[:, 0] *= 1 + 0.5 * wave
    return m, Q.reshape(-1), phys


def test_ramp_stays_double_float():
    m, q, phys = _flow()
    ctx = Hp.gpu_ctx(m, phys)
    low, qn, st = _stage(ctx, q, 1e-8, 1e-8)
    ref, _, st64 = _stage(ctx, q, 1e-8, 0.0)
    assert st["converged"] and st64["converged"] and st["norm_final"] <= 1e-8 * st["norm0"]
    assert st["f64_evaluations"] <= 2 and st["low_evaluations"] >= st["newton"], st
    # both are converged to 1e-8 of ||F||: their difference is a few 1e-8 of the stage's increment
    assert float((low - ref).norm()) <= 1e-7 * float((ref - qn).norm())


def test_double_float_floor_hands_over_to_fp64():
    m, q, phys = _flow()
    ctx = Hp.gpu_ctx(m, phys)
    # the double-float F cannot reach 1e-12 of ||F0|| at this Mach number; FP64 can
    _, _, st = _stage(ctx, q, 1e-12, 1e-15)
    assert st["converged"] and st["f64_evaluations"] >= 1 and st["norm_final"] <= 1e-12 * st["norm0"], st
