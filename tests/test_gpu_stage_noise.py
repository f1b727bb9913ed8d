"""A stage that starts near its solution, so that the double-float residual's
rounding noise is a large part of ||F0||: the iterates that no longer reduce
||F|| hand over to FP64 at once, and the stage converges within a small
iteration limit."""
import numpy as np
import pytest
import torch

import cases
import helpers as Hp

pytestmark = pytest.mark.gpu

DT = 0.1


@pytest.mark.parametrize("level,max_newton", [(20.0, 8), (20.0, 6), (200.0, 8)])
def test_noise_bound_stage_converges(level, max_newton):
    from paper_1910_03693_gb300.api import esdirk_tableau
    m, q, phys = cases.workload_tgv(6, 3)
    ctx = Hp.gpu_ctx(m, phys)
    A, _ = esdirk_tableau(3)
    qn = ctx.pack(torch.from_numpy(q).cuda())
    Rn = ctx.residual(qn)
    kw = dict(dtau_init=1e10, dtau_max=1e10, m=60, rtol=0.1, max_it=100)
    sol = qn.clone()
    assert ctx.esdirk_stage(A, 2, DT, qn, [Rn, None, None, None], sol, tol=1e-10, **kw)["converged"]
    # ||F|| grows linearly with the distance from the solution; the noise is the
    # difference of the two residuals there
    rhs = (qn + DT * A[1][0] * Rn) / (A[1][1] * DT)
    F = lambda x: rhs - x / (A[1][1] * DT) + ctx.residual(x)
    noise = float((ctx.residual(sol, double_float=True) - ctx.residual(sol)).norm())
    d = torch.from_numpy(cases.uniform(701, sol.numel()) - 0.5).cuda()
    d *= 1e-8 * float(sol.norm() / d.norm())
    start = sol + d * (level * noise / float((F(sol + d) - F(sol)).norm()))
    assert 0.5 * level * noise < float(F(start).norm()) < 2.0 * level * noise
    # a fifth of the noise: out of reach in double-float, six times the FP64
    # residual's own rounding (2^-53 against 2^-47, a factor of 30 at least)
    tol = 0.2 / level
    st = ctx.esdirk_stage(A, 2, DT, qn, [Rn, None, None, None], start.clone(), tol=tol, max_newton=max_newton,
                          low_above=1e-15, **kw)
    assert st["converged"] and st["norm_final"] <= tol * st["norm0"], st
    assert st["low_evaluations"] >= 2 and st["f64_evaluations"] >= 1, st
