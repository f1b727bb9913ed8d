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


def test_noise_bound_step_converges():
    """The same in a whole step, where the noise is measured at q^n: a nearly
    uniform flow whose ||F0|| is 40 times the noise."""
    from paper_1910_03693_gb300.api import esdirk_tableau
    m = cases.workload_tgv(6, 3)[0]
    ctx = Hp.gpu_ctx(m, dict(gamma=1.4, mu=1.0 / 1600.0, Pr=0.71))
    flow = ctx.pack(torch.from_numpy(cases.freestream_state(m, mach=0.1, noise=0.0, seed=1)).cuda())
    d = torch.from_numpy(cases.uniform(702, flow.numel()) - 0.5).cuda() * flow.abs().mean()
    q = flow + 1e-12 * d
    # stage 2 starts from q^n with F0 = (1 + a_21 / a_22) R(q^n)
    noise = float((ctx.residual(q, double_float=True) - ctx.residual(q)).norm())
    A, b = esdirk_tableau(3)
    F0 = (1.0 + A[1][0] / A[1][1]) * float(ctx.residual(q).norm())
    q = flow + 1e-12 * (40.0 * noise / F0) * d
    st = ctx.esdirk_step(A, DT, q, b=b, tol=0.0125, dtau_init=1e10, dtau_max=1e10, m=60, rtol=0.1, max_it=100,
                         max_newton=8, low_above=1e-15)
    assert all(x["converged"] for x in st), st
    assert max(x["low_evaluations"] for x in st) >= 2, st


def test_ramp_of_a_step_stays_double_float():
    from paper_1910_03693_gb300.api import esdirk_tableau
    from test_gpu_stage_ramp import _flow
    m, q0, phys = _flow()
    ctx = Hp.gpu_ctx(m, phys)
    A, b = esdirk_tableau(3)
    out = []
    for low_above in (1e-8, 0.0):
        q = ctx.pack(torch.from_numpy(q0).cuda())
        qn = q.clone()
        st = ctx.esdirk_step(A, 0.01, q, b=b, tol=1e-8, dtau_init=1e-3, dtau_max=0.01, m=60, rtol=0.1, max_it=100,
                             low_above=low_above)
        assert all(x["converged"] for x in st), st
        out.append(q - qn)
        if low_above:       # FP64 only to certify
            assert all(x["f64_evaluations"] <= 2 and x["low_evaluations"] >= x["newton"] for x in st), st
    assert float((out[0] - out[1]).norm()) <= 1e-7 * float(out[1].norm())
