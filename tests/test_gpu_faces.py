"""The one-launch face pass: every degree pair of 1..5 (mortars across jumps of
up to four degrees), walls and far field in the same launch as interior faces,
against the oracle; the smallest meshes, whose CTAs hold one face or element."""
import numpy as np
import pytest
import torch

import cases
import helpers as Hp

pytestmark = pytest.mark.gpu


def _mesh(kind):
    if kind == "box3d_all_pairs":
        m = cases.periodic_box(3, 3, 0.0, 1.0, 1)
        p = 1 + np.floor(cases.uniform(301, m.n_elem) * 5)
        phys = dict(gamma=1.4, mu=0.02, Pr=0.71)
    elif kind == "quads_all_pairs":
        m = cases.periodic_box(2, 9, 0.0, 1.0, 1, jitter_frac=0.1, seed=3)
        p = 1 + np.floor(cases.uniform(302, m.n_elem) * 5)
        phys = dict(gamma=1.4, mu=0.02, Pr=0.71, flux="roe")
    elif kind == "ogrid_all_pairs":
        m = cases.cylinder_ogrid(3, 8, 2, g=2, p=2)
        p = 1 + np.floor(cases.uniform(303, m.n_elem) * 5)
        phys = dict(gamma=1.4, mu=1e-2, Pr=0.71, q_inf=cases.free_stream_q(3, mach=0.2))
    elif kind == "euler_pairs":
        m = cases.periodic_box(3, 3, 0.0, 1.0, 1)
        p = 1 + np.floor(cases.uniform(304, m.n_elem) * 4)
        phys = dict(gamma=1.4, mu=0.0, Pr=0.71)
    else:   # two elements a direction: each pair of neighbours shares two faces
        m = cases.periodic_box(2, 2, 0.0, 1.0, 1)
        p = np.array([1, 2, 5, 3])
        phys = dict(gamma=1.4, mu=0.02, Pr=0.71)
    m = m.with_p(p.astype(np.int8))
    return m, cases.random_state(m, 305), phys


@pytest.mark.parametrize("kind", ["box3d_all_pairs", "quads_all_pairs", "ogrid_all_pairs", "euler_pairs", "quads_2x2"])
def test_all_degree_pairs_against_oracle(kind):
    from oracle import linearize as L
    m, q, phys = _mesh(kind)
    fr, ctx = Hp.oracle_fr(m, phys), Hp.gpu_ctx(m, phys)
    qt, scale = torch.from_numpy(q), np.abs(q).mean()
    v = torch.from_numpy((cases.uniform(306, q.size) - 0.5) * scale)
    w = torch.from_numpy((cases.uniform(307, q.size) - 0.5) * scale)
    R, J, A = fr.residual(qt).numpy(), L.jvp(fr, qt, v).numpy(), L.vjp(fr, qt, w).numpy()
    qd, vd, wd = ctx.pack(qt.cuda()), ctx.pack(v.cuda()), ctx.pack(w.cuda())
    # the suite's bounds: 1e-12 of the result, 1e-11 on curved meshes (metrics
    # computed independently on both sides), 2e-5 in FP32
    tol = 1e-11 if kind == "ogrid_all_pairs" else 1e-12
    get = lambda t: ctx.unpack(t).cpu().numpy()
    for gpu, ref in ((ctx.residual(qd), R), (ctx.jvp(qd, vd), J), (ctx.vjp(qd, wd), A)):
        ok = Hp.parity_ok(get(gpu), ref, m, q, tol)
        assert ok[0], ok
    # double-float (48 bits): the suite's 2e-10, 2e-9 on curved meshes
    ok = Hp.parity_ok(get(ctx.residual(qd, double_float=True)), R, m, q, 2e-9 if kind == "ogrid_all_pairs" else 2e-10)
    assert ok[0], ok
    q32 = qd.float()
    for gpu, ref in ((ctx.residual(q32), R), (ctx.jvp(q32, vd.float()), J), (ctx.vjp(q32, wd.float()), A)):
        ok = Hp.parity_ok(get(gpu), ref, m, q, 2e-5)
        assert ok[0], ok
