"""Calls in flight on another stream while the context is rebucketed finish on
the layout that they were queued with: their outputs are those they give alone,
and the context then works on the new layout."""
import numpy as np
import pytest
import torch

import cases
import helpers as Hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["walls", "box"])
def test_rebucket_beside_work_in_flight(kind):
    if kind == "walls":                 # curved, mortars, boundary records
        m = cases.cylinder_ogrid(12, 24, 6, g=2, p=2)
        m.p = cases.smooth_random_p_field(m, 781, levels=(1, 2, 3, 1))
        q0 = cases.freestream_state(m, mach=0.2, noise=0.02, seed=782)
        phys = dict(gamma=1.4, mu=1e-2, Pr=0.71, q_inf=cases.free_stream_q(3, mach=0.2))
    else:                               # conforming: the neighbour table
        m = cases.periodic_box(3, 12, 0.0, 1.0, 2)
        q0, phys = cases.random_state(m, 783), dict(gamma=1.4, mu=0.01, Pr=0.71)
    ctx = Hp.gpu_ctx(m, phys, p_min=1, p_max=3)
    table = [0] * 42
    table[(1 * 3 + 2) * 7 + 1] = 1      # box: the FP32 product by the fused kernel, which reads it
    ctx.set_tuning({"epb": table})
    q = ctx.pack(torch.from_numpy(q0).cuda())
    v = ctx.pack(torch.from_numpy(cases.uniform(784, q0.size) - 0.5).cuda())
    q32, v32 = q.float(), v.float()
    calls = [lambda o: ctx.residual(q, out=o), lambda o: ctx.jvp(q, v, out=o), lambda o: ctx.vjp(q, v, out=o),
             lambda o: ctx.jvp(q32, v32, out=o), lambda o: ctx.unpack(q, out=o), lambda o: ctx.precond_apply(v, out=o)]
    like = [q, q, q, q32, q, q]
    ctx.precond_build(q, 1e4)
    alone = [torch.empty_like(x) for x in like]
    for fn, o in zip(calls, alone):
        fn(o)
    torch.cuda.synchronize()
    buf = ctx.empty(capacity=True)
    buf[:ctx.n_dof] = q
    eta = torch.from_numpy(cases.uniform(785, m.n_elem)).cuda()
    one = torch.ones(1, dtype=torch.float64, device="cuda")
    p_old = ctx.p_map()
    side, done = torch.cuda.Stream(), torch.cuda.Event()
    for step in range(2):               # the second change fills the tables that the first one released
        rounds = [[torch.full_like(x, float("nan")) for x in like] for _ in range(40)]
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            for outs in rounds:
                for fn, o in zip(calls, outs):
                    fn(o)
            done.record()
        assert not done.query()         # still running when the tables change
        ctx.rebucket(eta, one, buf, nu_max=0.7, nu_min=0.3, p_min=1, p_max=3)
        torch.cuda.synchronize()
        assert not np.array_equal(ctx.p_map(), p_old)
        for outs in rounds:
            for got, want in zip(outs, alone):
                assert torch.equal(got, want)
        m2 = m.with_p(ctx.p_map())
        new = Hp.gpu_ctx(m2, phys, p_min=1, p_max=3)
        qt = torch.from_numpy(cases.random_state(m2, 786)).cuda()
        q = ctx.pack(qt)
        v = torch.roll(q, 1)
        q32, v32 = q.float(), v.float()
        assert torch.equal(ctx.residual(q), new.residual(new.pack(qt)))
        assert torch.equal(ctx.vjp(q, v), new.vjp(q, v))
        like = [q, q, q, q32, q, q]
        ctx.precond_build(q, 1e4)
        alone = [torch.empty_like(x) for x in like]
        for fn, o in zip(calls, alone):
            fn(o)
        torch.cuda.synchronize()
        p_old = ctx.p_map()
        buf[:ctx.n_dof] = q
        eta = eta.flip(0)
