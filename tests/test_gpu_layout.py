"""The layout built on the device: several blocks of the element and face sorts,
mixed degrees with walls and far field, and a context that reached its degrees
by rebucketing against one created with them."""
import numpy as np
import pytest
import torch

import cases
import helpers as Hp

pytestmark = pytest.mark.gpu


def test_many_blocks_against_oracle():
    m = cases.cylinder_ogrid(12, 24, 5, g=2, p=1)          # 1,440 elements: two sort blocks, 34 face blocks
    m.p = cases.smooth_random_p_field(m, 401, levels=(1, 2, 3, 1))
    q = cases.freestream_state(m, mach=0.2, noise=0.02, seed=402)
    phys = dict(gamma=1.4, mu=1e-2, Pr=0.71, q_inf=cases.free_stream_q(3, mach=0.2))
    fr, ctx = Hp.oracle_fr(m, phys), Hp.gpu_ctx(m, phys)
    qt = torch.from_numpy(q)
    qd = ctx.pack(qt.cuda())
    assert torch.equal(ctx.unpack(qd).cpu(), qt)
    R = ctx.unpack(ctx.residual(qd)).cpu().numpy()
    ok = Hp.parity_ok(R, fr.residual(qt).numpy(), m, q, 1e-11)   # the suite's bound on curved meshes
    assert ok[0], ok


@pytest.mark.parametrize("nd,n", [(2, 1), (2, 45), (3, 2), (3, 12)])
def test_rebucketed_equals_created(nd, n):
    from oracle import adapt as A
    m = cases.periodic_box(nd, n, 0.0, 1.0, 2)
    phys = dict(gamma=1.4, mu=0.01, Pr=0.71)
    ctx = Hp.gpu_ctx(m, phys, p_min=1, p_max=4)
    eta = cases.uniform(403, m.n_elem)
    eta[eta > 0.9] = 1.0
    eta[0] = 1.0
    buf = ctx.empty(capacity=True)
    buf[:ctx.n_dof] = ctx.pack(torch.from_numpy(cases.random_state(m, 404)).cuda())
    perm = torch.empty(m.n_elem, dtype=torch.int32, device="cuda")
    p = m.p.astype(np.int64)
    for nu_max, nu_min in ((0.9, 0.3), (0.8, 0.6), (0.2, 0.0)):
        ctx.rebucket(torch.from_numpy(eta).cuda(), torch.ones(1, dtype=torch.float64, device="cuda"), buf,
                     nu_max=nu_max, nu_min=nu_min, p_min=1, p_max=4, perm=perm)
        p = A.limit_jumps(m, A.decide(eta, p, nu_max, nu_min, 1, 4))
        assert np.array_equal(ctx.p_map(), p)
        assert np.array_equal(perm.cpu().numpy(), A.bucket_order(p))
        m2 = m.with_p(p)
        new = Hp.gpu_ctx(m2, phys, p_min=1, p_max=4)
        q = torch.from_numpy(cases.random_state(m2, 405)).cuda()
        v = torch.from_numpy(cases.uniform(406, q.numel()) - 0.5).cuda()
        got, ref = ctx.pack(q), new.pack(q)
        assert torch.equal(got, ref) and torch.equal(ctx.unpack(got), q)
        assert torch.equal(ctx.residual(got), new.residual(ref))
        assert torch.equal(ctx.jvp(got, ctx.pack(v)), new.jvp(ref, new.pack(v)))
        assert torch.equal(ctx.vjp(got, ctx.pack(v)), new.vjp(ref, new.pack(v)))
