"""The device's element and face sorts beyond one group of 32 blocks (32,768
elements, 8,192 element faces), against the order formed on the host; and the
preconditioner's blocks probed on one stream (capacities above two
full-occupancy waves of points) against the same blocks probed on four."""
import numpy as np
import pytest
import torch

import cases
import helpers as Hp

pytestmark = pytest.mark.gpu


def _state_order(m, canon):
    """The (p, id)-ordered state of a canonical vector, formed on the host."""
    off = m.offsets()
    parts = []
    for p in sorted(set(m.p.tolist())):
        e = np.nonzero(m.p == p)[0]
        n = (p + 1) ** m.nd
        ix = off[e][:, None, None] + np.arange(n)[None, None, :] * m.nv + np.arange(m.nv)[None, :, None]
        parts.append(canon[ix].reshape(-1))
    return np.concatenate(parts)


def test_sort_carries_across_groups():
    from oracle import adapt as A
    n = 190                             # 36,100 elements: 36 sort blocks, 565 face blocks
    m = cases.periodic_box(2, n, 0.0, 1.0, 1)
    m = m.with_p((1 + np.floor(cases.uniform(771, m.n_elem) * 3)).astype(np.int8))
    phys = dict(gamma=1.4, mu=0.01, Pr=0.71)
    ctx = Hp.gpu_ctx(m, phys, p_min=1, p_max=3)
    canon = cases.random_state(m, 772)
    buf = ctx.empty(capacity=True)
    buf[:ctx.n_dof] = ctx.pack(torch.from_numpy(canon).cuda())
    assert np.array_equal(buf[:ctx.n_dof].cpu().numpy(), _state_order(m, canon))
    eta = cases.uniform(773, m.n_elem)
    eta[0] = 1.0
    perm = torch.empty(m.n_elem, dtype=torch.int32, device="cuda")
    ctx.rebucket(torch.from_numpy(eta).cuda(), torch.ones(1, dtype=torch.float64, device="cuda"), buf,
                 nu_max=0.8, nu_min=0.4, p_min=1, p_max=3, perm=perm)
    p = A.limit_jumps(m, A.decide(eta, m.p.astype(np.int64), 0.8, 0.4, 1, 3))
    assert np.array_equal(ctx.p_map(), p) and np.array_equal(perm.cpu().numpy(), A.bucket_order(p))
    m2 = m.with_p(p)
    canon = cases.random_state(m2, 774)
    qt = torch.from_numpy(canon).cuda()
    q = ctx.pack(qt)
    assert np.array_equal(q.cpu().numpy(), _state_order(m2, canon)) and torch.equal(ctx.unpack(q), qt)
    # the face records: against a context created with these degrees, and the oracle
    new = Hp.gpu_ctx(m2, phys, p_min=1, p_max=3)
    assert torch.equal(ctx.residual(q), new.residual(new.pack(qt)))
    ok = Hp.parity_ok(ctx.unpack(ctx.residual(q)).cpu().numpy(), Hp.oracle_fr(m2, phys).residual(qt.cpu()).numpy(),
                      m2, canon, 1e-12)
    assert ok[0], ok


def test_blocks_probed_on_one_stream():
    m = cases.periodic_box(3, 15, 0.0, 1.0, 1)          # 3,375 elements: 729,000 points at p_max = 5
    phys = dict(gamma=1.4, mu=0.02, Pr=0.71)
    z = []
    for p_max in (1, 5):
        ctx = Hp.gpu_ctx(m, phys, p_min=1, p_max=p_max)
        q = ctx.pack(torch.from_numpy(cases.random_state(m, 775)).cuda())
        w = ctx.pack(torch.from_numpy(cases.uniform(776, ctx.n_dof) - 0.5).cuda())
        ctx.precond_build(q, 5e3)
        z.append(ctx.precond_apply(w))
    assert torch.isfinite(z[0]).all() and torch.equal(z[0], z[1])
