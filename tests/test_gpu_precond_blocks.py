"""Inverted element blocks of every size (2D and 3D, p = 1..5, and all degrees of
a mesh in one apply): the residual B z - w of z = M^-1 w with the dense blocks B
read off the FP64 product."""
import numpy as np
import pytest
import torch

import cases
import helpers as Hp

pytestmark = pytest.mark.gpu


def _check(m, phys, elements):
    ctx = Hp.gpu_ctx(m, phys)
    q = torch.from_numpy(cases.random_state(m, 501)).cuda()
    qs = ctx.pack(q)
    sigma = 40.0 * float(ctx.jvp(qs, torch.ones_like(qs)).abs().max()) / float(qs.abs().mean())
    ctx.precond_build(qs, sigma)
    w = ctx.pack(torch.from_numpy(cases.uniform(502, ctx.n_dof) - 0.5).cuda())
    z = ctx.precond_apply(w)
    assert torch.equal(ctx.precond_apply(w.clone(), out=w.clone()), z)
    order = np.lexsort((np.arange(m.n_elem), m.p))
    sizes = (m.p[order].astype(int) + 1) ** m.nd * (m.nd + 2)
    off = np.concatenate([[0], np.cumsum(sizes)])
    for e in elements:
        s = int(np.nonzero(order == e)[0][0])
        a, b = int(off[s]), int(off[s + 1])
        B = torch.empty(b - a, b - a, dtype=torch.float64, device="cuda")
        u = torch.zeros_like(qs)
        for k in range(b - a):
            u.zero_()
            u[a + k] = 1.0
            B[:, k] = -ctx.jvp(qs, u)[a:b]
        B += sigma * torch.eye(b - a, dtype=torch.float64, device="cuda")
        # backward error: elimination with partial pivoting in FP32 (n u a row, a
        # growth of 4), and blocks of the FP32 product (2e-5, the suite's bound)
        res = (B @ z[a:b] - w[a:b]).abs().max()
        bound = (4 * (b - a) * 2.0 ** -24 + 2e-5) * B.abs().sum(1).max() * z[a:b].abs().max()
        assert float(res) <= float(bound), (e, int(m.p[e]), float(res), float(bound))

@pytest.mark.parametrize("nd,p", [(2, 1), (2, 2), (2, 3), (2, 4), (2, 5), (3, 1), (3, 2), (3, 3), (3, 4), (3, 5)])
def test_blocks_of_every_size(nd, p):
    m = cases.periodic_box(nd, 3 if nd == 2 else 2, 0.0, 1.0, p)
    _check(m, dict(gamma=1.4, mu=0.02, Pr=0.71), [0, m.n_elem - 1])


def test_blocks_of_mixed_degrees():
    m = cases.periodic_box(3, 3, 0.0, 1.0, 1)
    m = m.with_p((1 + np.floor(cases.uniform(503, m.n_elem) * 4)).astype(np.int8))
    first = [int(np.nonzero(m.p == p)[0][0]) for p in range(1, 5)]
    _check(m, dict(gamma=1.4, mu=0.02, Pr=0.71), first + [m.n_elem - 1])

