"""Axis-aligned elements whose paired faces do not have the same tangential
metric: layers of different extent glued to each other, faces of different axes
glued together, tangential axes exchanged or reflected across a face.  The
connectivity is symmetric, so the meshes are accepted; both sides' gradients
count, as in the oracle, in every precision and with either kernel set."""
import numpy as np
import pytest
import torch

import cases
import helpers as Hp

pytestmark = pytest.mark.gpu


def _mesh(kind, p):
    m = cases.periodic_box(3, 2 if kind != "layers" else 3, 0.0, 1.0, p)
    if kind == "layers":          # the y extent differs from one x layer to the next
        layer = np.arange(m.n_elem) % 3
        m.nodes = m.nodes.copy()
        m.nodes[..., 1] *= np.array([1.0, 1.5, 0.75])[layer][:, None]
    elif kind == "axes":          # across the box's sides, x- meets y+ and x+ meets y-
        for j in range(2):
            for k in range(2):
                for x, f, y, g in ((0, 0, 1, 3), (1, 1, 0, 2)):
                    e, n = x + 2 * j + 4 * k, j + 2 * y + 4 * k
                    m.nbr[e, f], m.nbr_face[e, f] = n, g
                    m.nbr[n, g], m.nbr_face[n, g] = e, f
    elif kind == "swapped":       # elements twice as long in y; x and y trade places across the faces normal to z
        m.nodes = m.nodes * np.array([1.0, 2.0, 1.0])
        m.orient = m.orient.copy()
        m.orient[:, 4:] = 1
    else:                         # reflected: y reversed across every face normal to z
        m.orient = m.orient.copy()
        m.orient[:, 4:] = 4
    cases.check_connectivity(m)
    return m


@pytest.mark.parametrize("p", [1, 3])
@pytest.mark.parametrize("kind", ["layers", "axes", "swapped", "reflected"])
def test_against_oracle(kind, p):
    from oracle import linearize as L
    m = _mesh(kind, p)
    phys = dict(gamma=1.4, mu=0.03, Pr=0.71)
    q = cases.random_state(m, 720 + p)
    fr, ctx = Hp.oracle_fr(m, phys), Hp.gpu_ctx(m, phys)
    qt = torch.from_numpy(q)
    v = torch.from_numpy((cases.uniform(730 + p, q.size) - 0.5) * np.abs(q).mean())
    qs, vs = ctx.pack(qt.cuda()), ctx.pack(v.cuda())
    R, J, A = fr.residual(qt).numpy(), L.jvp(fr, qt, v).numpy(), L.vjp(fr, qt, v).numpy()
    get = lambda t: ctx.unpack(t).cpu().numpy()
    # the suite's bounds: FP64 1e-12, double-float 2e-10, FP32 2e-5
    for gpu, ref, tol in ((ctx.residual(qs), R, 1e-12), (ctx.residual(qs, double_float=True), R, 2e-10),
                          (ctx.jvp(qs, vs), J, 1e-12), (ctx.residual(qs.float()), R, 2e-5),
                          (ctx.jvp(qs.float(), vs.float()), J, 2e-5), (ctx.vjp(qs, vs), A, 1e-12),
                          (ctx.vjp(qs.float(), vs.float()), A, 2e-5)):
        ok = Hp.parity_ok(get(gpu), ref, m, q, tol)
        assert ok[0], ok
