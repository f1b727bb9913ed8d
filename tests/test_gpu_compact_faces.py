"""Viscous boxes of axis-aligned elements: the residual, product and transposed
product from compact traces and the common gradient whose tangential part is taken from q^com, against the
oracle, for every degree, both fluxes, stretched boxes, and elements turned by
180 degrees (negative diagonal metrics, flipped orientation codes)."""
import numpy as np
import pytest
import torch

import cases
import helpers as Hp

pytestmark = pytest.mark.gpu


def _turned(m):
    """Every other element of a checkerboard turned by 180 degrees about zeta:
    xi and eta reversed, so that the faces across xi and eta trade places and
    tangential axes meet reversed."""
    n = round(m.n_elem ** (1 / 3))
    i = np.arange(m.n_elem)
    odd = (i % n + i // n % n + i // (n * n)) % 2 == 1
    nodes, nbr, nbr_face = m.nodes.copy(), m.nbr.copy(), m.nbr_face.copy()
    nodes[odd] = m.nodes[odd][:, [3, 2, 1, 0, 7, 6, 5, 4]]
    swap = np.array([1, 0, 3, 2, 4, 5])
    nbr[odd], nbr_face[odd] = nbr[odd][:, swap], nbr_face[odd][:, swap]
    # every neighbour has the other parity: its face index is mapped when it is turned
    there = odd[nbr]
    nbr_face = np.where(there, swap[nbr_face], nbr_face).astype(np.int8)
    orient = np.broadcast_to(np.array([2, 2, 2, 2, 6, 6], np.int8), nbr.shape).copy()
    out = cases.Mesh(3, 1, nodes, nbr, nbr_face, orient, m.p.copy(), "turned")
    cases.check_connectivity(out)
    return out


def _mesh(p, n, kind):
    m = cases.periodic_box(3, n, 0.0, 1.0, p)
    if kind == "stretched":
        m.nodes = m.nodes * np.array([1.0, 2.0, 0.5])
    return _turned(m) if kind == "turned" else m


@pytest.mark.parametrize("p,n,kind,flux", [(1, 1, "plain", "rusanov"), (1, 4, "plain", "roe"), (2, 3, "stretched", "rusanov"),
                                           (3, 3, "stretched", "roe"), (4, 2, "plain", "rusanov"), (5, 2, "plain", "roe"),
                                           (1, 4, "turned", "rusanov"), (2, 2, "turned", "roe"), (3, 2, "turned", "rusanov"),
                                           (4, 2, "turned", "rusanov")])
def test_against_oracle(p, n, kind, flux):
    from oracle import linearize as L
    m = _mesh(p, n, kind)
    phys = dict(gamma=1.4, mu=0.03, Pr=0.71, flux=flux)
    q = cases.random_state(m, 600 + p)
    fr, ctx = Hp.oracle_fr(m, phys), Hp.gpu_ctx(m, phys)
    qt = torch.from_numpy(q)
    v = torch.from_numpy((cases.uniform(610 + p, q.size) - 0.5) * np.abs(q).mean())
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
