"""FP32 products in units far from one.  Density scaled by a and velocity by b
(pressure by a b^2, viscosity by a b) scale the product by b, variable by
variable; with powers of two every operation scales exactly unless something
leaves FP32's range on the way."""
import numpy as np
import pytest
import torch

import helpers as Hp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ea,eb", [(-66, 20), (74, -20), (0, -34), (0, 37)])
@pytest.mark.parametrize("flux", ["rusanov", "roe"])
@pytest.mark.parametrize("name", ["vortex2d_mixed_p1-4", "ns2d_mixed_p1-4", "tgv_5^3_p3"])
def test_product_in_scaled_units(name, flux, ea, eb):
    import cases
    m, q, ph = Hp.small_workloads()[name]
    a, b = 2.0 ** ea, 2.0 ** eb
    nv = m.nv
    scale = np.array([a] + [a * b] * m.nd + [a * b * b])
    q = Hp.generic_state(q).reshape(-1, nv)
    v = ((cases.uniform(711, q.size) - 0.5).reshape(-1, nv) * np.abs(q).max(0)).astype(np.float32).astype(np.float64)
    q = q.astype(np.float32).astype(np.float64)

    def product(s, mu, unscale):
        ctx = Hp.gpu_ctx(m, dict(ph, mu=mu, flux=flux))
        put = lambda x: ctx.pack(torch.from_numpy(np.ascontiguousarray(x * s).reshape(-1)).cuda(), torch.float32)
        return ctx.unpack(ctx.jvp(put(q), put(v))).cpu().numpy().reshape(-1, nv) / unscale

    ref = product(np.ones(nv), ph.get("mu", 0.0), np.ones(nv))
    got = product(scale, ph.get("mu", 0.0) * a * b, scale * b)
    err = np.abs(got - ref).max(0) / np.abs(ref).max(0)
    assert np.isfinite(got).all() and (err <= 2e-5).all(), err      # the suite's FP32 bound
