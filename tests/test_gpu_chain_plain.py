"""Kernels scheduled while their predecessor drains give what plain launches
give.  Launches captured into a graph are plain, so its replay is the reference;
the small meshes run the branch of grids with at most one CTA an SM, the large
ones that of grids of several waves, where a kernel's CTAs share SMs with the
predecessor's last wave."""
import numpy as np
import pytest
import torch

import cases
from helpers import generic_state, gpu_ctx, small_workloads

pytestmark = pytest.mark.gpu


def _large(name):
    if name == "tgv_20^3_p3":          # 512,000 points, one degree, compact passes
        return cases.workload_tgv(20, 3)
    if name == "quads_200^2_p1-4":     # 400,000 points, mortars, multi-degree launches
        m, _, ph = cases.workload_vortex2d(200, 2)
        m = m.with_p(cases.smooth_random_p_field(m, 751))
        return m, cases.random_state(m, 752), dict(ph, mu=0.02)
    m = cases.cylinder_ogrid(24, 48, 16, g=2, p=2)      # 675,000 points, curved, walls, mortars
    m.p = cases.smooth_random_p_field(m, 753)
    return m, cases.freestream_state(m, mach=0.2, noise=0.02, seed=754), dict(
        gamma=1.4, mu=1e-2, Pr=0.71, q_inf=cases.free_stream_q(3, mach=0.2))


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("name", ["vortex2d_mixed_p1-4", "cylinder_4x12x2_mixed", "tgv_20^3_p3", "quads_200^2_p1-4",
                                  "ogrid_24x48x16_p1-4"])
def test_chained_equals_plain(name, dtype):
    m, q0, ph = small_workloads()[name] if name in ("vortex2d_mixed_p1-4", "cylinder_4x12x2_mixed") else _large(name)
    ctx = gpu_ctx(m, ph)
    qs = [ctx.pack(torch.from_numpy(generic_state(q0, seed=760 + k)).cuda(), dtype) for k in range(3)]
    df = dtype == torch.float64
    q, v = qs[0].clone(), qs[1].clone()
    out = [torch.zeros_like(q) for _ in range(3 if df else 2)]

    def evaluate():
        ctx.residual(q, out=out[0])
        ctx.jvp(q, v, out=out[1])
        if df:
            ctx.residual(q, out=out[2], double_float=True)

    evaluate()                          # workspaces
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        evaluate()
    plain = []
    for k in range(3):
        q.copy_(qs[k])
        v.copy_(qs[(k + 1) % 3])
        g.replay()
        torch.cuda.synchronize()
        plain.append([x.clone() for x in out])
    got = [[torch.full_like(x, float("nan")) for x in out] for _ in range(9)]
    for i in range(9):                  # back to back, nothing synchronised
        q.copy_(qs[i % 3])
        v.copy_(qs[(i + 1) % 3])
        evaluate()
        for dst, x in zip(got[i], out):
            dst.copy_(x)
    torch.cuda.synchronize()
    for i in range(9):
        for x, y in zip(got[i], plain[i % 3]):
            assert torch.equal(x, y), (i, float((x - y).abs().max()))
