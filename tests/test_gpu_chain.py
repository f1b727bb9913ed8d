"""GPU: kernels of one stream that are scheduled while their predecessor drains
wait for its end before they touch memory.  Evaluations enqueued back to back,
with the input overwritten in place between them and nothing synchronised, give
bit for bit what each gives alone: the arithmetic of every point is the same."""
import pytest
import torch

from helpers import generic_state, gpu_ctx, small_workloads

pytestmark = pytest.mark.gpu

NAMES = ["vortex2d_mixed_p1-4", "ns2d_mixed_p1-4", "box_curved_mixed_p1-3", "tgv_5^3_p3", "diff_3^3_p4_mu0.05",
         "cylinder_4x12x2_mixed", "vortex_batch_5"]


@pytest.fixture(scope="module")
def works():
    from paper_1910_03693_gb300 import build as B
    B.build()
    return small_workloads()


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("name", NAMES)
def test_back_to_back_evaluations_match_alone(works, name, dtype):
    m, q0, ph = works[name]
    ctx = gpu_ctx(m, ph)
    qs = [ctx.pack(torch.from_numpy(generic_state(q0, seed=400 + k)).cuda(), dtype) for k in range(4)]

    def evaluate(q, v):
        return ctx.residual(q), ctx.jvp(q, v)

    alone = []
    for k in range(4):
        torch.cuda.synchronize()
        alone.append([x.clone() for x in evaluate(qs[k], qs[(k + 1) % 4])])
        torch.cuda.synchronize()
    q, v = qs[0].clone(), qs[1].clone()
    outs = [[torch.zeros_like(x) for x in alone[0]] for _ in range(12)]
    stream = torch.cuda.Stream()
    for on in (torch.cuda.current_stream(), stream):
        torch.cuda.synchronize()
        with torch.cuda.stream(on):
            for i in range(12):
                q.copy_(qs[i % 4])
                v.copy_(qs[(i + 1) % 4])
                for dst, x in zip(outs[i], evaluate(q, v)):
                    dst.copy_(x)
        torch.cuda.synchronize()
        for i in range(12):
            for got, want in zip(outs[i], alone[i % 4]):
                assert torch.equal(got, want)
