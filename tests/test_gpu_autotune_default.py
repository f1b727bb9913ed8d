"""The autotuner measures the default rule's elements per CTA among its
candidates and leaves a slot at 0 (the rule) where that value is the fastest: at
3D p = 5, one element is all a CTA holds, so there is nothing to choose."""
import pytest
import torch

import cases
import helpers as Hp

pytestmark = pytest.mark.gpu


def test_rule_value_stays_the_rule():
    m = cases.periodic_box(3, 6, 0.0, 1.0, 5)
    ctx = Hp.gpu_ctx(m, dict(gamma=1.4, mu=0.01, Pr=0.71))
    q = ctx.pack(torch.from_numpy(cases.random_state(m, 741)).cuda())
    for _ in range(4):
        ctx.autotune(q)
        table = ctx.tuning()["epb"]
        # [precision][kernel][P], P = 6: trace, volume residual, volume JVP in FP64 and FP32
        assert [table[(prec * 3 + kind) * 7 + 6] for prec in range(2) for kind in range(3)] == [0] * 6, table
