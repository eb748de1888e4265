"""The H scatter's conversion to fixed point where it changes path: contributions
of 2^14 Ha and more (the general conversion), and beyond its range.

Scaling v by a power of two scales every operand, product and partial sum of
the contraction by exactly that power, so h(2^k v) and 2^k h(v) differ only by
the conversion, at most two units of 2^-40 Ha a contribution (one for each
accumulator) on either side."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("both_signs", [False, True])
@pytest.mark.parametrize("k", [4, 14])
def test_large_values_scale_exactly(k, both_signs):
    import paper_2208_12335_gb300 as fgi
    prob = W.tiny_water()
    v = torch.from_numpy(prob.v + (3.0 if both_signs else 0.0)).cuda()
    ctx = fgi.Context(0).load(prob, "split_bf16")
    h = ctx.integrate_h(v).cpu().numpy()
    big = ctx.integrate_h(v * 2.0 ** k).cpu().numpy()
    ctx.sync()
    assert k < 14 or np.abs(big).max() > 2.0 ** 14
    n = len(ctx.schedule("h")["sb_rank"])
    assert np.abs(big - h * 2.0 ** k).max() <= n * 2 * 2.0 ** -40 * (1 + 2.0 ** k)


def test_values_beyond_the_fixed_point_range_are_reported():
    import paper_2208_12335_gb300 as fgi
    prob = W.tiny_water()
    ctx = fgi.Context(0).load(prob, "split_bf16")
    ctx.integrate_h(torch.from_numpy(prob.v * 2.0 ** 26).cuda())
    with pytest.raises(fgi.FGIError) as e:
        ctx.sync()
    assert e.value.code == -6
