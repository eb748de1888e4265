"""H does not depend on what the workspace held before: zeros, NaN or large finite
values in every byte of it.  Function counts from a few to just beyond a block,
so that most tiles have columns past the last function (rows of the images that are
not written)."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["split_bf16", "bf16"])
@pytest.mark.parametrize("both_signs", [False, True])
@pytest.mark.parametrize("n_atoms", [1, 5, 33])                   # 4, 20 and 132 functions
def test_h_of_a_used_workspace(n_atoms, both_signs, precision):
    import paper_2208_12335_gb300 as fgi
    rc = 4.0 * W.BOHR_PER_ANG
    radials = [W.make_radial(W.RadialSpec(l, (0.5 + 0.2 * l,), (1.0,), rc, rc - W.BOHR_PER_ANG, 700)) for l in (0, 1)]
    g = np.stack(np.meshgrid(*[2.0 * np.arange(4)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)[:n_atoms]
    prob = W.build_problem("stale", radials, [W.Species("A", 3.0, [0, 1])], [(np.zeros(n_atoms, dtype=np.int32), g)],
                           lambda k: (8, 26), 9, (200, 50, None))
    ctx = fgi.Context(0).load(prob, precision)
    v = torch.from_numpy(prob.v + (0.4 if both_signs else 0.0)).cuda()
    h = []
    for fill in (0, 0xFF, 0x7E):
        ws = torch.full((ctx.workspace_size(),), fill, dtype=torch.uint8, device="cuda")
        h.append(ctx.integrate_h(v, ws=ws))
        ctx.sync()
    assert float(h[0].abs().max()) > 0
    assert torch.equal(h[0], h[1]) and torch.equal(h[0], h[2])
