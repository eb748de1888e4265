"""fgi_hartree sums in the order of the points: a second call, a replayed graph and
another context set up alike give the same bits.  The points of a shell lie in many
places of the list (random order), on one thread's worth of points and on more
(65536 points a piece, the last piece partly filled)."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rad,n_ang", [(20, 50), (70, 700)])
def test_calls_and_contexts_agree(n_rad, n_ang):
    import paper_2208_12335_gb300 as fgi
    prob = W.tiny_water(n_rad=n_rad, n_ang=n_ang)
    rng = np.random.default_rng(8)
    n = torch.from_numpy(rng.standard_normal(prob.n_pts)).cuda()
    owner = np.where(rng.random(prob.n_pts) < 0.1, -1, prob.owner).astype(np.int32)
    out = []
    for _ in range(3):
        ctx = fgi.Context(0).load(prob, "fp64")
        ctx.set_atom_grids(owner, prob.shell, prob.atom_rgrid)
        ctx._pending_grids = None
        out += [ctx.hartree(n, l_max=4), ctx.hartree(n, l_max=4)]
        s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        vh = torch.zeros_like(n)
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=s):
            ctx.hartree(n, l_max=4, vh=vh, stream=s)
        g.replay()
        torch.cuda.synchronize()
        ctx.sync()
        out.append(vh)
    assert float(out[0].abs().max()) > 0
    assert all(torch.equal(out[0], x) for x in out[1:])
