"""The warps of the Hartree moments and of the radial equation at their edges:
radial grids of 4 to 100 shells (the lanes cover 32 a step), shells of fewer and
more points than a warp has lanes, every l_max (the split of the warp's sum),
a random density of both signs.  Against the FP64 oracle at the tolerance of
tests/test_gpu_hartree.py: 1e-10 of the largest |v_H| plus 2^-18 of the oracle's
scale of the l >= 1 terms."""
import numpy as np
import pytest
import torch

import oracle.hartree as OH
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rad,n_ang,l_max", [(4, 50, 4), (31, 26, 5), (32, 32, 3), (33, 33, 6), (64, 14, 2), (65, 70, 1),
                                               (100, 31, 6), (40, 110, 0)])
def test_hartree_shells(n_rad, n_ang, l_max):
    import paper_2208_12335_gb300 as fgi
    prob = W.tiny_water(n_rad=n_rad, n_ang=n_ang)
    n = np.random.default_rng(n_rad).standard_normal(prob.n_pts) * np.exp(-0.3 * np.linalg.norm(prob.pts, axis=1))
    ref, bound = OH.hartree(prob, n, l_max=l_max, l1_bound=True)
    ctx = fgi.Context(0).load(prob, "fp64")
    vh = ctx.hartree(torch.from_numpy(n).cuda(), l_max=l_max).cpu().numpy()
    ctx.sync()
    assert np.all(np.abs(vh - ref) <= 1e-10 * np.abs(ref).max() + 2.0 ** -18 * bound)


def test_more_shells_than_shared_memory_holds():
    """Beyond 256 shells the radial equation works in global scratch."""
    import paper_2208_12335_gb300 as fgi
    prob = W.tiny_water(n_rad=300, n_ang=6)
    n = np.random.default_rng(2).standard_normal(prob.n_pts) * np.exp(-0.3 * np.linalg.norm(prob.pts, axis=1))
    ref, bound = OH.hartree(prob, n, l_max=3, l1_bound=True)
    ctx = fgi.Context(0).load(prob, "fp64")
    vh = ctx.hartree(torch.from_numpy(n).cuda(), l_max=3).cpu().numpy()
    ctx.sync()
    assert np.all(np.abs(vh - ref) <= 1e-10 * np.abs(ref).max() + 2.0 ** -18 * bound)
