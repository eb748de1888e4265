"""The Hartree moments of l >= 1 keep their bits where the positions are large
against the shells, and over the range of the weights and the density.

* Two points of the fourth shell (r about 4e-6 Bohr) of an atom 2e5 Bohr from the
  origin carry opposite charges, so v_H is all l >= 1.  Their offsets from the nucleus are
  exact in FP64; positions of 48 bits would turn the directions by 2^-12.  Against
  the oracle at the tolerance of tests/test_gpu_hartree.py for the l >= 1 terms
  (2^-18 of the oracle's scale of them), at the points from 0.02 Bohr on.
* Scaling the density by a power of two scales v_H by it, down to w n of
  2^-143, below the range of FP32: there v_H itself is still a normal number
  inside the radial grid (a sum over 200 points, divided by 1e-6 Bohr), whose own FP32
  rounding below 2^-126 is 2^-150 a term, for at most 10^4 weighted terms 2^-22 of the
  largest v_H.  (Points on or beyond the last shell take v_H from the exterior
  moments, which are v_H times the distance and so leave that range first.)"""
import math

import numpy as np
import pytest
import torch

import oracle.hartree as OH
import workloads as W

pytestmark = pytest.mark.gpu


def _one_atom(center, n_rad, half_sphere):
    """One s function; shells r_k = 2^-20 exp(k / 2), each with the directions
    of half_sphere and their opposites."""
    radial = W.make_radial(W.RadialSpec(0, (0.8,), (1.0,), 4.0, 3.0, 400))
    dirs = np.concatenate([half_sphere, -half_sphere])
    r = 2.0 ** -20 * np.exp(0.5 * np.arange(n_rad))
    off = (r[:, None, None] * dirs[None]).reshape(-1, 3)
    n = len(off)
    w = np.repeat(r ** 3 * 0.5 * 4.0 * math.pi / len(dirs), len(dirs))
    cuts = np.arange(0, n + 100, 100).clip(max=n).astype(np.int64)
    cuts = np.unique(cuts)
    return W.Problem("one", [radial], [W.Species("A", 1.0, [0])], np.array([0, 1], dtype=np.int64),
                     np.zeros(1, dtype=np.int32), np.array([center]), np.array(center) + off, w, cuts,
                     np.zeros(len(cuts) - 1, dtype=np.int32), np.full(n, -0.3), owner=np.zeros(n, dtype=np.int32),
                     shell=np.repeat(np.arange(n_rad, dtype=np.int32), len(dirs)),
                     atom_rgrid=np.array([[2.0 ** -20, 0.5, n_rad]]))


@pytest.mark.parametrize("l_max", [1, 4, 6])
def test_atom_far_from_the_origin(l_max):
    import paper_2208_12335_gb300 as fgi
    half = W.fibonacci_sphere(23)[:7]
    prob = _one_atom([131072.3, -90210.7, 122333.1], 30, half)
    n = np.zeros(prob.n_pts)
    first = 3 * 14 + 2                                            # a point of shell 3 and its opposite
    n[first], n[first + 7] = 1.0 / prob.w[first], -1.0 / prob.w[first + 7]
    ref, bound = OH.hartree(prob, n, l_max=l_max, l1_bound=True)
    ctx = fgi.Context(0).load(prob, "fp64")
    vh = ctx.hartree(torch.from_numpy(n).cuda(), l_max=l_max).cpu().numpy()
    ctx.sync()
    outer = np.linalg.norm(prob.pts - prob.atom_xyz[0], axis=1) > 0.02
    assert outer.sum() >= 100 and np.abs(ref[outer]).max() > 0
    assert np.all(np.abs(vh - ref)[outer] <= 2.0 ** -18 * bound[outer])


@pytest.mark.parametrize("l_max", [1, 4, 6])
def test_density_scales_by_powers_of_two(l_max):
    import paper_2208_12335_gb300 as fgi
    prob = _one_atom([3.1, -1.4, 2.2], 12, W.fibonacci_sphere(301)[:100])
    d = prob.pts - prob.atom_xyz[0]
    d /= np.linalg.norm(d, axis=1)[:, None]
    n = np.where(prob.shell < 4, 0.1 + d[:, 0] + 0.5 * d[:, 1] * d[:, 2], 0.0)
    ctx = fgi.Context(0).load(prob, "fp64")
    v = [ctx.hartree(torch.from_numpy(n * 2.0 ** k).cuda(), l_max=l_max).cpu().numpy() * 2.0 ** -k for k in (0, -78, 78)]
    ctx.sync()
    inside = prob.shell < 11
    for x in v[1:]:
        assert np.abs(x - v[0])[inside].max() <= 2.0 ** -22 * np.abs(v[0]).max()
