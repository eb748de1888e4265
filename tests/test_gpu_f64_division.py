"""The FP64 path forms u(d)/d by a division.  With u(r) = r on knots of spacing 1 the
spline gives u = d exactly, so phi = Y_00 at every point whatever the rounding of d, and
the density of D = 1 is one number, bit for bit."""
import math

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def test_u_over_d_is_a_division():
    import paper_2208_12335_gb300 as fgi
    knots = 12
    coef = np.zeros((knots, 4))
    coef[:, 0], coef[:, 1] = np.arange(knots), 1.0
    spec = W.RadialSpec(0, (1.0,), (1.0,), float(knots), None, knots)
    rng = np.random.default_rng(12)
    xyz = np.array([[0.3, -0.7, 1.1]])
    dirs = rng.standard_normal((2000, 3))
    dirs /= np.linalg.norm(dirs, axis=1)[:, None]
    pts = xyz + dirs * rng.uniform(0.01, knots - 0.01, 2000)[:, None]
    off = np.arange(0, 2001, 200, dtype=np.int64)
    prob = W.Problem("division", [W.Radial(0, 1.0, coef, spec, 1.0)], [W.Species("A", 1.0, [0])], np.array([0, 1]),
                     np.zeros(1, dtype=np.int32), xyz, pts, np.ones(2000), off, np.zeros(10, dtype=np.int32),
                     np.ones(2000))
    ctx = fgi.Context(0).load(prob, "fp64")
    n = ctx.density(torch.ones(1, dtype=torch.float64, device="cuda"))[0].cpu().numpy()
    ctx.sync()
    assert np.all(n == n[0])
    assert abs(n[0] - 0.25 / math.pi) <= 4 * 2.0 ** -53 * 0.25 / math.pi
