"""The FP64 path forms u(d)/d as a correctly rounded quotient.

* With u(r) = r on knots of spacing 1 the spline gives u = d exactly, so phi = Y_00 at
  every point whatever the rounding of d, and the density of D = 1 is one number.
* With u constant on each interval and the points on an axis through the atom, u and d
  are exact, and the density is the square of fl(fl(u / d) Y_00), bit for bit that of
  the host's division."""
import math

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


KNOTS = 12


def _density(coef, xyz, pts):
    """n of D = 1 for one s function with spline coefficients coef on knots of spacing 1."""
    import paper_2208_12335_gb300 as fgi
    spec = W.RadialSpec(0, (1.0,), (1.0,), float(KNOTS), None, KNOTS)
    off = np.arange(0, len(pts) + 1, 200, dtype=np.int64)
    prob = W.Problem("division", [W.Radial(0, 1.0, coef, spec, 1.0)], [W.Species("A", 1.0, [0])], np.array([0, 1]),
                     np.zeros(1, dtype=np.int32), xyz, pts, np.ones(len(pts)), off,
                     np.zeros(len(off) - 1, dtype=np.int32), np.ones(len(pts)))
    ctx = fgi.Context(0).load(prob, "fp64")
    n = ctx.density(torch.ones(1, dtype=torch.float64, device="cuda"))[0].cpu().numpy()
    ctx.sync()
    return n


def test_u_equal_to_d():
    coef = np.zeros((KNOTS, 4))
    coef[:, 0], coef[:, 1] = np.arange(KNOTS), 1.0
    rng = np.random.default_rng(12)
    xyz = np.array([[0.3, -0.7, 1.1]])
    dirs = rng.standard_normal((2000, 3))
    dirs /= np.linalg.norm(dirs, axis=1)[:, None]
    n = _density(coef, xyz, xyz + dirs * rng.uniform(0.01, KNOTS - 0.01, 2000)[:, None])
    assert np.all(n == n[0])
    assert abs(n[0] - 0.25 / math.pi) <= 4 * 2.0 ** -53 * 0.25 / math.pi


def test_quotient_of_exact_operands():
    rng = np.random.default_rng(13)
    coef = np.zeros((KNOTS, 4))
    coef[:, 0] = rng.uniform(-1.0, 1.0, KNOTS) * 10.0 ** rng.integers(-8, 3, KNOTS)
    pts = np.zeros((4000, 3))
    x = rng.uniform(1e-4, KNOTS - 1e-4, 4000)
    pts[np.arange(4000), rng.integers(0, 3, 4000)] = x * rng.choice([-1.0, 1.0], 4000)
    n = _density(coef, np.zeros((1, 3)), pts)
    phi = coef[np.floor(x).astype(int), 0] / x * 0.28209479177387814
    assert np.array_equal(n, phi * phi)
