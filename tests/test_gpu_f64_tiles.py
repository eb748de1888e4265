"""The FP64 contractions at the edges of their tiles: function counts around the 64
of a tile and the 4 of a thread's block, batches around the 16 points of a step
and the 64 of a point tile.  H, the density and the adjoint's dL/dv against the
oracle, entry by entry within 1e-12 of the sum of the magnitudes of the terms
(at most 130^2 of them, each of some ten roundings of 2^-53)."""
import numpy as np
import pytest
import torch

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_fn", [1, 3, 60, 63, 64, 65, 68, 130])
def test_tile_edges(n_fn):
    import paper_2208_12335_gb300 as fgi
    rc = 4.0 * W.BOHR_PER_ANG
    radials = [W.make_radial(W.RadialSpec(l, (0.5 + 0.2 * l, 1.7), (1.0, 0.2), rc, rc - W.BOHR_PER_ANG, 700))
               for l in (0, 1)]
    species = [W.Species("A", 1.0, [0]), W.Species("B", 3.0, [0, 1])]
    rng = np.random.default_rng(n_fn)
    sp = np.array([1] * (n_fn // 4) + [0] * (n_fn % 4), dtype=np.int32)
    xyz = rng.uniform(-1.5, 1.5, (len(sp), 3))
    sizes = [1, 15, 16, 17, 63, 64, 65, 200]
    off = np.cumsum([0] + sizes).astype(np.int64)
    pts = rng.uniform(-1.5, 1.5, (off[-1], 3))
    w, v = rng.uniform(0.1, 1.0, off[-1]), rng.standard_normal(off[-1])
    prob = W.Problem("tiles", radials, species, np.array([0, len(sp)], dtype=np.int64), sp, xyz, pts, w, off,
                     np.zeros(len(sizes), dtype=np.int32), v)
    ctx = fgi.Context(0).load(prob, "fp64")
    basis = O.system_basis(prob)
    rowptr, col = (np.asarray(x) for x in ctx.pattern())
    rows = np.repeat(np.arange(n_fn), np.diff(rowptr))
    d = rng.standard_normal(len(col))
    D = np.zeros((n_fn, n_fn))
    D[rows, col] = d
    D = D + D.T - np.diag(np.diag(D))
    G = 0.5 * (D + np.diag(np.diag(D)))
    phi = np.abs(O.phi(basis, pts)).T
    h = ctx.integrate_h(torch.from_numpy(v).cuda()).cpu().numpy()
    n = ctx.density(torch.from_numpy(d).cuda())[0].cpu().numpy()
    dv = ctx.adjoint(torch.from_numpy(d).cuda(), torch.from_numpy(v).cuda())[0].cpu().numpy()
    ctx.sync()
    href = O.h_matrix(basis, pts, w, v)[rows, col]
    assert np.all(np.abs(h - href) <= 1e-12 * ((phi * (w * np.abs(v))) @ phi.T)[rows, col])
    scale = np.einsum("ip,ij,jp->p", phi, np.abs(D), phi)
    assert np.all(np.abs(n - O.density(basis, pts, D)) <= 1e-12 * scale)
    assert np.all(np.abs(dv - O.adjoint(basis, pts, w, v, G)[0]) <= 1e-12 * w * scale)
