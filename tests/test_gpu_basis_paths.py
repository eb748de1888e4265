"""The basis kernels' path for species whose shells share one knot grid against
the general path, over the forms the first accepts: thirteen shells (four a
bound look-up, a remainder of one), points on the nuclei and beyond every
cutoff, batches at the edges of a warp and of a 64-point chunk, potentials of
one sign (one image) and of both (two).

The general path is taken for the same functions by padding one shell's spline
with an interval of zeros: the knot grids then differ, the functions do not.
Both paths do the same operations in the same order, and the contractions sum
in fixed order: H and the density are equal bit by bit.
"""
import dataclasses

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def molecule():
    rc = 4.0 * W.BOHR_PER_ANG
    ls = [0, 0, 0, 0, 1, 1, 1, 1, 2, 2, 2, 3, 3]
    radials = [W.make_radial(W.RadialSpec(l, (0.4 + 0.11 * i, 1.9), (1.0, -0.2), rc, rc - W.BOHR_PER_ANG, 1700))
               for i, l in enumerate(ls)]
    species = [W.Species("A", 6.0, list(range(13))), W.Species("B", 3.0, [8, 0, 4])]
    xyz = np.array([[0.0, 0.0, 0.0], [2.4, 0.3, -0.2], [-0.7, 2.2, 1.0], [1.1, -1.9, 1.7], [-2.0, -1.2, -1.4]])
    sp = np.array([0, 1, 0, 1, 0], dtype=np.int32)
    prob = W.build_problem("paths", radials, species, [(sp, xyz)], lambda k: (14, 38), 9, (200, 50, None))
    pts = np.concatenate([prob.pts, xyz, [[30.0, 1.0, 0.0], [5.0, 6.5, 3.0]]])
    w = np.concatenate([prob.w, np.full(len(xyz) + 2, 1e-3)])
    v = np.concatenate([prob.v, np.full(len(xyz) + 2, -0.3)])
    # batches of 1, 31, 32, 33, 64, 65 points, then of 199
    off = np.cumsum([0, 1, 31, 32, 33, 64, 65])
    off = np.concatenate([off, np.arange(off[-1] + 199, len(w), 199), [len(w)]]).astype(np.int64)
    return W.Problem("paths", radials, species, prob.atom_off, prob.atom_species, prob.atom_xyz, pts, w, off,
                     np.zeros(len(off) - 1, dtype=np.int32), v)


@pytest.mark.parametrize("precision", ["split_bf16", "bf16"])
@pytest.mark.parametrize("both_signs", [False, True])
@pytest.mark.parametrize("points", [0, 512])                      # batches as given, and merged
def test_shared_knots_equal_general_path(molecule, both_signs, points, precision, tmp_path):
    import paper_2208_12335_gb300 as fgi
    v = molecule.v + (0.4 if both_signs else 0.0)
    assert (v.max() > 0) == both_signs
    tune = tmp_path / "tune.txt"
    tune.write_text("h_sb_points %d\ndensity_sb_points %d\n" % (points, points))
    padded = list(molecule.radials)
    for i in (8, 12):                                             # a shell of each species
        r = padded[i]
        padded[i] = W.Radial(r.l, r.h, np.concatenate([r.coef, np.zeros((1, 4))]), r.spec, r.norm)
    out = []
    for radials in (molecule.radials, padded):
        ctx = fgi.Context(0).load(dataclasses.replace(molecule, radials=radials), precision, tune_path=str(tune))
        d = torch.from_numpy(np.random.default_rng(5).standard_normal(ctx.sizes()[1])).cuda()
        h = ctx.integrate_h(torch.from_numpy(v).cuda())
        n = ctx.density(d)[0]
        ctx.sync()
        out.append((ctx.batch_work()[1], h.cpu().numpy(), n.cpu().numpy()))
    (a, h0, n0), (b, h1, n1) = out
    assert np.array_equal(a, b)                                   # the same active functions
    assert np.abs(h0).max() > 0 and np.array_equal(h0, h1)
    assert np.abs(n0).max() > 0 and np.array_equal(n0, n1)


def test_column_bounds_of_many_atoms(tmp_path):
    """More active atoms at a point than the column bounds stage at a time
    (128), the last group partly filled; the same two paths, equal bit by bit."""
    import paper_2208_12335_gb300 as fgi
    rc = 4.0 * W.BOHR_PER_ANG
    radials = [W.make_radial(W.RadialSpec(l, (0.5 + 0.2 * l, 1.7), (1.0, -0.2), rc, rc - W.BOHR_PER_ANG, 900))
               for l in (0, 1)]
    species = [W.Species("A", 1.0, [0, 1])]
    xyz = np.stack(np.meshgrid(*[1.2 * np.arange(n) for n in (6, 5, 5)], indexing="ij"), -1).reshape(-1, 3)
    prob = W.build_problem("many", radials, species, [(np.zeros(150, dtype=np.int32), xyz)], lambda k: (4, 14), 9,
                           (200, 50, None))
    r = radials[1]
    padded = [radials[0], W.Radial(r.l, r.h, np.concatenate([r.coef, np.zeros((1, 4))]), r.spec, r.norm)]
    out = []
    for rads in (radials, padded):
        ctx = fgi.Context(0).load(dataclasses.replace(prob, radials=rads), "split_bf16")
        d = torch.from_numpy(np.random.default_rng(5).standard_normal(ctx.sizes()[1])).cuda()
        n = ctx.density(d)[0]
        ctx.sync()
        out.append((ctx.batch_work()[1], n.cpu().numpy()))
    (a, n0), (b, n1) = out
    assert np.array_equal(a, b) and a.max() > 4 * 128
    assert np.abs(n0).max() > 0 and np.array_equal(n0, n1)


@pytest.mark.parametrize("points", [0, 512])
def test_position_gradient_paths(molecule, points, tmp_path):
    """The adjoint's position gradient on shared knots and shell by shell: the
    same FP32 operations, summed into dR by FP64 atomics in no fixed order
    (below 10^5 terms of 2^-53 each, against the largest component)."""
    import paper_2208_12335_gb300 as fgi
    tune = tmp_path / "tune.txt"
    tune.write_text("h_sb_points %d\ndensity_sb_points %d\n" % (points, points))
    padded = list(molecule.radials)
    for i in (8, 12):
        r = padded[i]
        padded[i] = W.Radial(r.l, r.h, np.concatenate([r.coef, np.zeros((1, 4))]), r.spec, r.norm)
    out = []
    for radials in (molecule.radials, padded):
        ctx = fgi.Context(0).load(dataclasses.replace(molecule, radials=radials), "split_bf16", tune_path=str(tune))
        g = torch.from_numpy(np.random.default_rng(7).standard_normal(ctx.sizes()[1])).cuda()
        dv, dR = ctx.adjoint(g, torch.from_numpy(molecule.v).cuda())
        ctx.sync()
        out.append((dv.cpu().numpy(), dR.cpu().numpy()))
    (v0, r0), (v1, r1) = out
    assert np.abs(v0).max() > 0 and np.array_equal(v0, v1)
    assert np.abs(r0).max() > 0 and np.abs(r0 - r1).max() <= 1e5 * 2.0 ** -53 * np.abs(r0).max()
