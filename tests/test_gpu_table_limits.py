"""Plans beyond what the kernels keep in shared memory: more than 64 active atoms in
a super-batch (the position gradient takes them 64 at a time, the last group
partly filled) and more than 64 shells in all species (tables read from global memory).

* dL/dR of 100 overlapping atoms against the oracle at the stated 1e-6 of its largest
  component, dL/dv at 1e-6 of its largest value.
* A species that no atom has, with 60 shells, changes no function: H, the density and
  dL/dv stay the same bit by bit, on shared knots and on the general path; dL/dR is
  summed by FP64 atomics in no fixed order (below 10^5 terms of 2^-53 each)."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


def test_position_gradient_of_many_active_atoms():
    import paper_2208_12335_gb300 as fgi
    rc = 4.0 * W.BOHR_PER_ANG
    radials = [W.make_radial(W.RadialSpec(l, (0.5 + 0.2 * l,), (1.0,), rc, rc - W.BOHR_PER_ANG, 800)) for l in (0, 1)]
    rng = np.random.default_rng(4)
    xyz = np.stack(np.meshgrid(*[1.5 * np.arange(n) for n in (5, 5, 4)], indexing="ij"), -1).reshape(-1, 3)
    xyz = xyz + rng.normal(0.0, 0.1, xyz.shape)
    pts = xyz[rng.integers(0, 100, 500)] + rng.normal(0.0, 1.0, (500, 3))
    off = np.array([0, 1, 90, 500], dtype=np.int64)
    v = rng.uniform(-1.0, 0.2, 500)
    prob = W.Problem("many", radials, [W.Species("A", 4.0, [0, 1])], np.array([0, 100]), np.zeros(100, dtype=np.int32),
                     xyz, pts, np.full(500, 0.02), off, np.zeros(3, dtype=np.int32), v)
    ctx = fgi.Context(0).load(prob, "split_bf16")
    assert ctx.batch_work()[1].max() > 4 * 64 and ctx.batch_work()[1].max() % (4 * 64)
    B = O.system_basis(prob)
    rowptr, col = ctx.pattern(0)
    rows = np.repeat(np.arange(len(rowptr) - 1), np.diff(rowptr))
    g = rng.standard_normal(len(col))
    G = np.zeros((B.n_fn, B.n_fn))
    G[rows, col] = g
    G = 0.5 * (G + G.T)                                           # stored values halved off the diagonal
    dv, dR = (x.cpu().numpy() for x in ctx.adjoint(torch.from_numpy(g).cuda(), torch.from_numpy(v).cuda()))
    ctx.sync()
    dv_ref, dR_ref = O.adjoint(B, pts, prob.w, v, G)
    assert np.abs(dv - dv_ref).max() <= 1e-6 * np.abs(dv_ref).max()
    assert np.abs(dR.reshape(-1, 3) - np.asarray(dR_ref).reshape(-1, 3)).max() <= 1e-6 * np.abs(dR_ref).max()


@pytest.mark.parametrize("precision", ["split_bf16", "bf16"])
@pytest.mark.parametrize("shared", [True, False])
def test_more_shells_than_shared_memory_holds(shared, precision):
    import paper_2208_12335_gb300 as fgi
    rc = 4.0 * W.BOHR_PER_ANG
    ls = [0, 0, 1, 2, 3]
    radials = [W.make_radial(W.RadialSpec(l, (0.4 + 0.11 * i, 1.9), (1.0, -0.2), rc, rc - W.BOHR_PER_ANG,
                                          1700 if shared else 1700 + 3 * i)) for i, l in enumerate(ls)]
    species = [W.Species("A", 6.0, [0, 1, 2, 3, 4]), W.Species("B", 3.0, [3, 0, 2])]
    xyz = np.array([[0.0, 0.0, 0.0], [2.4, 0.3, -0.2], [-0.7, 2.2, 1.0]])
    prob = W.build_problem("shells", radials, species, [(np.array([0, 1, 0], dtype=np.int32), xyz)], lambda k: (12, 38), 9,
                           (200, 50, None))
    v = torch.from_numpy(prob.v + 0.3).cuda()
    out = []
    for sp in (species, species + [W.Species("none", 1.0, [0] * 60)]):
        ctx = fgi.Context(0).load(dataclasses.replace(prob, species=sp), precision)
        d = torch.from_numpy(np.random.default_rng(5).standard_normal(ctx.sizes()[1])).cuda()
        dv, dR = ctx.adjoint(d, v)
        out.append([x.cpu().numpy() for x in (ctx.integrate_h(v), ctx.integrate_h(v - 2.0), ctx.density(d)[0], dv, dR)])
        ctx.sync()
    for a, b in zip(out[0][:4], out[1][:4]):
        assert np.abs(a).max() > 0 and np.array_equal(a, b)
    assert np.abs(out[0][4] - out[1][4]).max() <= 1e5 * 2.0 ** -53 * np.abs(out[0][4]).max()
