"""The gather of D per super-batch where it can go wrong: odd function counts,
so that a pair of columns spans two atoms; a super-batch of more than 512
active atoms (its tables stay in global memory); blocks and chunks that end
inside an atom; atom pairs beyond the pattern.  Against the oracle at the
stated bound of the split density (relative L2 1e-7), which also holds for the
adjoint's full gather through dL/dv (1e-6 of its largest value)."""
import numpy as np
import pytest
import torch

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


def _problem(n_atoms, shells, spacing, rc_ang):
    rc = rc_ang * W.BOHR_PER_ANG
    radials = [W.make_radial(W.RadialSpec(l, (0.6 + 0.2 * i,), (1.0,), rc, rc - 0.7 * W.BOHR_PER_ANG, 800))
               for i, l in enumerate(shells)]
    k = int(np.ceil(n_atoms ** (1 / 3)))
    g = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), axis=-1).reshape(-1, 3)[:n_atoms] * spacing
    xyz = g + np.random.default_rng(3).normal(0.0, 0.1, g.shape)
    species = [W.Species("A", 4.0, list(range(len(shells))))]
    rng = np.random.default_rng(4)
    pts = xyz[rng.integers(0, n_atoms, 700)] + rng.normal(0.0, 1.0, (700, 3))
    off = np.array([0, 1, 90, 300, 700], dtype=np.int64)
    return W.Problem("gather", radials, species, np.array([0, n_atoms]), np.zeros(n_atoms, dtype=np.int32), xyz, pts,
                     np.full(700, 0.02), off, np.zeros(4, dtype=np.int32), np.full(700, -0.4))


@pytest.mark.parametrize("n_atoms,shells,spacing,rc_ang", [(27, [0, 1, 2], 3.0, 3.0), (29, [0, 0, 1], 4.5, 1.6),
                                                           (60, [1], 2.5, 2.5), (600, [0], 1.6, 5.0)])
def test_gather(n_atoms, shells, spacing, rc_ang):
    import paper_2208_12335_gb300 as fgi
    prob = _problem(n_atoms, shells, spacing, rc_ang)
    B = O.system_basis(prob)
    ctx = fgi.Context(0).load(prob, "split_bf16")
    rowptr, col = ctx.pattern(0)
    rows = np.repeat(np.arange(len(rowptr) - 1), np.diff(rowptr))
    D, _ = W.density_matrix_occ(B.n_fn, max(1, B.n_fn // 4), np.random.default_rng(6))
    stored = np.zeros_like(D)
    stored[rows, col] = D[rows, col]
    full = stored + np.triu(stored, 1).T                          # zero where the pattern has no pair
    values = torch.from_numpy(D[rows, col]).cuda()
    n, _ = ctx.density(values)
    dv, _ = ctx.adjoint(values, torch.from_numpy(prob.v).cuda())
    ctx.sync()
    ref = O.density(B, prob.pts, full)
    assert np.linalg.norm(n.cpu().numpy() - ref) <= 1e-7 * np.linalg.norm(ref)
    half = 0.5 * (full + np.diag(np.diag(full)))                  # G of the adjoint: off-diagonal values halved
    dv_ref = prob.w * O.density(B, prob.pts, half)
    assert np.abs(dv.cpu().numpy() - dv_ref).max() <= 1e-6 * np.abs(dv_ref).max()
