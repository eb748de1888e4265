"""A grid point far outside every cutoff, in the same 64 points as points inside:
its functions are zero wherever it lies, also where its offset, the square of it
or the angular polynomials leave the range of FP32 (d shells from 1e19 Bohr, f
shells from 7e12).  H, the density and dL/dv are bit by bit those of the same
grid with that point at 60 Bohr; dL/dR is summed by FP64 atomics in no fixed
order (below 10^4 terms of 2^-53 each, against the largest component)."""
import dataclasses

import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def _results(prob, v, precision, tune):
    import paper_2208_12335_gb300 as fgi
    ctx = fgi.Context(0).load(prob, precision, tune_path=tune)
    d = torch.from_numpy(np.random.default_rng(5).standard_normal(ctx.sizes()[1])).cuda()
    vd = torch.from_numpy(v).cuda()
    h = ctx.integrate_h(vd)
    n = ctx.density(d)[0]
    dv, dR = ctx.adjoint(d, vd)
    ctx.sync()                                                    # no non-finite value was seen
    return [x.cpu().numpy() for x in (h, n, dv, dR)]


@pytest.mark.parametrize("precision", ["split_bf16", "bf16"])
@pytest.mark.parametrize("both_signs", [False, True])
@pytest.mark.parametrize("far", [1e13, 1e20, 1e200])
def test_far_point_contributes_nothing(far, both_signs, precision, tmp_path):
    rc = 4.0 * W.BOHR_PER_ANG
    radials = [W.make_radial(W.RadialSpec(l, (0.4 + 0.1 * l, 1.9), (1.0, -0.2), rc, rc - W.BOHR_PER_ANG, 1700))
               for l in (0, 1, 2, 3)]
    species = [W.Species("A", 6.0, [0, 1, 2, 3])]
    xyz = np.array([[0.0, 0.0, 0.0], [2.4, 0.3, -0.2]])
    prob = W.build_problem("far", radials, species, [(np.zeros(2, dtype=np.int32), xyz)], lambda k: (8, 26), 9,
                           (200, 50, None))
    tune = tmp_path / "tune.txt"
    tune.write_text("h_sb_points 0\ndensity_sb_points 0\n")       # the batches as given
    k = int(prob.batch_off[0] + prob.batch_off[1]) // 2
    v = prob.v + (0.4 if both_signs else 0.0)
    assert (v.max() > 0) == both_signs
    out = []
    for at in (60.0, far):
        pts = prob.pts.copy()
        pts[k] = [at, -at, 0.5 * at]
        out.append(_results(dataclasses.replace(prob, pts=pts), v, precision, str(tune)))
    for a, b in zip(out[0][:3], out[1][:3]):
        assert np.abs(a).max() > 0 and np.array_equal(a, b)
    assert out[1][1][k] == 0.0 and out[1][2][k] == 0.0
    assert np.abs(out[0][3] - out[1][3]).max() <= 1e4 * 2.0 ** -53 * np.abs(out[0][3]).max()
