"""The active functions of a batch that holds one point far from all atoms: those
of the other points, however far it lies (beside 1e20 Bohr a cutoff is below
the rounding of the batch's radius, at 1e200 its square overflows)."""
import dataclasses

import numpy as np
import pytest

import workloads as W


@pytest.mark.parametrize("far", [1e3, 1e13, 1e16, 1e20, 1e200])
def test_active_functions_do_not_depend_on_a_far_point(far):
    import paper_2208_12335_gb300 as fgi
    prob = W.tiny_water(n_rad=12, n_ang=26)
    work = []
    for at in (60.0, far):
        pts = prob.pts.copy()
        pts[prob.batch_off[:-1]] = [at, -at, 0.5 * at]            # one point of every batch
        work.append(fgi.Context(-1).load(dataclasses.replace(prob, pts=pts), "split_bf16").batch_work()[1])
    assert work[0].max() > 0 and np.array_equal(work[0], work[1])
