"""The autotuner on grid classes: the iteration launch has no lanes per side-row to choose, so they stay as
the layout gave them; the two-barrier launch (theta rule) has."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stop", ["primal", "theta"])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_lanes_are_tuned_only_where_they_are_used(stop, seed):
    from paper_2302_14344_gb300 import subadmm as sa
    p = sg.stir(seed, n_side=4, layers=3, tol_primal=-1, max_iters=30)
    p.options.stop, p.options.theta_th = stop, 1e-30
    a, b = sa.Simulation(p, grid_side_rows=1), sa.Simulation(p, grid_side_rows=1)
    (before,) = a.launch_classes()
    a.step(1)
    (row,) = a.autotune(steps=2)
    assert row["cached"] == 2 and row["ns_per_step"] > 0
    assert row["split"] in ((8, 16, 32) if stop == "theta" else (before["split"],))
    a.step(2)
    b.step(3)
    va, vb = a.scene_vhat(0), b.scene_vhat(0)
    assert np.max(np.abs(va - vb)) < 1e-9 * np.max(np.abs(vb))
