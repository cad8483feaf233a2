"""The theta stop rule on the device (the step ends in the v-step whose theta is below the threshold,
before its z-step) against the oracle: the block kernel, and the grid kernel with one scene over the
whole GPU, with D rows staged through shared memory and read directly."""
import numpy as np
import pytest

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-30))


def _problem(kind):
    p = {"chain": lambda: sg.chain(2, n_links=8, links_per_sub=2),
         "sides": lambda: sg.generic(7, n_scenes=2, n_sub=7, n_range=(1, 12), max_sides=8, extra=10, warm="prev"),
         "rows": lambda: sg.batched(3, n_scenes=2, n_sub=(20, 24), contacts=(150, 160)),
         "beam": lambda: sg.fem_beam(0, ny=8, nz=8, planes=6, slabs=2, length=0.02, with_gripper=False)}[kind]()
    p.options.stop, p.options.max_iters = "theta", 400
    p.options.theta_th = {"chain": 1e-7, "sides": 1e-9, "rows": 1e-7, "beam": 1e-6}[kind]
    return p


def _same(sim, problem, steps):
    ends = []
    for k, o in enumerate(oracle.run(problem, steps=steps)):
        r, q = sim.residuals(k), o.residuals()
        assert (r["iters"], r["converged"]) == (q["iters"], q["converged"])
        ends.append(r["converged"])
        if r["converged"]:
            assert np.isclose(r["theta"], q["theta"], rtol=1e-5, atol=1e-18)
        assert _rel(sim.scene_vhat(k), o.vhat_all()) < 1e-9
        assert _rel(sim.scene_lam(k), o.lam_all()) < 1e-9
    assert any(ends)


@pytest.mark.parametrize("kind", ["chain", "sides", "rows", "beam"])
@pytest.mark.parametrize("grid", [None, 1])
def test_theta_rule_fp64(kind, grid):
    """Iteration counts, theta, v-hat and lambda of three steps (FP64 parity bound, 1e-9)."""
    from paper_2302_14344_gb300 import subadmm as sa
    p = _problem(kind)
    sim = sa.Simulation(p, grid_side_rows=grid)
    assert all(c["cached"] == 2 if grid else c["cached"] in (0, 3) for c in sim.launch_classes())
    sim.step(3)
    _same(sim, p, 3)


@pytest.mark.parametrize("blocks", [0, 1])
def test_staged_rows_of_the_two_barrier_kernel(blocks):
    """Rows of D long enough for a warp each go through the stages of shared memory (several rows a
    warp on one block), with the same bits as without, and the oracle's iterations."""
    from paper_2302_14344_gb300 import subadmm as sa
    p = _problem("beam")
    sims = []
    for staging in (True, False):
        sim = sa.Simulation(p, grid_side_rows=1)
        sim.grid_staging(staging)
        sim.grid_blocks(blocks)
        sim.step(2)
        (c,) = sim.launch_classes()
        assert c["split"] == 32 and (c["smem_bytes"] > 0) == staging
        sims.append(sim)
    assert np.array_equal(sims[0].scene_vhat(0), sims[1].scene_vhat(0))
    _same(sims[0], p, 2)
