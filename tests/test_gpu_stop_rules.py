"""When a step ends, in every kernel that can run it: the check of a learned start after 10
iterations, with a fixed iteration count as well as with a tolerance; iterates that are not finite."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-30))


@pytest.mark.parametrize("seed,gain", [(2, 0.1), (3, 1.0), (4, 0.02), (5, 0.3)])
def test_learned_start_is_judged_alike_on_grid_and_block(seed, gain):
    """The residual after 10 iterations, max(|x - z|, |z - z of the iteration before|), decides whether a
    learned start is kept: the grid and the block kernels take the same decisions in every scene
    and so run as many iterations and end in the same v-hat (1e-5: the network's inputs are the
    state rounded to FP32, 6e-8 relative, and its output enters lambda^0)."""
    from paper_2302_14344_gb300 import learned as lr
    from paper_2302_14344_gb300 import subadmm as sa
    p = sg.robots(seed, n_robots=6, drop=(0.0, 1e-3), tol_primal=-1, max_iters=60)
    net = lr.init_network(seed=seed)
    net.set_params((gain * net.get_params()).astype(np.float32))
    a, b = sa.Simulation(p), sa.Simulation(p, grid_side_rows=1)
    for _ in range(6):
        a.step_learned(net, 1)
        b.step_learned(net, 1)
        sa_, sb = a.iteration_stats(), b.iteration_stats()
        assert sa_["fallbacks"] == sb["fallbacks"] and sa_["total_iters"] == sb["total_iters"]
        for k in range(6):
            assert _rel(b.scene_vhat(k), a.scene_vhat(k)) < 1e-5


@pytest.mark.parametrize("kind,precision", [("cached", 0), ("cached", 1), ("generic", 0), ("generic", 1),
                                            ("grid", 0), ("grid", 1), ("grid, rows streamed", 0)])
def test_not_a_number_is_above_no_tolerance(kind, precision):
    """With every velocity a NaN, no residual is finite and above the tolerance after the first
    iteration: the step ends there, not at its limit, and reports SIM_ENAN."""
    import torch
    from paper_2302_14344_gb300 import subadmm as sa
    small = kind in ("cached", "grid")
    p = (sg.chain(2, n_links=8, links_per_sub=2, tol_primal=1e-6, max_iters=200) if small else
         sg.batched(5, n_scenes=2, tol_primal=1e-6, max_iters=200))
    grid = kind.startswith("grid")
    sim = sa.Simulation(p, precision=precision, grid_side_rows=1 if grid else None)
    sim.grid_blocks(1 if "streamed" in kind else 0)
    assert all(c["cached"] in ([2] if grid else [1] if small else [0, 3]) for c in sim.launch_classes())
    sz = sim.sizes()
    st = torch.empty(13 * sz["bodies"] + 6 * sz["nodes"], dtype=torch.float64).pin_memory()
    sa.sim_read_state(sim.h, st.data_ptr())
    st[:13 * sz["bodies"]].view(-1, 13)[:, 7:] = float("nan")
    st[13 * sz["bodies"]:].view(-1, 6)[:, 3:] = float("nan")
    sa.sim_write_state(sim.h, st.data_ptr())
    sim.step(1)
    for k in range(len(p.scenes)):
        with pytest.raises(sa.SimError) as ei:
            sim.residuals(k)
        assert ei.value.code == sa.SIM_ENAN
    assert sim.iteration_stats()["total_iters"] == len(p.scenes)
