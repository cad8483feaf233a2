"""Steps of grid scenes captured by the caller into a CUDA graph: the first step, right after the layout,
allocates nothing, and a graph keeps its iteration layout when the block count changes later."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-30))


def _pair(p, **kw):
    import torch
    from paper_2302_14344_gb300 import subadmm as sa
    st = torch.cuda.Stream()
    return st, sa.Simulation(p, stream=st.cuda_stream, grid_side_rows=1, **kw), sa.Simulation(p, grid_side_rows=1, **kw)


def _capture(st, sim):
    import torch
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=st):
        sim.step(1)
    return g


def _replay(st, g, n=1):
    import torch
    with torch.cuda.stream(st):
        for _ in range(n):
            g.replay()
    torch.cuda.synchronize()


def test_first_step_of_refactorised_fp64_blocks():
    """Co-rotational slabs in FP64 (the banded factorisation): two replays are two direct steps (1e-12: the
    element pass adds with atomics)."""
    p = sg.fem_beam(0, ny=7, nz=7, planes=6, slabs=2, length=0.02, corotational=True, with_gripper=False,
                    tol_primal=-1, max_iters=15)
    st, a, b = _pair(p)
    a.launch_classes()
    g = _capture(st, a)
    _replay(st, g, 2)
    b.step(2)
    assert _rel(a.scene_vhat(0), b.scene_vhat(0)) < 1e-12
    assert _rel(a.scene_nodes(0), b.scene_nodes(0)) < 1e-12


@pytest.mark.parametrize("precision,tol", [(0, -1.0), (0, 1e-5), (1, -1.0)])
def test_graph_outlives_a_change_of_the_block_count(precision, tol):
    """Captured on the default block count, replayed after direct steps on 3 and on 7 blocks: the steps of
    a simulation without graphs (1e-12 in FP64; 1e-4 in FP32, whose sums a layout orders)."""
    p = sg.stir(1, n_side=3, layers=3, tol_primal=tol, max_iters=40)
    st, a, b = _pair(p, precision=precision)
    a.launch_classes()
    g = _capture(st, a)
    _replay(st, g)
    for blocks in (3, 7):
        a.grid_blocks(blocks)
        a.step(1)
        a.sync()
        _replay(st, g)
    b.step(5)
    assert _rel(a.scene_vhat(0), b.scene_vhat(0)) < (1e-4 if precision else 1e-12)
