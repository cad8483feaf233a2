"""The grid's iteration kernel (one scene over the whole GPU, one barrier or tagged exchange per
iteration) against the FP64 oracle at the edges of its layouts: items of up to 8 sides, subsystems
narrower and wider than a vector per lane, few warps (rows streamed, and more side-rows than
lanes: the two-barrier kernel), stop at the tolerance, warm starts over several steps and
single-iteration steps.  FP64 tolerance 1e-9 relative (the project's parity bound); FP32 iterates
carry 2^-24 per operation through a K^-1 of modest condition: 1e-4 relative after 40 iterations."""
import numpy as np
import pytest

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-30))


def _run(problem, steps=2, blocks=0, precision=0, calls=1):
    from paper_2302_14344_gb300 import subadmm as sa
    sim = sa.Simulation(problem, precision=precision, grid_side_rows=1)
    sim.grid_blocks(blocks)
    for _ in range(calls):
        sim.step(steps)
    orcs = oracle.run(problem, steps=steps * calls)
    out = []
    for k, o in enumerate(orcs):
        assert sim.residuals(k)["status"] == 0
        out.append((sim, k, o))
    return out


@pytest.mark.parametrize("blocks", [0, 1, 5])
@pytest.mark.parametrize("dof,subs,sides", [((1, 5), 9, 8), ((20, 90), 7, 4), ((130, 170), 3, 3)])
@pytest.mark.parametrize("warm", ["cold", "prev"])
def test_layouts_fp64(blocks, dof, subs, sides, warm):
    p = sg.generic(7, n_scenes=2, n_sub=subs, n_range=dof, max_sides=sides, extra=40,
                   tol_primal=-1, max_iters=25, warm=warm)
    for sim, k, o in _run(p, blocks=blocks):
        assert _rel(sim.scene_vhat(k), o.vhat_all()) < 1e-9
        assert _rel(sim.scene_lam(k), o.lam_all()) < 1e-9


@pytest.mark.parametrize("blocks", [0, 2])
def test_layouts_mixed(blocks):
    p = sg.generic(8, n_scenes=2, n_sub=8, n_range=(4, 60), max_sides=5, extra=60,
                   tol_primal=-1, max_iters=40, warm="prev")
    for sim, k, o in _run(p, blocks=blocks, precision=1):
        assert _rel(sim.scene_vhat(k), o.vhat_all()) < 1e-4


@pytest.mark.parametrize("iters", [1, 2, 3])
def test_first_iterates_and_residuals(iters):
    """After one, two and three iterations the iterates of the iteration before are the initial
    ones, then the first: residuals, z and lambda against the oracle, over repeated calls (the
    exchange's tags go on from call to call)."""
    p = sg.stir(1, n_side=3, layers=2, tol_primal=-1, max_iters=iters)
    for sim, k, o in _run(p, steps=1, calls=4):
        assert _rel(sim.scene_vhat(k), o.vhat_all()) < 1e-9
        r, q = sim.residuals(k), o.residuals()
        assert np.isclose(r["r_p"], q["r_p"], rtol=1e-7) and np.isclose(r["r_d"], q["r_d"], rtol=1e-7)
        assert r["iters"] == iters


def test_stop_at_the_tolerance():
    p = sg.chain(2, n_links=24, links_per_sub=2, rho=None, max_iters=4000, tol_primal=1e-7)
    for sim, k, o in _run(p, steps=1, calls=3):
        r, q = sim.residuals(k), o.residuals()
        assert r["converged"] and r["iters"] == q["iters"]
        assert _rel(sim.scene_vhat(k), o.vhat_all()) < 1e-9


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ny,nz,planes,slabs", [(7, 7, 4, 1), (8, 9, 6, 2), (10, 10, 8, 3)])
def test_refactorised_bands(precision, ny, nz, planes, slabs):
    """Co-rotational slabs (n = 588 .. 1200, ragged against the panels of 16 and 32 columns), refactorised
    every step by the banded factorisation, against the oracle over two steps."""
    p = sg.fem_beam(0, ny=ny, nz=nz, planes=planes, slabs=slabs, length=0.004 * planes, corotational=True,
                    with_gripper=False, tol_primal=-1, max_iters=15)
    for sim, k, o in _run(p, steps=1, calls=2, precision=precision):
        assert _rel(sim.scene_vhat(k), o.vhat_all()) < (1e-4 if precision else 1e-9)
        assert _rel(sim.scene_nodes(k), o.nodes_all()) < (1e-5 if precision else 1e-9)


def test_wide_envelopes_take_the_tensor_core_factorisation():
    """Dense blocks (envelopes wider than the banded factorisation takes) in the mixed form, every
    step refactorised: the blocked factorisation on the tensor cores, against the oracle."""
    p = sg.generic(9, n_scenes=1, n_sub=3, n_range=(400, 420), extra=12, tol_primal=-1, max_iters=20, warm="prev")
    for sim, k, o in _run(p, steps=1, calls=2, precision=1):
        assert _rel(sim.scene_vhat(k), o.vhat_all()) < 1e-4
