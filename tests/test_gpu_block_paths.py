"""The block kernel's narrow-band factorisation and solves, its iterations with side-rows owned by
threads, and D copied to shared memory from the workspace, against the FP64 oracle (1e-9 relative,
the project's parity bound) at the sizes where they can go wrong: bands at and around the 32 rows
a warp holds, more side-rows than threads, more than a thread owns."""
import numpy as np
import pytest

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-30))


def _check(problem, steps=2, precision=0, tol=1e-9, iters=False):
    from paper_2302_14344_gb300 import subadmm as sa
    sim = sa.Simulation(problem, precision=precision)
    sim.step(steps)
    for k, o in enumerate(oracle.run(problem, steps=steps)):
        r = sim.residuals(k)
        assert r["status"] == 0
        assert _rel(sim.scene_vhat(k), o.vhat_all()) < tol
        if iters:
            assert r["iters"] == o.residuals()["iters"]
    return sim


# DOF 6 .. 252 in one subsystem: shorter than a warp's window, just past it, many windows
@pytest.mark.parametrize("links", [1, 2, 5, 6, 11, 42])
def test_chains_in_one_subsystem(links):
    _check(sg.chain(3, n_links=2 * links, links_per_sub=links, tol_primal=-1, max_iters=20))


# generic blocks are dense: bands of n - 1 around the narrow limit of 31
@pytest.mark.parametrize("n", [31, 32, 33, 34, 48])
def test_dense_blocks_around_the_narrow_limit(n):
    _check(sg.generic(n, n_scenes=2, n_sub=4, n_range=(n, n), max_sides=2, extra=4, tol_primal=-1,
                      max_iters=20, warm="prev"))


@pytest.mark.parametrize("precision,tol", [(0, 1e-9), (1, 3e-3)])
@pytest.mark.parametrize("contacts", [(0, 0), (60, 64), (200, 220)])
def test_uneven_scenes(precision, tol, contacts):
    """Scenes of 20 to 32 subsystems, without and with many contacts (node contacts between rows of
    other types).  Mixed: the poorly conditioned scenes' FP32 iterates, 3e-3 after 15 iterations
    from a cold start (their step is known to 1e-2 at r_p <= 1e-6)."""
    p = sg.batched(5, n_scenes=4, n_sub=(20, 32), contacts=contacts, tol_primal=-1, max_iters=15)
    sim = _check(p, precision=precision, tol=tol)
    if precision == 0 and contacts[0] >= 60:
        assert max(sim_place(sim, k) for k in range(4)) == 2      # D in the workspace


def sim_place(sim, k):
    from paper_2302_14344_gb300 import subadmm as sa
    return sa.sim_scene_info(sim.h, k)["placement"]


def test_stop_at_the_tolerance_after_as_many_iterations_as_the_oracle():
    _check(sg.batched(6, n_scenes=6, n_sub=(2, 6), n_range=(6, 60), tol_primal=1e-6, max_iters=2000),
           steps=1, tol=1e-9, iters=True)


@pytest.mark.parametrize("iters", [1, 2, 3])
def test_last_iterates_and_residuals(iters):
    from paper_2302_14344_gb300 import subadmm as sa
    for p in (sg.batched(7, n_scenes=2, tol_primal=-1, max_iters=iters),
              sg.robots(1, n_robots=2, drop=(0.0, 1e-3), tol_primal=-1, max_iters=iters)):
        sim = sa.Simulation(p)
        sim.step(3)
        for k, o in enumerate(oracle.run(p, steps=3)):
            r, q = sim.residuals(k), o.residuals()
            for key in ("r_p", "r_d"):
                assert np.isclose(r[key], q[key], rtol=1e-6, atol=1e-18)
            assert _rel(sim.scene_vhat(k), o.vhat_all()) < 1e-9
