"""Blocks that are not positive definite, in the factorisations that run after the setup launch: the
banded one (FP32 and FP64, clusters) and the blocked one on the tensor cores (envelopes wider than the
banded one takes).  The step ends with SIM_ENOTSPD and leaves the state, and a later step with a
proper block is the oracle's."""
import numpy as np
import pytest

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-30))


def _problem(n, at):
    """One dense block of n DOF with the leading minor of order at + 2 negative (eigenvalue -1), unit
    diagonal (not stiff), and 18 rows away from there."""
    rng = np.random.default_rng(n)
    A = np.eye(n)
    A[at, at + 1] = A[at + 1, at] = 2.0
    ifs = []
    for k in range(6):
        J = np.zeros((3, n))
        lo = (at + 8 + (n // 8) * k) % (n - 8)
        J[:, lo:lo + 8] = rng.standard_normal((3, 8))
        J[:, max(0, at - 1):at + 3] = 0.0
        ifs.append(sg.RowsIf(sg.EQUALITY, [0], [J], np.zeros(3)))
    b = np.ones(n)
    return A, b, sg.Problem([sg.Scene([sg.GenericSub(A, b)], ifs)],
                            sg.Options(gravity=(0, 0, 0), max_iters=10, tol_primal=-1))


# (FP32 panels of 32 columns, FP64 of 16, the tensor-core path's of 128: the first panel, a later one, the
# last, ragged one)
@pytest.mark.parametrize("precision,n,at", [(0, 160, 0), (0, 160, 75), (0, 385, 381), (1, 160, 75), (1, 383, 379),
                                            (1, 420, 0), (1, 420, 200), (1, 420, 416)])
def test_indefinite_blocks(precision, n, at):
    from paper_2302_14344_gb300 import subadmm as sa
    A, b, p = _problem(n, at)
    sim = sa.Simulation(p, precision=precision, grid_side_rows=1)
    for _ in range(2):
        sim.step(1)
        with pytest.raises(sa.SimError) as ei:
            sim.residuals(0)
        assert ei.value.code == sa.SIM_ENOTSPD
    A[at, at + 1] = A[at + 1, at] = 0.5
    sa.sim_set_generic(sim.h, sim.sub_ids[0][0], A, b)
    sim.step(1)
    assert sim.residuals(0)["status"] == 0
    o = oracle.OracleScene(p.scenes[0], p.options)
    o.step()
    assert _rel(sim.scene_vhat(0), o.vhat_all()) < (1e-4 if precision else 1e-9)
