"""Co-rotational blocks whose rest stiffness is given by fewer entries than their rotated elements
fill: the entries of A come from the elements, whatever the triplets list."""
import numpy as np
import pytest

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-30))


def _thin(p, keep):
    for s in p.scenes[0].subs:
        if not getattr(s, "corot", False):
            continue
        i, j = np.asarray(s.Ki), np.asarray(s.Kj)
        use = j % 3 == 0 if keep == "one column of a node pair" else i >= j
        if keep == "one column of a node pair":
            use |= (i % 3 == 0) & (i < j)             # (and its mirror image)
        s.Ki, s.Kj, s.Kv = i[use], j[use], np.asarray(s.Kv)[use]
    return p


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("keep", ["one column of a node pair", "lower triangle"])
def test_rotated_elements_count_whole(keep, precision):
    """The same beam with all of K's entries and with some left out (the envelope the same): v-hat of
    three steps, in FP64 to 1e-9 of the oracle, in the mixed form to 1e-4 (FP32 iterates, see the
    banded factorisation's test)."""
    from paper_2302_14344_gb300 import subadmm as sa
    args = dict(ny=6, nz=7, planes=6, slabs=2, length=0.02, corotational=True, with_gripper=False,
                tol_primal=-1, max_iters=15)
    whole = sg.fem_beam(0, **args)
    sim = sa.Simulation(_thin(sg.fem_beam(0, **args), keep), precision=precision, grid_side_rows=1)
    o = oracle.OracleScene(whole.scenes[0], whole.options)
    for _ in range(3):
        sim.step(1)
        o.step()
        assert _rel(sim.scene_vhat(0), o.vhat_all()) < (1e-4 if precision else 1e-9)
