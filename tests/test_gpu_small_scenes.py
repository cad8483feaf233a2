"""The register-cached iteration at its smallest scenes, whose rows are shorter than the vectors that
a lane group takes together."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu


def _body(mu, k=0):
    b = sg.Body(m=1.0 + 0.1 * k, I=np.full(3, 1e-3), p=np.array([0.0, 0.0, -1e-4]), q=np.array([1.0, 0, 0, 0]),
                v=np.array([0.3, 0.0, -0.1]), w=np.zeros(3))
    return sg.Scene([sg.RigidSub([b])],
                    [sg.JointIf(sg.PLANE_CONTACT, a=(0, 0), anchor_a=np.zeros(3), plane_z=0.0, mu=mu)])


def _problem(scenes):
    return sg.Problem(scenes, sg.Options(h=1e-3, tol_primal=-1, max_iters=30, beta_mode="trace"))


@pytest.mark.parametrize("precision", [0, 1])
def test_unlimited_friction(precision):
    """One body on a plane with a friction coefficient that is infinite in FP32: sticks, as with any
    large one, bit for bit."""
    from paper_2302_14344_gb300 import subadmm as sa
    got = []
    for mu in (1e15, 1e39):
        sim = sa.Simulation(_problem([_body(mu)]), precision=precision)
        assert sim.launch_classes()[0]["cached"] == 1
        sim.step(3)
        assert sim.residuals(0)["status"] == 0
        got.append(sim.scene_vhat(0))
    assert np.all(np.isfinite(got[0])) and np.array_equal(got[0], got[1])


def test_small_scenes_beside_large_ones():
    """Scenes of one body, alone and in a launch with larger scenes before and between them: the same
    bits (nothing of a step depends on what shared memory held)."""
    from paper_2302_14344_gb300 import subadmm as sa
    alone = sa.Simulation(_problem([_body(0.5, k) for k in range(8)]), precision=1)
    alone.step(2)
    rest = sg.robots(3, n_robots=200).scenes
    sim = sa.Simulation(_problem(rest + [_body(0.5, k) for k in range(8)]), precision=1)
    for _ in range(2):
        sim.step(1)
    for k in range(8):
        assert np.array_equal(sim.scene_vhat(200 + k), alone.scene_vhat(k))
