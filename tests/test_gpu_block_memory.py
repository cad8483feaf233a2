"""What the block kernel's scenes keep in shared memory, and what they leave to the L1 cache."""
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu


def _sim(problem, precision):
    from paper_2302_14344_gb300 import subadmm as sa
    sim = sa.Simulation(problem, precision=precision)
    return sim, [sa.sim_scene_info(sim.h, k) for k in range(len(problem.scenes))]


def test_D_is_copied_only_where_the_setup_does_not_need_the_cache():
    """Scenes with D in the workspace: uneven scenes of narrow bands copy it to the shared memory that is
    left in the mixed form, not in FP64, and a scene with a wide band (a slab, whose factorisation
    lives on L1) does not: its launch takes what its tables need."""
    kw = dict(tol_primal=-1, max_iters=10)
    beam = sg.fem_beam(0, ny=5, nz=8, planes=6, slabs=2, length=0.016, corotational=True, **kw)
    for precision, contacts in ((0, (60, 64)), (1, (200, 220))):
        sim, info = _sim(sg.batched(5, n_scenes=4, n_sub=(20, 32), contacts=contacts, **kw), precision)
        far = [i["smem_bytes"] for i in info if i["placement"] == 2]
        assert far and all((b > 200000) == (precision == 1) for b in far), far
        sim, info = _sim(beam, precision)
        assert info[0]["placement"] == 2 and info[0]["smem_bytes"] < 90000, info


def test_setup_arrays_stay_on_chip():
    """Tables that only the iterations' start reads take no shared memory: scenes of dense blocks a few
    bytes below half an SM's shared memory keep all of their arrays there."""
    p = sg.generic(3, n_scenes=16, n_sub=5, n_range=(1, 42), extra=6, tol_primal=-1, max_iters=10)
    sim, info = _sim(p, 1)
    assert [i["placement"] for i in info] == [0] * 16, info
    assert max(i["smem_bytes"] for i in info) > 110000
