"""A batch ends where its boxes end alone, bit for bit, also with more particles
than one block takes: there a box alone runs its subcycles in one launch and a
batch in a launch each, after a launch of the first position update."""
import numpy as np
import pytest

from cases import build_gpu, spheres

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('storage', ['f32', 'bf16'])
@pytest.mark.parametrize('n_sub', [3, 6, 7])
def test_many_particles_in_a_batch_end_where_they_end_alone(n_sub, storage):
    from paper_2003_01490_gb300 import lbmdem as L
    # light spheres pulled from rest out of the planes through the origin, where
    # the last bits of a position are small enough to show those of its increments
    rng = np.random.default_rng(n_sub)
    k = np.stack(np.meshgrid(np.arange(24), np.arange(24), np.arange(1), indexing='ij'), -1).reshape(-1, 3)
    n = len(k)
    case = dict(shape=(120, 120, 9), periodic=(1, 1, 1), tau=0.9, storage=storage,
                spheres=spheres(k * 5.0, rng.uniform(1.3, 1.6, n), density=rng.uniform(1.2, 1.8, n),
                                omega=rng.normal(0.0, 1e-3, (n, 3))),
                dem=dict(gravity=(1e-3, 1.1e-3, 1.2e-3), n_sub=n_sub, fluid_counterforce=1))
    alone, other = build_gpu(case), build_gpu(case)
    L.lbm_step(alone, 2)
    L.lbm_step(other, 1)
    b = L.lbm_batch_create([other])
    L.lbm_batch_set_launch(b, 0, 128, 1, 4)      # the single launch's chunk of planes
    L.lbm_batch_step(b, 1)
    L.lbm_batch_sync(b)
    x, y = L.lbm_get_particle_state(alone), L.lbm_get_particle_state(other)
    for key in ('pos', 'vel', 'omega', 'force_hyd', 'torque_hyd'):
        assert np.array_equal(x[key], y[key]), key
