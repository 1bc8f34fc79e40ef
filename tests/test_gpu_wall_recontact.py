"""Spheres that leave a wall and meet it again within one time step: a new wall
contact starts from a spring of zero length (the one of the last contact ended
with it, Eq. (49)), whichever launch runs the subcycles: one block, one cluster, a
grid, and in a batch one block per box or a launch per subcycle."""
import numpy as np
import pytest

from cases import build_gpu, build_oracle, rel_l2, spheres

pytestmark = pytest.mark.gpu


def slit(n, storage, n_sub=20):
    """n spheres in a slit 0.004 cells wider than they are, between sliding walls:
    with contacts of 0.2 time steps each bounces between the walls several
    times a step."""
    rows, pitch = (1, 1) if n == 1 else (3, n // 3), 10.0
    radius = 0.5 * (9.0 - 0.004)
    shape = (14, 14, 9) if n == 1 else (int(pitch * rows[1]), int(pitch * rows[0]), 9)
    at = [[shape[0] * (i + 0.5) / rows[1], shape[1] * (j + 0.5) / rows[0], 4.5] for j in range(rows[0]) for i in range(rows[1])]
    rng = np.random.default_rng(n)
    vel = rng.uniform(-0.01, 0.01, (n, 3)) + [0.0, 0.0, 0.05]
    return dict(shape=shape, periodic=(1, 1, 0), tau=0.8, storage=storage,
                wall_vel_lo=[[0.0] * 3, [0.0] * 3, [0.03, 0.0, 0.0]],
                wall_vel_hi=[[0.0] * 3, [0.0] * 3, [-0.02, 0.02, 0.0]],
                spheres=spheres(at, np.full(n, radius), density=np.full(n, 8.0), vel=vel,
                                omega=rng.uniform(-0.002, 0.002, (n, 3))),
                dem=dict(Tc=0.2, n_sub=n_sub, lubrication=0, mu_p=0.4))


def count_recontacts(ora):
    """Contacts with a wall that the particle touched before in the same step, but
    not in the subcycle before (counted in ora.recontacts)."""
    ora.recontacts = 0
    seen, forces, cycles = set(), ora.dem_forces, ora.dem_subcycles

    def dem_forces(*args, **kw):
        before = set(ora.hist)
        out = forces(*args, **kw)
        now = {k for k in ora.hist if k[1] == 'wall'}
        ora.recontacts += len((now - before) & seen)
        seen.update(now)
        return out

    def dem_subcycles(*args):
        seen.clear()
        seen.update(k for k in ora.hist if k[1] == 'wall')
        return cycles(*args)

    ora.dem_forces, ora.dem_subcycles = dem_forces, dem_subcycles


# float64: a few ulp per operation, times the stiffness of a contact (16 of its
# radians a step) in two steps of 20 subcycles. float32 laws: a spring of 2^-24
# relative and gaps of 1e-3 known to 2^-24 of themselves are 1e-6 of a force, which
# two steps of contact turn into 1e-4 of the velocities
@pytest.mark.parametrize('storage,tol', [('f64', 1e-10), ('f32', 1e-4)])
@pytest.mark.parametrize('n', [1, 33])
def test_a_new_wall_contact_starts_without_a_spring(n, storage, tol):
    from paper_2003_01490_gb300 import lbmdem as L
    case = slit(n, storage)
    ora, ctx = build_oracle(case), build_gpu(case)
    count_recontacts(ora)
    ora.step(2)
    L.lbm_step(ctx, 2)
    st = L.lbm_get_particle_state(ctx)
    assert ora.recontacts >= 2 * n
    assert rel_l2(st['pos'], ora.X) < tol
    assert rel_l2(st['vel'], ora.U) < tol
    assert rel_l2(st['omega'], ora.Om) < tol


@pytest.mark.parametrize('storage', ['f32', 'f16'])
@pytest.mark.parametrize('n', [1, 33])
def test_a_batch_ends_where_its_boxes_end_alone(n, storage):
    from paper_2003_01490_gb300 import lbmdem as L
    case = slit(n, storage)
    alone, other = build_gpu(case), build_gpu(case)
    L.lbm_step(alone, 4)
    L.lbm_step(other, 1)
    b = L.lbm_batch_create([other])
    L.lbm_batch_set_launch(b, 0, 32 if n == 1 else 128, 1, 4)      # the single launch's chunk of planes
    L.lbm_batch_step(b, 3)
    L.lbm_batch_sync(b)
    x, y = L.lbm_get_particle_state(alone), L.lbm_get_particle_state(other)
    for k in ('pos', 'vel', 'omega', 'force_hyd', 'torque_hyd'):
        assert np.array_equal(x[k], y[k]), k
