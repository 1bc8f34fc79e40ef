"""The particle step at the sizes where its launch changes shape, between six
walls, against the oracle: one block up to 32 particles, with float32 laws one
cluster up to 512, a grid above; odd and even numbers of subcycles; contacts with
walls of either side of every axis, all of them moving, close partners, unequal
radii."""
import numpy as np
import pytest

from cases import build_gpu, build_oracle, rel_l2, spheres

pytestmark = pytest.mark.gpu


def packed_case(n, n_sub, storage):
    """n spheres on a jittered lattice; the outer ones run into the six walls."""
    rng = np.random.default_rng(n)
    pitch, radius = 5.0, 2.35 + 0.1 * rng.random(n)     # small gaps, no overlap at the start
    sites = (4, 4, 3) if n <= 48 else (9, 9, 7)
    cells = np.array([(i, j, k) for k in range(sites[2]) for j in range(sites[1]) for i in range(sites[0])])
    # few spheres sit in opposite corners
    pick = np.arange(n) if n > 2 else np.array([0, 47])[:n]
    side = pitch * np.array(sites)
    pos = (cells[pick] + 0.5) * pitch + rng.uniform(-0.045, 0.045, (n, 3))
    # the outer ones close to their walls and on their way into them
    reach = radius[:, None] + 0.004
    low, high = pos < 3.0, pos > side - 3.0
    pos = np.where(low, reach, np.where(high, side - reach, pos))
    toward = 0.03 * high - 0.03 * low
    lo = [[0.0, 0.004, -0.002], [0.003, 0.0, 0.0], [0.0, -0.005, 0.0]]
    hi = [[0.0, 0.0, 0.003], [0.0, 0.0, -0.004], [0.006, 0.0, 0.0]]
    return dict(shape=tuple(int(v) for v in side), periodic=(0, 0, 0), tau=0.7, storage=storage, wall_vel_lo=lo, wall_vel_hi=hi,
                spheres=spheres(pos, radius, density=rng.uniform(20.0, 40.0, n), vel=toward + rng.normal(0.0, 0.005, (n, 3)),
                                omega=rng.normal(0.0, 0.003, (n, 3))),
                dem=dict(gravity=(1e-4, -5e-5, -2e-4), Tc=8.0, n_sub=n_sub))


# float64: the laws agree to a few ulp and five steps of at most 10 subcycles
# amplify that by the contact stiffness (below 1e3). float32 laws: some twenty
# roundings of 6e-8 per force with up to tenfold cancellation are 1e-5 of the
# velocity change per step, 5e-5 in five steps
@pytest.mark.parametrize('storage,tol', [('f64', 1e-11), ('f32', 1e-4)])
@pytest.mark.parametrize('n,n_sub', [(1, 10), (2, 7), (32, 7), (33, 10), (48, 7)])
def test_packed_box_between_walls(n, n_sub, storage, tol):
    check(packed_case(n, n_sub, storage), tol)


# the float64 one has more missing-link cells than warps that walk them
@pytest.mark.parametrize('n,n_sub,storage,tol', [(512, 10, 'f32', 1e-4), (513, 7, 'f32', 1e-4), (513, 7, 'f64', 1e-11)])
def test_cluster_and_grid(n, n_sub, storage, tol):
    check(packed_case(n, n_sub, storage), tol)


def check(case, tol):
    from paper_2003_01490_gb300 import lbmdem as L
    ora = build_oracle(case)
    ctx = build_gpu(case)
    ora.step(5)
    L.lbm_step(ctx, 5)
    st = L.lbm_get_particle_state(ctx)
    assert any(k[1] == 'wall' for k in ora.hist)
    assert rel_l2(st['pos'], ora.X) < tol
    assert rel_l2(st['vel'], ora.U) < tol
    assert rel_l2(st['omega'], ora.Om) < tol
