"""The dense kernel at the sizes where its link work can go wrong, against the
oracle: box widths around the 32 bits of a row's words, an odd number of rows,
one plane per block and several, more particles in a warp's cells than it
keeps open, more links in a plane than its queue holds, walls on every axis,
and spheres that overlap (their links' constant force parts come from the cells
next to another body).

Float64 bound: both sides round differently in summation order only, 1e-16 per
operation over a few steps (1e-11). Float32: forces are sums of remainders of
~1e-3 with a relative rounding of 2^-24 in each of a few operations (1e-5);
velocities 1e-6.
"""
import numpy as np
import pytest

from cases import build_gpu, build_oracle, spheres, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope='module')
def L():
    torch = pytest.importorskip('torch')
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    from paper_2003_01490_gb300 import lbmdem
    lbmdem.load_library()
    return lbmdem


def packed(shape, pitch, radius, seed):
    """Spheres on a jittered lattice of the given pitch, with random velocities."""
    r = np.random.default_rng(seed)
    n = [int(s // pitch) for s in shape]
    k = np.stack(np.meshgrid(*[np.arange(v) for v in n], indexing='ij'), -1).reshape(-1, 3)
    step = np.array(shape) / np.array(n)
    room = 0.5 * (step - 2.0 * radius) - 0.05
    pos = (k + 0.5) * step + room * r.uniform(-1.0, 1.0, k.shape)
    m = len(pos)
    return spheres(pos, np.full(m, radius), density=np.full(m, 2.0), vel=0.02 * r.standard_normal((m, 3)),
                   omega=0.01 * r.standard_normal((m, 3)))


CASES = {
    # width, rows, planes; periodicity; sphere pitch and radius
    'one word less one': ((31, 9, 10), (1, 1, 1), 7.0, 2.3),
    'one word and one': ((33, 11, 12), (1, 1, 1), 8.0, 2.4),
    'two words and a half': ((80, 10, 9), (1, 0, 1), 8.0, 2.2),
    'walls on every axis': ((40, 13, 11), (0, 0, 0), 6.0, 2.0),
    'many small spheres': ((64, 8, 8), (1, 1, 1), 3.0, 1.3),
    'five words': ((131, 9, 8), (0, 1, 1), 6.0, 1.9),
}


@pytest.mark.parametrize('storage', ['f64', 'f32'])
@pytest.mark.parametrize('name', sorted(CASES))
def test_link_work_at_the_edges_matches_the_oracle(L, name, storage):
    shape, periodic, pitch, radius = CASES[name]
    case = dict(shape=shape, periodic=periodic, tau=0.7, storage=storage, body_force=(2e-5, -1e-5, 3e-5),
                wall_vel_hi=[[0.0, 0.01, 0.0], [0.01, 0.0, 0.02], [0.02, 0.01, 0.0]],
                spheres=packed(shape, pitch, radius, 5), dem=dict(fixed_particles=1))
    ora, ctx = build_oracle(case), build_gpu(case)
    ora.step(4)
    L.lbm_step(ctx, 4)
    st = L.lbm_get_particle_state(ctx)
    _, u, _ = L.lbm_get_fields(ctx)
    _, u_o = ora.fields()
    f_tol, u_tol = (1e-11, 1e-11) if storage == 'f64' else (1e-5, 1e-6)
    assert rel_l2(st['force_hyd'], ora.Ffp) < f_tol
    assert rel_l2(st['torque_hyd'], ora.Tfp) < f_tol
    assert rel_l2(u, u_o) < u_tol


@pytest.mark.parametrize('missing', [1, 0])
@pytest.mark.parametrize('storage', ['f64', 'f32'])
def test_forces_of_overlapping_spheres_match_the_oracle(L, storage, missing):
    # two spheres pushed into each other and one into the wall by prescribed
    # velocities, with cells inside both spheres, with and without the
    # missing-link correction
    case = dict(shape=(40, 24, 26), periodic=(1, 1, 0), tau=0.6, storage=storage,
                spheres=spheres([[12.2, 11.9, 12.3], [22.9, 12.4, 13.1], [31.5, 12.2, 4.1]], [5.0, 5.4, 3.8],
                                vel=[[0.04, 0.0, 0.0], [-0.04, 0.003, 0.0], [0.0, 0.01, -0.08]],
                                omega=[[0.0, 0.002, 0.0], [0.001, 0.0, 0.0], [0.0, 0.0, 0.003]]),
                dem=dict(fixed_particles=2, missing_links=missing))
    ora, ctx = build_oracle(case), build_gpu(case)
    ora.step(24)
    L.lbm_step(ctx, 24)
    st = L.lbm_get_particle_state(ctx)
    assert (L.lbm_get_fields(ctx)[2] & L.FLAG_MULTI).any()
    tol = 1e-10 if storage == 'f64' else 2e-5
    assert rel_l2(st['force_hyd'], ora.Ffp) < tol
    assert rel_l2(st['torque_hyd'], ora.Tfp) < tol
