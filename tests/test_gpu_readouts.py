"""Read-outs and velocity updates on both sides of the size up to which they go
through a context's page-locked memory, against the other read-outs."""
import numpy as np
import pytest

from cases import build_gpu, spheres

pytestmark = pytest.mark.gpu


def lattice(n, storage='f64'):
    cells = np.array([(i, j, k) for k in range(12) for j in range(12) for i in range(12)])[:n]
    rng = np.random.default_rng(n)
    return build_gpu(dict(shape=(72, 72, 72), periodic=(1, 1, 1), tau=0.7, storage=storage,
                          spheres=spheres(6.0 * cells + 3.0, np.ones(n), vel=rng.normal(0.0, 0.01, (n, 3)),
                                          omega=rng.normal(0.0, 0.01, (n, 3)))))


@pytest.mark.parametrize('n', [1, 546, 547])
def test_particle_state(n):
    from paper_2003_01490_gb300 import lbmdem as L
    ctx = lattice(n)
    L.lbm_step(ctx, 2)
    keys = ('pos', 'vel', 'omega', 'force_hyd', 'torque_hyd')
    out = {k: np.zeros((n, 3)) for k in keys}
    L.lbm_get_particle_state_async(ctx, out)
    L.lbm_sync(ctx)
    got = L.lbm_get_particle_state(ctx)
    assert all(np.array_equal(got[k], out[k]) for k in keys) and np.any(got['force_hyd'])


@pytest.mark.parametrize('rows', [1, 1365, 1366])
def test_set_velocity(rows):
    from paper_2003_01490_gb300 import lbmdem as L
    ctx = lattice(1366)
    before = L.lbm_get_particle_state(ctx)
    vel, omega = np.random.default_rng(rows).normal(0.0, 0.01, (2, rows, 3))
    L.lbm_set_particle_velocity(ctx, vel, None)
    L.lbm_set_particle_velocity(ctx, None, omega)
    got = L.lbm_get_particle_state(ctx)
    assert np.array_equal(got['vel'], np.concatenate([vel, before['vel'][rows:]]))
    assert np.array_equal(got['omega'], np.concatenate([omega, before['omega'][rows:]]))


# float64 storage: eight weighted densities near 1, a few ulp
@pytest.mark.parametrize('n', [1, 2047, 2048])
def test_sampled_density(n):
    from paper_2003_01490_gb300 import lbmdem as L
    ctx = lattice(40)
    L.lbm_step(ctx, 2)
    rho, _, flags = L.lbm_get_fields(ctx)
    rho = np.where((flags & L.FLAG_SOLID) != 0, 1.0, rho)
    x = np.random.default_rng(n).uniform(0.0, 72.0, (n, 3))
    i = np.floor(x - 0.5).astype(int)
    t = x - 0.5 - i
    want = np.zeros(n)
    for c in range(8):
        o = np.array([c & 1, c >> 1 & 1, c >> 2])
        w = np.where(o, t, 1.0 - t).prod(1)
        j = (i + o) % 72
        want += w * rho[j[:, 2], j[:, 1], j[:, 0]]
    assert np.abs(L.lbm_sample_density(ctx, x) - want).max() < 1e-14
