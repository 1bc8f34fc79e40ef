"""The DEM step without its one-launch forms: where the cooperative launch has no
room, the step runs as one launch per subcycle, and ends in the same bits."""
import ctypes

import numpy as np
import pytest

from cases import build_gpu, spheres

pytestmark = pytest.mark.gpu

KEYS = ('pos', 'vel', 'omega', 'force_hyd', 'torque_hyd')


@pytest.fixture(scope='module')
def L():
    torch = pytest.importorskip('torch')
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    from paper_2003_01490_gb300 import lbmdem
    return lbmdem


def set_capacity(L, ctx, grid, cluster):
    f = L.load_library().lbmdem_set_dem_capacity
    f.argtypes, f.restype = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int], None
    f(ctx.handle, grid, cluster)


def lattice(sites, storage, n_sub, walls=0):
    k = np.stack(np.meshgrid(*[np.arange(s) for s in sites], indexing='ij'), -1).reshape(-1, 3)
    rng = np.random.default_rng(len(k))
    pos = 5.0 * k + 2.5 + rng.uniform(-0.09, 0.09, (len(k), 3))
    return dict(shape=tuple(5 * s for s in sites), periodic=(1, 1, 1 - walls), tau=0.7, storage=storage,
                spheres=spheres(pos, np.full(len(k), 2.4), density=np.full(len(k), 20.0),
                                vel=rng.normal(0.0, 0.02, (len(k), 3)), omega=rng.normal(0.0, 0.005, (len(k), 3))),
                relax=dict(shell_width=1.0), dem=dict(gravity=(1e-4, 0.0, -2e-4), n_sub=n_sub))


# float64: the fluid's forces are sums of atomics in any order (1e-16 of themselves a step)
@pytest.mark.parametrize('storage', ['f32', 'f64'])
@pytest.mark.parametrize('sites,n_sub,walls', [((4, 4, 3), 10, 1), ((6, 5, 5), 7, 0), ((9, 9, 8), 10, 1)])
def test_subcycle_launches_end_where_the_one_launch_ends(L, sites, n_sub, walls, storage):
    case = lattice(sites, storage, n_sub, walls)
    a, b = build_gpu(case), build_gpu(case)
    set_capacity(L, b, 0, 0)
    for ctx in (a, b):
        L.lbm_step(ctx, 5)
    x, y = L.lbm_get_particle_state(a), L.lbm_get_particle_state(b)
    assert L.lbm_launch_count(b) >= L.lbm_launch_count(a) + 5 * n_sub
    for k in KEYS:
        if storage == 'f32':
            assert np.array_equal(x[k], y[k]), k
        else:
            assert np.abs(x[k] - y[k]).max() <= 1e-11 * np.abs(x[k]).max(), k


@pytest.mark.parametrize('before', [0, 1, 2])     # refused in the first step, in a capture, after a graph
def test_a_refused_cooperative_launch_falls_back(L, before):
    case = lattice((30, 24, 22), 'f32', 4)     # more particles than one launch holds
    a, b = build_gpu(case), build_gpu(case)
    L.lbm_step(a, before + 3)
    L.lbm_step(b, before)
    set_capacity(L, b, 1 << 22, 0)
    L.lbm_step(b, 3)
    x, y = L.lbm_get_particle_state(a), L.lbm_get_particle_state(b)
    for k in KEYS:
        assert np.array_equal(x[k], y[k]), k
