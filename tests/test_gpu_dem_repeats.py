"""The float64 particle step repeats bit for bit. Its pairs are evaluated from a
queue of the block; here a block has three times as many as threads and a lane
sums three contacts, so the order of its sums depends on the places in the queue.
The spheres are so heavy that the fluid's forces, whose float64 sums depend on the
order of atomics, are below the last bit of the contact forces."""
import numpy as np
import pytest

from cases import build_gpu, spheres

pytestmark = pytest.mark.gpu


def clusters(n, small=24):
    """n spheres (indices 0 .. n - 1) that 24 small ones each run into."""
    k = np.stack(np.meshgrid(np.arange(4), np.arange((n + 3) // 4), indexing='ij'), -1).reshape(-1, 2)[:n]
    centre = np.concatenate([16.0 * k + 8.0, np.full((n, 1), 8.0)], 1)
    i = np.arange(small) + 0.5
    z, a = 1.0 - 2.0 * i / small, np.pi * (1.0 + np.sqrt(5.0)) * i
    d = np.stack([np.sqrt(1.0 - z * z) * np.cos(a), np.sqrt(1.0 - z * z) * np.sin(a), z], -1)
    rng = np.random.default_rng(n)
    gap = rng.uniform(0.002, 0.004, (n, small, 1))
    pos = np.concatenate([centre, (centre[:, None] + (5.2 + gap) * d).reshape(-1, 3)])
    vel = np.concatenate([np.zeros((n, 3)), (-0.02 * d + rng.normal(0.0, 0.003, (n, small, 3))).reshape(-1, 3)])
    radius = np.concatenate([np.full(n, 4.0), np.full(n * small, 1.2)])
    return (64, 16 * ((n + 3) // 4), 16), spheres(pos, radius, density=np.full(len(pos), 1e12), vel=vel)


def test_float64_particle_step_repeats_bit_for_bit():
    from paper_2003_01490_gb300 import lbmdem as L
    shape, sp = clusters(48)
    case = dict(shape=shape, periodic=(1, 1, 1), tau=0.8, storage='f64', spheres=sp, relax=dict(shell_width=0.0),
                dem=dict(Tc=4.0))
    runs = []
    for _ in range(20):
        ctx = build_gpu(case)
        L.lbm_step(ctx, 6)
        st = L.lbm_get_particle_state(ctx)
        runs.append([st[key] for key in ('pos', 'vel', 'omega')])
        del ctx
    assert np.abs(runs[0][1][:48]).min() > 0.0      # every large one has been hit
    for r in runs[1:]:
        for a, b in zip(r, runs[0]):
            assert np.array_equal(a, b)
