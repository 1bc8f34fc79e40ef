"""Float32 pair laws in long boxes: the separation of a pair is a difference of
positions held as sums of two floats, so it is known to 2^-49 of the side. A pair
that collides at the far end of a box of 65,528 cells moves like one in a short
box, up to that: 2e-10 cells of gaps and overlaps of 1e-3 are 2e-7 of a force, and
a few steps of contact give velocities to 1e-5."""
import numpy as np
import pytest

from cases import build_gpu, rel_l2, spheres

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('side', [520, 4096, 65528])
def test_a_pair_far_from_the_origin_collides_as_one_near_it(side):
    from paper_2003_01490_gb300 import lbmdem as L
    got = []
    for nx, shift in ((40, 0.0), (side, side - 40.0)):
        at = np.array([[16.9375, 7.0625, 7.0], [22.953125, 7.25, 7.125], [10.90625, 6.96875, 7.0]])
        case = dict(shape=(nx, 14, 14), periodic=(1, 1, 1), tau=0.7, storage='f32',
                    spheres=spheres(at + [shift, 0.0, 0.0], [3.0, 3.0, 3.0], density=[20.0, 20.0, 20.0],
                                    vel=[[0.03, 0.01, 0.0], [-0.03, 0.0, 0.005], [0.04, 0.0, 0.0]],
                                    omega=[[0.0, 0.0, 0.01], [0.005, 0.0, 0.0], [0.0, 0.01, 0.0]]),
                    dem=dict(Tc=3.0))
        ctx = build_gpu(case)
        L.lbm_step(ctx, 6)
        st = L.lbm_get_particle_state(ctx)
        got.append((st['pos'] - [shift, 0.0, 0.0], st['vel'], st['omega']))
        del ctx
    assert np.abs(got[0][1] - case['spheres']['vel']).max(1).min() > 1e-3      # all have met
    for a, b in zip(got[1], got[0]):
        assert rel_l2(a, b) < 1e-5
