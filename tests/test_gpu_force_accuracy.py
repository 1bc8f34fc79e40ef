"""Accuracy of the float32 collision with a body force, and of the forces on a
box's only particle (a form of the dense kernel of its own).

The collision adds the body force's source at the size of a pair's correction.
Each operation rounds once, so one step of a box without particles is restated
here in float32 operation by operation (multiply-adds through float64: the
product is exact, and the second rounding meets a tie in about one of 2^29) and
must come out bit for bit but for such ties, 1e-5 of the values at most.

Forces: the float64 kernel is the reference, on a sphere that both moves and
spins, so that neither force nor torque is a small rest of the links' parts.
Float32 forces are sums of remainders of ~1e-3 with a relative rounding of 2^-24
in each of a few operations (1e-5); velocities 1e-6.
"""
import numpy as np
import pytest

from cases import build_gpu, rel_l2, spheres

pytestmark = pytest.mark.gpu

C = [(0, 0, 0), (0, 1, 0), (0, -1, 0), (-1, 0, 0), (1, 0, 0), (0, 0, 1), (0, 0, -1), (-1, 1, 0), (1, 1, 0),
     (-1, -1, 0), (1, -1, 0), (0, 1, 1), (0, -1, 1), (-1, 0, 1), (1, 0, 1), (0, 1, -1), (0, -1, -1), (-1, 0, -1),
     (1, 0, -1)]
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)
OPP = [C.index(tuple(-v for v in c)) for c in C]
F = np.float32


@pytest.fixture(scope='module')
def L():
    torch = pytest.importorskip('torch')
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    from paper_2003_01490_gb300 import lbmdem
    lbmdem.load_library()
    return lbmdem


def fma(a, b, c):
    return (np.float64(a) * np.float64(b) + np.float64(c)).astype(F)


def collided(f, a, tau):
    """One float32 collision of the streamed PDFs f (19, ...) with the body force a."""
    sp, sm = F(1.0 / tau), F(1.0 / (0.5 + 3.0 / 16.0 / (tau - 0.5)))
    a = np.asarray(a, dtype=F)
    w2 = {2: F(0.0555555522441864)}
    w2[1] = F(2) * w2[2]
    w0, w6 = F(1) - F(12) * w2[2], {2: F(1) / F(6)}
    w6[1] = F(1) - F(4) * w6[2]
    gp, gm = F(1) - F(0.5) * sp, F(1) - F(0.5) * sm
    drho, j = f[0], [F(0) * f[0]] * 3
    pairs = [q for q in range(1, 19) if OPP[q] > q]
    for q in pairs:
        drho = drho + (f[q] + f[OPP[q]])
        j = [v + F(c) * (f[q] - f[OPP[q]]) if c else v for v, c in zip(j, C[q])]
    u = [v + F(0.5) * b for v, b in zip(j, a)]
    usq = fma(u[2], u[2], fma(u[0], u[0], u[1] * u[1]))
    m3ua = F(-3) * fma(u[2], a[2], fma(u[0], a[0], u[1] * a[1]))
    drp = fma(F(-1.5), usq, drho)
    out = np.empty_like(f)
    out[0] = fma(gp, w0 * m3ua, fma(sp, fma(w0, drp, -f[0]), f[0]))
    for q in pairs:
        p, k = OPP[q], sum(v * v for v in C[q])
        cu, ca = F(0) * u[0], F(0)
        for c, v, b in zip(C[q], u, a):
            if c:
                cu, ca = cu + F(c) * v, ca + F(c) * b
        X = fma(F(4.5) * cu, cu, drp)
        Y = fma(F(9) * cu, ca, m3ua)
        dp = fma(F(-0.5) * sp, fma(-w2[k], X, f[q] + f[p]), fma(F(0.5) * gp * w2[k], Y, F(0)))
        dm = fma(F(-0.5) * sm, fma(-w6[k], cu, f[q] - f[p]), F(0.5) * gm * w6[k] * ca)
        out[q], out[p] = f[q] + (dp + dm), f[p] + (dp - dm)
    return out


@pytest.mark.parametrize('force', [(2e-5, -1e-6, 7e-6), (0.0, 0.0, -3e-5), (0.0, 0.0, 0.0)])
def test_float32_collision_adds_the_body_force_as_its_own_source(L, force):
    shape, tau = (37, 7, 6), 0.62
    rng = np.random.default_rng(3)
    v = (W[:, None, None, None] * 0.05 * rng.standard_normal((19,) + shape[::-1])).astype(F)
    case = dict(shape=shape, periodic=(1, 1, 1), tau=tau, storage='f32', body_force=force,
                init_pdfs=v.astype(np.float64) + W[:, None, None, None])
    ctx = build_gpu(case)
    L.lbm_step(ctx, 1)
    got = (L.lbm_get_pdfs(ctx).reshape(v.shape) - W[:, None, None, None]).astype(F)
    want = collided(np.stack([np.roll(v[q], C[q][::-1], (0, 1, 2)) for q in range(19)]), force, tau)
    assert np.mean(got != want) < 1e-5


# rows of 32 cells with up to 7, 30, 43, 118 and 160 links (a row's links are taken
# in runs of one per 32 and queued 128 at a time)
@pytest.mark.parametrize('shape,radius', [((31, 9, 10), 1.4), ((33, 29, 31), 8.2), ((64, 52, 51), 20.0),
                                          ((96, 95, 90), 40.0), ((160, 151, 150), 70.0)])
def test_forces_on_the_only_particle_match_float64(L, shape, radius):
    at = 0.5 * np.array(shape) + [0.02, 0.13, -0.27]
    got = []
    for storage in ('f64', 'f32'):
        case = dict(shape=shape, periodic=(1, 1, 1), tau=0.8, storage=storage, body_force=(2e-5, -1e-5, 3e-5),
                    spheres=spheres([at], [radius], vel=[[0.04, -0.03, 0.05]],
                                    omega=[[0.1 / radius, -0.05 / radius, 0.07 / radius]]),
                    dem=dict(fixed_particles=1))
        ctx = build_gpu(case)
        L.lbm_step(ctx, 5)
        st = L.lbm_get_particle_state(ctx)
        got.append((st['force_hyd'], st['torque_hyd'], L.lbm_get_fields(ctx)[1]))
        del ctx
    (F64, T64, u64), (F32, T32, u32) = got
    assert rel_l2(F32, F64) < 1e-5
    assert rel_l2(T32, T64) < 1e-5
    assert rel_l2(u32, u64) < 1e-6
