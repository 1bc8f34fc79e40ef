"""The mapping at the sizes where its loads and blocks change, against the
oracle: sides that are no multiple of four cells (byte-wide flags) or of a tile,
the smallest box, periodic axes too short for one image per tile, spheres that
overlap, boxes deep enough for a block to walk several tiles with a short last
chunk, and the mapping into caller's buffers that are not aligned."""
import numpy as np
import pytest
import torch

from cases import build_gpu, spheres
from oracle import Domain
from oracle.particles import cell_centres, map_cells

pytestmark = pytest.mark.gpu

SHAPES = [((3, 3, 3), (1, 1, 1), 2, 0.9), ((33, 7, 5), (1, 1, 1), 5, 3.0), ((32, 8, 40), (1, 0, 1), 20, 3.5),
          ((36, 9, 133), (0, 1, 0), 40, 4.0), ((64, 12, 44), (1, 1, 1), 70, 2.5), ((68, 60, 402), (1, 1, 0), 90, 9.0)]


# a context takes spheres apart from each other and from the walls, of radius
# 1 and more, in periodic sides longer than their diameter and four cells
APART = [((33, 9, 8), (1, 1, 1), 40, 1.9), ((32, 12, 40), (1, 0, 1), 60, 3.5), ((36, 9, 133), (0, 1, 0), 200, 2.4),
         ((64, 12, 44), (1, 1, 1), 200, 3.9), ((68, 60, 402), (1, 1, 0), 90, 9.0)]


def drawn(shape, n, rmax):
    rng = np.random.default_rng(sum(shape))
    return rng.random((n, 3)) * np.array(shape), rng.uniform(0.5 * rmax, rmax, n)


def apart(shape, periodic, pos, rad):
    """The spheres that fit beside those before them."""
    side, keep = np.array(shape, float), []
    rad = np.maximum(rad, 1.0)
    for i in range(len(rad)):
        e = pos[keep] - pos[i]
        e -= np.where(periodic, side * np.round(e / side), 0.0)
        inside = (pos[i] > rad[i] + 1e-3) & (pos[i] < side - rad[i] - 1e-3) | (np.array(periodic) != 0)
        if inside.all() and ((e * e).sum(1) > (rad[keep] + rad[i] + 1e-3) ** 2).all():
            keep.append(i)
    return pos[keep], rad[keep]


def wanted(shape, periodic, pos, rad):
    """(owner, shell) of the oracle."""
    dom = Domain(*shape, periodic=tuple(bool(p) for p in periodic))
    owner, shell = map_cells(cell_centres(dom), pos, rad, dom, 2.0)
    return owner, shell


@pytest.mark.parametrize('shape,periodic,n,rmax', APART)
def test_mapping_of_a_context(shape, periodic, n, rmax):
    from paper_2003_01490_gb300 import lbmdem as L
    pos, rad = apart(shape, periodic, *drawn(shape, n, rmax))
    ctx = build_gpu(dict(shape=shape, periodic=periodic, tau=0.7, storage='f32',
                         spheres=spheres(pos, rad), dem=dict(fixed_particles=1)))
    owner, shell = wanted(shape, periodic, pos, rad)
    flags = L.lbm_get_fields(ctx)[2]
    got = L.lbm_get_owner(ctx)
    solid = (flags & L.FLAG_SOLID) != 0
    assert np.array_equal(solid, owner >= 0)
    assert np.array_equal(got, owner)
    assert np.array_equal((flags & L.FLAG_SHELL) != 0, shell)


@pytest.mark.parametrize('shape,periodic,n,rmax', SHAPES)
@pytest.mark.parametrize('shift', [0, 1])
def test_mapping_into_buffers(shape, periodic, n, rmax, shift):
    from paper_2003_01490_gb300 import lbmdem as L
    pos, rad = drawn(shape, n, rmax)
    cells = int(np.prod(shape))
    flags = torch.full((cells + shift,), 0xa5, dtype=torch.uint8, device='cuda')[shift:]
    owner = torch.full((cells + shift,), 77, dtype=torch.int32, device='cuda')[shift:]
    L.lbm_map_spheres_noalloc(L.make_grid(shape, periodic), 2.0, torch.tensor(pos, device='cuda').reshape(-1),
                              torch.tensor(rad, device='cuda'), flags, owner)
    want, shell = wanted(shape, periodic, pos, rad)
    f = flags.cpu().numpy().reshape(shape[::-1])
    assert np.array_equal((f & L.FLAG_SOLID) != 0, want >= 0)
    assert np.array_equal(owner.cpu().numpy().reshape(shape[::-1]), want)
    assert np.array_equal((f & L.FLAG_SHELL) != 0, shell)
