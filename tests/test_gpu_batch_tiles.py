"""Domains with walls and solids stepped as the only member of a batch (tiles, classified on the host) against the
same domain stepped alone (whole-grid kernels): the same bits, with narrow 16-wide tiles at the ends of rows that
touch walls and cross solids, and the batch-stepped state against the oracle."""
import numpy as np
import pytest

import workloads as W
from tests import parity_util as U
from tests.test_gpu_batch import _members

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("which", [2, 3])
def test_one_member_batch_equals_domain_alone(which):
    from paper_2306_16274_gb300 import Batch
    d, rho, u, solid = _members()[which]
    alone, tiles = U.run_gpu(d, rho, u, solid), U.run_gpu(d, rho, u, solid)
    b = Batch([tiles])
    for n in (7, 40):
        alone.step(n)
        b.step(n)
        assert np.array_equal(alone.populations(device=False), tiles.populations(device=False)), n
    b.close()


@pytest.mark.parametrize("Q", [19, 27])
@pytest.mark.parametrize("nx", [33, 44, 48])   # 32 + 1 .. 16: narrow tiles at the ends of rows
def test_narrow_tiles_next_to_walls_and_solids(Q, nx):
    from paper_2306_16274_gb300 import Batch
    kw, rl, rv = U.cs_eos("T0.7")
    shape = (nx, 14, 10)
    rho, u = W.droplet(shape, 4.0, rl, rv)
    z, y, x = np.meshgrid(np.arange(10), np.arange(14), np.arange(nx), indexing="ij")
    solid = ((x - (nx - 5)) ** 2 + (y - 7) ** 2 <= 2.5 ** 2).astype(np.uint8)   # a post along z near x = nx
    d = dict(lattice=Q, shape=shape, bc=(1, 1, 1), sigma=0.1, kappa=0.3, G_ads=0.05, **kw)
    alone, tiles = U.run_gpu(d, rho, u, solid), U.run_gpu(d, rho, u, solid)
    b = Batch([tiles])
    for n in (3, 20):
        alone.step(n)
        b.step(n)
        assert np.array_equal(alone.populations(device=False), tiles.populations(device=False)), n
    # the oracle's tolerances are those of the same domain stepped alone
    ref = U.run_oracle(d, rho, u, solid, steps=23)
    er, eu, _, _ = U.compare_moments(tiles, ref)
    assert er < 1e-4 and eu < 1e-4, (er, eu)
    b.close()


@pytest.mark.parametrize("Q", [19, 27])
@pytest.mark.parametrize("shape,bc,points", [
    ((50, 13, 70), (0, 0, 0), 6),    # planes with and without solids within marches, more than 32 planes
    ((44, 9, 40), (0, 0, 1), 4),     # and walls in z
    ((33, 17, 20), (1, 1, 0), 0),    # side walls: every plane of some tiles
    ((64, 10, 3), (0, 0, 1), 0),     # wall planes only, the smallest domain with one between them
    ((64, 10, 2), (1, 0, 1), 2),
])
def test_tiles_that_switch_from_plane_to_plane(Q, shape, bc, points):
    # every tile shape, z-chunks down to single planes and up to whole columns, others for tiles with solids
    from paper_2306_16274_gb300 import Batch
    kw, rl, rv = U.cs_eos("T0.7")
    nx, ny, nz = shape
    rho, u = W.droplet(shape, max(1.0, min(shape) / 4.0), rl, rv)
    mask = None
    if points:
        rng = np.random.default_rng(nz)
        mask = np.zeros((nz, ny, nx), dtype=np.uint8)
        for _ in range(points):
            mask[rng.integers(nz), rng.integers(ny), rng.integers(nx)] = 1
    d = dict(lattice=Q, shape=shape, bc=bc, sigma=0.1, kappa=0.3, G_ads=0.05, **kw)
    alone, tiles = U.run_gpu(d, rho, u, mask), U.run_gpu(d, rho, u, mask)
    b = Batch([tiles])
    for tile_shape, plain, solid in [(0, 0, 0), (1, 1, 5), (2, 7, 1), (3, 40, 33), (4, 1 << 30, 4)]:
        b.set_group(0, tile_shape, plain)
        b.set_group(1, tile_shape, solid)
        for n in (1, 4):
            alone.step(n)
            b.step(n)
            assert np.array_equal(alone.populations(device=False), tiles.populations(device=False)), (tile_shape, n)
            assert np.array_equal(alone.psi(device=False), tiles.psi(device=False)), (tile_shape, n)
    b.close()


def test_wall_planes_in_launches_of_few_and_many_tiles():
    # D3Q27 with walls in z: launches of more than 4.5 waves take the kernel that switches from plane to plane
    from paper_2306_16274_gb300 import Batch
    kw, rl, rv = U.cs_eos("T0.7")
    shape = (96, 96, 50)
    rho, u = W.droplet(shape, 8.0, rl, rv)
    d = dict(lattice=27, shape=shape, bc=(0, 0, 1), sigma=0.1, kappa=0.3, G_ads=0.05, **kw)
    alone, tiles = U.run_gpu(d, rho, u), U.run_gpu(d, rho, u)
    b = Batch([tiles])
    for zchunk, many in ((0, False), (1, True)):
        b.set_group(0, 0, zchunk)
        assert (b.info()["tiles"] > 3420) == many
        for n in (1, 4):
            alone.step(n)
            b.step(n)
            assert np.array_equal(alone.populations(device=False), tiles.populations(device=False)), (zchunk, n)
    b.close()
