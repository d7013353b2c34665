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
