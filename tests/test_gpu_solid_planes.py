"""Whole-grid steps of domains with walls and solids: only the planes of a 32 x 4 column that hold cells with
solid neighbours take the code with solid tests (one bit per plane, 32 planes a word).  Stepping such a domain
alone must equal stepping it as the only member of a batch, whose tiles are classified on the host, bit for bit:
sparse masks that switch from plane to plane, across words, at ragged edges, with every set of walls."""
import numpy as np
import pytest

import workloads as W
from tests import parity_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("Q", [19, 27])
@pytest.mark.parametrize("shape,bc,zchunk,solids", [
    ((70, 13, 70), (0, 0, 0), 0, "points"),      # three columns wide, three words high
    ((33, 9, 64), (0, 0, 1), 9, "points"),       # marches that end within a word
    ((65, 6, 33), (1, 0, 0), 0, "points"),       # a second word of one plane
    ((40, 10, 35), (0, 1, 1), 0, None),          # walls only, none of them in z alone
    ((32, 4, 3), (0, 0, 1), 0, "points"),        # one column
    ((31, 5, 2), (0, 0, 1), 0, None),            # z walls too close for planes of their own
])
def test_solid_planes_equal_batch_tiles(Q, shape, bc, zchunk, solids):
    from paper_2306_16274_gb300 import Batch
    kw, rl, rv = U.cs_eos("T0.7")
    nx, ny, nz = shape
    rho, u = W.droplet(shape, max(1.5, min(shape) / 3.0), rl, rv)
    mask = None
    if solids:   # a few isolated solid cells, one of them next to a corner of the domain
        rng = np.random.default_rng(nx + nz)
        mask = np.zeros((nz, ny, nx), dtype=np.uint8)
        for _ in range(5):
            mask[rng.integers(nz), rng.integers(ny), rng.integers(nx)] = 1
        mask[nz - 1, 0, nx - 1] = 1
    d = dict(lattice=Q, shape=shape, bc=bc, sigma=0.1, kappa=0.3, G_ads=0.05, zchunk=zchunk, **kw)
    a, b = U.run_gpu(d, rho, u, mask), U.run_gpu(d, rho, u, mask)
    bb = Batch([b])
    for n in (1, 4, 11):
        a.step(n)
        bb.step(n)
        assert np.array_equal(a.populations(device=False), b.populations(device=False)), n
    assert np.array_equal(a.psi(device=False), b.psi(device=False))
    bb.close()
