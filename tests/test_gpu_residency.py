"""Launches that choose a kernel with other registers by the domain's size and type: the bits must not depend on the
choice.  z-chunks force it either way on one domain; single-phase domains are compared with the only member of a
batch, whose kernels do not choose."""
import numpy as np
import pytest

import workloads as W
from tests import parity_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


# FP16 pairs at walls in y: 16 (8) rows of columns x planes, up to 608 (D3Q19) / 456 (D3Q27) in the kernel with fewer blocks
@pytest.mark.parametrize("Q,shape", [(19, (34, 64, 38)), (19, (34, 64, 39)), (27, (64, 48, 38)), (27, (64, 48, 39)),
                                     (27, (6, 5, 3)), (19, (66, 9, 1))], ids=str)
@pytest.mark.parametrize("bc", [(0, 1, 0), (0, 1, 1)], ids=str)
def test_pairs_at_side_walls(Q, shape, bc):
    kw, rl, rv = U.cs_eos("T0.7")
    rho, u = W.droplet(shape, max(1.0, min(shape) / 4.0), rl, rv)
    d = dict(lattice=Q, shape=shape, bc=bc, sigma=0.1, kappa=0.3, G_ads=0.05, store="fp16", **kw)
    pairs, single = U.run_gpu(d, rho, u), U.run_gpu(dict(d, store_layout="single"), rho, u)
    for n in (1, 1, 6):
        pairs.step(n)
        single.step(n)
        assert np.array_equal(pairs.populations(device=False), single.populations(device=False)), n
        assert np.array_equal(pairs.psi(device=False), single.psi(device=False)), n


@pytest.mark.parametrize("Q", [19, 27])
@pytest.mark.parametrize("shape", [(64, 64, 64), (64, 64, 60), (20, 7, 1), (33, 130, 40)], ids=str)
@pytest.mark.parametrize("bc,points,zchunk", [((1, 0, 0), 0, 0), ((0, 1, 1), 0, 0), ((0, 0, 1), 5, 0), ((0, 0, 0), 5, 3),
                                              ((0, 0, 1), 0, 0)], ids=str)
def test_single_phase_walls_and_solids(Q, shape, bc, points, zchunk):
    from paper_2306_16274_gb300 import Batch
    nx, ny, nz = shape
    rho, u = W.perturbed(shape, seed=5)
    mask = None
    if points:
        rng = np.random.default_rng(nx + nz)
        mask = np.zeros((nz, ny, nx), dtype=np.uint8)
        for _ in range(points):
            mask[rng.integers(nz), rng.integers(ny), rng.integers(nx)] = 1
    d = dict(lattice=Q, shape=shape, bc=bc, zchunk=zchunk)
    alone, member = U.run_gpu(d, rho, u, mask), U.run_gpu(d, rho, u, mask)
    b = Batch([member])
    for n in (1, 1, 6):
        alone.step(n)
        b.step(n)
        assert np.array_equal(alone.populations(device=False), member.populations(device=False)), n
    b.close()
