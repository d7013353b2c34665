"""lbm_get_moments: its FP64 totals are sums of per-block sums in a fixed order, taken by one launch or, for many
blocks, by chains of them first; fields do not depend on whether totals are asked for."""
import numpy as np
import pytest

import workloads as W
from tests import parity_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


# blocks of 32 x 4 x 2 cells: 1; 2048 (the last domain of one launch); 2049 and more, with chains of 8 and 9, of
# 16 and 17 blocks (a whole group of loads and one beyond it)
@pytest.mark.parametrize("shape", [(5, 3, 1), (64, 128, 64), (32, 12, 1366), (128, 128, 64), (33, 128, 130)])
@pytest.mark.parametrize("Q", [19, 27])
def test_totals(Q, shape):
    rho, u = W.perturbed(shape, seed=3)
    sim = U.run_gpu(dict(lattice=Q, shape=shape), rho, u, steps=2)
    r, v, sums = sim.moments()
    r2, v2, none = sim.moments(sums=False)
    assert none is None and np.array_equal(r.cpu(), r2.cpu()) and np.array_equal(v.cpu(), v2.cpu())
    r64 = r.cpu().numpy().astype(np.float64)
    # rho enters the totals as the float that the field holds: FP64 additions of n terms of at most 1.2, so n^2 eps
    # is far above what can be lost; momentum is rounded once per cell on the way to the velocity field
    n = r64.size
    assert abs(sums[0] - r64.sum()) <= 1.2 * n * n * 2.0 ** -53
    j = (r64 * v.cpu().numpy().astype(np.float64)).reshape(3, -1).sum(axis=1)
    assert np.abs(sums[1:] - j).max() <= 3 * n * 2.0 ** -24 * float(np.abs(r64 * v.cpu().numpy()).max())
    assert list(sums) == list(sim.moments()[2])
