"""Batches whose members share launches: tiles with and without solid neighbours of one lattice and physics go
into one launch, several lattices and physics run side by side, and calls of many steps replay graphs of 2 and
16 steps.  Every member must evolve bitwise as when stepped alone, over call lengths on both sides of the
graphs' and from either AA phase."""
import numpy as np
import pytest

import workloads as W
from tests import parity_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("calls", [(1, 2, 3), (15, 17), (64, 1, 65), (5, 67)], ids=str)
def test_call_lengths_and_phases(calls):
    from paper_2306_16274_gb300 import Batch
    kw, rl, rv = U.cs_eos("T0.7")
    members = []
    for Q in (19, 27):
        for k, shape in enumerate(((33, 9, 20), (48, 17, 12), (21, 30, 35))):
            solid = W.cylinder_mask(shape, 2.5, axis="y") if k == 2 else None
            bc = (0, 0, 1) if k else (0, 0, 0)
            rho, u = W.droplet(shape, 3.0, rl, rv, center=(shape[0] / 2, shape[1] / 2, shape[2] - 5.0))
            members.append((dict(lattice=Q, shape=shape, bc=bc, sigma=0.1, kappa=0.3 * (k == 1), G_ads=0.05, **kw), rho, u,
                            solid))
    members.append((dict(lattice=19, shape=(20, 20, 20), g=(1e-5, 0.0, 0.0)), *W.perturbed((20, 20, 20), seed=4), None))
    alone = [U.run_gpu(*m) for m in members]
    together = [U.run_gpu(*m) for m in members]
    b = Batch(together)
    for n in calls:
        b.step(n)
        for s in alone:
            s.step(n)
    b.sync()
    for k, (s, t) in enumerate(zip(alone, together)):
        assert t.step_count == s.step_count == sum(calls)
        assert np.array_equal(s.populations(device=False), t.populations(device=False)), k
        assert np.array_equal(s.psi(device=False), t.psi(device=False)), k
    b.close()
