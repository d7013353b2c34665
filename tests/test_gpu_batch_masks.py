"""A batch member re-initialised with another solid mask in place of the one it had: the mask's buffers stay, but
which tiles and runs need solid handling changes with its cells.  Every member must go on bitwise as when
stepped alone, and tuned shapes and z-chunks stay."""
import numpy as np
import pytest

import workloads as W
from tests import parity_util as U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _init(sim, rho, u, solid):
    import torch
    sim.init_fields(torch.tensor(rho, dtype=torch.float32, device="cuda"),
                    torch.tensor(u, dtype=torch.float32, device="cuda"),
                    None if solid is None else torch.tensor(solid, dtype=torch.uint8, device="cuda"))


@pytest.mark.parametrize("Q", [19, 27])
@pytest.mark.parametrize("n", [1, 6, 65], ids=str)   # plain launches, the short graph, both graphs
def test_member_with_another_mask_in_the_same_buffers(Q, n):
    from paper_2306_16274_gb300 import Batch
    kw, rl, rv = U.cs_eos("T0.7")
    shape = (70, 17, 40)
    d = dict(lattice=Q, shape=shape, sigma=0.1, kappa=0.3, G_ads=0.05, **kw)
    rho, u = W.droplet(shape, 5.0, rl, rv)
    first, second = np.zeros((2, 40, 17, 70), dtype=np.uint8)
    first[3:6, 2:5, 4:8] = 1        # first column, low planes
    second[30:34, 9:12, 60:66] = 1  # last column (narrow), high planes
    masks = [first, second, first | second, second]
    alone = [U.run_gpu(d, rho, u, first), U.run_gpu(d, rho, u)]
    together = [U.run_gpu(d, rho, u, first), U.run_gpu(d, rho, u)]
    b = Batch(together)
    for g in range(b.info()["groups"]):
        b.set_group(g, 3, 5)
    for mask in masks:
        for s in (alone, together):
            for k, sim in enumerate(s):   # the other member keeps the phases equal
                _init(sim, rho, u, mask if k == 0 else None)
        b.step(n)
        b.step(n)
        for s in alone:
            s.step(2 * n)
        for k, (s, t) in enumerate(zip(alone, together)):
            assert np.array_equal(s.populations(device=False), t.populations(device=False)), k
            assert np.array_equal(s.psi(device=False), t.psi(device=False)), k
        assert all((g["shape"], g["zchunk"]) == (3, 5) for g in b.groups())
    # and through no mask at all, which groups anew
    for s in (alone, together):
        _init(s[0], rho, u, None)
        _init(s[0], rho, u, first)
        _init(s[1], rho, u, None)
    b.step(n)
    for s in alone:
        s.step(n)
    assert all(np.array_equal(s.populations(device=False), t.populations(device=False)) for s, t in zip(alone, together))
    b.close()
