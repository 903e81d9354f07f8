"""Steps enqueued one after another (each may start while the one before
drains) and the branch-free wall handling of the one-cell kernel."""
import numpy as np
import pytest

import oracle
from paper_2208_09267_gb300 import lbm

pytestmark = pytest.mark.gpu


def _make(lattice, shape, storage, walls, **kw):
    n = int(np.prod(shape))
    rng = np.random.default_rng(n + walls)
    lat = lbm.Lattice(lattice, shape, tau=0.6, storage=storage, walls=walls, **kw)
    lat.set_epsilon((0.6 + 0.3 * rng.random(n)).astype(np.float32))
    lat.set_force((1e-5, -3e-6, 2e-6))
    lat.init_equilibrium()
    return lat


@pytest.mark.parametrize("kernel", ["cell", "row"])
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("lattice,shape,walls", [
    ("D2Q9", (33, 9, 1), 0), ("D2Q9", (250, 131, 1), 2), ("D3Q19", (64, 12, 10), 2), ("D3Q27", (40, 7, 6), 4),
    ("D3Q19", (61, 75, 67), 0)])
def test_chained_steps_equal_single_ones(lattice, shape, walls, storage, kernel):
    """70 steps in one call (a captured graph and a rest, chained launches)
    give the populations of 70 calls of one step."""
    a = _make(lattice, shape, storage, walls, kernel=kernel)
    b = _make(lattice, shape, storage, walls, kernel=kernel)
    a.step(70, check_every=-1)
    for _ in range(70):
        b.step(1, check_every=-1)
    assert np.array_equal(a.populations(), b.populations())
    a.close()
    b.close()


@pytest.mark.parametrize("lattice,shape,walls", [
    ("D1Q3", (5, 1, 1), 1), ("D2Q9", (3, 5, 1), 3), ("D3Q19", (7, 3, 4), 6), ("D3Q27", (3, 3, 3), 7),
    ("D3Q19", (45, 6, 5), 5)])
def test_cell_kernel_at_walls_follows_the_oracle(lattice, shape, walls):
    """Bounce-back at faces, edges and corners, through odd and even steps and
    a change of phi: FP32 populations within float rounding of the oracle
    (20 steps of 2^-24 relative roundings: 2e-6 of the largest)."""
    n = int(np.prod(shape))
    a = _make(lattice, shape, "fp32", walls, kernel="cell")
    rng = np.random.default_rng(n + walls)
    e = (0.6 + 0.3 * rng.random(n)).astype(np.float32)
    P = oracle.Problem(lattice, *shape, tau=0.6, walls=walls, eps_ref=e.astype(np.float64), g=(1e-5, -3e-6, 2e-6))
    f = P.run(P.init(), 0, 9)
    a.step(9)
    e2 = (0.6 + 0.3 * rng.random(n)).astype(np.float32)
    a.set_epsilon(e2, n_ref=9)
    P.set_epsilon(e2.astype(np.float64), None, 9)
    f = P.run(f, 9, 11)
    a.step(11)
    assert np.abs(a.populations() - f).max() <= 2e-6 * np.abs(f).max()
    a.close()
