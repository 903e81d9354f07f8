"""The FP64 step deals cells in linear order to blocks whose size depends on
the lattice: sizes around a warp, a block and the thresholds of the block
size, with and without walls, stay bit-identical to the oracle."""
import numpy as np
import pytest

import oracle
from paper_2208_09267_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,shape,walls,block", [
    ("D1Q3", (31, 1, 1), 0, (0, 0)),
    ("D1Q3", (257, 1, 1), 0, (0, 0)),
    ("D2Q9", (1, 5, 1), 2, (0, 0)),
    ("D2Q9", (33, 31, 1), 1, (0, 0)),
    ("D2Q9", (33, 31, 1), 0, (32, 4)),
    ("D2Q9", (311, 257, 1), 0, (0, 0)),       # 64 threads a block
    ("D3Q19", (3, 3, 3), 4, (0, 0)),
    ("D3Q19", (47, 53, 67), 2, (0, 0)),       # 128 threads a block, a part-filled last one
    ("D3Q27", (13, 7, 5), 6, (0, 0)),
    ("D3Q27", (13, 7, 5), 0, (96, 1)),
    ("D2Q9", (64, 152, 1), 3, (0, 0)),        # the largest lattice whose cells four warps share
    ("D2Q9", (64, 153, 1), 0, (0, 0)),        # and the next
    ("D3Q27", (21, 20, 23), 2, (0, 0)),
])
def test_fp64_step_at_block_edges_is_bit_identical(lattice, shape, walls, block):
    N = int(np.prod(shape))
    rng = np.random.default_rng(N + walls)
    eps = 0.5 + 0.4 * rng.random(N)
    force = 1e-5 * rng.standard_normal(3 * N)
    g = (1e-5, -2e-6, 3e-6)
    gpu = lbm.Lattice(lattice, shape, tau=0.7, storage="fp64", walls=walls, block=block)
    gpu.set_epsilon(eps)
    gpu.set_force(g, force)
    gpu.init_equilibrium()
    P = oracle.Problem(lattice, *shape, tau=0.7, walls=walls, eps_ref=eps, g=g, force=force)
    gpu.step(6, check_every=-1)
    f = P.run(P.init(), 0, 6)
    assert np.array_equal(gpu.populations(), f)
