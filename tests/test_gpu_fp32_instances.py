"""Every instantiation of the FP32 row update rounds alike: plain and check
steps, steps behind a refresh by the same phi, lattices with walls away from
them, a tuned launch shape and a batch leave the same populations."""
import numpy as np
import pytest

from paper_2208_09267_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deps", [False, True])
@pytest.mark.parametrize("lattice,shape,walls", [("D2Q9", (40, 33, 1), 2), ("D3Q19", (64, 19, 17), 0),
                                                 ("D3Q19", (256, 9, 8), 6), ("D3Q27", (300, 6, 7), 2)])
def test_instantiations_agree_bit_for_bit(lattice, shape, walls, deps):
    n = int(np.prod(shape))
    rng = np.random.default_rng(n)
    phi = (0.5 + 0.4 * rng.random(n)).astype(np.float32)
    dphi = (1e-5 * rng.standard_normal(n)).astype(np.float32) if deps else None
    out = {}
    for how in ("plain", "check", "refresh", "check after refresh", "tuned", "batch"):
        lat = lbm.Lattice(lattice, shape, tau=0.6, storage="fp32", walls=walls, kernel="row", tuned=False,
                          row_shape=(5, 2) if how == "tuned" else None)
        lat.set_epsilon(phi, dphi, 0)
        lat.set_force((1e-5, -3e-6, 2e-6))
        lat.init_equilibrium()
        if how == "batch":
            b = lbm.Batch(max_members=1, storage="fp32")
            b.add(lat, 9)
            b.step(10)
            b.close()
        else:
            for _ in range(9):
                if "refresh" in how:
                    lat.set_epsilon(phi, dphi, 0)
                lat.step(1, check_every=0 if "check" in how else -1)
        out[how] = lat.populations()
        lat.close()
    for how, f in out.items():
        assert np.array_equal(f, out["plain"]), how
