"""FP16 row-staged steps: two cells per lane and consumer groups (plain steps)
against one cell per lane (check steps), at tile and ring edges."""
import numpy as np
import pytest

from paper_2208_09267_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rounding", ["stochastic", "nearest"])
@pytest.mark.parametrize("lattice,shape,walls,deps", [
    ("D2Q9", (8, 3, 1), 0, False),           # one short tile
    ("D2Q9", (13, 40, 1), 2, True),          # 8 rows a tile, odd rows
    ("D2Q9", (511, 6, 1), 0, False),         # pitch 512
    ("D3Q19", (64, 9, 7), 0, True),          # 4 rows a tile and a rest
    ("D3Q19", (75, 11, 9), 2, False),        # 3 rows of 80
    ("D3Q19", (129, 5, 6), 4, True),         # one row of 136
    ("D3Q19", (250, 6, 5), 6, False),        # one row at the compile-time pitch
    ("D3Q19", (256, 40, 45), 0, True),       # more tiles than stages in every block
    ("D3Q27", (33, 8, 6), 2, True),
    ("D3Q27", (200, 30, 33), 0, False),
    ("D3Q27", (300, 26, 20), 2, True),       # pitch 512 with d_t phi
])
def test_plain_steps_equal_check_steps(lattice, shape, walls, deps, rounding):
    """The pair update makes the roundings of the one-cell update (divisions
    included), so plain steps and check steps leave the same halves."""
    n = int(np.prod(shape))
    rng = np.random.default_rng(n)
    e = (0.5 + 0.4 * rng.random(n)).astype(np.float32)
    d = (1e-5 * rng.standard_normal(n)).astype(np.float32) if deps else None
    f = (1e-5 * rng.standard_normal(3 * n)).astype(np.float32)
    out = []
    for check in (False, True):
        lat = lbm.Lattice(lattice, shape, tau=0.6, storage="fp16", walls=walls, kernel="row", fp16_rounding=rounding)
        lat.set_epsilon(e, d, 0)
        lat.set_force((1e-5, -3e-6, 2e-6), f)
        lat.init_equilibrium()
        if check:
            for _ in range(7):
                lat.step(1)
        else:
            lat.step(1)                       # (the step after a refresh takes the one-cell update)
            lat.step(6, check_every=-1)
        out.append(lat.populations())
        lat.close()
    assert np.array_equal(*out)


@pytest.mark.parametrize("lattice,shape,walls", [
    ("D2Q9", (13, 40, 1), 2), ("D3Q19", (75, 11, 9), 2), ("D3Q19", (256, 9, 8), 0), ("D3Q27", (300, 6, 7), 0),
    ("D3Q27", (33, 8, 6), 4)])
def test_the_step_after_a_refresh_equals_its_check_step(lattice, shape, walls):
    """Decoding with the old shift and encoding with the new one, two cells per
    lane, at an even and at an odd step."""
    n = int(np.prod(shape))
    rng = np.random.default_rng(n + 1)
    phis = [(0.5 + 0.4 * rng.random(n)).astype(np.float32) for _ in range(3)]
    out = []
    for check in (False, True):
        lat = lbm.Lattice(lattice, shape, tau=0.6, storage="fp16", walls=walls, kernel="row")
        lat.set_epsilon(phis[0])
        lat.set_force((1e-5, -3e-6, 2e-6))
        lat.init_equilibrium()
        lat.step(4)
        for phi in phis[1:]:                  # refreshed before step 4 and step 7
            lat.set_epsilon(phi, n_ref=lat.steps_done)
            for _ in range(3):
                lat.step(1, check_every=0 if check else -1)
        out.append(lat.populations())
        lat.close()
    assert np.array_equal(*out)


@pytest.mark.parametrize("lattice,shape", [("D3Q19", (128, 64, 64)), ("D3Q27", (40, 24, 20))])
def test_wait_limit_ends_the_fp16_step(lattice, shape):
    """With the copies withheld (nothing is in flight) every wait of the groups,
    producers and storers runs out: the step reports the timeout and the handle
    keeps working with the normal limit."""
    lat = lbm.Lattice(lattice, shape, tau=0.6, storage="fp16", kernel="row")
    lat.set_force((1e-6, 0, 0))
    lat.set_wait_limit(64, withhold_copies=True)
    with pytest.raises(lbm.LbmError) as e:
        lat.step(2)
    assert e.value.code == -5
    lat.set_wait_limit(0, withhold_copies=False)
    lat.init_equilibrium()
    st = lat.step(4)
    assert not st["nan_seen"] and st["mass"] > 0
    lat.close()
