"""A phi refresh followed by many steps in one call: the steps behind the
refresh run as captured graphs, whose kernels are fixed to one parity of the
time, so the call has to reach that parity first."""
import numpy as np
import pytest

import oracle
from paper_2208_09267_gb300 import lbm

pytestmark = pytest.mark.gpu


def _lattice(lattice, shape, storage, kernel, phi):
    lat = lbm.Lattice(lattice, shape, tau=0.6, storage=storage, kernel=kernel)
    lat.set_epsilon(phi)
    lat.set_force((1e-5, -3e-6, 2e-6))
    lat.init_equilibrium()
    return lat


def _phis(shape):
    n = int(np.prod(shape))
    rng = np.random.default_rng(n)
    return [(0.6 + 0.3 * rng.random(n)).astype(np.float32) for _ in range(2)]


@pytest.mark.parametrize("kernel", ["cell", "row"])
@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("start", [0, 4, 5])
@pytest.mark.parametrize("steps", [63, 64, 65, 66, 129, 200])
def test_steps_behind_a_refresh_equal_single_ones(storage, kernel, start, steps):
    shape = (40, 9, 6)
    phis = _phis(shape)
    out = []
    for calls in ([steps], [1] * steps):
        lat = _lattice("D3Q19", shape, storage, kernel, phis[0])
        for _ in range(start):
            lat.step(1, check_every=-1)
        lat.set_epsilon(phis[1], n_ref=start)
        for k in calls:
            lat.step(k, check_every=-1)
        assert lat.steps_done == start + steps
        out.append(lat.populations())
        lat.close()
    assert np.array_equal(*out)


@pytest.mark.parametrize("kernel", ["cell", "row"])
@pytest.mark.parametrize("start", [4, 5])
def test_steps_behind_a_refresh_follow_the_oracle(kernel, start):
    """FP32 populations within float rounding of the oracle (200 steps of
    2^-24 relative roundings, random in sign: 4e-6 of the largest)."""
    shape = (40, 9, 1)
    phis = _phis(shape)
    lat = _lattice("D2Q9", shape, "fp32", kernel, phis[0])
    P = oracle.Problem("D2Q9", *shape, tau=0.6, eps_ref=phis[0].astype(np.float64), g=(1e-5, -3e-6, 0.0))
    f = P.run(P.init(), 0, start)
    lat.step(start, check_every=-1)
    lat.set_epsilon(phis[1], n_ref=start)
    P.set_epsilon(phis[1].astype(np.float64), None, start)
    f = P.run(f, start, 200)
    lat.step(200, check_every=-1)
    assert np.abs(lat.populations() - f).max() <= 4e-6 * np.abs(f).max()
    lat.close()
