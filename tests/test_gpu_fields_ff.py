"""Single-precision moments and the initial state of FP32/FP16 lattices are
formed in float-float arithmetic: they agree with the FP64 kernels to the
rounding of their results.  Bounds: float-float carries about 2^-44 of the O(1)
sums, far below the 2^-24 of a float result; 1e-12 covers it for values that
cancel (p, u near zero)."""
import numpy as np
import pytest

from paper_2208_09267_gb300 import lbm

pytestmark = pytest.mark.gpu
ULP = 2.0 ** -23


def _lattice(lattice, shape, storage, walls=0, **kw):
    rng = np.random.default_rng(int(np.prod(shape)) + walls)
    n = int(np.prod(shape))
    lat = lbm.Lattice(lattice, shape, tau=0.65, storage=storage, walls=walls, **kw)
    lat.set_epsilon((0.5 + 0.4 * rng.random(n)).astype(np.float32), (1e-4 * rng.standard_normal(n)).astype(np.float32), 0)
    lat.set_force((1e-5, -2e-6, 3e-6), (1e-5 * rng.standard_normal(3 * n)).astype(np.float32))
    return lat, rng, n


def _f32_moments(lat):
    import torch
    out = [torch.empty(k * lat.n, device="cuda") for k in (1, 1, 3)]
    lat.moments_into(*out)
    torch.cuda.synchronize()
    return [t.cpu().numpy().astype(np.float64) for t in out]


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("lattice,shape,walls,kw", [
    ("D1Q3", (37, 1, 1), 0, {}),
    ("D2Q9", (33, 9, 1), 1, {}),
    ("D3Q19", (45, 7, 6), 2, {}),
    ("D3Q27", (19, 6, 5), 4, {}),
    ("D3Q19", (21, 6, 5), 0, {"drag": (150.0, 1.75, 5.0)}),
])
def test_float_moments_round_the_fp64_ones(lattice, shape, walls, kw, storage):
    lat, rng, n = _lattice(lattice, shape, storage, walls, **kw)
    lat.init_equilibrium()
    for steps in (4, 1):               # an even and an odd layout
        lat.step(steps)
        m = lat.moments()
        for got, ref in zip(_f32_moments(lat), (m["rho"], m["p"], m["u"].ravel())):
            assert np.all(np.abs(got - ref) <= ULP * np.abs(ref) + 1e-12)
    lat.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("mode", [0, 1, 2, 3])
@pytest.mark.parametrize("lattice,shape", [("D2Q9", (33, 9, 1)), ("D3Q27", (19, 6, 5))])
def test_initial_state_rounds_the_fp64_one(lattice, shape, mode, storage):
    lat, rng, n = _lattice(lattice, shape, storage)
    ref, _, _ = _lattice(lattice, shape, "fp64")
    p0 = (1e-2 * rng.standard_normal(n)).astype(np.float32)
    u0 = (5e-2 * rng.standard_normal(3 * n)).astype(np.float32)
    for h in (lat, ref):
        h.init_equilibrium(p0=p0, u0=u0.copy(), integral=bool(mode & 1), half_force=bool(mode & 2))
    f, fr = lat.populations(), ref.populations()
    # stored: f/w minus the rest state, at 24 or 11 bits of a deviation below 1
    # (phi varies by 0.4 between neighbours); populations are weighted by w <= 1
    half_ulp = 2.0 ** -25 if storage == "fp32" else 2.0 ** -12
    w = fr.sum(axis=0) / fr.sum()
    assert np.all(np.abs(f - fr) <= w.max() * half_ulp + 1e-12)
    lat.close()
    ref.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
def test_non_finite_states_read_back_as_in_fp64(storage):
    import torch
    lat, rng, n = _lattice("D3Q19", (21, 6, 5), storage)
    p0 = torch.zeros(n, device="cuda")
    p0[7], p0[50], p0[99] = float("inf"), float("nan"), 3e38
    lat.init_equilibrium(p0=p0)
    m = lat.moments()
    for got, ref in zip(_f32_moments(lat), (m["rho"], m["p"], m["u"].ravel())):
        with np.errstate(over="ignore"):
            ref = ref.astype(np.float32).astype(np.float64)
        assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref))
    lat.close()
