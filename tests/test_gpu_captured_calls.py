"""Calls that the caller captured into a graph of its own follow the lattice's
state at the replay: its time and its fields, not those of the capture."""
import numpy as np
import pytest

from paper_2208_09267_gb300 import lbm

pytestmark = pytest.mark.gpu


def _capture(stream, call):
    import torch
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        call()
    return g


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("lattice,shape,walls", [("D1Q3", (37, 1, 1), 0), ("D2Q9", (33, 9, 1), 2), ("D3Q19", (45, 7, 6), 0),
                                                 ("D3Q27", (19, 6, 5), 4)])
def test_a_captured_read_back_gives_the_fields_of_its_replay(lattice, shape, walls, storage):
    import torch
    n = int(np.prod(shape))
    rng = np.random.default_rng(n)
    s = torch.cuda.Stream()
    dt = torch.float64 if storage == "fp64" else torch.float32
    out = [torch.zeros(k * n, dtype=dt, device="cuda") for k in (1, 1, 3)]
    ref = [torch.zeros_like(t) for t in out]
    lat = lbm.Lattice(lattice, shape, tau=0.65, storage=storage, walls=walls, stream=s.cuda_stream)
    lat.set_epsilon((0.5 + 0.4 * rng.random(n)).astype(np.float32))
    lat.set_force((1e-5, -2e-6, 3e-6))
    lat.init_equilibrium()
    for _ in range(2):                      # both parities, so that the kernels are loaded
        lat.step(1, check_every=-1)
        lat.moments_into(*out)
    g = _capture(s, lambda: lat.moments_into(*out))
    for steps in (1, 1, 2, 3):              # odd, even, even, odd times
        lat.step(steps, check_every=-1)
        with torch.cuda.stream(s):
            g.replay()
        lat.moments_into(*ref)
        torch.cuda.synchronize()
        for got, want in zip(out, ref):
            assert torch.equal(got, want)
    del g
    lat.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("steps", [2, 66])
@pytest.mark.parametrize("lattice,shape", [("D2Q9", (40, 9, 1)), ("D3Q19", (256, 5, 4)), ("D3Q27", (64, 6, 5)),
                                           ("D3Q27", (320, 5, 4))])
def test_captured_steps_follow_a_phi_that_starts_to_vary(lattice, shape, steps, storage):
    """Steps captured on a static phi replay on one with a time derivative, and
    on a static one again (phi_ref, and with it the shift, stays the same)."""
    import torch
    n = int(np.prod(shape))
    rng = np.random.default_rng(n)
    e = (0.5 + 0.4 * rng.random(n)).astype(np.float32)
    d = (1e-5 * rng.standard_normal(n)).astype(np.float32)
    s = torch.cuda.Stream()
    lats = []
    for stream in (s.cuda_stream, None):
        lat = lbm.Lattice(lattice, shape, tau=0.6, storage=storage, kernel="row", fp16_rounding="nearest", stream=stream)
        lat.set_epsilon(e)
        lat.set_force((1e-5, -2e-6, 3e-6))
        lat.init_equilibrium()
        lat.step(steps, check_every=-1)
        lats.append(lat)
    lat, ref = lats
    g = _capture(s, lambda: lat.step(steps, check_every=-1))
    for phi in (None, (e, d), (e, None)):
        # the handle's time stays that of the capture's end
        if phi:
            lat.set_epsilon(*phi, n_ref=lat.steps_done)
            ref.set_epsilon(*phi, n_ref=ref.steps_done)
        with torch.cuda.stream(s):
            g.replay()
        ref.step(steps, check_every=-1)
        assert np.array_equal(lat.populations(), ref.populations())
    del g
    lat.close()
    ref.close()
