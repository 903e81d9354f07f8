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
