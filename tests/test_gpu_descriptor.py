"""The device descriptor is uploaded only where its values changed; calls that
the caller captured into a graph of its own move nothing until it is replayed."""
import numpy as np
import pytest

from paper_2208_09267_gb300 import lbm

pytestmark = pytest.mark.gpu

SHAPE = (32, 16, 1)


def _lattice(eps, deps, stream=None):
    lat = lbm.Lattice("D2Q9", SHAPE, tau=0.7, storage="fp64", stream=stream)
    lat.set_epsilon(eps, deps, 0)
    lat.set_force((1e-5, 0.0, 0.0))
    lat.init_equilibrium()
    return lat


def _fields():
    n = int(np.prod(SHAPE))
    rng = np.random.default_rng(3)
    return 0.5 + 0.3 * rng.random(n), 1e-3 * rng.standard_normal(n)


def test_read_back_after_a_dropped_capture():
    """Two steps are captured and never run: the populations stand at time 0,
    the handle at time 2, so the moments are those of the initial populations
    with phi + 2 d_t phi."""
    import torch
    eps, deps = _fields()
    s = torch.cuda.Stream()
    warm = _lattice(eps, deps)
    warm.step(2, check_every=-1)              # the kernels are loaded
    warm.close()
    lat, ref = _lattice(eps, deps, s.cuda_stream), _lattice(eps, deps)
    lat.moments()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        lat.step(2, check_every=-1)
    assert lat.steps_done == 2
    got = lat.moments()
    ref.set_epsilon(eps + 2 * deps, None, 0)
    want = ref.moments()
    for k in ("rho", "p", "u"):
        np.testing.assert_allclose(got[k], want[k], rtol=1e-12, atol=1e-13)
    del g
    lat.close()
    ref.close()


def test_replays_of_a_captured_step_advance_the_lattice():
    """Static phi: a graph of two steps replayed three times is six steps."""
    import torch
    eps, _ = _fields()
    s = torch.cuda.Stream()
    lat, ref = _lattice(eps, None, s.cuda_stream), _lattice(eps, None)
    lat.step(2, check_every=-1)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        lat.step(2, check_every=-1)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    ref.step(8)
    got, want = lat.moments(), ref.moments()
    for k in ("rho", "p", "u"):
        np.testing.assert_array_equal(got[k], want[k])
    lat.close()
    ref.close()
