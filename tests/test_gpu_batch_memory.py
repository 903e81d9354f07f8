"""Joining a batch leaves no device memory behind."""
import pytest

from paper_2208_09267_gb300 import lbm

pytestmark = pytest.mark.gpu


def test_memberships_of_a_lattice_hold_no_memory_of_their_own():
    """A hundred memberships of a lattice of 2^18 cells: no more than the pool's
    granularity is taken (32 MiB; one buffer a membership would be 300)."""
    import torch
    lat = lbm.Lattice("D3Q19", (64, 64, 64), tau=0.6, storage="fp32")
    b = lbm.Batch(max_members=1, storage="fp32")
    b.add(lat, 1000)
    b.step(2, check=True)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(100):
        b.remove(lat)
        b.add(lat, 1000)
        b.step(2, check=True)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= 32 << 20
    b.close()
    lat.close()
