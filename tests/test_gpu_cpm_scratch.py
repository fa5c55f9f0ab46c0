"""The growth driver's scratch under a memory cap: 4 bytes a voxel (rounded up to
256) and 40 a cell table entry are enough on lattices of any size, the smallest
included.  The step itself is compared with the oracle elsewhere; here with the
one of an uncapped context, bit for bit."""
import numpy as np
import pytest

from paper_2505_03067_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2505_03067_gb300 import build, mpm
    build.build()
    return mpm


def _al(b):
    return (b + 255) // 256 * 256


@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 4, 3), (64, 1, 1), (65, 1, 1), (33, 7, 9), (40, 31, 17)])
def test_a_context_of_four_bytes_a_voxel_steps(M, dims):
    wl = W.random_case(71, dims, nspecies=2, ncell=24)
    wl.lattice.mask[:] = 1
    L, ncell = dims[0] * dims[1] * dims[2], wl.params.k_cell.shape[1]
    cap = _al(4 * L) + _al(8 * ncell) + _al(24 * ncell) + 2 * _al(4 * (ncell + 1))
    got = []
    for c in (cap, 0):
        lat, prm = M.DeviceLattice(wl.lattice), M.DeviceParams(wl.params)
        g = M.GrowthDriver(M.Context(c), lat, prm, ncell=ncell, seed=3, p_grow=0.9, v_div=6)
        for _ in range(2):
            g.step()
        got.append((lat.cell_id.cpu().numpy(), sorted(g.counts().items())))
    assert np.array_equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
