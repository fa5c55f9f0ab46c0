"""The growth driver's two forms (small and other lattices), and its scratch under
a memory cap: 4 bytes a voxel (rounded up to 256) and 40 a cell table entry are
enough on lattices of any size, the smallest included.  There the step is
compared with the one of an uncapped context, bit for bit."""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 4, 3), (64, 1, 1), (65, 1, 1), (33, 7, 9), (4095, 1, 1),
                                  (64, 64, 1), (40, 31, 17)])
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


@pytest.mark.parametrize("dims", [(128, 128, 128), (2048, 8, 128), (129, 128, 128), (3, 701, 1000), (33, 64, 995)])
def test_both_sides_of_the_line_between_the_two_forms(M, dims):
    """Lattices of 2^16 words of 32 voxels and just above run different kernels:
    both against the oracle's step, bit for bit, with tumour on every face and
    rows shorter than a word, longer, and no multiple of it."""
    rng = np.random.default_rng(dims[0])
    shape = dims[::-1]
    wl = W.random_case(72, (8, 8, 8), nspecies=2, ncell=40)
    cell = np.where(rng.random(shape) < 0.02, rng.integers(1, 30, size=shape), 0).astype(np.int32)
    mask = (rng.random(shape) < 0.9).astype(np.uint8)
    lattice = W.Lattice(cell, mask, rng.uniform(0.0, 2.0, size=(2,) + shape), None)
    cp = dict(p_grow=0.5, K_o2=0.2, K_nut=0.3, o2_min=0.05, v_div=50)
    lat, prm = M.DeviceLattice(lattice), M.DeviceParams(wl.params)
    g = M.GrowthDriver(M.Context(), lat, prm, ncell=30, seed=9, **cp)
    k, q, nc = np.array(wl.params.k_cell), np.array(wl.params.q_cell), 30
    for t in range(2):
        g.step()
        cell, k, q, nc, _ = oracle.cpm_step(cell, mask, lattice.fields[0], lattice.fields[1], k, q, nc, cp, 9, t)
        assert np.array_equal(lat.cell_id.cpu().numpy(), cell)
        assert g.counts()["ncell"] == nc == 40
