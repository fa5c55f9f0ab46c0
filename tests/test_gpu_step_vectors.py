"""The device-resident step's extraction on four-voxel vectors (rows of a
multiple of four voxels, a box starting at any x) and on single voxels (other
rows) against the composed extraction and assembly: box, stored tiles, face
flags, cell ids, rows, and the in-mask count."""
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


def _case(lx, lo, hi, nspecies):
    """A lattice whose tumour spans x in [lo, hi)."""
    wl = W.random_case(lx + 7 * lo + hi, (lx, 13, 9), nspecies=nspecies)
    c = wl.lattice.cell_id
    c[:, :, :lo] = 0
    c[:, :, hi:] = 0
    c[4, 6, lo] = c[5, 7, hi - 1] = 1
    wl.lattice.mask[:, ::3, :] = wl.lattice.mask[:, ::3, :] * 7      # any non-zero byte is in the mask
    return wl


@pytest.mark.parametrize("tile", [None, (8, 4, 2), (2, 4, 4), (1, 8, 4), (16, 2, 2), (64, 1, 1)])
@pytest.mark.parametrize("lx,lo,hi,margin", [(32, 0, 32, 0), (32, 5, 31, 1), (32, 9, 30, 0), (32, 10, 11, 1),
                                             (32, 14, 27, 3), (140, 2, 139, 1), (136, 3, 136, 0), (31, 6, 20, 2),
                                             (33, 1, 33, 0)])
def test_step_extraction_equals_the_composed_one(M, lx, lo, hi, margin, tile):
    ns = 1 + (lx + lo) % 4
    wl = _case(lx, lo, hi, ns)
    ctx = M.Context()
    prm = M.DeviceParams(wl.params)
    la, lb = M.DeviceLattice(wl.lattice), M.DeviceLattice(wl.lattice)
    a, b = ctx.subgrid_create(), ctx.subgrid_create()
    opts = M.make_opts(rtol=1e-8, restart=8, maxit=200, precision=1, inner_rtol=1e-6)
    rep = a.mpm_step(la, prm, margin, opts, tile)
    box = b.mpm_box_extract(lb, ns, margin, tile)
    b.mpm_assemble_coeffs(prm)
    assert rep["box"] == box
    ia, ib = a.info(), b.info()
    assert ia == ib and rep["mask_voxels"] == ib["mask_voxels"]
    for what in (M.EXPORT_FLAGS, M.EXPORT_CELL):
        assert np.array_equal(a.mpm_subgrid_export(what).cpu().numpy(), b.mpm_subgrid_export(what).cpu().numpy())
    for s in range(ns):
        for what in (M.EXPORT_RHS, M.EXPORT_DIAG):
            x, y = a.mpm_subgrid_export(what, s).cpu().numpy(), b.mpm_subgrid_export(what, s).cpu().numpy()
            # three roundings of terms no larger than the sum on either side
            assert np.max(np.abs(x - y) / np.maximum(np.abs(y), 1.0)) <= 8 * 2.0 ** -53
