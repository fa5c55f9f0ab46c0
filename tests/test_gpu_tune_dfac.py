"""The solver tuner and a per-voxel diffusivity: a batch that has one runs kernels
of its own in one variant, so the tuner must not choose a variant from it, nor
share a cache line with a batch that has none."""
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


@pytest.mark.parametrize("precision", [0, 1])
def test_a_batch_with_dfac_has_one_variant_and_cache_lines_of_its_own(M, tmp_path, precision):
    wl = W.random_case(31, (21, 13, 11), nspecies=3, dfac=True)
    uniform = wl.lattice.copy()
    uniform.dfac = None
    ctx, cache = M.Context(), str(tmp_path / "tune.txt")
    prm = M.DeviceParams(wl.params)

    def tune(lattice):
        sub = ctx.subgrid_create()
        lat = M.DeviceLattice(lattice)
        sub.mpm_box_extract(lat, 3, wl.margin)
        sub.mpm_assemble_coeffs(prm)
        opts = M.make_opts(rtol=1e-8, restart=8, maxit=400, precision=precision, inner_rtol=1e-4)
        m, var = ctx.mpm_tune_solver([sub], opts, cache)
        with open(cache) as f:
            return m, var, sum(1 for _ in f)

    m, var, lines = tune(wl.lattice)
    assert var == 0 and lines == 1
    assert tune(uniform)[2] == 2                      # a miss: timed and added
    assert tune(wl.lattice) == (m, 0, 2)              # both are hits now
    assert tune(uniform)[2] == 2
