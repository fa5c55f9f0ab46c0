"""The harmonic means of a per-voxel diffusivity stored by the assembly against
the oracle, and against a context with a memory cap, whose solver forms them in
every pass: composed, device-resident and batched steps, both precisions."""
import numpy as np
import pytest

import oracle
from paper_2505_03067_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-13          # absolute residual both sides are driven to
BOUND = 1e-10        # |x - x*| <= ||r|| (the system is an M-matrix with smallest eigenvalue >= 1)


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2505_03067_gb300 import build, mpm
    build.build()
    return mpm


def _step(M, ctx, wl, form, opts, tile):
    lat, prm = M.DeviceLattice(wl.lattice), M.DeviceParams(wl.params)
    if form == "batch":
        b = M.BatchStepper(ctx, [lat], [prm], [wl.margin], tile=tile)
        for _ in range(2):
            st, _ = b.step(opts)
    else:
        s = M.StepSolver(ctx, lat, prm, wl.margin, tile=tile, fused=form == "step")
        for _ in range(2):
            st = s.step(opts)["status_code"]
    assert st == M.OK
    return lat.fields_numpy()


@pytest.mark.parametrize("form", ["composed", "step", "batch"])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("dims,tile", [((21, 13, 11), None), ((9, 34, 7), (8, 4, 2)), ((5, 6, 4), (2, 4, 4))])
def test_stored_means_equal_the_oracle_and_the_means_formed_in_the_pass(M, form, precision, dims, tile):
    wl = W.random_case(sum(dims), dims, nspecies=3, dfac=True)
    ref = wl.lattice.copy()
    for _ in range(2):
        oracle.step(ref, wl.params, wl.margin, rtol=0.0, atol=TOL)
    opts = M.make_opts(rtol=0.0, atol=TOL, restart=8 if precision else 16, maxit=800, precision=precision,
                       inner_rtol=1e-6)
    for cap in (0, 1 << 32):
        got = _step(M, M.Context(cap), wl, form, opts, tile)
        assert np.max(np.abs(got - ref.fields)) <= BOUND, cap
