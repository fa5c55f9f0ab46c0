"""Which form of the stencil a per-voxel diffusivity runs, and that each is right:
stored face means (the counter says that they are held) and means formed in the
pass (a context with a memory cap holds none), at the largest restart bucket, and
in a batch that mixes systems with and without a factor.  Bounds as in
test_gpu_face_means.py."""
import numpy as np
import pytest

import oracle
from paper_2505_03067_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-13
BOUND = 1e-10


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2505_03067_gb300 import build, mpm
    build.build()
    return mpm


def _opts(M, precision, restart):
    return M.make_opts(rtol=0.0, atol=TOL, restart=restart, maxit=800, precision=precision, inner_rtol=1e-6)


def _reference(wl):
    ref = wl.lattice.copy()
    for _ in range(2):
        oracle.step(ref, wl.params, wl.margin, rtol=0.0, atol=TOL)
    return ref.fields


@pytest.mark.parametrize("cap", [0, 1 << 32])
@pytest.mark.parametrize("form", ["composed", "step"])
@pytest.mark.parametrize("precision", [0, 1])
def test_restart_32_in_both_forms(M, cap, form, precision):
    wl = W.random_case(57, (19, 14, 9), nspecies=2, dfac=True)
    ctx = M.Context(cap)
    lat, prm = M.DeviceLattice(wl.lattice), M.DeviceParams(wl.params)
    s = M.StepSolver(ctx, lat, prm, wl.margin, fused=form == "step")
    for _ in range(2):
        assert s.step(_opts(M, precision, 32))["status_code"] == M.OK
    assert (ctx.counter(M.COUNTER_FACE_MEANS_BYTES) > 0) == (cap == 0)
    assert np.max(np.abs(lat.fields_numpy() - _reference(wl))) <= BOUND


@pytest.mark.parametrize("cap", [0, 1 << 32])
@pytest.mark.parametrize("precision,restart", [(0, 8), (0, 16), (1, 8), (1, 32)])
def test_a_batch_of_systems_with_and_without_a_factor(M, cap, precision, restart):
    wls = [W.random_case(61, (13, 11, 9), nspecies=3, dfac=True), W.random_case(62, (16, 9, 8), nspecies=3),
           W.random_case(63, (8, 12, 10), nspecies=2, dfac=True)]
    ctx = M.Context(cap)
    lats = [M.DeviceLattice(w.lattice) for w in wls]
    b = M.BatchStepper(ctx, lats, [M.DeviceParams(w.params) for w in wls], [w.margin for w in wls])
    for _ in range(2):
        assert b.step(_opts(M, precision, restart))[0] == M.OK
    assert (ctx.counter(M.COUNTER_FACE_MEANS_BYTES) > 0) == (cap == 0)
    for lat, wl in zip(lats, wls):
        assert np.max(np.abs(lat.fields_numpy() - _reference(wl))) <= BOUND
