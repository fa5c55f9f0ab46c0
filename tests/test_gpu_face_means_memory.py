"""Memory of the stored face means of a per-voxel diffusivity: they are optional
and given up when the device is full, and nothing else depends on them.  A
refused device allocation is made by the test hook; every system must come out
at the oracle's step (the bound is that of test_gpu_face_means.py: the residual
is driven to TOL, and A is an M-matrix with smallest eigenvalue >= 1)."""
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


@pytest.fixture(scope="module")
def case():
    wl = W.random_case(31, (21, 13, 11), nspecies=3, dfac=True)
    ref, states = wl.lattice.copy(), []
    for _ in range(3):
        oracle.step(ref, wl.params, wl.margin, rtol=0.0, atol=TOL)
        states.append(ref.fields.copy())
    return wl, states


class System:
    """One subgrid of ctx on a lattice of its own, stepped in one of three forms."""

    def __init__(self, M, ctx, wl, form):
        self.M, self.n = M, 0
        self.lat, self.prm = M.DeviceLattice(wl.lattice), M.DeviceParams(wl.params)
        if form == "batch":
            self.b = M.BatchStepper(ctx, [self.lat], [self.prm], [wl.margin])
            self.sub, self._step = self.b.subs[0], lambda o: self.b.step(o)[0]
        else:
            s = M.StepSolver(ctx, self.lat, self.prm, wl.margin, fused=form == "step")
            self.sub, self._step = s.sub, lambda o: s.step(o)["status_code"]

    def step(self, restart=16):
        opts = self.M.make_opts(rtol=0.0, atol=TOL, restart=restart, maxit=800)
        assert self._step(opts) == self.M.OK
        self.n += 1

    def error(self, states):
        return np.max(np.abs(self.lat.fields_numpy() - states[self.n - 1]))


def held(M, ctx):
    return ctx.counter(M.COUNTER_FACE_MEANS_BYTES)


@pytest.mark.parametrize("form", ["composed", "step", "batch"])
def test_a_call_that_had_to_give_the_means_up_succeeds(M, case, form):
    wl, states = case
    ctx = M.Context(0)
    a = System(M, ctx, wl, form)
    a.step()
    assert held(M, ctx) > 0
    ctx.debug_set(M.DEBUG_REFUSE_ALLOC, 1)
    b = System(M, ctx, wl, form)
    b.step()
    a.step()
    b.step()
    assert a.error(states) <= BOUND and b.error(states) <= BOUND


@pytest.mark.parametrize("form", ["composed", "step", "batch"])
def test_whichever_allocation_is_refused_the_call_succeeds(M, case, form):
    """A second subgrid makes at most ten device allocations of its own (the
    device-resident step: tile tables, elements, means, scratch, barriers, Krylov
    bases, descriptors, partials, rates, extraction scratch)."""
    wl, states = case
    for n in range(1, 12):
        ctx = M.Context(0)
        a = System(M, ctx, wl, form)
        a.step()
        ctx.debug_set(M.DEBUG_REFUSE_ALLOC, n)
        b = System(M, ctx, wl, form)
        b.step()
        assert a.error(states) <= BOUND and b.error(states) <= BOUND, n
        a.step()
        assert a.error(states) <= BOUND, n


def test_a_network_takes_the_memory_of_the_means(M, case):
    wl, states = case
    ctx = M.Context(0)
    a = System(M, ctx, wl, "step")
    a.step()
    ctx.debug_set(M.DEBUG_REFUSE_ALLOC, 1)
    M.CNN(ctx, wl.lattice.dims, 1, M.cnn_init_params(1))
    assert held(M, ctx) == 0
    a.step()
    assert a.error(states) <= BOUND


def test_the_step_holds_48_bytes_a_stored_voxel(M, case):
    wl, _ = case
    ctx = M.Context(0)
    System(M, ctx, wl, "step").step()
    assert held(M, ctx) == 48 * 24 * 16 * 12      # the lattice of 21 x 13 x 11 in tiles of 4 x 4 x 4


def test_a_batch_makes_no_means_of_its_own(M, case):
    """Given up while the batch is planned again, the means stay given up until
    the next extraction: a buffer of a later call would not have been filled."""
    wl, states = case
    ctx = M.Context(0)
    a = System(M, ctx, wl, "batch")
    a.step(8)
    assert held(M, ctx) > 0
    ctx.debug_set(M.DEBUG_REFUSE_ALLOC, 1)
    a.step(32)                                    # longer restart: the Krylov bases grow
    assert held(M, ctx) == 0
    a.step(32)
    assert held(M, ctx) == 0 and a.error(states) <= BOUND


def test_refresh_and_assembly_can_be_captured(M, case):
    import torch
    wl, states = case
    ctx = M.Context(0)
    System(M, ctx, wl, "composed").step()         # every kernel is loaded
    lat, prm, sub = M.DeviceLattice(wl.lattice), M.DeviceParams(wl.params), ctx.subgrid_create()
    sub.mpm_box_extract(lat, 3, wl.margin)
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        sub.mpm_subgrid_refresh(lat)
        sub.mpm_assemble_coeffs(prm)
    opts = M.make_opts(rtol=0.0, atol=TOL, restart=16, maxit=800)
    for want in states:
        g.replay()
        sub.mpm_solve_step(opts, scatter_to=lat)
        assert np.max(np.abs(lat.fields_numpy() - want)) <= BOUND


@pytest.mark.parametrize("form", ["composed", "step"])
@pytest.mark.parametrize("nth", [1, 3])           # the next growing buffer; the means' own request
def test_means_without_room_are_not_requested_again(M, case, form, nth):
    wl, states = case
    ctx = M.Context(0)
    a = System(M, ctx, wl, form)
    if nth == 1:
        a.step(8)
    ctx.debug_set(M.DEBUG_REFUSE_ALLOC, nth)
    a.step(32)                                    # tile tables, elements, means; Krylov bases
    assert held(M, ctx) == 0
    a.step(32)
    assert held(M, ctx) == 0 and a.error(states) <= BOUND


def test_means_that_a_recorded_graph_writes_stay(M, case):
    import torch
    wl, states = case
    System(M, M.Context(0), wl, "composed").step()     # every kernel is loaded
    ctx = M.Context(0)
    lat, prm, sub = M.DeviceLattice(wl.lattice), M.DeviceParams(wl.params), ctx.subgrid_create()
    sub.mpm_box_extract(lat, 3, wl.margin)
    before = held(M, ctx)
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        sub.mpm_subgrid_refresh(lat)
        sub.mpm_assemble_coeffs(prm)
    ctx.debug_set(M.DEBUG_REFUSE_ALLOC, 1)
    with pytest.raises(M.MpmError):                    # nothing that could be given up
        M.CNN(ctx, wl.lattice.dims, 1, M.cnn_init_params(1))
    assert held(M, ctx) == before > 0
    opts = M.make_opts(rtol=0.0, atol=TOL, restart=16, maxit=800)
    for want in states:
        g.replay()
        sub.mpm_solve_step(opts, scatter_to=lat)
        assert np.max(np.abs(lat.fields_numpy() - want)) <= BOUND
    uniform = M.DeviceLattice(W.random_case(31, (21, 13, 11), nspecies=3).lattice)
    sub.mpm_box_extract(uniform, 3, wl.margin)         # leaves the buffer to the graph
    assert held(M, ctx) == 0


def test_a_subgrid_destroyed_without_its_context_leaves_nothing_behind(M, case):
    """mpm_subgrid_destroy(NULL, sub) is allowed, before the context is destroyed
    and after it."""
    wl, states = case
    ctx = M.Context(0)
    a, b = System(M, ctx, wl, "step"), System(M, ctx, wl, "step")
    a.step()
    b.step()
    one = held(M, ctx) // 2
    h, a.sub.h = a.sub.h, None                          # the binding's own destroy has nothing left to do
    assert ctx.lib.mpm_subgrid_destroy(None, h) == M.OK
    assert held(M, ctx) == one
    ctx.debug_set(M.DEBUG_REFUSE_ALLOC, 1)
    c = System(M, ctx, wl, "step")
    c.step()
    b.step()
    assert b.error(states) <= BOUND and c.error(states) <= BOUND
    handles = [s.sub.h for s in (b, c)]
    b.sub.h = c.sub.h = None
    lib = ctx.lib
    ctx.close()
    assert [lib.mpm_subgrid_destroy(None, h) for h in handles] == [M.OK, M.OK]
