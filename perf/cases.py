"""The work this framework is measured on: one pass of each of its public paths, at small, ordinary and
large sizes.

A case is a dict of plain values; `prepare` makes the inputs on the GPU from a seed, `run` is one pass
through the public entry points, `exact` the same result from plain torch in 64 bits, `work` the bytes
and operations that the pass cannot do without.

The per-cell rates alternate between two tables from pass to pass (the CPM revises its cells' rates
every Monte Carlo step), so that a lattice stepped many times keeps having something to solve.
"""
import math

import numpy as np
import torch

from paper_2505_03067_gb300 import mpm
from paper_2505_03067_gb300 import workloads as W

MIXED = dict(rtol=1e-6, restart=8, maxit=1000, precision=1, inner_rtol=1e-6)
FP64 = dict(rtol=1e-6, restart=8, maxit=1000, precision=0)
CHANNELS = (9, 24, 24, 24, 24, 24, 3)
S_OUT = 0.01
MAX_VOXELS = 512 * 384 * 384


def _shell(name, kind, dims, extent, cell=100.0, species=3, mixed=True, **more):
    return dict(name=name, kind=kind, shape="shell", nx=dims[0], ny=dims[1], nz=dims[2], extent=extent, cell=cell,
                species=species, mixed=mixed, **more)


def _sphere(name, kind, n, species=1, mixed=False, **more):
    return dict(name=name, kind=kind, shape="sphere", nx=n, ny=n, nz=n, extent=0.25, cell=43.0, species=species,
                mixed=mixed, **more)


def listed():
    return [
        # the smallest step a user takes: one species in a 32^3 box, full FP64, long restart, tight tolerance
        _sphere("sphere32_fp64", "step", 32, tight=True),
        # an ordinary CPM lattice: three species on a pleural shell, steps queued back to back
        _shell("shell256_mixed", "step", (256, 256, 256), 0.5, queued=True),
        # the same with FP64 throughout, the host reading each step's report
        _shell("shell256_fp64", "step", (256, 256, 256), 0.5, mixed=False),
        # the largest lattice with its tumour fully grown, on the tuner's tile
        _shell("growth512_mixed", "step", (512, 384, 384), 0.65, cell=200.0, queued=True, tuned=True),
        # extract, assemble and solve called one by one: odd dims, four species, a diffusivity per voxel
        _shell("ragged_composed", "composed", (97, 150, 121), 0.7, species=4, mixed=False, dfac=True),
        # the learned form: the network's guess inside the step, on the growth region of the large lattice
        _shell("crop_learned", "step", (324, 264, 264), 0.9, cell=200.0, queued=True, tuned=True, learned=True),
        # cell ids and fields in page-locked host memory, as a CPM on the host keeps them
        _shell("shell256_host", "host", (256, 256, 256), 0.5),
        # many patients' patches at once, replayed from one graph
        dict(name="patches64_mixed", kind="batch", systems=64, lo=16, hi=96, mixed=True),
        # the network alone on the largest pleural box, features included
        _shell("crop_cnn_forward", "forward", (324, 264, 264), 0.9, cell=200.0),
        # one training step of the network as the training loop takes it
        dict(name="cnn_train_32x8", kind="train", n=32, images=8),
        # flexible GMRES with the network as the preconditioner
        _sphere("sphere32_fgmres", "fgmres", 32, mixed=True),
        # the growth driver on the largest lattice
        _shell("growth512_cpm", "cpm", (512, 384, 384), 0.65, cell=200.0, species=2),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sphere", "step", "step", "step", "composed", "learned", "host", "batch", "forward", "train",
                       "fgmres", "cpm"])
    if kind == "sphere":
        tight = rng.random() < 0.5
        c = _sphere("", "step", _log(rng, 16, 72), species=rng.randint(1, 4), mixed=not tight and rng.random() < 0.5,
                    tight=tight)
    elif kind == "batch":
        lo = _log(rng, 8, 24)
        c = dict(name="", kind="batch", systems=_log(rng, 3, 64), lo=lo, hi=_log(rng, lo + 8, 96),
                 mixed=rng.random() < 0.7)
    elif kind == "train":
        c = dict(name="", kind="train", n=rng.randint(12, 32), images=rng.randint(1, 8))
    elif kind == "fgmres":
        c = _sphere("", "fgmres", _log(rng, 12, 48), species=rng.randint(1, 3), mixed=rng.random() < 0.5)
    else:
        top = {"step": (512, 384), "cpm": (512, 384), "host": (256, 256), "composed": (200, 200),
               "learned": (324, 264), "forward": (324, 264)}[kind]
        dims = (_log(rng, 48, top[0]), _log(rng, 48, top[1]), _log(rng, 48, top[1]))
        more = {}
        if kind == "step":
            more = dict(queued=rng.random() < 0.5, tuned=rng.random() < 0.5)
            if rng.random() < 0.25:
                more["every"] = 50
        elif kind == "learned":
            more = dict(queued=rng.random() < 0.5, tuned=rng.random() < 0.5, learned=True)
        elif kind == "composed":
            more = dict(dfac=rng.random() < 0.5)
        species = 2 if kind == "cpm" else 3 if kind in ("learned", "forward") else rng.randint(1, 4)
        c = _shell("", "step" if kind == "learned" else kind, dims, rng.uniform(0.3, 0.9),
                   cell=rng.choice([100.0, 200.0]), species=species, mixed=rng.random() < 0.6, **more)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------ inputs
class _Lattice(mpm.DeviceLattice):
    """A device lattice from tensors that are on the GPU already."""

    def __init__(self, cell_id, mask, fields, dfac=None):
        self.cell_id, self.mask, self.fields, self.dfac = cell_id, mask, fields, dfac
        self.nspecies = int(fields.shape[0])
        self.dims = (int(cell_id.shape[2]), int(cell_id.shape[1]), int(cell_id.shape[0]))


class _State:
    """What a user's program keeps between passes; gives the library's objects back when it is dropped."""

    def __init__(self):
        self.ctx = mpm.Context()
        self.subs, self.nets, self.i = [], [], 0

    def __del__(self):
        try:
            torch.cuda.synchronize()
            for n in self.nets:
                n.close()
            for s in self.subs:
                s.destroy()
            self.ctx.close()
        except Exception:
            pass


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _voronoi(pts, pitch, g):
    """Nearest of the seeds of a jittered grid of the given pitch, as labels 0, 1, ... of the seeds in use."""
    p = pts / pitch
    base = p.floor().long()
    lo = base.amin(0) - 2
    n = base.amax(0) + 3 - lo
    n = [int(v) for v in n]
    jitter = torch.rand((n[0] * n[1] * n[2], 3), generator=g, device="cuda")
    best = torch.full((len(pts),), 1e9, device="cuda")
    label = torch.zeros(len(pts), dtype=torch.long, device="cuda")
    for o in range(27):
        c = base + torch.tensor([o % 3 - 1, o // 3 % 3 - 1, o // 9 - 1], device="cuda")
        k = ((c[:, 0] - lo[0]) * n[1] + (c[:, 1] - lo[1])) * n[2] + (c[:, 2] - lo[2])
        d = (c + jitter[k] - p).square().sum(1)
        near = d < best
        best = torch.where(near, d, best)
        label = torch.where(near, k, label)
    return torch.unique(label, return_inverse=True)[1]


def _axes(dims):
    nx, ny, nz = dims
    return (torch.arange(nx, device="cuda")[None, None, :], torch.arange(ny, device="cuda")[None, :, None],
            torch.arange(nz, device="cuda")[:, None, None])


def _shell_mask(dims, full=None, origin=(0, 0, 0)):
    """Pleural space: between two ellipsoids 10 voxels apart (15 on a lattice of over 300), in the proportions
    of the 256^3 workload; `full` and `origin`: a crop of a larger lattice."""
    full = full or dims
    x, y, z = _axes(dims)
    a = [0.43 * full[0], 0.4 * full[1], 0.45 * full[2]]
    t = 10.0 if max(full) <= 300 else 15.0
    q = [(v + o - (f - 1) / 2.0) for v, o, f in zip((x, y, z), origin, full)]
    outer = sum((v / s) ** 2 for v, s in zip(q, a)) <= 1.0
    inner = sum((v / max(1.0, s - t)) ** 2 for v, s in zip(q, a)) <= 1.0
    return (outer & ~inner).to(torch.uint8)


def _params(species, ncell, rng, sphere=False):
    """Rates as in the framework's own workloads: uptake of species 0 and 1, secretion of the others."""
    k, q = np.zeros((species, ncell + 1)), np.zeros((species, ncell + 1))
    for s in range(species):
        (k if s < 2 else q)[s, 1:] = rng.uniform(0.01, 0.1, ncell)
    D = np.array([1.0, 0.5, 0.2, 0.2])[:species]
    mu = np.array([0.0, 0.0, 0.01, 0.01])[:species]
    bc = np.array([1.0, 1.0, 0.0, 0.0])[:species]
    return W.Params(species, 0.1 if sphere else 0.05, 1.0, D, mu, bc, k, q)


def _geometry(case, seed):
    """(cell ids, mask, number of cells) of a case's lattice."""
    g = _generator(seed)
    dims = (case["nx"], case["ny"], case["nz"])
    x, y, z = _axes(dims)
    if case["shape"] == "sphere":
        n = dims[0]
        mask = torch.ones((n, n, n), dtype=torch.uint8, device="cuda")
        c = (n - 1) / 2.0
        region = (x - c) ** 2 + (y - c) ** 2 + (z - c) ** 2 <= (case["extent"] * n) ** 2
    else:
        mask = _shell_mask(dims)
        e = case["extent"]
        region = ((mask > 0) & (x >= dims[0] * (1 - e)) & ((y - dims[1] / 2).abs() <= dims[1] * e / 2)
                  & ((z - dims[2] / 2).abs() <= dims[2] * e / 2))
    at = region.reshape(-1).nonzero()[:, 0]
    pts = torch.stack([at % dims[0], at // dims[0] % dims[1], at // (dims[0] * dims[1])], 1).float()
    label = _voronoi(pts, case["cell"] ** (1 / 3), g)
    ids = torch.zeros(mask.numel(), dtype=torch.int32, device="cuda")
    ids[at] = (label + 1).int()
    return ids.view(mask.shape), mask, int(label.max()) + 1


def _fields(species, shape):
    f = torch.ones((species,) + tuple(shape), dtype=torch.float64, device="cuda")
    f[2:] = 0.0
    return f


def _two_tables(st, prm, species, rng):
    """The rates of the even passes (those of `prm`) and of the odd ones."""
    n = int(prm.k.shape[1]) - 1
    alt = _params(species, n, rng)
    st.k = [prm.k.clone(), torch.from_numpy(alt.k_cell).cuda()]
    st.q = [prm.q.clone(), torch.from_numpy(alt.q_cell).cuda()]


def _problem(st, case, seed):
    """Lattice, parameters and margin of a single-lattice case, in the state."""
    rng = np.random.default_rng(seed)
    ids, mask, ncell = _geometry(case, seed)
    S = case["species"]
    dfac = None
    if case.get("dfac"):
        dfac = torch.rand(ids.shape, generator=_generator(seed + 1), device="cuda", dtype=torch.float64) * 1.5 + 0.5
    st.lat = _Lattice(ids, mask, _fields(S, ids.shape), dfac)
    st.host_params = _params(S, ncell, rng, case["shape"] == "sphere")
    st.prm = mpm.DeviceParams(st.host_params)
    st.margin = case["nx"] if case["shape"] == "sphere" else 4
    _two_tables(st, st.prm, S, rng)


def _opts(case):
    if case.get("tight"):
        return mpm.make_opts(rtol=1e-10, restart=30, maxit=1000)
    o = dict(MIXED if case["mixed"] else FP64)
    if case.get("every"):
        o.update(box_every=case["every"], box_guard=2)
    if case["kind"] == "fgmres":
        o["rtol"] = 1e-8
    return mpm.make_opts(**o)


def _patch_systems(case, seed):
    """(lattice, parameters, margin, second rate tables) of the systems of a batch: crops of a 256^3 shell around
    random shell voxels, cells of ~100 voxels, 5 to 40 % of them tumour.  The dims come from the case alone."""
    rng, g = np.random.default_rng(seed), _generator(seed)
    full = (256, 256, 256)
    sizes = np.random.default_rng(case["systems"]).uniform(math.log(case["lo"]), math.log(case["hi"] + 1),
                                                           (case["systems"], 3))
    sizes = np.clip(np.exp(sizes).astype(int), case["lo"], case["hi"])
    out = []
    for d in sizes:
        u = rng.normal(size=3)
        u /= np.linalg.norm(u)
        c = 127.5 + u / np.sqrt(sum((u[i] / (f * 256 - 5)) ** 2 for i, f in enumerate((0.43, 0.4, 0.45))))
        o = np.clip((c - d / 2).round().astype(int), 0, 256 - d)
        d, o = [int(v) for v in d], [int(v) for v in o]
        mask = _shell_mask(d, full, o)
        at = mask.view(-1).nonzero()[:, 0]
        pts = torch.stack([at % d[0], at // d[0] % d[1], at // (d[0] * d[1])], 1).float()
        label = _voronoi(pts, 100.0 ** (1 / 3), g)
        n = int(label.max()) + 1
        tumour = np.zeros(n, np.int32)
        few = max(1, int(round(n * rng.uniform(0.05, 0.4))))
        tumour[rng.permutation(n)[:few]] = np.arange(1, few + 1)
        ids = torch.zeros(mask.numel(), dtype=torch.int32, device="cuda")
        ids[at] = torch.from_numpy(tumour).cuda()[label]
        out.append((_Lattice(ids.view(mask.shape), mask, _fields(3, mask.shape)), _params(3, few, rng), max(d),
                    _params(3, few, rng)))
    return out


def _prepare_batch(st, case, seed):
    systems = _patch_systems(case, seed)
    st.lats = [s[0] for s in systems]
    st.host_params = [s[1] for s in systems]
    st.margins = [s[2] for s in systems]
    st.prms = [mpm.DeviceParams(p) for p in st.host_params]
    # the rate tables of all systems side by side, so that a pass revises them by two copies
    tables = [[torch.from_numpy(np.concatenate([getattr(s[j], a).reshape(-1) for s in systems])).cuda()
               for j in (1, 3)] for a in ("k_cell", "q_cell")]
    st.k, st.q = tables
    st.now_k, st.now_q = st.k[0].clone(), st.q[0].clone()
    at = 0
    for p in st.prms:
        n = p.k.numel()
        p.k, p.q = st.now_k[at:at + n].view(p.k.shape), st.now_q[at:at + n].view(p.q.shape)
        p.struct.k_cell, p.struct.q_cell = p.k.data_ptr(), p.q.data_ptr()
        at += n
    st.batch = mpm.BatchStepper(st.ctx, st.lats, st.prms, st.margins, tune_tiles=True)
    st.subs += st.batch.subs
    st.opts = mpm.make_opts(**(MIXED if case["mixed"] else FP64))


def _train_lattice(n, rng, g):
    """A training lattice: a tumour sphere at a random place in an n^3 box, all of it in the domain."""
    r = rng.uniform(0.125, 0.375) * n
    c = rng.uniform(0.5 * r, n - 1 - 0.5 * r, 3)
    x, y, z = _axes((n, n, n))
    region = (x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2 <= max(1.0, r * r)
    at = region.reshape(-1).nonzero()[:, 0]
    pts = torch.stack([at % n, at // n % n, at // (n * n)], 1).float()
    label = _voronoi(pts, max(2.0, (len(at) / 50) ** (1 / 3)), g)
    ids = torch.zeros(n ** 3, dtype=torch.int32, device="cuda")
    ids[at] = (label + 1).int()
    lat = _Lattice(ids.view(n, n, n), torch.ones((n, n, n), dtype=torch.uint8, device="cuda"), _fields(3, (n, n, n)))
    return lat, _params(3, int(label.max()) + 1, rng, sphere=True)


def _train_images(case, seed):
    rng, g = np.random.default_rng(seed), _generator(seed)
    return [_train_lattice(case["n"], rng, g) for _ in range(case["images"])]


def _prepare_train(st, case, seed):
    n = case["n"]
    st.box = ((0, 0, 0), (n, n, n))
    st.images = []
    for lat, params in _train_images(case, seed):
        prm = mpm.DeviceParams(params)
        nxt = _Lattice(lat.cell_id, lat.mask, lat.fields.clone())
        solver = mpm.StepSolver(st.ctx, nxt, prm, n)
        solver.step(mpm.make_opts(rtol=1e-12, restart=16, maxit=500))
        solver.sub.destroy()
        st.images.append((lat, nxt, prm))
    st.cnn = mpm.CNN(st.ctx, (n, n, n), case["images"], mpm.cnn_init_params(seed % (1 << 31)), s_out=S_OUT, train=True)
    st.nets.append(st.cnn)


def _bounds(ids, margin):
    """The tumour's box, as ((lo), (hi)) in x, y, z."""
    lo, hi = [], []
    for axis in (2, 1, 0):
        other = [a for a in (0, 1, 2) if a != axis]
        at = (ids > 0).any(dim=other[1]).any(dim=other[0]).nonzero()[:, 0]
        lo.append(max(0, int(at[0]) - margin))
        hi.append(min(int(ids.shape[axis]), int(at[-1]) + margin + 1))
    return tuple(lo), tuple(hi)


def prepare(case, seed):
    st = _State()
    st.kind = case["kind"]
    if st.kind == "batch":
        _prepare_batch(st, case, seed)
        return st
    if st.kind == "train":
        _prepare_train(st, case, seed)
        return st
    _problem(st, case, seed)
    if st.kind == "cpm":
        n = st.host_params.ncell
        # room for the daughters: a table of the tumour's voxels over the cell size, whatever the draw of the cells
        room = W.with_capacity(st.host_params, 12 * int((st.lat.cell_id > 0).sum() / case["cell"]) + 1000)
        st.prm = mpm.DeviceParams(room)
        st.lat.fields.mul_(torch.rand(st.lat.fields.shape, generator=_generator(seed + 2), device="cuda",
                                      dtype=torch.float64) * 0.5 + 0.5)
        # slow growth, as in earnest: a Monte Carlo step moves the tumour's front by a small part of a voxel
        st.driver = mpm.GrowthDriver(st.ctx, st.lat, st.prm, n, p_grow=0.02, seed=seed)
        return st
    if st.kind == "forward":
        st.box = _bounds(st.lat.cell_id, st.margin)
        st.cnn = mpm.CNN(st.ctx, st.lat.dims, 1, mpm.cnn_init_params(seed % (1 << 31)), s_out=S_OUT)
        st.nets.append(st.cnn)
        st.pred = torch.zeros((st.lat.cell_id.numel(), 3), dtype=torch.float32, device="cuda")
        return st
    st.opts = _opts(case)
    if st.kind == "fgmres":
        st.sub = st.ctx.subgrid_create()
        st.subs.append(st.sub)
        st.cnn = mpm.CNN(st.ctx, st.lat.dims, 1, mpm.cnn_init_params(seed % (1 << 31)), s_out=S_OUT)
        st.nets.append(st.cnn)
        return st
    tile = st.ctx.mpm_tune_tile(st.lat, st.margin)[0] if case.get("tuned") else None
    st.solver = mpm.StepSolver(st.ctx, st.lat, st.prm, st.margin, tile=tile, fused=st.kind != "composed")
    st.subs.append(st.solver.sub)
    st.queued = bool(case.get("queued"))
    if case.get("learned"):
        cnn = mpm.CNN(st.ctx, st.lat.dims, 1, mpm.cnn_init_params(seed % (1 << 31)), s_out=S_OUT)
        st.nets.append(cnn)
        st.solver.set_network(cnn)
    if st.kind == "host":
        st.host_ids = torch.empty(st.lat.cell_id.shape, dtype=torch.int32, pin_memory=True)
        st.host_ids.copy_(st.lat.cell_id)
        st.host_fields = torch.empty(st.lat.fields.shape, dtype=torch.float64, pin_memory=True)
        st.host_fields.copy_(st.lat.fields)
    return st


# ------------------------------------------------------------------------------------------------ one pass
def run(st):
    kind = st.kind
    if kind == "cpm":
        st.driver.step()
        return {"cell_id": st.lat.cell_id, "ncell": st.driver.ncell, "stats": st.driver.stats, "k": st.prm.k,
                "q": st.prm.q}
    if kind == "forward":
        st.cnn.load_image(0, st.lat, st.prm, st.box, mpm.CNN_INPUT)
        return st.cnn.forward(1, pred=st.pred)
    if kind == "train":
        for b, (lat, nxt, prm) in enumerate(st.images):
            st.cnn.load_image(b, lat, prm, st.box, mpm.CNN_INPUT)
            st.cnn.load_image(b, nxt, prm, st.box, mpm.CNN_TARGET)
        # the rate of the cosine schedule's end
        loss = st.cnn.train_step(len(st.images), 1e-4)
        return {"loss": loss, "grad": st.cnn.get(1)}
    j = st.i & 1
    st.i += 1
    if kind == "batch":
        st.now_k.copy_(st.k[j])
        st.now_q.copy_(st.q[j])
        st.batch.step(st.opts)
        return [lat.fields for lat in st.lats]
    st.prm.k.copy_(st.k[j])
    st.prm.q.copy_(st.q[j])
    if kind == "fgmres":
        st.sub.mpm_box_extract(st.lat, st.lat.nspecies, st.margin)
        st.sub.mpm_assemble_coeffs(st.prm)
        st.cnn.solve_fgmres(st.sub, st.lat, st.prm, st.opts, scatter_to=st.lat)
        return st.lat.fields
    if kind == "host":
        rep = st.solver.step_host(st.host_ids, st.host_fields, st.opts)
        return {"fields": st.host_fields, "box": np.array(rep["box"])}
    if st.queued:
        st.solver.step_async(st.opts)
        return st.lat.fields
    rep = st.solver.step(st.opts)
    return {"fields": st.lat.fields, "box": np.array(rep["box"])}


# ------------------------------------------------------------------------------------------------ exact
def _conjugate_gradients(ids, mask, c, box, p, s, dfac=None):
    """c^{n+1} of species s on the in-mask voxels of the box: the implicit Euler finite-volume system solved to
    the last digits; `c` with those voxels replaced."""
    (x0, y0, z0), (x1, y1, z1) = box
    sl = (slice(z0, z1), slice(y0, y1), slice(x0, x1))
    m = (mask[sl] > 0).double()
    i = ids[sl].long()
    a = p.dt / p.h ** 2
    d = torch.full_like(m, float(p.D[s])) if dfac is None else float(p.D[s]) * dfac[sl]
    k, q = torch.from_numpy(p.k_cell[s]).cuda()[i], torch.from_numpy(p.q_cell[s]).cuda()[i]
    diag = 1.0 + p.dt * (float(p.mu[s]) + k)
    b = c[sl] + p.dt * q
    faces = []
    for ax in range(3):
        n = m.shape[ax]
        lo, hi = d.narrow(ax, 0, n - 1), d.narrow(ax, 1, n - 1)
        w = a * 2.0 * lo * hi / (lo + hi) * m.narrow(ax, 0, n - 1) * m.narrow(ax, 1, n - 1)
        diag.narrow(ax, 0, n - 1).add_(w)
        diag.narrow(ax, 1, n - 1).add_(w)
        faces.append(w)
        for at in (0, n - 1):
            diag.narrow(ax, at, 1).add_(2.0 * a * d.narrow(ax, at, 1))
            b.narrow(ax, at, 1).add_(2.0 * a * d.narrow(ax, at, 1) * float(p.c_bc[s]))
    diag, b = torch.where(m > 0, diag, torch.ones_like(m)), b * m

    def apply(v):
        y = diag * v
        for ax, w in enumerate(faces):
            n = w.shape[ax]
            y.narrow(ax, 0, n).sub_(w * v.narrow(ax, 1, n))
            y.narrow(ax, 1, n).sub_(w * v.narrow(ax, 0, n))
        return y

    x = c[sl] * m
    r = b - apply(x)
    p_, rho = r.clone(), float((r * r).sum())
    end = 1e-32 * float((b * b).sum())
    for _ in range(200):
        if rho <= end:
            break
        ap = apply(p_)
        alpha = rho / float((p_ * ap).sum())
        x += alpha * p_
        r -= alpha * ap
        new = float((r * r).sum())
        p_ = r + (new / rho) * p_
        rho = new
    out = c.clone()
    out[sl] = torch.where(m > 0, x, c[sl])
    return out


def _exact_fields(ids, mask, p, margin, dfac=None):
    box = _bounds(ids, margin)
    c = _fields(p.nspecies, ids.shape)
    for s in range(p.nspecies):
        c[s] = _conjugate_gradients(ids, mask, c[s].clone(), box, p, s, dfac)
    return c, box


def _features(lat_ids, lat_mask, fields, p, box):
    """The nine input channels of the active voxels, their flat positions and c^n there."""
    (x0, y0, z0), (x1, y1, z1) = box
    inside = torch.zeros_like(lat_mask)
    inside[z0:z1, y0:y1, x0:x1] = lat_mask[z0:z1, y0:y1, x0:x1]
    at = (inside.view(-1) > 0).nonzero()[:, 0]
    i = lat_ids.view(-1)[at].long()
    c = fields.view(fields.shape[0], -1)[:, at]
    k, q = torch.from_numpy(p.k_cell).cuda(), torch.from_numpy(p.q_cell).cuda()
    x = torch.stack([c[0], c[1], 20 * c[2], (i == 0).double(), (i > 0).double(), 10 * k[0][i], 10 * k[1][i],
                     10 * q[2][i], torch.ones_like(c[0])], 1)
    return x, at, c.t().contiguous()


def _taps(at, dims, where):
    """For each tap, the row of the neighbour among the active voxels (the last row, all zero, where it is none)."""
    nx, ny, nz = dims
    x, y, z = at % nx, at // nx % ny, at // (nx * ny)
    for t in range(27):
        i, j, k = x + t % 3 - 1, y + t // 3 % 3 - 1, z + t // 9 - 1
        ok = (i >= 0) & (i < nx) & (j >= 0) & (j < ny) & (k >= 0) & (k < nz)
        yield torch.where(ok, where[torch.where(ok, i + nx * (j + ny * k), torch.zeros_like(at))],
                          torch.full_like(at, len(at)))


def _network(x, at, dims, params):
    """z6 of the masked network on the active voxels (rows of x)."""
    where = torch.full((dims[0] * dims[1] * dims[2],), len(at), dtype=torch.long, device="cuda")
    where[at] = torch.arange(len(at), device="cuda")
    taps = list(_taps(at, dims, where))
    o = 0
    for l, (ci, co) in enumerate(zip(CHANNELS[:-1], CHANNELS[1:])):
        w = params[o:o + 27 * ci * co].view(27, ci, co)
        bias = params[o + 27 * ci * co:o + 27 * ci * co + co]
        o += 27 * ci * co + co
        padded = torch.cat([x, torch.zeros_like(x[:1])])
        y = bias.expand(len(at), co)
        for t in range(27):
            y = y + padded[taps[t]] @ w[t]
        x = torch.nn.functional.gelu(y) if l < 5 else y
    return x


def _exact_train(case, seed):
    images = _train_images(case, seed)
    n = case["n"]
    box = ((0, 0, 0), (n, n, n))
    params = torch.from_numpy(mpm.cnn_init_params(seed % (1 << 31))).double().cuda().requires_grad_()
    loss, grad = 0.0, 0.0
    for lat, p in images:
        x, at, c = _features(lat.cell_id, lat.mask, lat.fields, p, box)
        target = _exact_fields(lat.cell_id, lat.mask, p, n)[0].view(3, -1)[:, at].t()
        part = (c + S_OUT * _network(x, at, (n, n, n), params) - target).square().sum() / (3 * n ** 3 * len(images))
        grad = grad + torch.autograd.grad(part, params)[0]
        loss += float(part.detach())
    return {"loss": loss, "grad": grad.cpu().numpy()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "cpm":
        return None  # whole numbers, and rates copied as they are
    if kind == "batch":
        return [_exact_fields(lat.cell_id, lat.mask, p, margin)[0]
                for lat, p, margin, _ in _patch_systems(case, seed)]
    if kind == "train":
        return _exact_train(case, seed)
    st = _Problem()
    _problem(st, case, seed)
    ids, mask, p = st.lat.cell_id, st.lat.mask, st.host_params
    if kind == "forward":
        x, at, c = _features(ids, mask, st.lat.fields, p, _bounds(ids, st.margin))
        params = torch.from_numpy(mpm.cnn_init_params(seed % (1 << 31))).double().cuda()
        pred = torch.zeros((ids.numel(), 3), dtype=torch.float64, device="cuda")
        with torch.no_grad():
            pred[at] = c + S_OUT * _network(x, at, st.lat.dims, params)
        return pred
    fields, box = _exact_fields(ids, mask, p, st.margin, st.lat.dfac)
    if kind == "fgmres" or (kind == "step" and case.get("queued")):
        return fields
    return {"fields": fields, "box": np.array(box)}


class _Problem:
    """A case's lattice and parameters, without the library."""


# ------------------------------------------------------------------------------------------------ work
def _lattice_work(ids, mask, margin, species, dfac=False):
    (x0, y0, z0), (x1, y1, z1) = _bounds(ids, margin)
    voxels = (x1 - x0) * (y1 - y0) * (z1 - z0)
    unknowns = int(mask[z0:z1, y0:y1, x0:x1].sum())
    # the ids of the whole lattice for its box, the mask of the box, and of each unknown its fields in and out
    n = 4 * ids.numel() + voxels + unknowns * (16 * species + (8 if dfac else 0))
    # a 7-point row and an update per unknown and species, and about four Krylov steps of 40 operations
    return n, 200 * unknowns * species, unknowns


def work(case):
    kind = case["kind"]
    per_voxel = 2 * 27 * sum(a * b for a, b in zip(CHANNELS[:-1], CHANNELS[1:]))
    if kind == "train":
        v = case["images"] * case["n"] ** 3
        # features and targets read, three products of the same size a layer (no input gradient of the first)
        return {"bytes": v * (5 + 48), "flops": v * (3 * per_voxel - 2 * 27 * 9 * 24)}
    if kind == "batch":
        each = [_lattice_work(lat.cell_id, lat.mask, m, 3) for lat, _, m, _ in _patch_systems(case, 1)]
        return {"bytes": sum(e[2] * (5 + 48) for e in each), "flops": sum(e[1] for e in each)}
    ids, mask, _ = _geometry(case, 1)
    if kind == "cpm":
        # ids and mask read, the changed ids written (few); the fields only at the front
        return {"bytes": 5 * ids.numel(), "flops": 0}
    margin = case["nx"] if case["shape"] == "sphere" else 4
    n, ops, unknowns = _lattice_work(ids, mask, margin, case["species"], bool(case.get("dfac")))
    if kind == "forward":
        return {"bytes": unknowns * (5 + 24 + 12), "flops": unknowns * per_voxel}
    if case.get("learned"):
        return {"bytes": n, "flops": ops + unknowns * per_voxel}
    if kind == "fgmres":
        # one application of the network for each of about four Krylov steps
        return {"bytes": n, "flops": ops + 4 * case["species"] * unknowns * per_voxel}
    return {"bytes": n, "flops": ops}
