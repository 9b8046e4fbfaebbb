"""The calls whose speed matters to a program that uses this library: forward
shots over the range of grids, space orders, forms and storages, shots with
receivers, the FWI gradient, batches of uneven shots and stepping on the
caller's own buffers. Every case goes through the package's public entry
points, from a model in device memory (host memory where the entry point takes
host arrays) to the fields a program reads back.

Models, sources and dampings are made here from the seed alone, so that
:func:`exact` can repeat a case in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

import paper_1912_00695_gb300 as fd
from paper_1912_00695_gb300._abi import fd_forward_noalloc

H = 10.0  # grid spacing in metres


def listed():
    return [
        # a small shot of the test suite's plain configuration: launches and latency count
        _shot("plain84_so4", 64, 64, 64, 10, 4, 100, model="constant", f0=10.0),
        # the paper's 256^3 workload (four layers, 10-cell absorbing layer) over its
        # space orders: the smallest stencil, where memory traffic is everything ...
        _shot("sweep276_so2", 256, 256, 256, 10, 2, 300),
        # ... the order most finite-difference propagators run ...
        _shot("sweep276_so4", 256, 256, 256, 10, 4, 300),
        # ... the unfactored expression (a coefficient for every tap) ...
        _shot("sweep276_so8_expanded", 256, 256, 256, 10, 8, 300, form="expanded"),
        # ... and the widest stencil of the sweep, where arithmetic dominates
        _shot("sweep276_so16", 256, 256, 256, 10, 16, 300),
        # the precision study's volume, 384^3 with a 20-cell layer, in bfloat16 storage
        _shot("volume424_so12_bf16", 384, 384, 384, 20, 12, 200, storage="bf16"),
        # half-precision storage on a survey-shaped grid with no round extent
        _shot("ragged_so8_f16", 201, 233, 150, 10, 8, 250, storage="f16", model="smooth"),
        # the highest space order, on odd extents
        _shot("ragged_so24", 131, 170, 151, 10, 24, 150, model="smooth"),
        # a survey: an off-grid source and a plane of receivers, traces read to the host
        _shot("receivers276_so8", 256, 256, 256, 10, 8, 300, kind="receivers", every=2),
        # one full-waveform-inversion gradient, host data in and host gradient out
        _shot("gradient200_so8", 180, 180, 180, 10, 8, 200, kind="gradient", model="smooth", f0=10.0, every=3),
        # many uneven shots advanced together
        {"name": "batch12_so8", "kind": "batch", "shots": 12, "lo": 96, "hi": 256, "sizes": 1, "nbl": 10, "so": 8,
         "nt": 150, "storage": "f32", "form": "factored", "f0": 10.0},
        # a plug-in's buffers, stepped in place without allocating
        _shot("buffers186_so8", 166, 166, 166, 10, 8, 150, kind="buffers", form="expanded", model="smooth"),
    ]


def _shot(name, nx, ny, nz, nbl, so, nt, kind="shot", storage="f32", form="factored", model="layered", f0=15.0,
          every=0):
    c = {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "nbl": nbl, "so": so, "nt": nt, "storage": storage,
         "form": form, "model": model, "f0": f0, "every": every}
    if name is None:
        del c["name"]
    return c


def draw(rng):
    kind = rng.choice(["shot"] * 10 + ["half"] * 4 + ["receivers"] * 2 + ["gradient", "batch", "batch", "buffers"])
    orders = [2, 4, 4, 6, 8, 8, 8, 10, 12, 12, 14, 16, 16]
    so = rng.choice(orders + [18, 20, 24]) if kind in ("shot", "half") else rng.choice(orders)
    form = "expanded" if kind == "buffers" or (kind in ("shot", "receivers") and rng.random() < 0.3) else "factored"
    storage = rng.choice(["bf16", "bf16", "f16"]) if kind == "half" else "f32"
    nt = int(math.exp(rng.uniform(math.log(60), math.log(400))))
    if kind == "batch":
        lo = rng.choice([32, 48, 64, 96])
        hi = int(lo * rng.uniform(1.3, 2.5))
        shots = rng.randint(4, 24 if lo > 48 else 48)
        most = shots * (0.5 * (lo + hi) + 20) ** 3
        return {"kind": "batch", "shots": shots, "lo": lo, "hi": hi, "sizes": rng.randint(2, 10 ** 6), "nbl": 10, "so": so,
                "nt": max(20, min(nt, int(6e9 / most))), "storage": rng.choice(["f32", "f32", "bf16"]),
                "form": "factored", "f0": 10.0}
    n = math.exp(rng.uniform(math.log(36), math.log(230 if kind in ("gradient", "buffers") else 380)))
    nx, ny, nz = (max(24, int(n * rng.uniform(0.75, 1.3))) for _ in range(3))
    nbl = rng.choice([10, 10, 20])
    pts = (nx + 2 * nbl) * (ny + 2 * nbl) * (nz + 2 * nbl)
    most = {"gradient": 1.4e9, "buffers": 2.5e9, "receivers": 4e9}.get(kind, 3e9 if so > 16 or form == "expanded" else 6e9)
    return _shot(None, nx, ny, nz, nbl, so, max(20, min(nt, int(most / pts))), kind="shot" if kind == "half" else kind,
                 storage=storage, form=form, model=rng.choice(["layered", "smooth"]), f0=rng.choice([10.0, 15.0]),
                 every=rng.choice([2, 3, 5]) if kind in ("receivers", "gradient") else 0)


# ---- inputs -------------------------------------------------------------------

def _weights(so):
    """Centred second-derivative weights c_0..c_r (closed form)."""
    r, f = so // 2, math.factorial
    c = [2.0 * (-1) ** (j + 1) * f(r) ** 2 / (j * j * f(r - j) * f(r + j)) for j in range(1, r + 1)]
    return [-2.0 * math.fsum(c)] + c


def _dt(so, vmax):
    """0.9 of the leapfrog's stability limit (the Nyquist mode on every axis)."""
    c = _weights(so)
    return 0.9 * 2.0 * H / (vmax * math.sqrt(3.0 * (abs(c[0]) + 2.0 * sum(abs(x) for x in c[1:]))))


def _velocity(interior, nbl, model, gen):
    """Velocity over the domain (float64, on the device): one value, four layers along z, or a
    smooth random field of 1.5 to 4.5 km/s with a correlation length of about eight cells."""
    nx, ny, nz = interior
    r = torch.rand(4, generator=gen, dtype=torch.float64)
    if model == "constant":
        v = torch.full(interior, 1500.0 + 30.0 * float(r[0]), dtype=torch.float64, device="cuda")
    elif model == "layered":
        edge = torch.tensor([1500.0, 2500.0, 3500.0, 4500.0], dtype=torch.float64) - 60.0 * r
        v = edge.cuda()[torch.arange(nz, device="cuda") * 4 // nz].expand(nx, ny, nz)
    else:
        coarse = torch.rand([1, 1] + [n // 8 + 2 for n in interior], generator=gen, dtype=torch.float64)
        v = torch.nn.functional.interpolate(coarse.cuda(), size=interior, mode="trilinear", align_corners=True)[0, 0]
        v = 1500.0 + 3000.0 * (v - v.min()) / (v.max() - v.min())
    at = [(torch.arange(n + 2 * nbl, device="cuda") - nbl).clamp(0, n - 1) for n in interior]
    return v[at[0]][:, at[1]][:, :, at[2]].contiguous()


def _damping(m, nbl, vmax):
    """eta = m sum_a d (l_a / nbl)^2, l_a the depth in the layer, d = 3 vmax ln(1000) / (2 nbl h)."""
    s = torch.zeros_like(m)
    for axis, n in enumerate(m.shape):
        i = torch.arange(n, device=m.device, dtype=torch.float64)
        depth = torch.maximum((nbl - i).clamp(min=0), (i - (n - 1 - nbl)).clamp(min=0)) / nbl
        s = s + (3.0 * vmax * math.log(1000.0) / (2.0 * nbl * H) * depth * depth).reshape(
            [-1 if a == axis else 1 for a in range(3)])
    return m * s


def _ricker(f0, dt, nt):
    a = (math.pi * f0 * (np.arange(nt) * dt - 1.0 / f0)) ** 2
    return ((1.0 - 2.0 * a) * np.exp(-a)).astype(np.float32)


def _inputs(interior, nbl, so, nt, model, f0, seed):
    """m and eta (float32, over the domain), dt, the source's node and its wavelet."""
    gen = torch.Generator().manual_seed(int(seed))
    v = _velocity(interior, nbl, model, gen)
    vmax = float(v.max())
    m = (1.0 / (v * v)).float()
    eta = _damping(m.double(), nbl, vmax).float()
    dt = _dt(so, vmax)
    u = torch.rand(4, generator=gen, dtype=torch.float64).tolist()
    nx, ny, nz = interior
    # shallow and near the middle of the survey, as sources sit
    src = (int(nx * (0.4 + 0.2 * u[0])), int(ny * (0.4 + 0.2 * u[1])), int(nz * (0.06 + 0.1 * u[2])))
    return m, eta, dt, src, _ricker(f0 * (0.95 + 0.1 * u[3]), dt, nt)


def _interior(case):
    return (case["nx"], case["ny"], case["nz"])


def _batch_sizes(case):
    rng = np.random.default_rng(case["sizes"])
    return [tuple(int(v) for v in rng.integers(case["lo"], case["hi"] + 1, size=3)) for _ in range(case["shots"])]


def _receivers(case):
    """A grid of receivers half a cell below a plane of nodes, every `every` nodes."""
    z = min(10.5, case["nz"] - 1.5)
    x = np.arange(0.0, case["nx"] - 1, case["every"])
    y = np.arange(0.25, case["ny"] - 1, case["every"])
    return np.stack([g.reshape(-1) for g in np.meshgrid(x, y, [z], indexing="ij")], axis=1)


def _off_grid(src):
    return (src[0] + 0.375, src[1] + 0.5, src[2] + 0.25)


# ---- the calls ------------------------------------------------------------------

_STREAMS = []


def _stream():
    """The program's compute stream: its tensors and every handle's work are queued on it."""
    if not _STREAMS:
        _STREAMS.append(torch.cuda.Stream())
    return _STREAMS[0]


def _make_shot(case, m, eta, dt):
    shot = fd.Shot(_interior(case), case["so"], H, dt, case["nbl"], storage=case["storage"], form=case["form"])
    shot.set_stream(_stream().cuda_stream)
    shot.set_model_device(m.data_ptr(), eta.data_ptr())
    return shot


def prepare(case, seed):
    with torch.cuda.stream(_stream()):
        return _prepare(case, seed)


def _prepare(case, seed):
    if case["kind"] == "batch":
        batch = fd.Batch(case["so"], H, storage=case["storage"], form=case["form"], stream=_stream())
        slots = []
        for i, interior in enumerate(_batch_sizes(case)):
            m, eta, dt, src, wav = _inputs(interior, case["nbl"], case["so"], case["nt"], "smooth", case["f0"],
                                           1000003 * seed + i)
            slot = batch.add(interior, case["nbl"], dt, m.cpu().numpy(), eta.cpu().numpy())
            batch.inject(slot, *src, wav)
            slots.append(slot)
        return {"case": case, "batch": batch, "slots": slots}
    m, eta, dt, src, wav = _inputs(_interior(case), case["nbl"], case["so"], case["nt"], case["model"], case["f0"], seed)
    if case["kind"] == "buffers":
        u = [torch.zeros_like(m) for _ in range(2)]
        node = [c + case["nbl"] for c in src]
        return {"case": case, "m": m, "eta": eta, "dt": dt, "u": u, "node": node, "wavelet": torch.from_numpy(wav).cuda()}
    shot = _make_shot(case, m, eta, dt)
    state = {"case": case, "shot": shot, "m": m, "eta": eta}
    if case["kind"] == "receivers":
        shot.inject_at(*_off_grid(src), wav)
        shot.set_receivers(_receivers(case), case["nt"])
        return state
    shot.inject(*src, wav)
    if case["kind"] == "gradient":
        state["receivers"] = _receivers(case)
        state["observed"] = _observed(case, m, eta, dt, src, wav).cpu().numpy()
    return state


def _sought(m):
    """The model behind the observed data: up to 4 % slower than m at depth."""
    return (m.double() * (1.0 + 0.08 * torch.linspace(0.0, 1.0, m.shape[2], dtype=torch.float64, device=m.device))).float()


def _observed(case, m, eta, dt, src, wav):
    """The traces of the sought model (in 64 bits, rounded once): made without the library, since exact() uses them too."""
    node = tuple(c + case["nbl"] for c in src)
    at = _Sampling(tuple(m.shape), case["nbl"], _receivers(case))
    return _exact_shot(_sought(m), eta, case["so"], dt, case["nt"], wav, [(node, 1.0)], at)[2].float()


def _read(shot):
    out = [torch.empty(shot.shape, dtype=torch.float32, device="cuda") for _ in range(2)]
    for level, o in enumerate(out):
        shot.read_device(o.data_ptr(), level)
    return out


def run(state):
    with torch.cuda.stream(_stream()):
        return _run(state)


def _run(state):
    case = state["case"]
    if case["kind"] == "batch":
        batch = state["batch"]
        batch.reset()
        batch.forward(case["nt"])
        out = []
        for slot in state["slots"]:
            out.append(torch.empty(batch.shapes[slot], dtype=torch.float32, device="cuda"))
            fd.fd_batch_read_device(batch.handle, slot, out[-1].data_ptr(), 0)
        return out
    if case["kind"] == "buffers":
        u, up = state["u"]
        u.zero_()
        up.zero_()
        fd_forward_noalloc(u.data_ptr(), up.data_ptr(), state["m"].data_ptr(), state["eta"].data_ptr(), tuple(u.shape),
                           case["so"], H, state["dt"], sources=[state["node"]], d_wavelet=state["wavelet"].data_ptr(),
                           ld=case["nt"], nt=case["nt"], stream=_stream().cuda_stream,
                           want_amax=False)
        return [u, up]
    shot = state["shot"]
    if case["kind"] == "gradient":
        grad, syn, misfit = shot.fwi_gradient(state["receivers"], state["observed"])
        return {"gradient": grad, "synthetic": syn, "misfit": misfit}
    shot.reset()
    shot.forward(case["nt"])
    out = _read(shot)
    return out + [shot.traces()] if case["kind"] == "receivers" else out


# ---- work and 64-bit results ------------------------------------------------------

def work(case):
    """One pass: every time step reads u^n, u^{n-1} and the point's coefficient once and
    writes u^{n+1} once (the gradient's forward pass also writes the second time difference,
    its adjoint pass reads that and the gradient and writes the gradient), plus the damping
    coefficient in the absorbing layer. Operations: per distance five additions and one
    multiply-add per point, eight more for the update. The levels' traffic is that of steps
    run one after another; a schedule that keeps levels on the chip moves less."""
    dims = _batch_sizes(case) if case["kind"] == "batch" else [_interior(case)]
    total = [0.0, 0.0]
    for n in dims:
        pts = math.prod(a + 2 * case["nbl"] for a in n)
        layer = pts - math.prod(n)
        level = 4 if case["storage"] == "f32" else 2
        per_pt = 3 * level + 4
        steps = case["nt"]
        passes = [per_pt + 4, per_pt + 12] if case["kind"] == "gradient" else [per_pt]
        for b in passes:
            total[0] += steps * (pts * b + 4.0 * layer)
            total[1] += steps * pts * (3.5 * case["so"] + 8.0)
    return {"bytes": total[0], "flops": total[1]}


class _Steps:
    """The scheme in 64 bits: r0 u+ = dt^2 (L u + q) + m (2u - u-) + dt/2 eta u-, r0 = m + dt/2 eta."""

    def __init__(self, m, eta, so, dt):
        self.r, self.c, self.dt = so // 2, [w / (H * H) for w in _weights(so)], dt
        m, e = m.double(), 0.5 * dt * eta.double()
        inv = 1.0 / (m + e)
        self.w, self.a, self.b = dt * dt * inv, 2.0 * m * inv, (e - m) * inv
        self.shape, self.lap = tuple(m.shape), torch.empty_like(m)

    def field(self):
        """A field with its zero halo, and the view of the domain in it."""
        p = torch.zeros([n + 2 * self.r for n in self.shape], dtype=torch.float64, device=self.w.device)
        return p, self._at(p, 0, 0)

    def _at(self, p, axis, shift):
        r = self.r
        return p[tuple(slice(r + (shift if a == axis else 0), r + n + (shift if a == axis else 0))
                       for a, n in enumerate(self.shape))]

    def step(self, u, up, sources=()):
        """u^{n+1} over u^{n-1} (both from field()); sources: (node, value)."""
        lap = torch.mul(u[1], 3.0 * self.c[0], out=self.lap)
        for j in range(1, self.r + 1):
            for axis in range(3):
                for s in (-j, j):
                    lap.add_(self._at(u[0], axis, s), alpha=self.c[j])
        up[1].mul_(self.b).addcmul_(self.a, u[1]).addcmul_(self.w, lap)
        for node, value in sources:
            up[1][node] += self.w[node] * value


def _corners(shape, point):
    """(node, trilinear weight) of the eight corners of the cell around a point."""
    lo = [min(int(math.floor(t)), n - 2) for t, n in zip(point, shape)]
    f = [t - i for t, i in zip(point, lo)]
    out = []
    for c in range(8):
        d = (c >> 2, (c >> 1) & 1, c & 1)
        w = math.prod(f[a] if d[a] else 1.0 - f[a] for a in range(3))
        if w > 0.0:
            out.append((tuple(lo[a] + d[a] for a in range(3)), w))
    return out


class _Sampling:
    """Trilinear sampling at the receivers and its transpose."""

    def __init__(self, shape, nbl, points):
        t = torch.from_numpy(points + nbl).cuda()
        n = torch.tensor(shape, device="cuda")
        lo = torch.minimum(t.floor().long(), n - 2)
        f = t - lo
        self.shape, self.off, self.w = shape, [], []
        for c in range(8):
            d = torch.tensor([c >> 2, (c >> 1) & 1, c & 1], device="cuda")
            i = lo + d
            self.off.append((i[:, 0] * shape[1] + i[:, 1]) * shape[2] + i[:, 2])
            self.w.append(torch.where(d.bool(), f, 1.0 - f).prod(dim=1))

    def sample(self, u):
        flat = u.reshape(-1) if u.is_contiguous() else u.contiguous().reshape(-1)
        return sum(w * flat[o] for o, w in zip(self.off, self.w))

    def spread(self, values):
        out = torch.zeros(math.prod(self.shape), dtype=torch.float64, device="cuda")
        for o, w in zip(self.off, self.w):
            out.index_add_(0, o, w * values)
        return out.reshape(self.shape)


def _exact_shot(m, eta, so, dt, nt, wav, nodes, sampling=None, keep=None):
    """(u^nt, u^{nt-1}, traces [n, nt]) in 64 bits; nodes: (node, factor) of the source. `keep`
    collects the second time differences of the levels."""
    s = _Steps(m, eta, so, dt)
    u, up, traces = s.field(), s.field(), []
    for n in range(nt):
        q = float(wav[n])
        last = up[1].clone() if keep is not None else None
        s.step(u, up, [(node, f * q) for node, f in nodes])
        if keep is not None:
            keep.append(last.add_(up[1]).sub_(u[1], alpha=2.0))
        u, up = up, u
        if sampling is not None:
            traces.append(sampling.sample(u[1]))
    return u[1], up[1], torch.stack(traces, dim=1) if traces else None


def exact(case, seed):
    so, nt, nbl = case["so"], case["nt"], case["nbl"]
    if case["kind"] == "batch":
        out = []
        for i, interior in enumerate(_batch_sizes(case)):
            m, eta, dt, src, wav = _inputs(interior, nbl, so, nt, "smooth", case["f0"], 1000003 * seed + i)
            out.append(_exact_shot(m, eta, so, dt, nt, wav, [(tuple(c + nbl for c in src), 1.0)])[0].clone())
        return out
    m, eta, dt, src, wav = _inputs(_interior(case), nbl, so, nt, case["model"], case["f0"], seed)
    nodes = [(tuple(c + nbl for c in src), 1.0)]
    if case["kind"] == "shot":
        return list(_exact_shot(m, eta, so, dt, nt, wav, nodes)[:2])
    if case["kind"] == "buffers":
        new, old, _ = _exact_shot(m, eta, so, dt, nt, wav, nodes)
        return [new, old] if nt % 2 == 0 else [old, new]
    receivers = _Sampling(tuple(m.shape), nbl, _receivers(case))
    if case["kind"] == "receivers":
        nodes = _corners(m.shape, [c + nbl for c in _off_grid(src)])
        new, old, traces = _exact_shot(m, eta, so, dt, nt, wav, nodes, receivers)
        return [new, old, traces]
    # the gradient: the time-reversed system driven by the residuals
    observed = _observed(case, m, eta, dt, src, wav).double()
    diffs = []
    _, _, syn = _exact_shot(m, eta, so, dt, nt, wav, nodes, receivers, keep=diffs)
    resid = syn - observed
    s = _Steps(m, eta, so, dt)
    w, wp, grad = s.field(), s.field(), torch.zeros_like(s.w)
    for n in reversed(range(nt)):
        s.step(w, wp)
        wp[1].addcmul_(s.w, receivers.spread(resid[:, n]), value=1.0 / (dt * dt))
        w, wp = wp, w
        grad.addcmul_(w[1], diffs.pop(), value=-1.0)
    return {"gradient": grad, "synthetic": syn, "misfit": 0.5 * resid.square().sum()}
