"""The work that users of this package have it do, as measurable cases.

Every case runs through the public entry points of ``appga.py`` (the C ABI) on a
parallel-beam scanner geometry: a system matrix handle, made once per scanner, and
synthetic Poisson sinograms of random-ellipse phantoms.  The kinds:

  steps    the single hot-path calls: forward projection and ratio, back-projection,
           SHOITV gradient, pixel update, objective
  recon    appga_reconstruct, one slice on the device
  host     appga_reconstruct_host, one slice in pinned host buffers
  batched  appga_reconstruct_batched, K slices that share the matrix
  volume   appga_reconstruct_volume, a stack of slices with the 3-D regulariser
  afppa    appga_afppa_reconstruct, the non-smooth model
  serve    a Server: a burst of requests of mixed image sizes from host arrays, drained

The scanner's matrix (Siddon ray lengths) is built here on the GPU because states are made
often.  A program keeps one handle per scanner and passes many slices through it, so handles
are kept per geometry and shared by all states; inputs depend on the seed alone.
Small images run with the step size beta = 0.1: at 1 the EM-preconditioned map amplifies
rounding there, and two correct FP32 runs drift apart.
"""
import functools
import math

import numpy as np
import torch

from paper_2409_13344_gb300 import appga

KAPPA = 1e-3  # floor of the Poisson ratio's denominator, in units of gamma
LAM1, LAM2, EPS, STEP_EPS = 0.1, 0.05, 1e-3, 0.02
OMEGA, GN_A, GN_B = 0.5, 0.125, 1.0


def _case(name, kind, n, angles, bins, maps, **more):
    return {"name": name, "kind": kind, "n": n, "angles": angles, "bins": bins, "maps": maps,
            "slices": 1, "counts": 1e6, "track": False, "tol": 0.0, "bf16": False, "beta": 1.0,
            "momentum": "gn", "freeze": -1, **more}


def listed():
    return [
        # the smallest image, of quick looks and tests: a launch-bound loop
        _case("recon_64", "recon", 64, 90, 95, 100, counts=1e5, beta=0.1),
        # the ordinary slice, with the objective evaluated every iteration
        _case("recon_256", "recon", 256, 180, 367, 100, track=True, beta=0.3),
        # the same slice from and to pinned host buffers in one short call
        _case("host_256", "host", 256, 180, 367, 20, track=True),
        # odd sizes (no quarter-turn symmetry), BF16 values of A, Nesterov momentum, a
        # preconditioner frozen after early iterations
        _case("recon_odd_201_bf16", "recon", 201, 141, 285, 30, bf16=True, momentum="nesterov",
              freeze=10, beta=0.1),
        # a large slice that runs until its objective settles (the tolerance is polled)
        _case("recon_400_tol", "recon", 400, 288, 575, 40, counts=5e6, tol=1e-12),
        # an algorithm of the user's own over the single calls
        _case("steps_256", "steps", 256, 180, 367, 1),
        # a few dynamic frames of a small image
        _case("batched_5x128", "batched", 128, 90, 185, 50, slices=5, counts=3e5,
              beta=0.1),
        # many slices of one scanner, counts over two decades, the objective tracked
        _case("batched_64x256", "batched", 256, 180, 367, 20, slices=64, track=True,
              beta=0.3),
        # the largest batch: 120 frames of a 512 x 512 image, BF16 values of A
        _case("batched_120x512_bf16", "batched", 512, 360, 731, 5, slices=120, bf16=True),
        # a stack of slices with the 3-D regulariser
        _case("volume_64x256", "volume", 256, 180, 367, 10, slices=64, counts=6.4e7, track=True),
        # the non-smooth model
        _case("afppa_256", "afppa", 256, 180, 367, 40, beta=0.3, counts=1e6),
        # a burst of requests of three image sizes
        _case("serve_mix", "serve", 256, 180, 367, 60, slices=24, beta=0.1),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["steps", "recon", "recon", "host", "batched", "batched", "volume", "afppa"])
    n = log(40, 400 if kind != "steps" else 512)
    angles = max(8, int(n * rng.uniform(0.5, 0.9)))
    if rng.random() < 0.6:  # most scanners have the quarter-turn symmetry
        n += n % 2
        angles += angles % 2
    bins = int(n * math.sqrt(2.0)) + rng.choice([1, 2, 3, 5])
    case = _case("", kind, n, angles, bins, log(10, 120), counts=float(log(200, 2000)) * n)
    case["bf16"] = kind != "steps" and rng.random() < 0.3
    case["beta"] = 0.1 if n < 200 else 0.3
    if kind in ("batched", "volume"):
        case["slices"] = log(1, 128)
        # no dearer than the largest listed case
        case["maps"] = max(2, min(case["maps"], int(2.5e10 / (_entries(case) * max(32, case["slices"])))))
    if kind == "volume":
        case["counts"] *= case["slices"]
    if kind in ("recon", "host"):
        case["momentum"] = rng.choice(["gn", "gn", "nesterov", "none"])
        case["freeze"] = rng.choice([-1, -1, 5])
        case["tol"] = rng.choice([0.0, 0.0, 1e-12])
    if kind == "steps":
        case["maps"] = 1
    if kind == "afppa":
        case["beta"] = 0.1
        case["maps"] = min(case["maps"], 40)
    case["track"] = kind not in ("steps", "afppa") and rng.random() < 0.5
    del case["name"]
    return case


def _entries(case):
    """Entries of A: a pixel meets (|cos| + |sin|) rays of unit spacing per angle."""
    return case["n"] ** 2 * case["angles"] * 4.0 / math.pi


SERVED = ((128, 90, 185), (256, 180, 367), (400, 288, 575))


def _requests(case):
    """(geometry, maps) of the requests of a serve case."""
    return [(SERVED[i % 3], case["maps"] // 2 + (7 * i) % case["maps"])
            for i in range(case["slices"])]


def work(case):
    """Per map A is read (FP32 value and int32 column, as the caller holds it; BF16: two bytes
    of value) at least once for all slices, and every slice's sinogram, background, image and
    previous image once; two multiply-adds per entry and slice."""
    entry = 6 if case["bf16"] else 8
    if case["kind"] == "serve":
        by, fl = 0.0, 0.0
        for geom in SERVED:
            maps = [k for q, k in _requests(case) if q == geom]
            one = dict(case, n=geom[0], angles=geom[1], bins=geom[2])
            rows, pixels = geom[1] * geom[2], geom[0] ** 2
            by += entry * _entries(one) * max(maps) + sum(maps) * (8 * rows + 12 * pixels)
            fl += 4 * _entries(one) * sum(maps)
        return {"bytes": by, "flops": fl}
    rows, pixels = case["angles"] * case["bins"], case["n"] ** 2
    per_slice = 8 * rows + 12 * pixels
    if case["kind"] == "afppa":
        per_slice += 6 * 12 * pixels  # six dual fields: two read, one written
    if case["kind"] == "steps":  # four projections; sinogram vectors and images of each call
        return {"bytes": 4 * entry * _entries(case) + 44 * rows + 40 * pixels,
                "flops": 8 * _entries(case)}
    return {"bytes": case["maps"] * (entry * _entries(case) + case["slices"] * per_slice),
            "flops": case["maps"] * case["slices"] * 4 * _entries(case)}


# ------------------------------------------------------------------------- inputs


def _dev():
    return torch.device("cuda", torch.cuda.current_device())


@functools.lru_cache(maxsize=None)
def _context():
    return appga.Context(torch.cuda.current_device())


@functools.lru_cache(maxsize=4)
def _siddon(n, angles, bins):
    """CSR (row starts int32, columns int32, FP32 values) of the ray lengths in unit pixels, on
    the GPU.  With an even number of angles the second half is the first turned by a quarter
    (bin b to bins-1-b, pixel (r, c) to (n-1-c, r)), so the scanner's symmetry holds bit for bit."""
    dev, h = _dev(), n / 2.0
    s = torch.arange(bins, dtype=torch.float64, device=dev) - (bins - 1) / 2.0
    edges = torch.arange(n + 1, dtype=torch.float64, device=dev) - h
    half = angles // 2 if angles % 2 == 0 else angles
    keys, vals = [], []
    for a in range(half):
        c, q = (0.0 if abs(v) < 1e-12 else v for v in (math.cos(a * math.pi / angles), math.sin(a * math.pi / angles)))
        lo = torch.full((bins,), -math.inf, dtype=torch.float64, device=dev)
        hi, parts = -lo, []
        for start, slope in ((-s * q, c), (s * c, q)):  # x, then y, along the ray
            if slope != 0.0:
                t = (edges[None, :] - start[:, None]) / slope
                lo, hi = torch.maximum(lo, t.amin(1)), torch.minimum(hi, t.amax(1))
                parts.append(t)
            else:
                lo = torch.where((start >= -h) & (start < h), lo, math.inf)
        ray = torch.nonzero(hi > lo + 1e-12).flatten()
        lo, hi = lo[ray, None], hi[ray, None]
        t = torch.cat([lo, hi] + [p[ray] for p in parts], 1)
        t = torch.minimum(torch.maximum(t, lo), hi).sort(1).values
        length, mid = t.diff(dim=1), 0.5 * (t[:, 1:] + t[:, :-1])
        col = torch.floor((-s * q)[ray, None] + mid * c + h).long().clamp(0, n - 1)
        row = torch.floor((s * c)[ray, None] + mid * q + h).long().clamp(0, n - 1)
        keep = length > 1e-9
        b, col, row = ray[:, None].expand_as(length)[keep], col[keep], row[keep]
        length = length[keep]
        keys.append((a * bins + b) * (n * n) + row * n + col)
        vals.append(length)
        if half < angles:
            keys.append(((a + half) * bins + bins - 1 - b) * (n * n) + (n - 1 - col) * n + row)
            vals.append(length)
    key, order = torch.cat(keys).sort()
    val = torch.cat(vals)[order].float()
    row = torch.div(key, n * n, rounding_mode="floor")
    ptr = torch.zeros(angles * bins + 1, dtype=torch.int64, device=dev)
    ptr[1:] = torch.bincount(row, minlength=angles * bins).cumsum(0)
    return ptr.int(), (key - row * (n * n)).int(), val


class _Csr:
    """What appga.Matrix takes of a SciPy CSR."""

    def __init__(self, shape, ptr, col, val):
        self.shape = shape
        self.indptr, self.indices, self.data = (x.cpu().numpy() for x in (ptr, col, val))


@functools.lru_cache(maxsize=None)
def _matrix(n, angles, bins, bf16):
    csr = _Csr((angles * bins, n * n), *_siddon(n, angles, bins))
    return appga.Matrix(_context(), csr, n, angles, bf16=bf16)


def _ellipses(n, slices, stack, rng):
    """The parts of a phantom, as (activity, x, y, half axes, turn), each [slices, 1] FP64: a body
    of activity 1 and eight ellipses of activity 0 to 3 added to it.  With `stack` the slices cut
    one set of ellipsoids, else each slice has its own."""
    radius, each = n / 2.0, (1 if stack else slices, 1)
    z = np.arange(slices)[:, None] + 0.5 - slices / 2.0
    parts = []
    for k in range(9):
        if k == 0:
            act, x, y = np.ones(each), np.zeros(each), np.zeros(each)
            ax, ay = rng.uniform(0.8, 0.95, each) * radius, rng.uniform(0.6, 0.85, each) * radius
            cz, az = 0.0, rng.uniform(0.6, 1.0) * slices + 1.0
        else:
            r, turn = 0.5 * radius * np.sqrt(rng.uniform(size=each)), rng.uniform(0, 2 * math.pi, each)
            act, x, y = rng.uniform(0.0, 3.0, each), r * np.cos(turn), r * np.sin(turn)
            ax, ay = rng.uniform(0.05, 0.3, each) * radius, rng.uniform(0.05, 0.3, each) * radius
            cz, az = rng.uniform(-0.4, 0.4) * slices, rng.uniform(0.1, 0.5) * slices + 1.0
        cut = np.sqrt(np.clip(1.0 - ((z - cz) / az) ** 2, 0.0, None)) if stack else 1.0
        part = act, x, y, ax * cut + 1e-6, ay * cut + 1e-6, rng.uniform(0, math.pi, each)
        parts.append([torch.from_numpy(np.broadcast_to(v, (slices, 1)).copy()).to(_dev()) for v in part])
    return parts


def _image(parts, n):
    at = torch.arange(n, dtype=torch.float64, device=_dev()) + 0.5 - n / 2.0
    col, row = at.repeat(n)[None], at.repeat_interleave(n)[None]
    out = 0.0
    for act, x, y, ax, ay, turn in parts:
        u = (col - x) * torch.cos(turn) + (row - y) * torch.sin(turn)
        v = (row - y) * torch.cos(turn) - (col - x) * torch.sin(turn)
        out = out + act * ((u / ax) ** 2 + (v / ay) ** 2 <= 1.0)
    return out.float()


def _projection(parts, angles, bins):
    """The phantom's line integrals, [slices, rows] FP64, in closed form."""
    phi = (torch.arange(angles, dtype=torch.float64, device=_dev()) * (math.pi / angles)).repeat_interleave(bins)[None]
    s = (torch.arange(bins, dtype=torch.float64, device=_dev()) - (bins - 1) / 2.0).repeat(angles)[None]
    out = 0.0
    for act, x, y, ax, ay, turn in parts:
        wide = (ax * torch.sin(turn - phi)) ** 2 + (ay * torch.cos(turn - phi)) ** 2
        off = s - (y * torch.cos(phi) - x * torch.sin(phi))
        out = out + act * 2 * ax * ay * (wide - off * off).clamp_min(0.0).sqrt() / wide
    return out


def _sinograms(n, angles, bins, slices, counts, stack, seed):
    """Counts g and background gamma, [slices, rows] FP32: Poisson of the phantom's line integrals
    plus gamma, a tenth of their mean.  Slices of their own scale over two decades around `counts`."""
    rng = np.random.default_rng(seed)
    mean = _projection(_ellipses(n, slices, stack, rng), angles, bins)
    if stack or slices == 1:
        mean = mean * (counts / (1.1 * mean.sum()))
        gamma = (0.1 * mean.mean()).expand(mean.shape)
    else:
        each = torch.from_numpy(counts * 10.0 ** rng.uniform(-1, 1, (slices, 1))).to(_dev())
        mean = mean * (each / (1.1 * mean.sum(1, keepdim=True)))
        gamma = (0.1 * mean.mean(1, keepdim=True)).expand(mean.shape)
    gen = torch.Generator(device=_dev()).manual_seed(seed)
    return torch.poisson((mean + gamma).float(), generator=gen), gamma.float().contiguous()


def _params(case):
    momentum = {"gn": appga.APPGA_MOMENTUM_GN, "none": appga.APPGA_MOMENTUM_NONE,
                "nesterov": appga.APPGA_MOMENTUM_NESTEROV}[case["momentum"]]
    return appga.default_params(
        lambda1=LAM1, lambda2=LAM2, eps=STEP_EPS if case["kind"] == "steps" else EPS, omega=OMEGA,
        a=GN_A, b=GN_B, beta=case["beta"], max_iters=case["maps"], rel_obj_tol=case["tol"],
        track_objective=int(case["track"]), momentum=momentum, precond_freeze_iter=case["freeze"],
        a_precision=appga.APPGA_PREC_BF16 if case["bf16"] else appga.APPGA_PREC_FP32)


def _serve_inputs(case, seed):
    """(g, gamma) of each request, as host arrays."""
    by_geometry = {}
    for k, geom in enumerate(SERVED):
        count = sum(q == geom for q, _ in _requests(case))
        g, gamma = _sinograms(*geom, count, case["counts"], False, seed * 3 + k)
        by_geometry[geom] = iter(list(zip(g.cpu().numpy(), gamma.cpu().numpy())))
    return [next(by_geometry[geom]) for geom, _ in _requests(case)]


def prepare(case, seed):
    state = {"case": case, "params": _params(case)}
    if case["kind"] == "serve":
        server = appga.Server(_context())
        mats = {geom: _matrix(*geom, case["bf16"]) for geom in SERVED}
        ids = {geom: server.add_geometry(mats[geom]) for geom in SERVED}
        state["server"] = server
        state["requests"] = []
        for (geom, maps), (g, gamma) in zip(_requests(case), _serve_inputs(case, seed)):
            state["requests"].append((ids[geom], g, gamma, _params(dict(case, maps=maps))))
        return state
    geom = case["n"], case["angles"], case["bins"]
    state["mat"] = _matrix(*geom, case["bf16"])
    g, gamma = _sinograms(*geom, case["slices"], case["counts"], case["kind"] == "volume", seed)
    if case["kind"] in ("recon", "host", "steps", "afppa"):
        g, gamma = g[0], gamma[0]
    if case["kind"] == "host":
        g, gamma = g.cpu().pin_memory(), gamma.cpu().pin_memory()
        state["f"] = torch.empty(case["n"] ** 2, dtype=torch.float32).pin_memory()
    if case["kind"] == "steps":
        state["f"] = _step_image(case, seed)
    state["g"], state["gamma"] = g, gamma
    torch.cuda.synchronize()
    return state


def _step_image(case, seed):
    """A current and a previous image such as an iteration holds."""
    f = _image(_ellipses(case["n"], 1, False, np.random.default_rng(seed + 1)), case["n"])[0]
    f = f * (case["counts"] / (case["n"] ** 2 * case["angles"]))
    gen = torch.Generator(device=_dev()).manual_seed(seed + 1)
    noise = torch.rand(2, f.numel(), device=_dev(), generator=gen)
    level = 0.1 * case["counts"] / (case["n"] ** 2 * case["angles"])
    return f + level * noise[0], f + level * noise[1]


THETA = 0.4  # momentum of the single pixel update


def run(state):
    case, p, kind = state["case"], state["params"], state["case"]["kind"]
    if kind == "serve":
        server = state["server"]
        ids = [server.submit(*request) for request in state["requests"]]
        while server.step():
            pass
        return [server.collect(i)[0] for i in ids]
    mat, g, gamma = state["mat"], state["g"], state["gamma"]
    ctx, dev = mat.ctx.handle, _dev()
    if kind == "recon":
        f, stats = appga.reconstruct(mat, g, gamma, p)
        return [f, stats.iters] + ([stats.phi] if case["track"] else [])
    if kind == "host":
        stats = appga.appga_reconstruct_host(ctx, mat.handle, g, gamma, None, p, state["f"])
        return [state["f"], stats.iters] + ([stats.phi] if case["track"] else [])
    if kind == "batched":
        f = torch.empty(case["slices"], mat.d, device=dev)
        stats = appga.appga_reconstruct_batched(ctx, mat.handle, case["slices"], g, gamma, None, p, f)
        return [f, np.array([s.iters for s in stats])] + (
            [np.array([s.phi for s in stats], np.float32)] if case["track"] else [])
    if kind == "volume":
        f = torch.empty(case["slices"], mat.d, device=dev)
        stats = appga.appga_reconstruct_volume(ctx, mat.handle, case["slices"], g, gamma, None, p, f)
        return [f, stats.iters] + ([stats.phi] if case["track"] else [])
    if kind == "afppa":
        f, b, c = (torch.empty(k, mat.d, device=dev) for k in (1, 2, 4))
        appga.appga_afppa_reconstruct(ctx, mat.handle, g, gamma, None, p, f, b, c)
        return [f, b, c]
    f, before = state["f"]
    y = torch.empty(mat.m, dtype=torch.float64, device=dev)
    w = torch.empty(mat.m, device=dev)
    data = torch.empty(1, dtype=torch.float64, device=dev)
    back, grad, after = (torch.empty(mat.d, device=dev) for _ in range(3))
    appga.appga_forward_ratio(ctx, mat.handle, f, g, gamma, y, w, data)
    appga.appga_backproject(ctx, mat.handle, w, back)
    appga.appga_shoitv_grad(ctx, case["n"], f, p.lambda1, p.lambda2, p.eps, grad)
    appga.appga_pixel_update(ctx, mat.handle, before, f, w, THETA, p, after)
    phi = appga.appga_objective(ctx, mat.handle, after, g, gamma, p)
    return [y, w, data, back, grad, after, phi]


# ------------------------------------------------------------------------- 64-bit values


def _d(x, axis):
    """Backward difference along `axis` with a zero first row."""
    return torch.cat([torch.zeros_like(x.narrow(axis, 0, 1)), x.diff(dim=axis)], axis)


def _dt(x, axis):
    """Its transpose."""
    x = torch.cat([torch.zeros_like(x.narrow(axis, 0, 1)), x.narrow(axis, 1, x.shape[axis] - 1)], axis)
    return x - torch.cat([x.narrow(axis, 1, x.shape[axis] - 1), torch.zeros_like(x.narrow(axis, 0, 1))], axis)


Z, R, C = 0, 1, 2
FIRST = [[(_d, C)], [(_d, R)]]
SECOND = [[(_dt, C), (_d, C)], [(_dt, R), (_d, C)], [(_dt, R), (_d, R)], [(_d, R), (_dt, C)]]
FIRST_Z = [[(_d, Z)]]
SECOND_Z = [[(_dt, Z), (_d, Z)], [(_dt, Z), (_d, C)], [(_d, Z), (_dt, C)], [(_dt, Z), (_d, R)],
            [(_d, Z), (_dt, R)]]


def _fields(x, group):
    """A group's difference fields of x; second-order ones carry a minus sign."""
    out = []
    for ops in group:
        u = x
        for op, axis in reversed(ops):
            u = op(u, axis)
        out.append(u if len(ops) == 1 else -u)
    return torch.stack(out)


def _adjoint(v, group):
    total = 0.0
    for field, ops in zip(v, group):
        for op, axis in ops:
            field = (_dt if op is _d else _d)(field, axis)
        total = total + (field if len(ops) == 1 else -field)
    return total


def _groups(volume):
    return ((LAM1, FIRST + FIRST_Z if volume else FIRST), (LAM2, SECOND + SECOND_Z if volume else SECOND))


def _reg_grad(x, eps, volume):
    total = 0.0
    for lam, group in _groups(volume):
        u = _fields(x, group)
        total = total + _adjoint(lam * u / u.norm(dim=0).clamp_min(eps), group)
    return total


def _reg_value(x, eps, volume):
    """The regulariser of each slice of x."""
    total = 0.0
    for lam, group in _groups(volume):
        v = _fields(x, group).norm(dim=0)
        total = total + lam * torch.where(v > eps, v - eps / 2, v * v / (2 * eps)).sum((1, 2))
    return total


class _Problem:
    """One geometry's A and A^T in 64 bits; images are [slices, n, n], sinograms [slices, rows]."""

    def __init__(self, n, angles, bins, bf16):
        self.n, self.angles = n, angles
        ptr, col, val = _siddon(n, angles, bins)
        val = (val.bfloat16() if bf16 else val).double()
        self.a = torch.sparse_csr_tensor(ptr, col, val, size=(angles * bins, n * n))
        row = torch.repeat_interleave(torch.arange(angles * bins, device=_dev()), ptr.diff())
        order = col.sort(stable=True).indices
        tptr = torch.zeros(n * n + 1, dtype=torch.int64, device=_dev())
        tptr[1:] = torch.bincount(col, minlength=n * n).cumsum(0)
        self.at = torch.sparse_csr_tensor(tptr.int(), row[order].int(), val[order],
                                          size=(n * n, angles * bins))
        lam = self.back(torch.ones(1, angles * bins, dtype=torch.float64, device=_dev()))
        self.lam = torch.where(lam > 0, lam, 1.0)

    def project(self, f):
        return (self.a @ f.reshape(f.shape[0], -1).T).T

    def back(self, w):
        return (self.at @ w.T).T.reshape(-1, self.n, self.n)

    def initial(self, g, gamma):
        at = torch.arange(self.n, dtype=torch.float64, device=_dev()) + 0.5 - self.n / 2.0
        disk = (at[:, None] ** 2 + at[None, :] ** 2 <= self.n ** 2 / 4.0).double()
        return ((g - gamma).sum(1) / (disk.sum() * self.angles))[:, None, None] * disk

    def weights(self, f, g, gamma):
        return 1.0 - g / torch.maximum(self.project(f) + gamma, KAPPA * gamma)

    def data(self, f, g, gamma):
        y = self.project(f)
        return (y - g * torch.log(y + gamma)).sum(1)


def _thetas(case, maps):
    out, t = [], 1.0
    for k in range(1, maps + 1):
        if case["momentum"] == "nesterov":
            new = (1.0 + math.sqrt(1.0 + 4.0 * t * t)) / 2.0
            out.append((t - 1.0) / new)
            t = new
        elif case["momentum"] == "gn":
            out.append((GN_A * (k - 1) ** OMEGA + GN_B - 1.0) / (GN_A * k ** OMEGA + GN_B))
        else:
            out.append(0.0)
    return out


def _solve(problem, case, g, gamma, maps):
    """The image after `maps` APPGA maps from the initial image."""
    volume = case["kind"] == "volume"
    f = before = problem.initial(g, gamma)
    frozen = None
    for k, theta in enumerate(_thetas(case, maps), 1):
        ahead = f + theta * (f - before)
        p = case["beta"] * f / problem.lam if frozen is None else frozen
        if k == case["freeze"]:
            frozen = p
        grad = problem.back(problem.weights(ahead, g, gamma)) + _reg_grad(ahead, EPS, volume)
        f, before = (ahead - p * grad).clamp_min(0.0), f
    return f


def _solve_afppa(problem, case, g, gamma):
    f = before = problem.initial(g, gamma)
    duals = [(lam, group, torch.zeros(len(group), *f.shape, dtype=torch.float64, device=f.device))
             for lam, group in _groups(False)]
    old = [v for _, _, v in duals]
    for theta in _thetas(case, case["maps"]):
        ahead = f + theta * (f - before)
        tilde = [v + theta * (v - o) for (_, _, v), o in zip(duals, old)]
        p = case["beta"] * f / problem.lam
        grad = problem.back(problem.weights(ahead, g, gamma))
        grad = grad + sum(_adjoint(t, group) for (_, group, _), t in zip(duals, tilde))
        f, before = (ahead - p * grad).clamp_min(0.0), f
        u, new = 2.0 * f - ahead, []
        for (lam, group, _), t, norm in zip(duals, tilde, (8, 64)):
            z = t + _fields(u, group) / (2 * norm * p.max())
            new.append((lam, group, z / (z.norm(dim=0) / lam).clamp_min(1.0)))
        old, duals = [v for _, _, v in duals], new
    return [f.reshape(1, -1)] + [v.reshape(len(group), -1) for _, group, v in duals]


def exact(case, seed):
    if case["kind"] == "serve":
        problems = {geom: _Problem(*geom, case["bf16"]) for geom in SERVED}
        out = []
        for (geom, maps), (g, gamma) in zip(_requests(case), _serve_inputs(case, seed)):
            g, gamma = (torch.from_numpy(x).to(_dev()).double()[None] for x in (g, gamma))
            out.append(_solve(problems[geom], case, g, gamma, maps).reshape(-1))
        return out
    geom = case["n"], case["angles"], case["bins"]
    problem, volume = _Problem(*geom, case["bf16"]), case["kind"] == "volume"
    g, gamma = _sinograms(*geom, case["slices"], case["counts"], volume, seed)
    g, gamma = g.double(), gamma.double()
    if case["kind"] == "afppa":
        return _solve_afppa(problem, case, g, gamma)
    if case["kind"] == "steps":
        f, before = (x.double().reshape(1, case["n"], case["n"]) for x in _step_image(case, seed))
        y, w = problem.project(f), problem.weights(f, g, gamma)
        ahead = f + THETA * (f - before)
        grad = problem.back(w) + _reg_grad(ahead, STEP_EPS, False)
        after = (ahead - case["beta"] * f / problem.lam * grad).clamp_min(0.0)
        phi = problem.data(after, g, gamma) + _reg_value(after, STEP_EPS, False)
        return [y[0], w[0], problem.data(f, g, gamma), problem.back(w).reshape(-1),
                _reg_grad(f, STEP_EPS, False).reshape(-1), after.reshape(-1), float(phi)]
    f = _solve(problem, case, g, gamma, case["maps"])
    phi = problem.data(f, g, gamma) + _reg_value(f, EPS, volume)
    flat = f.reshape(case["slices"], -1)
    if case["kind"] == "batched":
        return [flat, None] + ([phi] if case["track"] else [])
    if volume:
        return [flat, None] + ([float(phi.sum())] if case["track"] else [])
    return [flat[0], None] + ([float(phi)] if case["track"] else [])
