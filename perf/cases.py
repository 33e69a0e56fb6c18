"""The work that users of this library have it do, as measurable cases.

Each case is one call (or the short run of calls a program makes in one go)
through the Python binding of liblrccs, on seeded synthetic inputs shaped like
the dynamic-MRI scans the library serves: an ellipse phantom whose inner
ellipses deform over the frames, smooth coil maps of unit sum of squares,
variable-density Cartesian line masks or golden-angle pseudo-radial masks
redrawn for every frame, and 1% complex Gaussian noise.

  solve   : a whole reconstruction: lrccs_init, lrccs_iterate, lrccs_get_images
  iterate : a solve resumed from a given subspace (lrccs_set_subspace,
            lrccs_iterate, then the images and the subspace)
  track   : one later mini-batch of subspace tracking (lrccs_track_minibatch)
            from the subspace and step size handed over by the first one
  online  : frames of online tracking with a fixed subspace and mean
            (lrccs_online_frames)
  mean    : the mean step with its residual measurements (lrccs_mean_step)
  mec1/2  : model-error correction after a solve (lrccs_mec1, lrccs_mec2)
  batch   : independent slices of uneven sizes as one launch
            (lrccs_batch_iterate), resumed from given subspaces

Inputs live on the GPU; `exact` restates each path in FP64 torch.
"""
import math

import numpy as np
import torch

from paper_2212_09664_gb300 import lrccs

FIRST = 32        # frames of the first mini-batch (tracking and online cases)
SIDES = (64, 96, 128, 160, 192, 224, 256)
BATCH_SIDES = (128, 160, 192, 224, 256)


def _case(name, op, ny, nx, q, coils, rank, mask, accel, iters, precision="fp32", data="phantom", slices=1):
    return dict(name=name, op=op, ny=ny, nx=nx, q=q, coils=coils, rank=rank, mask=mask, accel=accel, iters=iters,
                precision=precision, data=data, slices=slices)


def listed():
    return [
        # one new frame of an online scan, reconstructed as it arrives: the smallest call, latency only
        _case("online_lines128_q1", "online", 128, 128, 1, 12, 6, "lines", 8.0, 3),
        # the serving loop's unit of work: a mini-batch of 8 frames, 5 iterations, warm start
        _case("track_lines192_q8", "track", 192, 192, 8, 16, 10, "lines", 8.0, 5),
        # the same for a pseudo-radial acquisition with uneven sizes
        _case("track_radial224_q8", "track", 224, 224, 8, 18, 13, "radial", 9.5, 5),
        # single coil, exactly low rank, noiseless: the smallest whole solve
        _case("solve_lines64_q32", "solve", 64, 64, 32, 1, 4, "lines", 4.0, 50, data="lowrank"),
        # the cardiac-shaped scan: an ordinary whole solve
        _case("solve_lines192_q48", "solve", 192, 192, 48, 12, 10, "lines", 8.0, 50),
        # the large pseudo-radial scan (16 spokes): a whole solve on general masks
        _case("solve_radial256_q64", "solve", 256, 256, 64, 20, 12, "radial", 16.0, 50),
        # the largest Cartesian scan of the range, rows too long for one block's shared memory
        _case("iterate_lines256_q96", "iterate", 256, 256, 96, 32, 14, "lines", 6.0, 10),
        # the tensor-core form of the forward transform on the cardiac-shaped scan
        _case("iterate_bf16x3_192_q48", "iterate", 192, 192, 48, 12, 10, "lines", 8.0, 10, precision="bf16x3"),
        # the mean image of the cardiac-shaped scan and its residual measurements
        _case("mean_lines192_q48", "mean", 192, 192, 48, 12, 1, "lines", 8.0, 10),
        # unstructured model error of a mid-sized pseudo-radial scan, odd frame and coil counts
        _case("mec1_radial160_q27", "mec1", 160, 128, 27, 9, 3, "radial", 7.0, 3),
        # temporally sparse model error of the cardiac-shaped scan
        _case("mec2_lines192_q48", "mec2", 192, 192, 48, 12, 4, "lines", 8.0, 10),
        # eight uneven slices (line and radial masks in turn) in one launch
        _case("batch_uneven_s8", "batch", 256, 256, 64, 32, 14, "mixed", 8.0, 10, slices=8),
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def _cost(case):
    w = work(case)
    return w["flops"] + 10.0 * w["bytes"]


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        op = rng.choice(["online", "track", "track", "solve", "solve", "iterate", "iterate", "mean", "mec1", "mec2",
                         "batch"])
        ny = rng.choice(SIDES)
        nx = ny if rng.random() < 0.5 else rng.choice(SIDES)
        mask = rng.choice(["lines", "radial"])
        accel = round(rng.uniform(4.0, 12.0), 1)
        coils = int(round(_log(rng, 8, 32)))
        rank = rng.randint(4, 14)
        q, iters, slices, precision = int(round(_log(rng, 16, 96))), 0, 1, "fp32"
        if op == "online":
            q, iters = rng.randint(1, 4), rng.randint(1, 4)
        elif op == "track":
            q, iters = rng.randint(4, 16), rng.randint(3, 8)
        elif op == "solve":
            iters = 50
        elif op == "iterate":
            iters = rng.randint(4, 20)
            precision = rng.choice(["fp32", "fp32", "fp32", "bf16x3"])
        elif op == "mean":
            rank, iters = 1, 10
        elif op == "mec1":
            rank, iters = rng.randint(2, 5), rng.randint(1, 4)
        elif op == "mec2":
            rank, iters = rng.randint(2, 5), rng.randint(4, 10)
        else:
            ny = nx = 256
            q, coils, rank, mask, accel, iters, slices = 64, 32, 14, "mixed", 8.0, rng.randint(4, 12), rng.randint(3, 9)
        rank = min(rank, max(1, q // 2)) if op in ("solve", "iterate", "mec1", "mec2") else rank
        c = _case("", op, ny, nx, q, coils, rank, mask, accel, iters, precision=precision, slices=slices)
        del c["name"]
        if _cost(c) <= most:
            return c


# ---------------------------------------------------------------- inputs

def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _gauss(gen, *shape):
    z = torch.randn(*shape, 2, generator=gen, dtype=torch.float64, device=gen.device) / math.sqrt(2.0)
    return torch.view_as_complex(z)


def _line_mask(rng, ny, nx, q, accel):
    """Variable-density phase-encode lines, redrawn per frame: a sampled centre
    and further lines with weight (1 - |ky| / (ny / 2))^2."""
    n_lines = max(5, int(round(ny / accel)))
    n_center = min(n_lines, max(4, int(round(ny / (4.0 * accel)))))
    ky = np.arange(-ny // 2, ny - ny // 2)
    center = np.arange(-(n_center // 2), n_center - n_center // 2)
    others = np.setdiff1d(ky, center)
    w = (1.0 - np.abs(others) / (ny / 2.0)) ** 2 + 1e-9
    w /= w.sum()
    m = np.zeros((q, ny, nx), dtype=np.uint8)
    for k in range(q):
        pick = rng.choice(others, size=n_lines - n_center, replace=False, p=w)
        m[k, np.mod(np.concatenate([center, pick]), ny)] = 1
    return m.reshape(q, ny * nx)


def _radial_mask(ny, nx, q, accel, turn):
    """Golden-angle pseudo-radial spokes gridded by rounding."""
    n = max(ny, nx)
    spokes = max(4, int(round(n / accel)))
    t = np.arange(-n // 2, n - n // 2, dtype=np.float64)
    m = np.zeros((q, ny, nx), dtype=np.uint8)
    for k in range(q):
        th = np.radians(np.mod(np.arange(spokes) * 180.0 / spokes + k * 111.25 + turn, 180.0))[:, None]
        kyc = np.floor(t * np.sin(th) + 0.5).astype(np.int64).reshape(-1)
        kxc = np.floor(t * np.cos(th) + 0.5).astype(np.int64).reshape(-1)
        ok = (kyc >= -ny // 2) & (kyc < ny - ny // 2) & (kxc >= -nx // 2) & (kxc < nx - nx // 2)
        m[k, np.mod(kyc[ok], ny), np.mod(kxc[ok], nx)] = 1
    return m.reshape(q, ny * nx)


def _maps(gen, ny, nx, nc):
    """Complex Gaussian bumps on a ring around the field of view, unit sum of squares."""
    if nc == 1:
        return torch.ones(1, ny * nx, dtype=torch.complex128, device=gen.device)
    yy = torch.linspace(-1, 1, ny, dtype=torch.float64, device=gen.device)[None, :, None]
    xx = torch.linspace(-1, 1, nx, dtype=torch.float64, device=gen.device)[None, None, :]
    u = torch.rand(4, nc, generator=gen, dtype=torch.float64, device=gen.device)
    th = 2 * math.pi * (torch.arange(nc, device=gen.device) + 0.5 * u[0]) / nc
    cy, cx = (1.1 * torch.sin(th))[:, None, None], (1.1 * torch.cos(th))[:, None, None]
    wd = (0.7 + 0.5 * u[1])[:, None, None]
    mag = torch.exp(-((yy - cy) ** 2 + (xx - cx) ** 2) / (2 * wd ** 2))
    ph = 2 * math.pi * u[2][:, None, None] + 0.8 * (yy * torch.sin(th)[:, None, None] + xx * u[3][:, None, None])
    s = mag * torch.exp(1j * ph)
    return (s / torch.sqrt((s.abs() ** 2).sum(0, keepdim=True))).reshape(nc, -1)


def _images(gen, ny, nx, q, motion=1.0):
    """(q, n) images: a body ellipse and inner ellipses whose axes and contrast vary over the frames."""
    dev = gen.device
    yy = torch.linspace(-1, 1, ny, dtype=torch.float64, device=dev)[None, :, None]
    xx = torch.linspace(-1, 1, nx, dtype=torch.float64, device=dev)[None, None, :]
    k = torch.arange(q, dtype=torch.float64, device=dev)[:, None, None]
    period = max(24.0, float(min(q, 48)))

    def ellipse(cy, cx, ay, ax, th):
        c, s = math.cos(th), math.sin(th)
        y, x = yy - cy, xx - cx
        rho = torch.sqrt(((c * y + s * x) / ay) ** 2 + ((-s * y + c * x) / ax) ** 2)
        return torch.sigmoid((1.0 - rho) * 25.0)

    img = ellipse(0.0, 0.0, 0.85, 0.72, 0.0).expand(q, ny, nx).clone()
    for p in torch.rand(6, 9, generator=gen, dtype=torch.float64, device=dev).tolist():
        phi = 2 * math.pi * p[6]
        wob = 1.0 + 0.15 * motion * torch.sin(2 * math.pi * k / period + phi)
        con = 1.0 + 0.4 * motion * torch.sin(2 * math.pi * k * (1 + int(3 * p[8])) / period + 2 * phi)
        rho = (0.3 + 0.6 * p[5]) * (1.0 if p[7] < 0.7 else -1.0)
        img += rho * con * ellipse(0.72 * p[0] - 0.36, 0.6 * p[1] - 0.3, (0.08 + 0.16 * p[2]) * wob,
                                   (0.08 + 0.16 * p[3]) * wob, math.pi * p[4])
    ph = torch.rand(2, generator=gen, dtype=torch.float64, device=dev).tolist()
    return (img * torch.exp(1j * (ph[0] * yy + ph[1] * xx))).reshape(q, ny * nx)


def _slice_inputs(case, seed):
    """Everything a call is given, as complex64 / integer tensors, from the seed alone."""
    dev, ny, nx, q, nc, r = _dev(), case["ny"], case["nx"], case["q"], case["coils"], case["rank"]
    n = ny * nx
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 7919 + 17)
    rng = np.random.default_rng(int(seed) + 104729)
    lead = FIRST if case["op"] in ("track", "online") else 0
    if case["data"] == "lowrank":
        v = torch.linalg.qr(_gauss(gen, n, r))[0]
        x = (v @ _gauss(gen, r, lead + q)).T.contiguous()
    else:
        # model-error correction is for scans that a low rank misses: more motion, a smaller rank
        x = _images(gen, ny, nx, lead + q, 2.0 if case["op"] in ("mec1", "mec2") else 1.0)
    maps = _maps(gen, ny, nx, nc).to(torch.complex64)
    if case["mask"] == "lines":
        mask = _line_mask(rng, ny, nx, q, case["accel"])
    else:
        mask = _radial_mask(ny, nx, q, case["accel"], float(rng.uniform(0.0, 180.0)))
    fp = np.zeros(q + 1, dtype=np.int64)
    fp[1:] = np.cumsum(mask.sum(1, dtype=np.int64))
    mask_d = torch.from_numpy(mask).to(dev)
    y = torch.empty(nc * int(fp[-1]), dtype=torch.complex64, device=dev)
    at = 0
    for k in range(q):
        f = torch.fft.fft2((maps.to(torch.complex128) * x[lead + k][None]).reshape(nc, ny, nx), norm="ortho")
        yk = f.reshape(nc, n)[:, mask_d[k].bool()].reshape(-1)
        y[at:at + yk.numel()] = yk.to(torch.complex64)
        at += yk.numel()
    if case["data"] != "lowrank":
        rms = torch.sqrt((y.abs().double() ** 2).mean())
        y += (0.01 * rms * _gauss(gen, y.numel())).to(torch.complex64)
    # an imperfect subspace estimate: r random mixtures of the frames a solve has seen, orthonormalised
    seen = x[:lead] if lead else x
    base = seen.T @ _gauss(gen, seen.shape[0], r)
    base = base / torch.linalg.norm(base, dim=0, keepdim=True)
    u0 = torch.linalg.qr(base + 0.02 / math.sqrt(n) * _gauss(gen, n, r))[0]
    smax2 = float(torch.linalg.matrix_norm(seen @ seen.conj().T, ord="fro"))
    eta = 0.4 / (smax2 * q / seen.shape[0])
    zbar = seen.mean(0)
    if case["op"] == "online":   # the subspace of what the mean leaves
        base = (seen - zbar[None]).T @ _gauss(gen, seen.shape[0], r)
        u0 = torch.linalg.qr(base / torch.linalg.norm(base, dim=0, keepdim=True))[0]
    return dict(y=y, fp=torch.from_numpy(fp).to(dev), mask=mask_d, maps=maps.contiguous(),
                u0=u0.to(torch.complex64).contiguous(), eta=eta, zbar=zbar.to(torch.complex64).contiguous())


def _slices(case, seed):
    """The slices of a case: itself, or a batch's uneven slices (sizes fixed by the case, not by the seed)."""
    if case["op"] != "batch":
        return [(case, seed)]
    rng, out = np.random.default_rng(case["slices"]), []
    for i in range(case["slices"]):
        side = int(rng.choice(BATCH_SIDES))
        q = int(rng.integers(24, case["q"] + 1))
        out.append((dict(case, op="iterate", ny=side, nx=side, q=q, coils=int(rng.integers(8, case["coils"] + 1)),
                         rank=int(rng.integers(6, case["rank"] + 1)), mask="lines" if i % 2 == 0 else "radial",
                         accel=float(rng.uniform(4.0, 12.0))), int(seed) * 31 + i))
    return out


def _solver(c, stream, rank_max=0):
    prec = lrccs.PREC_BF16X3_GEMM if c["precision"] == "bf16x3" else lrccs.PREC_FP32_FFT
    return lrccs.Solver(c["ny"], c["nx"], c["q"], c["coils"], c["rank"], rank_max, stream=stream, precision=prec)


def _new(*shape):
    return torch.empty(shape, dtype=torch.complex64, device=_dev())


class _State:
    """A program's solvers, inputs and output buffers for one case."""

    def __init__(self, case, seed):
        self.case, self.stream, self.parts, self.batch = case, torch.cuda.Stream(), [], None
        for c, s in _slices(case, seed):
            d, n = _slice_inputs(c, s), c["ny"] * c["nx"]
            torch.cuda.synchronize()
            sv = _solver(c, self.stream)
            d.update(c=c, solver=sv, X=_new(c["q"], n), U=_new(n, c["rank"]), inp=(d["y"], d["fp"], d["mask"], d["maps"]))
            op = c["op"]
            if op in ("iterate", "mec1", "mec2"):
                sv.init(*d["inp"])                      # the scan is loaded; its solve is resumed
            if op in ("mec1", "mec2"):
                sv.set_subspace(d["u0"], d["eta"])
                sv.iterate(5)
                d["E"] = _new(c["q"], n)
            if op == "online":
                sv.set_subspace(d["u0"], 0.0)
                d["B"] = _new(c["q"], c["rank"])
            if op == "mean":
                d["ytil"] = torch.empty_like(d["y"])
                d["z"] = _new(n)
            self.parts.append(d)
        if case["op"] == "batch":
            self.batch = lrccs.lrccs_batch_create([d["solver"].ctx for d in self.parts], self.stream)
        torch.cuda.synchronize()

    def __del__(self):
        if getattr(self, "batch", None):
            lrccs.lrccs_batch_destroy(self.batch)


def prepare(case, seed):
    return _State(case, seed)


def run(state):
    case, d, op = state.case, state.parts[0], state.case["op"]
    sv, ctx, it = d["solver"], d["solver"].ctx, state.case["iters"]
    with torch.cuda.stream(state.stream):
        if op == "solve":
            sv.init(*d["inp"])
            sv.iterate(it)
            lrccs.lrccs_get_images(ctx, d["X"])
            return {"X": d["X"]}
        if op == "iterate":
            sv.set_subspace(d["u0"], d["eta"])
            sv.iterate(it)
            lrccs.lrccs_get_images(ctx, d["X"])
            lrccs.lrccs_get_subspace(ctx, d["U"])
            return {"X": d["X"], "U": d["U"]}
        if op == "track":
            sv.set_subspace(d["u0"], d["eta"])
            sv.track(*d["inp"], t_max=it, X=d["X"])
            lrccs.lrccs_get_subspace(ctx, d["U"])
            return {"X": d["X"], "U": d["U"]}
        if op == "online":
            lrccs.lrccs_online_frames(ctx, *d["inp"], d["zbar"], it, d["X"], d["B"])
            return {"X": d["X"], "B": d["B"]}
        if op == "mean":
            n_it = lrccs.lrccs_mean_step(ctx, *d["inp"], d["z"], d["ytil"], 1e-3, it)
            return {"zbar": d["z"], "ytil": d["ytil"], "iterations": n_it}
        if op == "mec1":
            lrccs.lrccs_mec1(ctx, it, d["zbar"], d["E"], d["X"])
            return {"E": d["E"], "X": d["X"]}
        if op == "mec2":
            n_it = lrccs.lrccs_mec2(ctx, it, 0.0025, 0.001, d["zbar"], d["E"], d["X"])
            return {"E": d["E"], "X": d["X"], "iterations": n_it}
        for p in state.parts:
            p["solver"].set_subspace(p["u0"], p["eta"])
        lrccs.lrccs_batch_iterate(state.batch, it)
        out = []
        for p in state.parts:
            lrccs.lrccs_get_images(p["solver"].ctx, p["X"])
            lrccs.lrccs_get_subspace(p["solver"].ctx, p["U"])
            out.append({"X": p["X"], "U": p["U"]})
        return out


# ---------------------------------------------------------------- work

def _samples(c):
    """Samples per coil of one frame (about, for pseudo-radial masks) and k-space points that some frame samples."""
    ny, nx, n = c["ny"], c["nx"], c["ny"] * c["nx"]
    if c["mask"] == "lines":
        lines = max(5, int(round(ny / c["accel"])))
        return lines * nx, min(ny, lines + 0.08 * lines * (c["q"] - 1)) * nx
    m = min(0.75 * n, 0.8 * max(4, round(max(ny, nx) / c["accel"])) * min(ny, nx))
    return m, n * (1.0 - (1.0 - m / n) ** (c["q"] * 0.7))


def _transform(c, cols):
    """Flops of `cols` coil images' transforms one way (ky only where the masks are lines)."""
    n = c["ny"] * c["nx"]
    lg = math.log2(c["ny"]) + (math.log2(c["nx"]) if c["mask"] != "lines" else 0.0)
    return 5.0 * n * lg * cols + 6.0 * n * cols


def _one_work(c):
    ny, nx, q, nc, r, it, op = c["ny"], c["nx"], c["q"], c["coils"], c["rank"], c["iters"], c["op"]
    n = ny * nx
    m, union = _samples(c)
    full = 5.0 * n * math.log2(n) + 8.0 * n          # one 2D transform of one coil image, and its map
    iteration = 2 * _transform(c, nc * r) + union * nc * 16.0 * r * r + 16.0 * n * q * r + 24.0 * n * r * r
    inputs = 8.0 * (nc * m * q + nc * n) + q * n
    per_frame = 2 * _transform(c, nc) * q            # one normal operator of every frame
    if op == "solve":
        return inputs + 8.0 * n * q, q * nc * full + 4.0 * n * q * q + it * iteration + 8.0 * n * q * r
    if op == "iterate":
        return inputs + 8.0 * (n * q + 2 * n * r), it * iteration + 8.0 * n * q * r
    if op == "track":
        return inputs + 8.0 * (n * q + 2 * n * r), q * nc * full + it * iteration + 8.0 * n * q * r
    if op == "online":
        return inputs + 8.0 * (n * q + n * r + n), q * nc * full + iteration / 2 + (it + 2) * per_frame
    if op == "mean":
        return inputs + 8.0 * (nc * m * q + n), q * nc * full + it * 2 * _transform(c, nc) + nc * full
    if op == "mec1":
        return inputs + 8.0 * (2 * n * q + n * r + n), (it + 1) * per_frame + 40.0 * it * n * q + 8.0 * n * q * r
    return inputs + 8.0 * (2 * n * q + n * r + n), it * (per_frame + 10.0 * n * q * math.log2(max(2, q))) + 8.0 * n * q * r


def work(case):
    parts = [_one_work(c) for c, _ in _slices(case, 0)]
    return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}


# ---------------------------------------------------------------- the same in FP64

class _Exact:
    def __init__(self, c, seed):
        d = _slice_inputs(c, seed)
        self.c, self.ny, self.nx, self.q, self.nc, self.r = c, c["ny"], c["nx"], c["q"], c["coils"], c["rank"]
        self.n = self.ny * self.nx
        self.maps = d["maps"].to(torch.complex128)
        self.mask = d["mask"].to(torch.float64)
        self.idx = [torch.nonzero(d["mask"][k]).reshape(-1) for k in range(self.q)]
        self.u0, self.eta = d["u0"].to(torch.complex128), d["eta"]
        self.zbar = d["zbar"].to(torch.complex128)
        self.y, at = [], 0
        for k in range(self.q):
            m = self.idx[k].numel()
            self.y.append(d["y"][at:at + self.nc * m].to(torch.complex128).reshape(self.nc, m))
            at += self.nc * m

    def fft(self, x):
        return torch.fft.fft2(x.reshape(*x.shape[:-1], self.ny, self.nx), norm="ortho").reshape(x.shape)

    def ifft(self, x):
        return torch.fft.ifft2(x.reshape(*x.shape[:-1], self.ny, self.nx), norm="ortho").reshape(x.shape)

    def adjoint(self, y):
        """n x q: A_k^H y_k."""
        out = torch.zeros(self.n, self.q, dtype=torch.complex128, device=self.maps.device)
        for k in range(self.q):
            f = torch.zeros(self.nc, self.n, dtype=torch.complex128, device=self.maps.device)
            f[:, self.idx[k]] = y[k]
            out[:, k] = (self.maps.conj() * self.ifft(f)).sum(0)
        return out

    def apply(self, k, x):
        return self.fft(self.maps * x[None])[:, self.idx[k]]

    def normal(self, x):
        """N_k x_k of every frame, x (q, n)."""
        out = torch.empty_like(x)
        for k in range(self.q):
            out[k] = (self.maps.conj() * self.ifft(self.fft(self.maps * x[k][None]) * self.mask[k][None])).sum(0)
        return out

    def spectral(self):
        tot = sum(int(i.numel()) for i in self.idx)
        gamma = 36.0 * sum(float((v.abs() ** 2).sum()) for v in self.y) / (self.nc * tot)
        mbar = tot / self.q
        x0 = self.adjoint([torch.where(v.real ** 2 + v.imag ** 2 <= gamma, v, torch.zeros_like(v)) for v in self.y])
        x0 = x0 / torch.sqrt(torch.tensor([i.numel() * mbar for i in self.idx], dtype=torch.float64,
                                          device=x0.device))[None]
        lam, v = torch.linalg.eigh(x0.conj().T @ x0)
        v = v.flip(1)[:, :self.r]
        return torch.linalg.qr(x0 @ v)[0]

    def bstep(self, u, z):
        fu = self.fft((self.maps[:, None] * u.T[None]).contiguous())          # (nc, r, n)
        h = u.conj().T @ z
        b = torch.empty(self.r, self.q, dtype=torch.complex128, device=u.device)
        for k in range(self.q):
            a = fu[:, :, self.idx[k]].permute(1, 0, 2).reshape(self.r, -1)
            b[:, k] = torch.linalg.solve(a.conj() @ a.T, h[:, k])
        return fu, b

    def iterate(self, u, z, eta, iters):
        """x (q, n) = (U_{t-1} B_t)^T and U_t; eta <= 0: 0.14 / ||first gradient||."""
        for _ in range(iters):
            fu, b = self.bstep(u, z)
            bb = (b.T[:, :, None] * b.T.conj()[:, None, :]).reshape(self.q, -1)
            w = (self.mask.T.to(torch.complex128) @ bb).reshape(self.n, self.r, self.r)
            f = torch.bmm(fu.permute(2, 0, 1), w).permute(1, 2, 0).contiguous()   # (nc, r, n)
            grad = (self.maps.conj()[:, None] * self.ifft(f)).sum(0).T - z @ b.conj().T
            if eta <= 0.0:
                eta = 0.14 / float(torch.linalg.matrix_norm(grad.conj().T @ grad, ord=2)) ** 0.5
            x = (u @ b).T
            qm, rm = torch.linalg.qr(u - eta * grad)
            ph = torch.diagonal(rm)
            u = qm * (ph / ph.abs())[None]
        return x, u

    def cgls(self, s, iters):
        """e_k from `iters` CG steps on N_k e = s_k from zero, s (q, n)."""
        e, p = torch.zeros_like(s), s.clone()
        g = (s.abs() ** 2).sum(1)
        for _ in range(iters):
            w = self.normal(p)
            d = (p.conj() * w).real.sum(1)
            a = torch.where((d > 0) & (g > 0), g / d, torch.zeros_like(g))
            e, s = e + a[:, None] * p, s - a[:, None] * w
            g2 = (s.abs() ** 2).sum(1)
            p = s + torch.where(g > 0, g2 / g, torch.zeros_like(g))[:, None] * p
            g = g2
        return e

    def mean(self, iters):
        cnt, z = self.mask.sum(0), torch.zeros(self.n, dtype=torch.complex128, device=self.maps.device)
        s = self.adjoint(self.y).sum(1)
        p, g = s.clone(), float((s.abs() ** 2).sum())
        g0, it = g, 0
        while it < iters and math.sqrt(g) > 1e-3 * math.sqrt(g0):
            w = (self.maps.conj() * self.ifft(self.fft(self.maps * p[None]) * cnt[None])).sum(0)
            a = g / float((p.conj() * w).real.sum())
            z, s = z + a * p, s - a * w
            g2 = float((s.abs() ** 2).sum())
            p, g, it = s + (g2 / g) * p, g2, it + 1
        res = [self.y[k] - self.apply(k, z) for k in range(self.q)]
        return {"zbar": z, "ytil": torch.cat([v.reshape(-1) for v in res]), "iterations": it}

    def mec2(self, s0, iters):
        e, prev, it = torch.zeros_like(s0), None, 0
        while it < iters:
            m = torch.fft.fft(e + s0 - (self.normal(e) if it else 0), dim=0, norm="ortho")
            if it == 0:
                omega = 0.001 * float(m.abs().max())
            elif float(torch.linalg.norm(m - prev)) < 0.0025 * float(torch.linalg.norm(prev)):
                break
            a = m.abs()
            e = torch.fft.ifft(torch.where(a > omega, m * (1.0 - omega / a.clamp_min(1e-300)), torch.zeros_like(m)),
                               dim=0, norm="ortho")
            prev, it = m, it + 1
        return e, it


def _one_exact(c, seed):
    x, op, it = _Exact(c, seed), c["op"], c["iters"]
    if op == "mean":
        return x.mean(it)
    if op == "online":
        z = x.adjoint([x.y[k] - x.apply(k, x.zbar) for k in range(x.q)])
        u = torch.linalg.qr(x.u0)
        u = u[0] * (torch.diagonal(u[1]) / torch.diagonal(u[1]).abs())[None]
        _, b = x.bstep(u, z)
        lr = (u @ b).T
        return {"X": x.zbar[None] + lr + x.cgls(z.T - x.normal(lr), it), "B": b.T.contiguous()}
    z = x.adjoint(x.y)
    if op == "solve":
        return {"X": x.iterate(x.spectral(), z, 0.0, it)[0]}
    u0 = torch.linalg.qr(x.u0)
    u0 = u0[0] * (torch.diagonal(u0[1]) / torch.diagonal(u0[1]).abs())[None]
    if op in ("iterate", "track"):
        img, u = x.iterate(u0, z, x.eta, it)
        return {"X": img, "U": u}
    img, _ = x.iterate(u0, z, x.eta, 5)
    s0 = z.T - x.normal(img)
    if op == "mec1":
        e = x.cgls(s0, it)
        return {"E": e, "X": x.zbar[None] + img + e}
    e, n_it = x.mec2(s0, it)
    return {"E": e, "X": x.zbar[None] + img + e, "iterations": n_it}


def exact(case, seed):
    got = [_one_exact(c, s) for c, s in _slices(case, seed)]
    return got if case["op"] == "batch" else got[0]
