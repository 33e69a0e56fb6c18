"""GPU tests of the vector kernels around the transforms (the mean step's CG, MEC)
against FP64 torch: one block and many, single frames and coils, frame counts
that leave a warp partly idle."""
import numpy as np
import pytest

from paper_2212_09664_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2212_09664_gb300 import lrccs  # noqa: E402

DEV = torch.device("cuda:0")


class Case:
    """A seeded problem on the device and its operators in complex128."""

    def __init__(self, ny, nx, q, nc, rank, kind, seed):
        spec = dict(kind="phantom", ny=ny, nx=nx, q=q, nc=nc, rank=rank, noise=0.02)
        spec.update(dict(mask_kind="lines_vd", accel=4.0) if kind == "lines" else dict(mask_kind="radial", spokes=9))
        p = synth.make_problem(spec, seed=seed)
        self.inp = tuple(torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (p.y, p.frame_ptr, p.mask, p.smaps))
        self.ny, self.nx, self.q, self.nc, self.n = ny, nx, q, nc, ny * nx
        self.d = self.inp[3].to(torch.complex128)
        self.m = self.inp[2].to(torch.float64)
        self.y, at = [], 0
        for k in range(q):
            cnt = int(self.m[k].sum())
            f = torch.zeros((nc, self.n), dtype=torch.complex128, device=DEV)
            f[:, self.m[k] > 0] = self.inp[0][at:at + nc * cnt].to(torch.complex128).reshape(nc, cnt)
            self.y.append(f)
            at += nc * cnt

    def fft(self, x, inv=False):
        f = torch.fft.ifft2 if inv else torch.fft.fft2
        return f(x.reshape(self.nc, self.ny, self.nx), norm="ortho").reshape(self.nc, self.n)

    def adjoint(self, k, f):
        return (self.d.conj() * self.fft(f * self.m[k], True)).sum(0)

    def apply(self, k, x):
        return self.fft(self.d * x) * self.m[k]


def rel(a, b):
    return float(torch.linalg.norm(a - b) / torch.linalg.norm(b))


@pytest.mark.parametrize("ny,nx,q,nc,kind", [(32, 32, 1, 1, "lines"), (64, 32, 33, 3, "radial"), (256, 256, 5, 2, "lines"),
                                             (96, 160, 40, 4, "lines")])
def test_mean_step_matches_torch(ny, nx, q, nc, kind):
    c = Case(ny, nx, q, nc, 1, kind, ny + q)
    s = lrccs.Solver(ny, nx, q, nc, 1)
    # one frame of one coil: A^H A is a projector, CG is done after one step and a second one divides 0 by 0
    steps = 1 if q * nc == 1 else 3
    zbar, ytil, it = s.mean_step(*c.inp, tol=0.0, max_iter=steps)
    s.sync()
    r = sum(c.adjoint(k, c.y[k]) for k in range(q))
    z, p, g = torch.zeros_like(r), r.clone(), (r.abs() ** 2).sum()
    for _ in range(steps):
        w = sum(c.adjoint(k, c.apply(k, p)) for k in range(q))
        a = g / (p.conj() * w).real.sum()
        z, r = z + a * p, r - a * w
        g2 = (r.abs() ** 2).sum()
        p, g = r + (g2 / g) * p, g2
    assert it == steps
    # up to three CG steps in FP32 vectors with FP64 scalars: each step's transforms round at about 3e-7
    assert rel(zbar, z) < 5e-6
    res = torch.cat([(c.y[k] - c.apply(k, z))[:, c.m[k] > 0].reshape(-1) for k in range(q)])
    scale = torch.linalg.norm(c.inp[0].to(torch.complex128))
    assert float(torch.linalg.norm(ytil - res)) < 5e-6 * float(scale)
    s.close()


# chunks of the frames' normal operators: one column, padded chunks, wider and narrower than the rank
@pytest.mark.parametrize("ny,nx,q,nc,rank,kind", [(64, 64, 1, 3, 1, "lines"), (32, 96, 16, 2, 2, "lines"),
                                                  (64, 64, 17, 3, 5, "radial"), (96, 64, 33, 2, 3, "lines"),
                                                  (64, 32, 5, 4, 4, "radial")])
def test_mec1_matches_torch(ny, nx, q, nc, rank, kind):
    c = Case(ny, nx, q, nc, rank, kind, nx + q)
    s = lrccs.Solver(ny, nx, q, nc, rank)
    s.init(*c.inp)
    s.iterate(3)
    E, X = s.mec1(2)
    U, B = s.factors()
    s.sync()
    low = (U.to(torch.complex128) @ B.to(torch.complex128).T).T
    scale = torch.linalg.norm(low) / q ** 0.5
    for k in range(q):
        r = c.adjoint(k, c.y[k]) - c.adjoint(k, c.apply(k, low[k]))
        e, p, g = torch.zeros_like(r), r.clone(), (r.abs() ** 2).sum()
        for _ in range(2):
            w = c.adjoint(k, c.apply(k, p))
            a = g / (p.conj() * w).real.sum()
            e, r = e + a * p, r - a * w
            g2 = (r.abs() ** 2).sum()
            p, g = r + (g2 / g) * p, g2
        # the residual is a difference of FP32 terms of the image's size
        assert float(torch.linalg.norm(E[k] - e)) < 3e-6 * float(scale)
        assert float(torch.linalg.norm(X[k] - low[k] - e)) < 3e-6 * float(scale)
    s.close()


# temporal transforms: one frame, odd, prime, even and the largest frame counts
@pytest.mark.parametrize("ny,nx,q,nc,kind", [(32, 32, 1, 2, "lines"), (32, 64, 2, 3, "radial"), (32, 32, 13, 2, "lines"),
                                             (64, 32, 30, 2, "lines"), (32, 32, 127, 1, "lines"), (32, 32, 128, 2, "lines")])
def test_mec2_matches_torch(ny, nx, q, nc, kind):
    c = Case(ny, nx, q, nc, 1, kind, ny + 3 * q)
    s = lrccs.Solver(ny, nx, q, nc, 1)
    s.init(*c.inp)
    s.iterate(2)
    E, X, it = s.mec2(3, 0.0, 0.02)
    U, B = s.factors()
    s.sync()
    low = (U.to(torch.complex128) @ B.to(torch.complex128).T).T
    s0 = torch.stack([c.adjoint(k, c.y[k]) - c.adjoint(k, c.apply(k, low[k])) for k in range(q)])
    e = torch.zeros_like(s0)
    for tau in range(3):
        ne = torch.stack([c.adjoint(k, c.apply(k, e[k])) for k in range(q)])
        m = torch.fft.fft(e + s0 - ne, dim=0, norm="ortho")
        if tau == 0:
            omega = 0.02 * float(m.abs().max())
        a = m.abs()
        e = torch.fft.ifft(torch.where(a > omega, m * (1 - omega / a.clamp_min(1e-300)), torch.zeros_like(m)), dim=0,
                           norm="ortho")
    assert it == 3
    # FP32 sums of q terms, three steps, on the residual of FP32 images
    scale = torch.linalg.norm(low) + torch.linalg.norm(e)
    assert float(torch.linalg.norm(E - e)) < 3e-6 * float(scale)
    s.close()
