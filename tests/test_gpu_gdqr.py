"""GPU tests of the GD step with its Cholesky QR (k_gdqr) against FP64 torch:
one pixel row per thread and many, Z in one piece and through two chunk
buffers, few and many frames, odd and extreme ranks, more columns than frames."""
import numpy as np
import pytest

from paper_2212_09664_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2212_09664_gb300 import lrccs  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("ny,nx,q,nc,r", [(32, 32, 1, 2, 1), (32, 32, 7, 3, 5), (64, 32, 15, 2, 16), (96, 96, 33, 2, 7),
                                          (192, 192, 8, 4, 10), (256, 256, 64, 2, 12), (256, 256, 128, 2, 16),
                                          (256, 224, 5, 3, 3), (64, 64, 2, 4, 8), (128, 160, 14, 2, 4)])
def test_gd_step_and_qr_match_torch(ny, nx, q, nc, r):
    n = ny * nx
    rng = np.random.default_rng(n + q + r)
    p = synth.make_problem(dict(kind="lowrank", ny=ny, nx=nx, q=q, nc=nc, rank=min(r, q), mask_kind="lines_vd", accel=2.0,
                                noise=0.05), seed=n + r)
    y, fp, mask, sm = (torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (p.y, p.frame_ptr, p.mask, p.smaps))
    u0 = torch.from_numpy(np.linalg.qr(rng.standard_normal((n, r)) + 1j * rng.standard_normal((n, r)))[0]).to(DEV)
    s = lrccs.Solver(ny, nx, q, nc, r, rank_max=r)
    s.set_subspace(u0.to(torch.complex64).contiguous(), 0.0)
    info = s.track(y, fp, mask, sm, t_max=2, info=True)
    Up, B = s.factors()
    G, U, Z = s.buffer(lrccs.BUF_GRAD), s.subspace(), s.buffer(lrccs.BUF_Z)
    s.sync()
    torch.cuda.synchronize()
    up, g = Up.to(torch.complex128), G.to(torch.complex128)
    step = up - info["eta"] * g
    qm, rm = torch.linalg.qr(step)
    ph = torch.diagonal(rm)
    ref = qm * (ph / ph.abs())[None]
    # FP32 rows, Gram sums and an r x r factorisation of a well-conditioned G1: a few eps sqrt(r)
    assert float(torch.linalg.norm(U - ref)) < 2e-6 * r ** 0.5
    eye = torch.eye(r, dtype=torch.complex128, device=DEV)
    uu = U.to(torch.complex128)
    assert float(torch.linalg.norm(uu.conj().T @ uu - eye)) < 3e-6 * r ** 0.5
    sd = torch.linalg.norm(ref - up @ (up.conj().T @ ref))
    assert abs(info["sd"] ** 2 - float(sd) ** 2) < 1e-5 * r
    # the right-hand sides of the second B-step came from the first iteration's h = U^H Z
    d = sm.to(torch.complex128)
    z = Z.to(torch.complex128)
    fu = torch.fft.fft2((d[:, None] * up.T[None]).reshape(nc, r, ny, nx), norm="ortho").reshape(nc, r, n)
    for k in range(q):
        a = fu[:, :, mask[k].bool()].permute(1, 0, 2).reshape(r, -1)
        gk, hk, b = a.conj() @ a.T, up.conj().T @ z[:, k], B[k].to(torch.complex128)
        assert float(torch.linalg.norm(gk @ b - hk)) < 3e-6 * float(torch.linalg.norm(gk) * torch.linalg.norm(b))
    s.close()
