"""GPU tests of the column passes (k_fwd_cols, k_adj_cols) against FP64 torch:
every side with its own factorisation, tiles that straddle pixels (odd ranks),
one pixel per column (rank 1) and the largest rank, cluster sizes with a ragged
last group of coils."""
import numpy as np
import pytest

from paper_2212_09664_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2212_09664_gb300 import lrccs  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("ny,nx,nc,r,groups", [
    (32, 32, 1, 1, 0), (64, 96, 5, 3, 3), (96, 32, 4, 16, 4), (128, 64, 7, 5, 8), (160, 96, 3, 7, 2),
    (192, 160, 12, 10, 0), (224, 64, 9, 13, 0), (256, 128, 20, 12, 0), (256, 32, 2, 16, 1)])
def test_column_passes_match_torch(ny, nx, nc, r, groups):
    n, q = ny * nx, max(r, 4) + 3
    p = synth.make_problem(dict(kind="lowrank", ny=ny, nx=nx, q=q, nc=nc, rank=r, mask_kind="lines_vd", accel=3.0,
                                noise=0.05), seed=ny + r)
    y, fp, mask, sm = (torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (p.y, p.frame_ptr, p.mask, p.smaps))
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    s = lrccs.Solver(ny, nx, q, nc, r, stream=st)
    lrccs.lrccs_set_plan(s.ctx, lrccs.Plan(0, groups, 0, 0))
    s.init(y, fp, mask, sm)
    T = torch.zeros((nc, ny, nx, r), dtype=torch.complex64, device=DEV)
    torch.cuda.synchronize()
    lrccs.lrccs_forward_transform(s.ctx, T)
    U = s.subspace()
    s.sync()
    used = mask.reshape(q, ny, nx).bool().any(2).any(0)
    d = sm.to(torch.complex128).reshape(nc, ny, nx, 1)
    ref = torch.fft.fft(d * U.to(torch.complex128).reshape(1, ny, nx, r), dim=1, norm="ortho")
    err = torch.linalg.norm((T - ref)[:, used]) / torch.linalg.norm(ref[:, used])
    # FP32 roundings of a length-N transform add up to about eps sqrt(log2 N), eps = 6e-8
    assert float(err) < 1e-6
    s.iterate(1)
    Up, B = s.factors()
    Z, G = s.buffer(lrccs.BUF_Z), s.buffer(lrccs.BUF_GRAD)
    s.sync()
    bk = B.to(torch.complex128)
    rows = mask.reshape(q, ny, nx)[:, :, 0].to(torch.complex128)
    W = torch.einsum("ky,ka,kb->yab", rows, bk, bk.conj())
    T = torch.fft.fft(d * Up.to(torch.complex128).reshape(1, ny, nx, r), dim=1, norm="ortho")
    K = torch.einsum("jyxa,yab->jyxb", T, W)
    gk = (d.conj() * torch.fft.ifft(K, dim=1, norm="ortho")).sum(0).reshape(n, r)
    grad = gk - Z.to(torch.complex128) @ bk.conj()
    # the gradient is a difference of terms of the size of gk; each carries FP32 sums of up to q + C ny terms
    assert float(torch.linalg.norm(G - grad)) < 3e-6 * float(torch.linalg.norm(gk))
    s.close()
