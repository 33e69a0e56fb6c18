"""GPU tests of the general-mask kernels (row passes, point Grams, frame sums,
point weighting) against FP64 torch: every row length with its own
factorisation, odd and extreme ranks, several coils at a time in one block,
coil counts that leave the last step or the staged chunk ragged."""
import numpy as np
import pytest

from paper_2212_09664_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2212_09664_gb300 import lrccs  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("ny,nx,q,nc,r,groups", [
    (32, 32, 5, 1, 1, 0), (32, 64, 9, 5, 3, 2), (64, 96, 20, 4, 16, 0), (32, 128, 8, 7, 5, 8), (64, 160, 12, 3, 7, 0),
    (96, 192, 14, 33, 10, 0), (32, 224, 16, 9, 13, 0), (128, 256, 16, 20, 12, 3), (32, 256, 18, 40, 16, 0)])
def test_general_iteration_matches_torch(ny, nx, q, nc, r, groups):
    n = ny * nx
    p = synth.make_problem(dict(kind="lowrank", ny=ny, nx=nx, q=q, nc=nc, rank=r, mask_kind="radial",
                                spokes=max(6, nx // 5), noise=0.05), seed=nx + r)
    y, fp, mask, sm = (torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (p.y, p.frame_ptr, p.mask, p.smaps))
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    s = lrccs.Solver(ny, nx, q, nc, r, stream=st)
    lrccs.lrccs_set_plan(s.ctx, lrccs.Plan(0, 0, groups, 0))
    s.init(y, fp, mask, sm)
    s.iterate(1)
    s.sync()
    U, B = s.factors()
    Z, G = s.buffer(lrccs.BUF_Z), s.buffer(lrccs.BUF_GRAD)
    s.sync()
    torch.cuda.synchronize()
    d, u, m = sm.to(torch.complex128), U.to(torch.complex128), mask.to(torch.complex128)
    z, b = Z.to(torch.complex128), B.to(torch.complex128)
    fu = torch.fft.fft2((d[:, None] * u.T[None]).reshape(nc, r, ny, nx), norm="ortho").reshape(nc, r, n)
    for k in range(q):
        a = fu[:, :, mask[k].bool()].permute(1, 0, 2).reshape(r, -1)
        gk, hk = a.conj() @ a.T, u.conj().T @ z[:, k]
        # FP32 Gram and elimination, both backward stable: a few eps of ||G|| ||b||
        res = torch.linalg.norm(gk @ b[k] - hk)
        assert float(res) < 3e-6 * float(torch.linalg.norm(gk) * torch.linalg.norm(b[k]))
    w = torch.einsum("ki,ka,kb->iab", m, b, b.conj())
    f = torch.einsum("jai,iab->jbi", fu, w)
    back = torch.fft.ifft2(f.reshape(nc, r, ny, nx), norm="ortho").reshape(nc, r, n)
    gk = (d.conj()[:, None] * back).sum(0).T
    grad = gk - z @ b.conj()
    # a difference of FP32 terms of the size of gk
    assert float(torch.linalg.norm(G - grad)) < 3e-6 * float(torch.linalg.norm(gk))
    s.close()
