"""GPU tests of the spectral step (Gram of X0, Jacobi eigensolver, U_0) against
numpy's SVD of the X0 the library formed: one frame, odd and even counts, one
and two tiles per thread of the Gram kernel, the largest q."""
import numpy as np
import pytest

from paper_2212_09664_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2212_09664_gb300 import lrccs  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("ny,nx,q,r", [(32, 32, 1, 1), (32, 64, 2, 2), (64, 32, 3, 1), (64, 64, 17, 5), (96, 64, 47, 9),
                                       (64, 96, 64, 12), (128, 128, 125, 16), (96, 96, 128, 16)])
def test_spectral_step_matches_svd(ny, nx, q, r):
    p = synth.make_problem(dict(kind="phantom", ny=ny, nx=nx, q=q, nc=3, rank=r, mask_kind="lines_vd", accel=3.0,
                                noise=0.02), seed=11 * q + r)
    inp = tuple(torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (p.y, p.frame_ptr, p.mask, p.smaps))
    s = lrccs.Solver(ny, nx, q, 3, r)
    s.init(*inp)
    X0, sig, U = s.buffer(lrccs.BUF_X0), s.buffer(lrccs.BUF_SIGMA), s.subspace()
    s.sync()
    torch.cuda.synchronize()
    x = X0.cpu().numpy().astype(np.complex128)
    ref = np.linalg.svd(x, compute_uv=False)
    sig, u = sig.cpu().numpy(), U.cpu().numpy().astype(np.complex128)
    # the leading r singular values: squares from FP32 Gram sums, then an FP64 refinement
    assert np.all(np.abs(sig[:r] - ref[:r]) < 2e-6 * ref[0] ** 2 / ref[:r] + 1e-6 * ref[:r])
    # U_0 captures what the best rank-r subspace does (insensitive to small gaps)
    left = np.linalg.norm(x - u @ (u.conj().T @ x))
    best = np.sqrt(np.sum(ref[r:] ** 2))
    assert left < best + 2e-6 * ref[0]
    assert np.linalg.norm(u.conj().T @ u - np.eye(r)) < 3e-6 * r ** 0.5
    s.close()
