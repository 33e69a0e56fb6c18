"""GPU test of the GD/QR kernel on a device with few multiprocessors, where a
block's pixels no longer fit its shared memory at once: results against the
whole device's (the same bits where the pixels are cut alike)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2212_09664_gb300 import lrccs  # noqa: E402
from test_gpu_vectors import DEV, Case, rel  # noqa: E402

MP = torch.cuda.get_device_properties(0).multi_processor_count


def track(c, r, U, blocks, eta):
    s = lrccs.Solver(c.ny, c.nx, c.q, c.nc, r)
    if blocks:
        lrccs.lrccs_test_few_blocks(s.ctx, blocks)
    X = torch.empty(c.q, c.n, dtype=torch.complex64, device=DEV)
    s.set_subspace(U, eta)
    s.track(*c.inp, t_max=3, X=X)
    s.sync()
    V = s.subspace()
    torch.cuda.synchronize()
    s.close()
    return X, V


# whole rows fit: one part a block; 65536 pixels at rank 15 and 16 on half, a quarter and a tenth of the device: several
@pytest.mark.parametrize("ny,nx,q,nc,r,kind,blocks", [
    (64, 64, 5, 2, 4, "lines", 3), (96, 128, 128, 1, 5, "lines", 20), (256, 256, 3, 2, 16, "lines", MP // 2),
    (256, 256, 3, 2, 15, "radial", MP // 4), (256, 256, 40, 1, 16, "radial", MP // 10), (256, 256, 3, 1, 16, "lines", 1)])
def test_few_blocks_match_the_whole_device(ny, nx, q, nc, r, kind, blocks):
    c = Case(ny, nx, q, nc, 2, kind, ny + q + r)
    gen = torch.Generator(device=DEV).manual_seed(r)
    U = torch.linalg.qr(torch.randn(ny * nx, r, dtype=torch.complex64, device=DEV, generator=gen))[0].contiguous()
    for eta in (0.0, 1e-6):     # the step size set from the first gradient, or given
        X, V = track(c, r, U, 0, eta)
        Xf, Vf = track(c, r, U, blocks, eta)
        assert np.isfinite(float(X.abs().sum()))
        if ny * nx == 65536 and blocks * 2 == MP:
            assert torch.equal(X, Xf) and torch.equal(V, Vf)
        # three iterations of FP32 sums in another order
        assert rel(Xf, X) < 1e-5 and rel(Vf, V) < 1e-5
    with pytest.raises(lrccs.LrccsError):
        track(c, r, U, MP + 1, 0.0)
