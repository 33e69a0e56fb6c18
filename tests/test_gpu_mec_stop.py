"""GPU test of MEC-2's stopping test: the number of ISTA updates against FP64
torch, on data near 1 and on the same data scaled by powers of two to the ends
of the range whose squares FP32 cannot hold."""
import math

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2212_09664_gb300 import lrccs  # noqa: E402
from test_gpu_vectors import DEV, Case  # noqa: E402

FRAC, STOP = 0.2, 4


@pytest.mark.parametrize("q,kind", [(12, "lines"), (15, "radial")])
def test_mec2_stops_where_fp64_does(q, kind):
    ny, nx, nc, r = 64, 32, 3, 2
    c = Case(ny, nx, q, nc, r, kind, 5 + q)
    gen = torch.Generator(device=DEV).manual_seed(11)
    U0 = torch.linalg.qr(torch.randn(ny * nx, r, dtype=torch.complex64, device=DEV, generator=gen))[0].contiguous()
    zbar = torch.zeros(ny * nx, dtype=torch.complex64, device=DEV)
    y, rest = c.inp[0], c.inp[1:]

    def call(scale, rel):
        s = lrccs.Solver(ny, nx, q, nc, r)
        s.set_subspace(U0, 0.0)
        s.online(y * scale, *rest, zbar, 0)
        E, _, it = s.mec2(20, rel, FRAC)
        U, B = s.factors()
        s.sync()
        s.close()
        return E.to(torch.complex128) / scale, it, (U.to(torch.complex128) @ B.to(torch.complex128).T).T

    _, _, low = call(1.0, 0.0)
    s0 = torch.stack([c.adjoint(k, c.y[k]) - c.adjoint(k, c.apply(k, low[k])) for k in range(q)])
    e, m0, ratio, peak = torch.zeros_like(s0), None, [], 0.0
    for tau in range(STOP + 1):
        ne = torch.stack([c.adjoint(k, c.apply(k, e[k])) for k in range(q)])
        m = torch.fft.fft(e + s0 - ne, dim=0, norm="ortho")
        if tau == 0:
            top = float(m.abs().max())
        else:
            ratio.append(float(torch.linalg.norm(m - m0) / torch.linalg.norm(m0)))
        a = m.abs()
        peak = max(peak, float(a.max()))
        ref = e
        e = torch.fft.ifft(torch.where(a > FRAC * top, m * (1 - FRAC * top / a.clamp_min(1e-300)), torch.zeros_like(m)),
                           dim=0, norm="ortho")
        m0 = m
    assert all(x > 1.1 * y for x, y in zip(ratio, ratio[1:]))
    rel = math.sqrt(ratio[STOP - 1] * ratio[STOP - 2])     # between the last two: STOP updates are made
    # as they are; |m|^2 of the threshold a few, of the changes less than one step of the smallest FP32 number; the
    # largest |m|^2 0.9 of the largest FP32 number, so that no sum of such squares is one
    expo = math.floor(math.log2(top))
    for scale, tol in ((1.0, 1e-4), (2.0 ** (-71 - expo), None), (0.95 * 2.0 ** 64 / peak, 1e-4)):
        E, it, _ = call(scale, rel)
        assert it == STOP
        if tol:     # FP32 transforms and sums, STOP steps
            assert float(torch.linalg.norm(E - ref)) < tol * float(torch.linalg.norm(ref))
