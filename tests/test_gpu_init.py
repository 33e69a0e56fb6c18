"""GPU tests of the data load (mask structure, gamma, Z and X0) against FP64
torch: single frames, frame counts around the chunk width, rows sampled by few
and by every frame, outliers that the truncation drops, values outside the FP32
range of squares."""
import numpy as np
import pytest

from paper_2212_09664_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2212_09664_gb300 import lrccs  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("ny,nx,q,nc,kind,scale", [
    (32, 32, 1, 1, "lines", 1.0), (64, 32, 16, 2, "lines", 1e-18), (96, 64, 17, 5, "lines", 1.0),
    (32, 96, 33, 3, "radial", 1e17), (64, 128, 9, 20, "radial", 1.0), (160, 160, 5, 4, "lines", 1.0),
    (192, 224, 20, 3, "radial", 1.0), (256, 256, 4, 33, "radial", 1.0), (128, 192, 128, 2, "lines", 1.0)])
def test_data_load_matches_torch(ny, nx, q, nc, kind, scale):
    n = ny * nx
    rng = np.random.default_rng(ny + nx + q)
    if kind == "lines":
        mask = synth.cartesian_lines_vd(rng, ny, nx, q, 4.0)
        mask[0] = 0
        mask[0].reshape(ny, nx)[[0, ny // 2]] = 1       # frames of different length
    else:
        mask = synth.radial_golden(ny, nx, q, 5)
        mask[:, 0] = 1
    idx, fp = synth.compact_mask(mask)
    y = rng.standard_normal(nc * fp[-1]) + 1j * rng.standard_normal(nc * fp[-1])
    y[rng.random(y.size) < 0.002] *= 40.0                # outliers above 6 x RMS
    y = (y * scale).astype(np.complex64)
    sm = (rng.standard_normal((nc, n)) + 1j * rng.standard_normal((nc, n))).astype(np.complex64)
    s = lrccs.Solver(ny, nx, q, nc, 1)
    inp = tuple(torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (y, fp, mask, sm))
    s.init(*inp)
    Z, X0, sc = s.buffer(lrccs.BUF_Z), s.buffer(lrccs.BUF_X0), s.buffer(lrccs.BUF_SCAL)
    got = torch.empty(int(fp[-1]), dtype=torch.int32, device=DEV)
    lrccs.lrccs_get_buffer(s.ctx, lrccs.BUF_IDX, got)
    s.sync()
    torch.cuda.synchronize()
    assert np.array_equal(got.cpu().numpy(), idx)
    y64 = y.astype(np.complex128)
    sq = y64.real ** 2 + y64.imag ** 2
    gamma = 36.0 * np.sum(sq) / y.size
    assert abs(float(sc[0]) / gamma - 1.0) < 1e-12
    keep = sq <= float(sc[0])
    assert (~keep).any() or y.size < 5000
    d = inp[3].to(torch.complex128)
    m = np.diff(fp)
    for ref, buf, drop in ((None, Z, False), (None, X0, True)):
        ref = torch.zeros((n, q), dtype=torch.complex128, device=DEV)
        for k in range(q):
            a, b = nc * fp[k], nc * fp[k + 1]
            v = (y64[a:b] * keep[a:b] if drop else y64[a:b]).reshape(nc, -1)
            f = torch.zeros((nc, n), dtype=torch.complex128, device=DEV)
            f[:, torch.from_numpy(idx[fp[k]:fp[k + 1]].astype(np.int64)).to(DEV)] = torch.from_numpy(v).to(DEV)
            z = torch.fft.ifft2(f.reshape(nc, ny, nx), norm="ortho").reshape(nc, n)
            ref[:, k] = (d.conj() * z).sum(0) * (1.0 / np.sqrt(m[k] * (fp[-1] / q)) if drop else 1.0)
        # two FP32 transforms and a coil sum: a few roundings of 6e-8
        assert float(torch.linalg.norm(buf - ref)) < 1e-6 * float(torch.linalg.norm(ref))
    s.close()
