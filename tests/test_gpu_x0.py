"""GPU test of LRCCS_BUF_X0 after every call that loads data: the loaded data's
adjoint, truncated at the gamma of the last lrccs_init and scaled, against FP64
torch; zeros in a context that has no gamma."""
import numpy as np
import pytest

from paper_2212_09664_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2212_09664_gb300 import lrccs  # noqa: E402

DEV = torch.device("cuda:0")
NY, NX, Q, NC, R = 64, 96, 18, 3, 2


def load(kind, seed, scale):
    rng = np.random.default_rng(seed)
    mask = synth.cartesian_lines_vd(rng, NY, NX, Q, 4.0) if kind == "lines" else synth.radial_golden(NY, NX, Q, 6)
    idx, fp = synth.compact_mask(mask)
    y = rng.standard_normal(NC * fp[-1]) + 1j * rng.standard_normal(NC * fp[-1])
    y[rng.random(y.size) < 0.01] *= 30.0
    y = (scale * y).astype(np.complex64)
    sm = (rng.standard_normal((NC, NY * NX)) + 1j * rng.standard_normal((NC, NY * NX))).astype(np.complex64)
    return idx, tuple(torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (y, fp, mask, sm))


def x0_of(idx, inp, gamma):
    y, fp, d = inp[0].to(torch.complex128), inp[1].cpu().numpy(), inp[3].to(torch.complex128)
    kept = torch.where(y.real ** 2 + y.imag ** 2 <= gamma, y, torch.zeros_like(y))
    assert 0 < int((kept != y).sum()) < y.numel() // 2
    out = torch.zeros((NY * NX, Q), dtype=torch.complex128, device=DEV)
    for k in range(Q):
        f = torch.zeros((NC, NY * NX), dtype=torch.complex128, device=DEV)
        at = torch.from_numpy(idx[fp[k]:fp[k + 1]].astype(np.int64)).to(DEV)
        f[:, at] = kept[NC * fp[k]:NC * fp[k + 1]].reshape(NC, -1)
        z = torch.fft.ifft2(f.reshape(NC, NY, NX), norm="ortho").reshape(NC, -1)
        out[:, k] = (d.conj() * z).sum(0) / np.sqrt(float(fp[k + 1] - fp[k]) * fp[-1] / Q)
    return out


@pytest.mark.parametrize("kind", ["lines", "radial"])
def test_x0_is_the_loaded_datas(kind):
    (_, first), (i2, second), (i3, third) = load(kind, 1, 1.0), load(kind, 2, 1.5), load(kind, 3, 0.7)
    U = torch.linalg.qr(torch.randn(NY * NX, R, dtype=torch.complex64, device=DEV))[0].contiguous()
    s = lrccs.Solver(NY, NX, Q, NC, R)

    def x0():
        b = s.buffer(lrccs.BUF_X0)
        s.sync()
        torch.cuda.synchronize()
        return b

    assert not x0().any()
    s.set_subspace(U, 1e-6)
    s.track(*second, t_max=1)
    assert not x0().any()
    s.init(*first)
    gamma = float(s.buffer(lrccs.BUF_SCAL)[0])
    s.track(*second, t_max=1)
    ref = x0_of(i2, second, gamma)
    # two FP32 transforms and a coil sum: a few roundings of 6e-8
    assert float(torch.linalg.norm(x0() - ref)) < 1e-6 * float(torch.linalg.norm(ref))
    s.mean_step(*third, max_iter=1)
    ref = x0_of(i3, third, gamma)
    assert float(torch.linalg.norm(x0() - ref)) < 1e-6 * float(torch.linalg.norm(ref))
    with pytest.raises(lrccs.LrccsError):      # the frame offsets of another mask; gamma is cleared
        s.init(second[0], second[1] + 1, second[2], second[3])
    s.set_subspace(U, 1e-6)
    s.track(*second, t_max=1)
    assert not x0().any()
    s.close()
