"""GPU test of the tracking call's inputs: the frame offsets, the mask and the
coil maps are copied, so the caller may overwrite them from any stream once the
call has returned, whatever else keeps the GPU busy then."""
import numpy as np
import pytest

from paper_2212_09664_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2212_09664_gb300 import lrccs  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("kind", ["lines", "radial"])
def test_track_inputs_are_the_callers_again_on_return(kind):
    ny, nx, q, nc, r = 256, 256, 8, 32, 4
    rng = np.random.default_rng(7)
    mask = synth.cartesian_lines_vd(rng, ny, nx, q, 8.0) if kind == "lines" else synth.radial_golden(ny, nx, q, 8)
    _, fp = synth.compact_mask(mask)
    gen = torch.Generator(device=DEV).manual_seed(3)
    y = torch.randn(nc * int(fp[-1]), dtype=torch.complex64, device=DEV, generator=gen)
    maps = torch.randn(nc, ny * nx, dtype=torch.complex64, device=DEV, generator=gen)
    U = torch.linalg.qr(torch.randn(ny * nx, r, dtype=torch.complex64, device=DEV, generator=gen))[0].contiguous()
    fp, mask = torch.from_numpy(np.ascontiguousarray(fp)).to(DEV), torch.from_numpy(mask).to(DEV)
    own, other, busy = torch.cuda.Stream(), torch.cuda.Stream(priority=-1), torch.cuda.Stream()
    a = torch.randn(4096, 4096, device=DEV, generator=gen)
    s = lrccs.Solver(ny, nx, q, nc, r, stream=own)
    X = [torch.zeros(q, ny * nx, dtype=torch.complex64, device=DEV) for _ in range(2)]
    torch.cuda.synchronize()
    for k in range(2):
        inp = [t.clone() for t in (fp, mask, maps)]
        torch.cuda.synchronize()
        s.set_subspace(U, 1e-9)
        if k == 1:
            with torch.cuda.stream(busy):
                for _ in range(40):
                    a @ a
        s.track(y, *inp, t_max=1, X=X[k])
        with torch.cuda.stream(other):
            for t in inp:
                t.zero_()
        s.sync()
        torch.cuda.synchronize()
    assert float(X[0].abs().sum()) > 0 and torch.equal(X[0], X[1])
    s.close()
