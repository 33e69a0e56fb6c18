"""GPU test of the FP32 chains in the GD/QR kernel's Gram sums: two columns that
agree in one large entry per block's pixels and whose other products vanish
against it, so that the chain that holds the large product loses the rest of
its own terms and nothing else; the angle between the orthonormalised columns
shows how many those were."""
import math

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2212_09664_gb300 import lrccs  # noqa: E402
from test_gpu_vectors import DEV, Case  # noqa: E402

BIG, SMALL = 4096.0, (1.4, 0.7)    # BIG^2 = 2^24, whose FP32 neighbours are 2 apart: 1.4 x 0.7 = 0.98 is lost


def test_gram_chains_are_no_longer_than_the_block_allows():
    ny, nx, r = 256, 256, 16
    n = ny * nx
    per = -(-n // min(n // 32, torch.cuda.get_device_properties(0).multi_processor_count))
    tiles = (r // 2) * (r // 2 + 1) // 2                    # 2 x 2 tiles of the upper triangle, 512 threads
    W = torch.zeros(n, r, dtype=torch.complex64, device=DEV)
    for c, v in enumerate(SMALL):
        W[:, c] = v
        W[::per, c] = BIG
    for c in range(2, r):                                   # the other columns: one entry each, in different blocks
        W[c * per + 7, c] = 100.0
    inp = Case(ny, nx, 2, 1, 2, "lines", 3).inp
    s = lrccs.Solver(ny, nx, 2, 1, r)
    s.set_subspace(W, 0.0)
    s.online(*inp, torch.zeros(n, dtype=torch.complex64, device=DEV), 0)    # orthonormalises the subspace and keeps it
    U = s.subspace()[:, :2].to(torch.complex128)
    torch.cuda.synchronize()
    a, b = U[:, 0], U[:, 1]
    angle = float((a.conj() @ b).abs() / (torch.linalg.norm(a) * torch.linalg.norm(b)))
    # lost: at most one chain's terms per block, with as many chains as the threads make slices; 6 more for the
    # roundings of the sums and the division at 2^24.  The second column's part off the first has norm 0.7 sqrt(per)
    bound = (SMALL[0] * SMALL[1] * -(-per // (512 // tiles)) + 6) / (BIG * SMALL[1] * math.sqrt(per))
    assert angle < bound
    s.close()
