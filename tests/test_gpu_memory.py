"""GPU tests of the optional transform buffers: they never take the memory that
the caller reserves, they are given back when a call needs their memory, and
the narrow transforms that run without them give the same results."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2212_09664_gb300 import lrccs  # noqa: E402
from test_gpu_vectors import DEV, Case, rel  # noqa: E402

MIB = 1 << 20


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def cache_outputs():
    """Let the caching allocator hold what the outputs of a run take, so that a run's device memory is the library's."""
    torch.empty(512 * MIB, dtype=torch.uint8, device=DEV)


def run(c, rank, rank_max, params=None, between=lambda: None):
    s = lrccs.Solver(c.ny, c.nx, c.q, c.nc, rank, rank_max, params)
    s.init(*c.inp)
    Z = s.buffer(lrccs.BUF_Z)
    s.iterate(2)
    between()
    E, X = s.mec1(2)
    s.sync()
    left = free_bytes()
    s.close()
    return Z, E, X, left


@pytest.mark.parametrize("kind", ["lines", "radial"])
def test_reserved_memory_stays_free(kind):
    c = Case(192, 192, 17, 32, 2, kind, 9)
    cache_outputs()
    wide = run(c, 2, 2)
    # room for the context, the general masks' buffers and the frames' vectors, not for 16 columns (144 MiB)
    params = lrccs.default_params()
    need = lrccs.lrccs_context_bytes(192, 192, 17, 32, 2, 2)
    params.admit_reserve_bytes = float(free_bytes() - need - 100 * MIB)
    narrow = run(c, 2, 2, params)
    assert wide[3] < params.admit_reserve_bytes <= narrow[3]
    # two transforms and, for E, two CG steps in FP32 with differently grouped coil sums
    assert rel(narrow[0], wide[0]) < 1e-6
    assert rel(narrow[2], wide[2]) < 3e-6
    assert float(torch.linalg.norm(narrow[1] - wide[1])) < 3e-6 * float(torch.linalg.norm(wide[2]))


@pytest.mark.parametrize("kind", ["lines", "radial"])
def test_optional_memory_is_given_back(kind):
    """The frames' vectors (5 q n complex values, 168 MB) fit only without the widened transform buffers."""
    c = Case(256, 256, 64, 16, 1, kind, 10)
    cache_outputs()
    wide = run(c, 1, 1)
    params = lrccs.default_params()
    params.admit_reserve_bytes = 0.0
    fill = []

    def leave():          # 30 MiB short of the vectors; giving 126 MB of T back covers it
        fill.append(torch.empty(free_bytes() - 130 * MIB, dtype=torch.uint8, device=DEV))

    got = run(c, 1, 1, params, leave)
    fill.clear()
    torch.cuda.empty_cache()
    assert rel(got[0], wide[0]) < 1e-6 and rel(got[2], wide[2]) < 3e-6


@pytest.mark.parametrize("kind", ["lines", "radial"])
def test_iterations_and_batches_go_on_after_a_buffer_has_grown(kind):
    """Captured iterations hold the work buffers' addresses; model-error correction grows them in between."""
    c = Case(96, 64, 17, 3, 2, kind, 11)
    res = []
    for grow in (False, True):
        solo, stream = torch.cuda.Stream(), torch.cuda.Stream()
        a = lrccs.Solver(c.ny, c.nx, c.q, c.nc, 2, stream=solo)
        b = lrccs.Solver(c.ny, c.nx, c.q, c.nc, 2, stream=stream)
        batch = lrccs.lrccs_batch_create([b.ctx], stream)
        torch.cuda.synchronize()
        for s, step in ((a, a.iterate), (b, lambda n: lrccs.lrccs_batch_iterate(batch, n))):
            with torch.cuda.stream(s.stream):
                s.init(*c.inp)
                step(4)
                s.sync()
                if grow:
                    s.mec1(1)
                step(4)
                s.sync()
                res.append(s.subspace())
        torch.cuda.synchronize()
        lrccs.lrccs_batch_destroy(batch)
        a.close()
        b.close()
    assert all(torch.equal(res[0], u) for u in res[1:])
