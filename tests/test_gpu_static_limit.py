"""tdse_propagate_static at the limit of its scratch: the largest batch that the FP64 sweep's tables leave room for is
accepted, without the fixed-point form where that form's tables do not fit, and the next one refused."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _need(groups, N):
    """Bytes of the scratch (64 MB) with a class's 20 N doubles of tables and one CTA of 8 warps."""
    a = lambda v: (v + 255) // 256 * 256
    return a(256) + a(56 * groups) + 2 * a(256 * groups) + 2 * a(4 * groups) + a(128 * groups) + a(160 * N) + 16 * 8 * N * 64


def test_largest_batch():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_04115_gb300 import build, tdse
    build.build()
    tdse.load()
    N, nt = 64, 3
    g = 90000
    while _need(g + 1, N) <= 64 << 20:
        g += 1
    psi = torch.zeros(2 * 32 * (g + 1) * N, dtype=torch.float64, device="cuda")
    E, d, a = (torch.zeros(32 * (g + 1) * (nt + 1), dtype=torch.float64, device="cuda") for _ in range(3))
    call = lambda n: tdse.tdse_propagate_static((N, 0.2, 1.19, 1.0), n, 0.05, nt, nt + 1, psi, E, d, a, 2, 2, absorber=None)
    call(32 * g)          # an empty step range: 94564 groups on the one CTA that is left would take minutes
    torch.cuda.synchronize()
    with pytest.raises(tdse.TDSEError):
        call(32 * (g + 1))
