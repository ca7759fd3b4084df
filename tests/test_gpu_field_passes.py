"""tdse_resample_field by its passes and routes, against the interpolant's sum in numpy."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tdse():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_04115_gb300 import build, tdse
    build.build()
    tdse.load()
    return tdse


def _interpolant(row, dt_c, t):
    M = row.size
    k = np.arange(M // 2 + 1)
    c = np.fft.rfft(row) / M * np.where((k == 0) | (2 * k == M), 1.0, 2.0)
    u = np.mod(t / (M * dt_c), 1.0)
    return (np.exp(2j * np.pi * np.outer(u, k)) @ c).real


@pytest.mark.parametrize("rows,M,n_fine", [(3, 2400, 1016802), (9, 600, 2100000)])
def test_outputs_of_several_passes(tdse, rows, M, n_fine):
    """More outputs than a pass holds (1016801): sampled across the passes' edges and at random."""
    rng = np.random.default_rng(n_fine)
    coarse = rng.standard_normal((rows, M))
    dt_c, dt_f = 0.8, 0.8 * 1.1 * M / n_fine
    out = tdse.resample_field(torch.from_numpy(coarse).cuda(), dt_c, dt_f, n_fine, out_stride=n_fine + 3)
    assert torch.all(out[:, n_fine:] == 0.0)
    edge = [e + k for e in (0, 1016801, 2033602, n_fine) for k in range(-3, 3)]
    n = np.unique([i for i in edge + list(rng.integers(0, n_fine, 200)) if 0 <= i < n_fine])
    got = out[:, torch.from_numpy(n).cuda()].cpu().numpy()
    for r in range(rows):
        assert np.max(np.abs(got[r] - _interpolant(coarse[r], dt_c, n * dt_f))) < 2e-11 * np.max(np.abs(coarse[r]))


@pytest.mark.parametrize("rows,M,n_fine", [(1, 2, 300), (40, 2, 257), (1, 3, 100), (1, 100, 400001), (8, 127, 9000), (7, 128, 9000),
                                           (7, 129, 9000), (1, 1500, 200000), (3, 300, 12000)])
def test_direct_sums(tdse, rows, M, n_fine):
    """Few coefficients and rows, summed directly: odd and even M, one coefficient more and fewer than a block of 64,
    outputs past the window, the largest M of the route."""
    rng = np.random.default_rng(M)
    coarse = rng.standard_normal((rows, M))
    dt_c, dt_f = 0.5, 0.5 * 1.3 * M / n_fine
    out = tdse.resample_field(torch.from_numpy(coarse).cuda(), dt_c, dt_f, n_fine, out_stride=n_fine + 3)
    assert torch.all(out[:, n_fine:] == 0.0)
    n = np.unique(np.concatenate([np.arange(3), rng.integers(0, n_fine, 300), [n_fine - 1]]))
    got = out[:, torch.from_numpy(n).cuda()].cpu().numpy()
    for r in range(rows):
        assert np.max(np.abs(got[r] - _interpolant(coarse[r], dt_c, n * dt_f))) < 2e-11 * np.max(np.abs(coarse[r]))
