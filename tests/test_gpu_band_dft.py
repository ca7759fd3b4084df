"""Fourier sums by block moments (tdse_spectrum and tdse_dipole_spectrum over a band of low frequencies)
against numpy: block edges (rows one sample short of, at and past a multiple of the block), ragged rows,
one row and many, every number of moments, and the direct sum where the band is too wide.  The bound is
1e-12 of the largest value of a row, the rounding of sums of this length with room."""
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


def _rows(rng, lens):
    offs = np.concatenate([[0], np.cumsum(lens)])
    t = np.arange(max(lens))
    a = np.concatenate([np.cos(0.013 * t[:L] + 0.1 * i) * np.sin(np.pi * t[:L] / L) ** 2 + 0.1 * rng.standard_normal(L)
                        for i, L in enumerate(lens)])
    return offs, a


@pytest.mark.parametrize("lens,k0,k1", [([4096] * 5, 0, 64), ([4095] * 4, 0, 200), ([4097] * 9, 13, 300), ([20011], 0, 400),
                                        ([6000, 5555, 9001, 6000], 0, 180), ([1000] * 3, 0, 400), ([300] * 2, 0, 40),
                                        ([55160] * 2, 0, 129), ([50000] * 4, 4000, 4040)])
def test_power_spectrum_of_a_band(tdse, lens, k0, k1):
    rng = np.random.default_rng(len(lens) + k1)
    offs, a = _rows(rng, lens)
    S = tdse.spectrum(torch.from_numpy(a).cuda(), offs, 0.02, k0, k1).cpu().numpy()
    for r, L in enumerate(lens):
        ref = 0.02 ** 2 * np.abs(np.fft.fft(a[offs[r]:offs[r + 1]])) ** 2
        want = ref[np.arange(k0, k1) % L]
        assert np.max(np.abs(S[r] - want)) <= 1e-12 * want.max(), (r, L)


@pytest.mark.parametrize("lens,top,n_w", [([4096] * 6, 0.05, 100), ([5000, 1, 0, 3333, 512], 0.03, 70), ([30000], 0.004, 33),
                                          ([2048] * 5, 0.4, 600), ([2048] * 5, 1.5, 40), ([900] * 4, 0.0, 40)])
def test_dipole_spectrum_of_a_band(tdse, lens, top, n_w):
    """Frequencies of both signs and zero; top: the largest turn per sample."""
    rng = np.random.default_rng(n_w)
    offs, a = _rows(rng, lens) if min(lens) > 0 else (np.concatenate([[0], np.cumsum(lens)]), rng.standard_normal(sum(lens)))
    dt = 0.02
    om = np.linspace(-0.3 * top, top, n_w) / dt
    wt = rng.uniform(0.5, 2.0, len(lens))
    got = tdse.dipole_spectrum(torch.from_numpy(a).cuda(), offs, dt, om, weight=torch.from_numpy(wt).cuda()).cpu().numpy()
    for r, L in enumerate(lens):
        ph = np.outer(np.arange(L), om * dt)
        want = wt[r] * dt / np.sqrt(2 * np.pi) * (a[offs[r]:offs[r + 1]] @ np.exp(1j * ph)) if L else np.zeros(n_w)
        assert np.max(np.abs(got[r] - want)) <= 1e-12 * max(np.max(np.abs(want)), 1e-300), (r, L)
