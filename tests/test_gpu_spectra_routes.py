"""Spectra and far field by every route: the direct sums on a capturing stream and without room for the moments, CUDA's j0
where the table does not pay and beyond its end."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_04115_gb300 import build, tdse
    build.build()
    tdse.load()
    import oracle
    oracle.build()
    return tdse, oracle


@pytest.mark.parametrize("n_rho,n_z,n_obs,ro_max", [(64, 128, 128, 8e-3), (40, 24, 150, 4e-3), (5, 4, 200, 8e-3), (1, 1, 3, 1e-3), (40, 24, 20, 0.0)])
def test_hankel_arguments_beyond_the_table(env, n_rho, n_z, n_obs, ro_max):
    """Arguments k rho rho' / D to 17000, where the table ends at 4096; few source points, which take j0 throughout;
    radius 0 alone.  A term's argument and phases, below 3e4 rad together, are rounded a few times each: about 2e-11 of
    it, below the bound of the other far-field tests."""
    tdse, oracle = env
    rng = np.random.default_rng(n_rho)
    k = 2 * np.pi / np.array([40e-9, 52e-9, 61e-9])
    rho = np.linspace(0.0, 8e-3, n_rho) if n_rho > 1 else np.array([8e-3])
    z = np.linspace(-5e-5, 5e-5, n_z) if n_z > 1 else np.array([0.0])
    ro = np.linspace(0.0, ro_max, n_obs) if ro_max > 0 else np.zeros(1)
    S = rng.standard_normal((n_rho, n_z, k.size)) + 1j * rng.standard_normal((n_rho, n_z, k.size))
    E = tdse.hankel(torch.from_numpy(S).cuda(), rho, z, k, 0.6, ro).cpu().numpy()
    ref = oracle.hankel_far_field(S, rho, z, k, 0.6, ro)
    for w in range(k.size):
        assert np.max(np.abs(E[w] - ref[w])) <= 1e-10 * np.max(np.abs(ref[w])), w


@pytest.mark.parametrize("dipole", [False, True])
def test_spectra_replay_from_a_graph(env, dipole):
    """A captured call sums directly and replays on new samples; the bound is that of the moments' test."""
    tdse, _ = env
    rng = np.random.default_rng(3)
    L, rows, dt = 9000, 5, 0.02
    offs = np.arange(rows + 1) * L
    om = np.linspace(0.1, 2.0, 64)
    x = torch.from_numpy(rng.standard_normal(rows * L)).cuda()
    a = x.clone()
    out = torch.zeros((rows, 64), dtype=torch.complex128 if dipole else torch.float64, device="cuda")

    def call(stream=None):
        if dipole:
            tdse.dipole_spectrum(a, offs, dt, om, out=out, stream=stream)
        else:
            tdse.spectrum(a, offs, dt, 0, 64, out=out, stream=stream)

    call()   # (not captured: by the moments)
    ref = out.clone()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        call(s)
    for scale in (1.0, 3.0):
        a.copy_(x * scale)
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        want = ref * (scale if dipole else scale * scale)
        assert float((out - want).abs().max()) <= 1e-12 * float(want.abs().max())


def test_spectra_without_room_for_the_moments(env):
    """With 160 MB of the device left a call whose moments take 262 MB sums directly: the bits of a captured call, which
    does so too, and not those of the moments."""
    tdse, _ = env
    rows, L, k0, k1, dt = 400, 65536, 6200, 6240, 0.02
    offs = np.arange(rows + 1) * L
    a = torch.randn(rows * L, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    om = np.arange(k0, k1) * (2 * np.pi / (L * dt))
    S = torch.empty((rows, k1 - k0), dtype=torch.float64, device="cuda")
    D = torch.empty((rows, k1 - k0), dtype=torch.complex128, device="cuda")

    def calls(stream=None):
        tdse.spectrum(a, offs, dt, k0, k1, out=S, stream=stream)
        tdse.dipole_spectrum(a, offs, dt, om, out=D, stream=stream)

    def result():
        torch.cuda.synchronize()
        r = S.cpu(), D.cpu()
        S.zero_()
        D.zero_()
        return r

    calls()
    moments = result()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        calls(s)
    graph.replay()
    direct = result()
    del graph
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (160 << 20), dtype=torch.uint8, device="cuda")
    try:
        calls()
        got = result()
    finally:
        del fill
        torch.cuda.empty_cache()
    for k in range(2):
        assert torch.equal(got[k], direct[k]) and not torch.equal(got[k], moments[k])
