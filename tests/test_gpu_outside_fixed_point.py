"""Propagation outside the fixed-point range: the FP64 sweeps that take such a class or such a slice, against
the oracle and at their own split of the instances."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RTOL_SERIES = 1e-9   # as in test_gpu_parity
GS_KW = dict(dtau=0.1, max_iter=1500, tol=0.0)


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


def _rel(x, ref):
    return float(np.max(np.abs(np.asarray(x) - np.asarray(ref))) / max(np.max(np.abs(ref)), 1e-4))


@pytest.mark.parametrize("scheme,n,N,lanes", [(0, 40, 2048, 1), (0, 3, 2048, 8), (0, 2, 8192, 32), (1, 40, 2048, 1), (1, 3, 2048, 8),
                                              (1, 2, 8192, 32)])
def test_slices_outside_the_range_run_at_the_fp64_split(env, scheme, n, N, lanes):
    """With every slice out of range (a field for FULL_CN, the norm for NUMEROV_SPLIT) the default launch, whose
    fixed-point split has 13 or 14 warps in most of these batches, gives the bits of a launch of the FP64 rule's 8
    warps: the instances are split the same way, so the sums are formed in the same order."""
    tdse, _ = env
    dt, nt = 0.05, 20
    out = []
    for warps in (0, 8):
        b = tdse.Batch([N] * n, 0.2, 1.19, [nt] * n, dt, absorber=(20.0, 0.125), scheme=scheme, lanes_per_instance=lanes)
        b.set_launch(warps_per_cta=warps)
        b.ground_state(**GS_KW)
        if scheme == 1:
            b.load_state(b.save_state() * 1e16)
        E = torch.full((n * (nt + 1),), 0.04 if scheme else 5.0, dtype=torch.float64, device="cuda")
        d, a = torch.zeros_like(E), torch.zeros_like(E)
        b.propagate(E, d, a)
        out.append((d, a, b.get_psi(0), b.get_psi(n - 1)))
        b.close()
    for x, y in zip(*out):
        assert torch.equal(x, y)


@pytest.mark.parametrize("N,lanes,dt,scale", [(401, 1, 0.1, 1.0), (401, 8, 0.1, 1.0), (1001, 32, 0.1, 1.0), (402, 1, 0.05, 1e16),
                                              (401, 8, 0.05, 1e16)])
def test_numerov_split_fp64_sweeps(env, N, lanes, dt, scale):
    """NUMEROV_SPLIT in double: a time step whose factors leave the fixed-point range (decay 0.42), odd grids
    among them, and states of a norm beyond it beside others in the range."""
    tdse, oracle = env
    from paper_2507_04115_gb300 import inputs
    dx, a, nt = 0.2, 1.19, 90
    sizes = [N, N, N, 502]
    rows = [inputs.sin2_pulse(nt, dt, 0.05 + 0.01 * i, 0.057, 1.0, 0.3 * i) for i in range(4)]
    offs = np.arange(5) * (nt + 1)
    Et = torch.from_numpy(np.concatenate(rows)).cuda()
    b = tdse.Batch(sizes, dx, a, nt, dt, absorber=(20.0, 0.125), scheme=tdse.TDSE_NUMEROV_SPLIT, lanes_per_instance=lanes)
    b.ground_state(**GS_KW)
    s = [1.0, scale, 1.0, 1.0]
    b.set_psi(1, b.get_psi(1) * s[1])
    d, acc = torch.zeros_like(Et), torch.zeros_like(Et)
    b.propagate(Et, d, acc)
    for i, n in enumerate(sizes):
        psi0, _, _ = oracle.ground_state(n, dx, a, scheme=oracle.NUMEROV_SPLIT, **GS_KW)
        psi, d_o, a_o = oracle.propagate(psi0, rows[i], dx, dt, a, scheme=oracle.NUMEROV_SPLIT,
                                         mask_values=oracle.mask(n, dx, 20.0, 0.125))
        sl = slice(offs[i], offs[i + 1])
        assert _rel(d[sl].cpu().numpy() / s[i] ** 2, d_o) < RTOL_SERIES, i
        assert _rel(acc[sl].cpu().numpy() / s[i] ** 2, a_o) < RTOL_SERIES, i
        assert float((b.get_psi(i).cpu() / s[i] - torch.from_numpy(psi)).abs().max()) < 1e-12, i
    b.close()


@pytest.mark.parametrize("N,dx,dt,lanes", [(512, 0.2, 0.05, 8), (511, 0.1, 0.02, 1), (511, 0.2, 0.01, 8)])
def test_full_cn_fp64_sweeps(env, N, dx, dt, lanes):
    """FULL_CN in double: lane-split groups of which some meet a field beyond the range for some slices, and grids
    above and below the range of dt / (4 dx^2)."""
    tdse, oracle = env
    a, nt, n = 1.19, 96, 12
    rows = [np.full(nt + 1, 0.02) for _ in range(n)]
    for i in (0, 9):
        rows[i][40:50] = 6.0
    offs = np.arange(n + 1) * (nt + 1)
    Et = torch.from_numpy(np.concatenate(rows)).cuda()
    b = tdse.Batch([N] * n, dx, a, nt, dt, absorber=(10.0, 0.125), lanes_per_instance=lanes)
    b.ground_state(**GS_KW)
    d, acc = torch.zeros_like(Et), torch.zeros_like(Et)
    b.propagate(Et, d, acc)
    assert b.check() == -1
    psi0, _, _ = oracle.ground_state(N, dx, a, **GS_KW)
    m = oracle.mask(N, dx, 10.0, 0.125)
    for i in (0, 1, 9, n - 1):
        _, d_o, a_o = oracle.propagate(psi0, rows[i], dx, dt, a, mask_values=m)
        sl = slice(offs[i], offs[i + 1])
        assert _rel(d[sl].cpu().numpy(), d_o) < RTOL_SERIES and _rel(acc[sl].cpu().numpy(), a_o) < RTOL_SERIES, i
    b.close()


@pytest.mark.parametrize("dx,dt,kc,field,lanes", [(0.2, 0.05, 37, 8.0, 1), (0.2, 0.05, 37, 8.0, 4), (0.1, 0.02, 37, 0.05, 1),
                                                  (0.1, 0.02, 37, 0.05, 4), (0.2, 0.05, 400, 0.05, 1), (0.2, 0.05, 400, 0.05, 4)])
def test_gamma_tape_of_the_fp64_adjoint(env, dx, dt, kc, field, lanes):
    """The FP64 adjoint with and without its gamma tape gives the same bits, through both entry points: groups that
    the fixed-point adjoint leaves (a field beyond the range), a class without that form, and an interval longer than
    the grid.  Dropping the tape gives memory back, so it was there."""
    tdse, oracle = env
    rng = np.random.default_rng(kc)
    n, N, a, nt = 35, 384, 1.19, 120
    E = rng.uniform(-field, field, n * (nt + 1))
    Et = torch.from_numpy(E).cuda()
    gd, ga = (torch.from_numpy(rng.standard_normal(E.size)).cuda() for _ in range(2))
    b = tdse.Batch([N] * n, dx, a, [nt] * n, dt, absorber=(10.0, 0.125), lanes_per_instance=lanes)
    b.ground_state(**GS_KW)
    psi0 = b.save_state()
    d, acc = torch.zeros_like(Et), torch.zeros_like(Et)
    out, free = [], []
    for tape in (True, False):
        b.set_adjoint_gamma_tape(tape)
        b.load_state(psi0)
        one = b.adjoint(Et, gd, ga, ckpt_every=kc)
        b.propagate_checkpointed(Et, d, acc, kc)
        out.append((one, b.adjoint_checkpointed(Et, gd, ga)))
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert free[1] - free[0] >= (4 << 20), free
    p, m = oracle.ground_state(N, dx, a, **GS_KW)[0], oracle.mask(N, dx, 10.0, 0.125)
    for i in (0, 17, n - 1):
        sl = slice(i * (nt + 1), (i + 1) * (nt + 1))
        ref = oracle.adjoint(p, E[sl], dx, dt, a, gd[sl].cpu().numpy(), ga[sl].cpu().numpy(), mask_values=m)
        for g in out[0]:
            assert _rel(g[sl].cpu().numpy(), ref) < RTOL_SERIES, i
    b.close()
