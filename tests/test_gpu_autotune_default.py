"""The autotuner times the planner's own launch among its candidates, so a tuned batch is not slower than an untuned one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N,precision,scheme", [(20000, 1024, 0, 0), (3, 2000, 0, 0), (300, 1024, 0, 1), (300, 1024, 1, 0)])
def test_default_launch_is_a_candidate(n, N, precision, scheme):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2507_04115_gb300 import build, tdse
    build.build()
    tdse.load()
    nt = 8
    b = tdse.Batch([N] * n, 0.2, 1.19, [nt] * n, 0.05, precision=precision, scheme=scheme)
    b.ground_state(max_iter=20, tol=0.0)
    p = b.plan()
    E = torch.full((n * (nt + 1),), 0.03, dtype=torch.float64, device="cuda")
    d, a = torch.zeros_like(E), torch.zeros_like(E)
    before = b.save_state()
    trials = b.autotune(E, d, a, repeats=2)
    default = [t for t in trials if (t["warps_per_cta"], t["ctas"], t["slice_steps"]) == (p["warps_per_cta"], p["ctas"], p["slice_steps"])]
    assert default and min(t["ms"] for t in trials) <= default[0]["ms"]
    assert len(trials) == len({(t["warps_per_cta"], t["ctas"], t["slice_steps"]) for t in trials})
    best = min(trials, key=lambda t: t["ms"])
    q = b.plan()
    assert (q["warps_per_cta"], q["ctas"], q["slice_steps"]) == (best["warps_per_cta"], best["ctas"], best["slice_steps"])
    assert torch.equal(b.save_state(), before)
    # the trial's numbers give its shape
    b.set_launch(best["warps_per_cta"], best["ctas_per_sm"], best["slice_steps"])
    r = b.plan()
    assert (r["warps_per_cta"], r["ctas"], r["slice_steps"], r["segments"]) == (q["warps_per_cta"], q["ctas"], q["slice_steps"], q["segments"])
    b.close()
