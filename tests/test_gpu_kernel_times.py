"""emri_ctx_kernel_times counts launches: together with the LISA phase table,
which has no kind of its own, they are the launches the context counts."""
import pytest

from paper_2311_17174_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("mixed,groups", [(False, 1), (True, 1), (True, 2)])
def test_launch_counts(mixed, groups):
    from paper_2311_17174_gb300 import emri as E
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = E.Context(0)
    n, dt, w = 1 << 14, 15.0, 6
    prec = E.MIXED if mixed else E.FP64
    psd = I.psd_bc04(n, dt)
    ds = ctx.dataset(E.grid(n, dt), I.noise_spectrum(7, psd, n, dt), psd, 1e-4, 1.0)
    theta = torch.tensor(I.draw_sources(8, w, n).T.copy(), device="cuda:0")
    lnl = torch.zeros(w, dtype=torch.float64, device="cuda:0")
    ctx.set_pipeline(prec, groups)
    ctx.profile(True)
    before = ctx.launches()
    calls = 3
    for _ in range(calls):
        ctx.loglike_batch(ds, theta, E.opts(precision=prec, n_max=4), lnl)
    launched = ctx.launches() - before
    kt = ctx.kernel_times()
    ctx.profile(False)
    assert sum(c for _, c in kt.values()) + calls == launched
    # the orbit step: nine launches a group, and the mixed interval records
    assert kt["orbit"][1] == calls * groups * (10 if mixed else 9)
    assert all(ms > 0 for name, (ms, c) in kt.items() if c)
    ds.close()
    ctx.close()
