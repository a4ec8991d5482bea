"""The per-walker constants of walkers whose gravitational-wave distance is
not positive (Xi0 far below zero): flagged EMRI_ST_BADPARAM, and like every
flagged walker they have no delay, in emri_prologue's output and in the
likelihood's."""
import numpy as np
import pytest

from paper_2311_17174_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("walkers", [1, 9])
def test_no_delay_without_a_distance(walkers):
    from paper_2311_17174_gb300 import emri as E
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = E.Context(0)
    n, dt = 1 << 15, 15.0
    th = I.draw_sources(41, walkers, n)
    th[:, I.I_ALPT] = 0.05
    bad = np.arange(walkers) % 3 == 0
    th[bad, I.I_XI0] = -5.0      # Xi(z) = Xi0 + (1 - Xi0)/(1 + z)^2 < 0 from z = 0.096 on
    assert np.all(th[bad, I.I_XI0] + (1 - th[bad, I.I_XI0]) / (1 + th[bad, I.I_Z]) ** 2 < 0)
    theta = torch.tensor(th.T.copy(), device="cuda:0")
    out = torch.full((6, walkers), float("nan"), dtype=torch.float64, device="cuda:0")
    ctx.prologue(E.grid(n, dt), theta, E.opts(), out)
    torch.cuda.synchronize()
    d_l, xi, d_gw, dt_gw, r_hi, r_lo = out.cpu().numpy()
    assert np.all(d_l > 0) and np.all(xi[bad] < 0) and np.all(d_gw[bad] < 0)
    for v in (dt_gw, r_hi, r_lo):
        assert np.all(v[bad] == 0)
    assert np.all(dt_gw[~bad] != 0) and np.all(r_hi[~bad] > 0)
    psd = I.psd_bc04(n, dt)
    ds = ctx.dataset(E.grid(n, dt), I.noise_spectrum(42, psd, n, dt), psd, 1e-4, 1.0)
    for prec in (E.FP64, E.MIXED):
        lnl, dh, hh = (torch.full((walkers,), float("nan"), dtype=torch.float64, device="cuda:0") for _ in range(3))
        st = torch.zeros(walkers, dtype=torch.int32, device="cuda:0")
        ctx.loglike_batch(ds, theta, E.opts(precision=prec, n_max=4), lnl, dh, hh, st)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(st.cpu().numpy() == E.ST_BADPARAM, bad)
        for v in (lnl, dh, hh):
            assert np.all(v.cpu().numpy()[bad] == 0)
    ds.close()
    ctx.close()
