"""The likelihood at the lengths where its FP64 passes run in fixed point and
its FP32 pass 2 in registers (rows of 256 points or more, n >= 2^15), and the
rows that leave the fixed-point range.

* frequency-dependent propagation at n = 2^14, 2^16, 2^18 (rows of 128, 256,
  512 points) against the oracle, with and without amplitude and phase terms:
  FP64 lnL within 1e-9 (|<d|h>| + <h|h>/2), <h|h> within 2e-9, mixed 1e-2;
* sources so far out that their series lies below the fixed-point range (v0 of
  1e-17): some rows of pass 2 in double, others in fixed point; <d|h> and
  <h|h> within 1e-9 of the oracle (<d|h> of sqrt(<d|d><h|h>));
* the side stream's order with the fixed-point delay table;
* the transform's rms error below a double's rounding unit, 2^-52, against a
  long double transform.
"""
import numpy as np
import pytest

import oracle as O
from paper_2311_17174_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DT = 15.0


@pytest.fixture(scope="module")
def E():
    from paper_2311_17174_gb300 import emri
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return emri


@pytest.fixture(scope="module")
def ctx(E):
    c = E.Context(0)
    yield c
    c.close()


def sums(ctx, E, ds, th, o, fd=None):
    w = len(th)
    theta = torch.tensor(th.T.copy(), device="cuda:0")
    out = [torch.zeros(w, dtype=torch.float64, device="cuda:0") for _ in range(3)]
    st = torch.zeros(w, dtype=torch.int32, device="cuda:0")
    if fd is None:
        ctx.loglike_batch(ds, theta, o, *out, st)
    else:
        qm, qt, fstar, coef = fd
        ctx.loglike_batch_fd(ds, theta, o, qm, qt, fstar, torch.tensor(coef.T.copy(), device="cuda:0"), *out, st)
    torch.cuda.synchronize()
    return [x.cpu().numpy() for x in out + [st]]


@pytest.fixture(scope="module", params=[14, 16, 18])
def problem(request, ctx, E):
    n, nm, w = 1 << request.param, 6, 6
    psd = I.psd_bc04(n, DT)
    d, inj, wts, _ = O.injection_data(I.draw_sources(91, 1, n)[0], n, DT, psd, 92, O.Opts(n_max=nm), snr=40.0)
    th = I.scatter_walkers(93, inj, w)
    ds = ctx.dataset(E.grid(n, DT), d, psd, 1e-4, 1.0 / (2 * DT))
    yield n, nm, d, wts, th, ds
    ds.close()


@pytest.mark.parametrize("qm,qt", [(2, 3), (1, 1), (3, 0), (0, 1)])
def test_propagation(ctx, E, problem, qm, qt):
    n, nm, d, wts, th, ds = problem
    w, fstar = len(th), 3e-3
    g = np.random.default_rng(94)
    # (f/f_*)^3 reaches 1400: amplitude terms of like size at the top of the band
    coef = np.concatenate([g.normal(0, 0.3, (w, qm)) * 0.1 ** np.arange(qm), g.normal(0, 0.05, (w, qt))], axis=1)
    ref, dh_o, hh_o, _ = O.loglike_fd(th, n, DT, d, wts, qm, qt, fstar, coef, O.Opts(n_max=nm))
    dgw = np.array([O.prologue(t, n, DT)[2] for t in th])
    lnl, dh, hh, st = sums(ctx, E, ds, th, E.opts(n_max=nm), (qm, qt, fstar, coef))
    assert not st.any()
    tol = 1e-9 * (np.abs(dh_o / dgw) + 0.5 * hh_o / dgw ** 2)
    assert np.all(np.abs(lnl - ref) <= tol), (np.abs(lnl - ref) / tol).max()
    np.testing.assert_allclose(hh, hh_o, rtol=2e-9)
    lnl, _, _, _ = sums(ctx, E, ds, th, E.opts(precision=E.MIXED, n_max=nm), (qm, qt, fstar, coef))
    assert np.max(np.abs(lnl - ref)) <= 1e-2


@pytest.mark.parametrize("fd", [False, True])
@pytest.mark.parametrize("logn", [15, 17])
def test_series_below_the_fixed_range(ctx, E, logn, fd):
    n, nm, w = 1 << logn, 4, 3
    psd = I.psd_bc04(n, DT)
    th = I.draw_sources(95, w, n)
    th[:, I.I_NU0] = [1e-50, 3e-50, 1e-49]
    d = I.noise_spectrum(96, psd, n, DT)
    fmin, fmax = 2e-5, 1.0 / (2 * DT)
    wts = O.weights(psd, n, DT, fmin, fmax)
    ds = ctx.dataset(E.grid(n, DT), d, psd, fmin, fmax)
    coef = np.random.default_rng(97).normal(0, 0.2, (w, 2))
    _, dh_o, hh_o, _ = (O.loglike_fd(th, n, DT, d, wts, 1, 1, 3e-3, coef, O.Opts(n_max=nm)) if fd else
                        O.loglike(th, n, DT, d, wts, O.Opts(n_max=nm)))
    _, dh, hh, st = sums(ctx, E, ds, th, E.opts(n_max=nm), (1, 1, 3e-3, coef) if fd else None)
    assert not st.any() and np.all(hh > 0)
    np.testing.assert_allclose(hh, hh_o, rtol=1e-9)
    assert np.all(np.abs(dh - dh_o) <= 1e-9 * np.sqrt(ds.dd() * hh_o))
    ds.close()


@pytest.mark.parametrize("logn", [15, 16])
def test_side_stream_order(ctx, E, logn):
    n, w = 1 << logn, 5
    psd = I.psd_bc04(n, DT)
    ds = ctx.dataset(E.grid(n, DT), I.noise_spectrum(9, psd, n, DT), psd, 1e-4, 1.0 / (2 * DT))
    th = [torch.tensor(I.draw_sources(60 + k, w, n).T.copy(), device="cuda:0") for k in range(6)]
    for prec in (E.FP64, E.MIXED):
        o = E.opts(precision=prec, n_max=6)
        alone = []
        for t in th:
            out = torch.zeros(w, dtype=torch.float64, device="cuda:0")
            ctx.loglike_batch(ds, t, o, out)
            torch.cuda.synchronize()
            alone.append(out.cpu().numpy())
        streams = [torch.cuda.Stream() for _ in range(2)]
        outs = [torch.zeros(w, dtype=torch.float64, device="cuda:0") for _ in th]
        torch.cuda.synchronize()
        for k, t in enumerate(th):
            ctx.loglike_batch(ds, t, o, outs[k], stream=streams[k % 2])
        torch.cuda.synchronize()
        for k in range(len(th)):
            np.testing.assert_array_equal(outs[k].cpu().numpy(), alone[k])
    ds.close()


@pytest.mark.parametrize("sign", [-1, 1])
@pytest.mark.parametrize("logn", [16, 18])
def test_rms_error_of_the_transform(ctx, E, logn, sign):
    fft = pytest.importorskip("scipy.fft")
    n, g = 1 << logn, np.random.default_rng(logn)
    t = np.arange(n) / n
    x = np.stack([g.standard_normal(n) + 1j * g.standard_normal(n),
                  np.exp(2j * np.pi * (0.2 * n * t + 0.05 * n * t * t)) * (1 + t)])
    z = torch.tensor(x, device="cuda:0")
    ctx.fft_batch(z, n, len(x), E.FP64, sign)
    torch.cuda.synchronize()
    y = x.astype(np.clongdouble)
    ref = fft.fft(y, axis=1) if sign < 0 else fft.ifft(y, axis=1) * n
    err = np.linalg.norm((z.cpu().numpy() - ref).astype(np.complex128), axis=1) / \
        np.linalg.norm(ref.astype(np.complex128), axis=1)
    assert np.all(err <= 2.0 ** -52), err
