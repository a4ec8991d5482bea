"""The FP64 kernels that compute in 64-bit fixed point.

* FFT: rounding of the inputs at 2^-62 of the transform's sum L <= 1.6 N rms,
  in each of two passes of N <= 4096 points: at most
  sqrt(2) 1.6 4096 2^-62 / sqrt(6) = 8e-16 of the spectrum's norm, the stages
  and numpy's own transform as much again: 3e-15.  Inputs outside the
  fixed-point range keep the double form: 1e-14 sqrt(log2 n), as elsewhere.
* waveform: circular and eccentric orbits, one to 32 harmonics, against the
  oracle at the path's own bound, 1e-9 at the knot spacing 128, and with the
  fourth power of the spacing beyond (the knots' cubic Hermite interpolation).
"""
import numpy as np
import pytest

import oracle as O
from paper_2311_17174_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    from paper_2311_17174_gb300 import emri
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = emri.Context(0)
    yield c
    c.close()


def gpu_fft(ctx, x, sign):
    from paper_2311_17174_gb300 import emri as E
    z = torch.tensor(x, dtype=torch.complex128, device="cuda:0")
    ctx.fft_batch(z, x.shape[1], x.shape[0], E.FP64, sign)
    torch.cuda.synchronize()
    return z.cpu().numpy()


def numpy_fft(x, sign):
    return np.fft.fft(x, axis=1) if sign < 0 else np.fft.ifft(x, axis=1) * x.shape[1]


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("sign", [-1, 1])
@pytest.mark.parametrize("logn", [10, 13, 15, 16, 17, 18, 19, 20, 21, 22])
def test_fft_fixed_point(ctx, logn, sign):
    n, g = 1 << logn, np.random.default_rng(logn)
    t = np.arange(n) / n
    x = np.stack([
        g.standard_normal(n) + 1j * g.standard_normal(n),
        np.exp(2j * np.pi * (0.37 * n * t + 0.1 * n * t * t)) * np.exp(-8 * t) * 1e-21,   # a chirp at strain size
        np.where(np.arange(n) == 3 * n // 7, 1e20, 1e-3 * g.standard_normal(n)) + 0j,      # one sample dominates
    ])
    got, ref = gpu_fft(ctx, x, sign), numpy_fft(x, sign)
    for b in range(len(x)):
        assert rel(got[b], ref[b]) <= 3e-15, (b, rel(got[b], ref[b]))
        err = np.abs(got[b] - ref[b]).max() / np.abs(ref[b]).max()
        assert err <= 1e-14 * np.sqrt(logn), (b, err)


@pytest.mark.parametrize("logn", [16, 19])
def test_fft_outside_the_fixed_range(ctx, logn):
    """Zeros, huge, tiny and non-finite inputs: as in double, row by row."""
    n, g = 1 << logn, np.random.default_rng(7)
    noise = g.standard_normal(n) + 1j * g.standard_normal(n)
    nan, inf = noise.copy(), noise.copy()
    nan[5 * n // 11] = np.nan
    inf[n // 3] = np.inf
    x = np.stack([np.zeros(n), 1e200 * noise, 1e-200 * noise, nan, inf, noise])
    got = gpu_fft(ctx, x, -1)
    ref = numpy_fft(x, -1)
    assert np.all(got[0] == 0)
    for b in (1, 2, 5):
        assert rel(got[b] / np.abs(ref[b]).max(), ref[b] / np.abs(ref[b]).max()) <= 1e-14 * np.sqrt(logn), b
    for b in (3, 4):
        assert not np.isfinite(got[b].real).any() and not np.isfinite(got[b].imag).any(), b


@pytest.mark.parametrize("n_max", [1, 2, 32])
@pytest.mark.parametrize("ks", [64, 128, 256])
def test_waveform_knot_spacings(ctx, ks, n_max):
    from paper_2311_17174_gb300 import emri as E
    n, dt = 1 << 13, 15.0
    th = I.draw_sources(31 + ks, 3, n)
    th[1, I.I_E0] = 1e-9
    z = torch.zeros((3, n), dtype=torch.complex128, device="cuda:0")
    ctx.ak_waveform(E.grid(n, dt), torch.tensor(th.T.copy(), device="cuda:0"),
                    E.opts(n_max=n_max, knot_spacing=ks), z, None)
    torch.cuda.synchronize()
    got = z.cpu().numpy()
    hI, hII, _ = O.waveform(th, n, dt, O.Opts(n_max=n_max))
    for k in range(3):
        ref = hI[k] + 1j * hII[k]
        if not np.abs(ref).max() > 0:
            assert np.abs(got[k]).max() == 0
            continue
        tol = 1e-9 * max(1.0, (ks / 128) ** 4)
        assert rel(got[k], ref) <= tol, (k, rel(got[k], ref))
        assert np.abs(got[k] - ref).max() <= tol * np.abs(ref).max(), k


def test_side_stream_order(ctx):
    """The delay tables run on the context's side stream: calls in a row on
    two user streams, with other walkers each, give the same bits as the same
    calls one at a time, and so does a captured call (which keeps one stream;
    a context captures on the stream of its last call)."""
    from paper_2311_17174_gb300 import emri as E
    n, dt, w = 1 << 13, 15.0, 5
    psd = I.psd_bc04(n, dt)
    noise = I.noise_spectrum(9, psd, n, dt)
    ds = ctx.dataset(E.grid(n, dt), noise, psd, 1e-4, 1.0 / (2 * dt))
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
        c2 = E.Context(0)
        ds2 = c2.dataset(E.grid(n, dt), noise, psd, 1e-4, 1.0 / (2 * dt))
        out = torch.zeros(w, dtype=torch.float64, device="cuda:0")
        torch.cuda.synchronize()
        c2.loglike_batch(ds2, th[3], o, out, stream=streams[0])
        torch.cuda.synchronize()
        out.zero_()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=streams[0]):
            c2.loglike_batch(ds2, th[3], o, out, stream=streams[0])
        g.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(out.cpu().numpy(), alone[3])
        ds2.close()
        c2.close()
    ds.close()
