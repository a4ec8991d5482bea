"""Device memory of the likelihood and waveform calls: per walker the constants
(up to 640 B), knots (128 B), mixed interval records (104 B), the delay tables,
the rows' partial sums and the time series, per call the LISA phase table of
the tiles, each buffer rounded up to 256 B -- and nothing else, so a budget or
a serving pool of that size admits the call.  The orbit step's own memory lies
in the series buffer; when that holds fewer walkers' state than the call has,
they take turns, with the same results bit for bit."""
import numpy as np
import pytest

from paper_2311_17174_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DT = 15.0


def emri():
    from paper_2311_17174_gb300 import emri as E
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return E


def dataset(E, ctx, n):
    psd = I.psd_bc04(n, DT)
    return ctx.dataset(E.grid(n, DT), I.noise_spectrum(61, psd, n, DT), psd, 1e-4, 1.0 / (2 * DT))


def theta_of(n, w):
    return torch.tensor(I.scatter_walkers(62, I.draw_sources(63, 1, n)[0], w, rel=1e-5).T.copy(), device="cuda:0")


def shared(w, n, ks, mixed):
    return w * (640 + 128 * (n // ks + 1) + (104 * (n // ks) if mixed else 0)) + n // 256 * 64


def likelihood(w, n, ks, mixed):
    cs = 8 if mixed else 16
    n2 = 1 << min(10, (n.bit_length() - 1) // 2)
    return shared(w, n, ks, mixed) + w * (n // n2 * cs + n2 * cs + n2 * 16 + n * cs) + 12 * 256


@pytest.mark.parametrize("logn,w", [(10, 300), (16, 32), (18, 9)])
@pytest.mark.parametrize("mixed", [False, True])
def test_budget_of_a_likelihood(logn, w, mixed):
    E, n = emri(), 1 << logn
    ks = 1024 if mixed else 128
    most = likelihood(w, n, ks, mixed)
    o = E.opts(precision=E.MIXED if mixed else E.FP64, n_max=4)
    ctx = E.Context(0)
    ds = dataset(E, ctx, n)
    assert ctx.serve_request_bytes(ds, w, o) <= most + 18 * 8 * w + 512
    used = ctx.memory()[0]
    ds.close()
    ctx.close()
    ctx = E.Context(0, used + max(most, n * 60 + 8192))   # a dataset is prepared in 44 n bytes beside its own
    ds = dataset(E, ctx, n)
    lnl = torch.zeros(w, dtype=torch.float64, device="cuda:0")
    ctx.loglike_batch(ds, theta_of(n, w), o, lnl)
    torch.cuda.synchronize()
    assert ctx.memory()[0] - used <= most
    assert torch.isfinite(lnl).all() and (lnl != 0).all()
    ds.close()
    ctx.close()


@pytest.mark.parametrize("mixed", [False, True])
def test_budget_of_a_waveform(mixed):
    E, n, w = emri(), 1 << 18, 9
    ks = 1024 if mixed else 128
    ctx = E.Context(0)
    used = ctx.memory()[0]
    most = shared(w, n, ks, mixed) + 6 * 256
    ctx.close()
    ctx = E.Context(0, used + most)
    z = torch.zeros((w, n), dtype=torch.complex64 if mixed else torch.complex128, device="cuda:0")
    ctx.ak_waveform(E.grid(n, DT), theta_of(n, w), E.opts(precision=E.MIXED if mixed else E.FP64, n_max=4), z, None)
    torch.cuda.synchronize()
    assert ctx.memory()[0] - used <= most
    assert (z != 0).all()
    ctx.close()


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("logn", [10, 14])
def test_orbits_in_turns(tmp_path, logn, mixed):
    """Waves of 1 to 3 of 37 walkers: the series buffer holds 2 to 45 walkers'
    orbit state.  Sequential and in groups (a wave of one walker is one group),
    and through the graph of emri_loglike_multi."""
    E, n, w = emri(), 1 << logn, 37
    prec = E.MIXED if mixed else E.FP64
    o = E.opts(precision=prec, n_max=4)
    theta = theta_of(n, w)
    ref = None
    for wave in (0, 1, 2, 3):
        ctx = E.Context(0)
        if wave:
            cache = tmp_path / f"plans{wave}.jsonl"
            cache.write_text('{"n": %d, "n_max": %d, "precision": %d, "knot_spacing": 0, "wave": %d, "n2": 0}\n'
                             % (n, 4, prec, wave))
            assert ctx.autotune(E.grid(n, DT), 4, prec, str(cache))["wave_walkers"] == wave
        ds = dataset(E, ctx, n)
        for groups in (1, 2, 5):
            ctx.set_pipeline(prec, groups)
            out = [torch.zeros(w, dtype=torch.float64, device="cuda:0") for _ in range(3)]
            ctx.loglike_batch(ds, theta, o, *out)
            torch.cuda.synchronize()
            got = [x.cpu().numpy() for x in out]
            if ref is None:
                ref = got
                assert np.isfinite(ref[0]).all() and (ref[0] != 0).all()
            for a, b in zip(got, ref):
                np.testing.assert_array_equal(a, b)
        lnl = torch.zeros(w, dtype=torch.float64, device="cuda:0")
        ctx.loglike_multi([(ds, theta, o, lnl, None, None, None)])
        torch.cuda.synchronize()
        np.testing.assert_array_equal(lnl.cpu().numpy(), ref[0])
        ds.close()
        ctx.close()


def test_waveform_into_an_unaligned_buffer():
    """A float2 output need only be aligned to 8 bytes."""
    E, n, w = emri(), 1 << 12, 5
    ctx = E.Context(0)
    o, theta = E.opts(precision=E.MIXED, n_max=4), theta_of(n, w)
    buf = torch.zeros(w * n + 3, dtype=torch.complex64, device="cuda:0")
    ref = torch.zeros((w, n), dtype=torch.complex64, device="cuda:0")
    ctx.ak_waveform(E.grid(n, DT), theta, o, ref, None)
    ctx.ak_waveform(E.grid(n, DT), theta, o, buf[1:1 + w * n], None)
    torch.cuda.synchronize()
    assert torch.equal(buf[1:1 + w * n].view(w, n), ref)
    assert buf[0] == 0 and (buf[1 + w * n:] == 0).all()
    ctx.close()
