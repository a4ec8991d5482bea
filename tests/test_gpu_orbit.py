"""The orbit solver (all segments at once, then the sequential tail) against
the oracle's RK4 orbit, through the waveform, at the sizes where its segment
split changes: one segment, two, eight, and 64 (a coarse segment over four),
knot spacings that put fewer or more than 32 knots in a segment, both
directions, and windows in which some walkers plunge in an early, middle or
the last segment while others do not.

Tolerance: the path's parity bar, 1e-9 relative (2-norm and largest element)
in FP64; 2e-5 in mixed precision at K_s = 1024."""
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


def run(ctx, th, n, n_max, precision, ks, backward):
    from paper_2311_17174_gb300 import emri
    z = torch.zeros((len(th), n), dtype=torch.complex128 if precision == 0 else torch.complex64, device="cuda:0")
    st = torch.zeros(len(th), dtype=torch.int32, device="cuda:0")
    theta = torch.tensor(np.ascontiguousarray(th.T), device="cuda:0")
    ctx.ak_waveform(emri.grid(n, 15.0), theta,
                    emri.opts(precision=precision, n_max=n_max, knot_spacing=ks,
                              mode=emri.BACKWARD_FROM_LSO if backward else emri.FORWARD), z, st)
    torch.cuda.synchronize()
    return z.cpu().numpy().astype(np.complex128), st.cpu().numpy()


def check(z, st, hI, hII, st_o, tol):
    np.testing.assert_array_equal(st, st_o)
    for k in range(len(z)):
        ref = hI[k] + 1j * hII[k]
        np.testing.assert_array_equal(z[k] == 0, ref == 0)      # the same plunge sample
        assert np.linalg.norm(z[k] - ref) <= tol * np.linalg.norm(ref), k
        assert np.max(np.abs(z[k] - ref)) <= tol * np.max(np.abs(ref)), k


@pytest.mark.parametrize("logn,ks,precision,backward,walkers", [
    (10, 64, 0, 0, 3), (12, 128, 0, 0, 3), (13, 64, 0, 1, 3), (15, 128, 0, 1, 2), (17, 128, 0, 0, 2),
    (19, 64, 0, 0, 1), (10, 1024, 1, 0, 3), (14, 1024, 1, 1, 3), (16, 512, 1, 0, 2)])
def test_segment_splits(ctx, logn, ks, precision, backward, walkers):
    n = 1 << logn
    th = I.config_paper(walkers=walkers, n=n, rel=1e-2, seed=51).theta if backward else \
        I.draw_sources(52, walkers, n, t_margin=(2.5, 4.0))
    hI, hII, st_o = O.waveform(th, n, 15.0, O.Opts(n_max=5, backward=backward))
    z, st = run(ctx, th, n, 5, precision, ks, backward)
    check(z, st, hI, hII, st_o, 1e-9 if precision == 0 else 2e-5)


@pytest.mark.parametrize("when", [0.05, 0.45, 0.97])
def test_plunge_in_a_segment(ctx, when):
    # walkers 0 and 2 plunge at about `when` of the window (the draw's
    # circular-orbit time estimate is refined on the oracle), walker 1 does not
    n = 1 << 15
    th = I.draw_sources(53, 3, n, t_margin=(3.0, 4.0))
    for k in (0, 2):
        m, mu, e = th[k, I.I_M], th[k, I.I_MU], th[k, I.I_E0]
        lo, hi = 0.05, 8.0
        for _ in range(12):
            mid = 0.5 * (lo + hi)
            th[k, I.I_NU0] = I.start_frequency(m, mu, e, mid * when * n * 15.0)
            h = O.waveform(th[k:k + 1], n, 15.0, O.Opts(n_max=1))[0][0]
            j = int(np.max(np.nonzero(h)[0], initial=0))
            lo, hi = (mid, hi) if j < when * n else (lo, mid)
    hI, hII, st_o = O.waveform(th, n, 15.0, O.Opts(n_max=4))
    assert st_o[0] & 1 and st_o[2] & 1 and not st_o[1] & 1
    # the last samples before a plunge move too fast for the knot spacing's
    # interpolation: values are compared up to 512 samples before it
    z, st = run(ctx, th, n, 4, 0, 64, 0)
    np.testing.assert_array_equal(st, st_o)
    for k in range(3):
        ref = hI[k] + 1j * hII[k]
        np.testing.assert_array_equal(z[k] == 0, ref == 0)
        j = n if k == 1 else max(0, int(np.max(np.nonzero(ref)[0])) - 512)
        if j:
            assert np.max(np.abs(z[k, :j] - ref[:j])) <= 1e-9 * np.max(np.abs(ref[:j])), (k, j)
