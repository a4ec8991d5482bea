"""The waveform kernel's instances: FP64 CTAs of one or four 1024-sample
segments, mixed CTAs of four or eight warps, chosen by how far the batch fills
the GPU (four segments from 608 CTAs of 4096 samples on, four warps from 912
segments on).  A walker's series may not depend on the choice, bit for bit,
also where it plunges in the first, a middle or the last segment of a
four-segment CTA; there the FP64 series is also compared with the oracle
(same plunge sample, the path's 1e-9 up to 512 samples before it: the last
ones move too fast for the knots' interpolation), the mixed one at 2e-5 of its
largest value."""
import numpy as np
import pytest

import oracle as O
from paper_2311_17174_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DT = 15.0


def run(ctx, E, th, n, o):
    z = torch.zeros((len(th), n), dtype=torch.complex64 if o.precision else torch.complex128, device="cuda:0")
    ctx.ak_waveform(E.grid(n, DT), torch.tensor(np.ascontiguousarray(th.T), device="cuda:0"), o, z, None)
    torch.cuda.synchronize()
    return z


@pytest.mark.parametrize("logn,walkers,mixed", [(14, 160, False), (15, 80, False), (14, 64, True), (15, 64, True),
                                                (16, 64, True)])
def test_batch_does_not_matter(logn, walkers, mixed):
    from paper_2311_17174_gb300 import emri as E
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n = 1 << logn
    seg = min(4096, n // 16) if mixed else 4096
    assert n // seg * walkers >= (912 if mixed else 608) > n // seg * 8
    ctx = E.Context(0)
    th = I.draw_sources(71, walkers, n, t_margin=(0.3, 3.0))
    th[::5, I.I_E0] = 0.6
    ks = 1024 if mixed else 64
    for n_max in (4, 20):
        o = E.opts(precision=E.MIXED if mixed else E.FP64, n_max=n_max, knot_spacing=ks)
        z = run(ctx, E, th, n, o)
        for k0 in range(0, walkers, 8):
            few = run(ctx, E, th[k0:k0 + 8], n, o)
            assert torch.equal(torch.view_as_real(few), torch.view_as_real(z[k0:k0 + 8])), (n_max, k0)
    o = E.opts(precision=E.MIXED if mixed else E.FP64, n_max=4, knot_spacing=ks)
    z = run(ctx, E, th, n, o).cpu().numpy().astype(np.complex128)
    last = np.array([np.max(np.nonzero(r)[0], initial=-1) for r in z])
    picks = []
    for s in range(4):   # plunges in segment s of a 4096-sample block, beyond the first block's start
        hit = [k for k in range(walkers) if 600 < last[k] < n - 1 and last[k] % 4096 // 1024 == s]
        picks += hit[:2]
        assert hit, s
    picks += [k for k in range(walkers) if last[k] == n - 1][:1]
    hI, hII, _ = O.waveform(th[picks], n, DT, O.Opts(n_max=4))
    for i, k in enumerate(picks):
        ref = hI[i] + 1j * hII[i]
        np.testing.assert_array_equal(z[k] == 0, ref == 0)
        j = last[k] + 1 if last[k] == n - 1 else last[k] - 512
        tol = 2e-5 if mixed else 1e-9
        assert np.max(np.abs(z[k, :j] - ref[:j])) <= tol * np.max(np.abs(ref)), (k, last[k])
    ctx.close()
