"""GPU: CLEAN as whole-chip kernels (one PSF with a large window, the gridded PSF on images of very
many rows) against the loop in numpy on the device's own cutouts: more iterations than one queued
chunk, a stop by the threshold inside a chunk, equal maxima, windows clipped at the edges.

The reference rounds as the device does (one fused multiply-add per pixel, formed in float64), so
choices agree and residuals agree to a few roundings (1e-6 of the brightest pixel)."""
import numpy as np
import pytest

import obsgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def plan():
    import paper_2009_07010_gb300 as psf

    obs = obsgen.tiny_obs(seed=61, nant=8, ntime=240, nchan=4, tavg=6, favg=2, radius_m=1200.0)
    with psf.Plan(obs, prec="fp32") as p:
        yield p


# the last window sizes below and the first above the line between the forms for these images,
# windows larger than the image, a very wide image, and images of many rows (gridded)
@pytest.mark.parametrize("facet,N,nl,nm", [(True, 96, 300, 220), (True, 98, 300, 220), (True, 256, 200, 180),
                                           (True, 512, 90, 400), (True, 16, 131072, 6), (False, 16, 4, 60000), (False, 64, 6, 131072)])
@pytest.mark.parametrize("iters", [1, 64, 150])
def test_matches_numpy(plan, facet, N, nl, nm, iters):
    import paper_2009_07010_gb300 as psf

    cell, gain, h, centre = 2.0 * obsgen.ARCSEC, np.float32(0.2), N // 2, (0.004, -0.003)
    g = np.random.default_rng(N + nl)
    img = (0.2 * g.standard_normal((nm, nl)) + 15.0 * (g.random((nm, nl)) < 20.0 / (nl * nm))).astype(np.float32)
    img[nm - 1, nl - 1] = img[0, nl - 1] = img[nm // 3, 0] = 30.0   # the first in row-major order comes first

    def cutout(lm):
        fn = plan.approx_img_grid if not facet else plan.approx_uv
        return fn(psf.Batch(np.array([lm]), N, cell))[:N * N].view(N, N).cpu().numpy()

    P = cutout(centre) if facet else None
    ref, want, peaks = img.copy(), [], []
    for _ in range(iters):
        k = int(np.argmax(ref))
        y, x = divmod(k, nl)
        want.append(k)
        peaks.append(ref[y, x])
        if not facet:
            P = cutout((centre[0] + (x - nl // 2) * cell, centre[1] + (y - nm // 2) * cell))
        s = np.float32(gain * ref[y, x]) / P[h, h]
        ya, yb, xa, xb = max(0, y - h), min(nm, y - h + N), max(0, x - h), min(nl, x - h + N)
        w = P[ya - y + h:yb - y + h, xa - x + h:xb - x + h].astype(np.float64)
        ref[ya:yb, xa:xb] = (ref[ya:yb, xa:xb].astype(np.float64) - np.float64(s) * w).astype(np.float32)
    kw = dict(method="uv" if facet else "img_grid", gain=float(gain), centre=centre, facet_psf=facet)
    res, model, pix, flux = plan.clean(torch.from_numpy(img.copy()).cuda(), cell, N, max_iter=iters, threshold=-1e30, **kw)
    assert pix.cpu().tolist() == want
    assert np.abs(res.cpu().numpy() - ref).max() <= 1e-6 * 30.0
    m = np.zeros(nl * nm)
    np.add.at(m, pix.cpu().numpy(), flux.cpu().numpy().astype(np.float64))
    assert np.abs(model.cpu().numpy().ravel() - m).max() <= 1e-5 * 30.0
    if iters > 64:   # the threshold stops the loop where the peak has first come down to it
        stop = next(t for t in range(1, iters) if peaks[t] <= peaks[100])
        pix = plan.clean(torch.from_numpy(img.copy()).cuda(), cell, N, max_iter=iters, threshold=float(peaks[100]), **kw)[2]
        assert pix.cpu().tolist() == want[:stop]
