"""GPU: what the CTAs of the CLEAN loop's cluster hand to one another.

First iterations: launches of a single iteration, back to back, whose PSF rows are written into
shared memory of CTAs that have only just been launched.  The arithmetic has a fixed order, so
every call gives the same bits."""
import numpy as np
import pytest

import obsgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def plan():
    import paper_2009_07010_gb300 as psf

    obs = obsgen.tiny_obs(seed=37, nant=8, ntime=240, nchan=4, tavg=6, favg=2, radius_m=1200.0)
    with psf.Plan(obs, prec="fp32") as p:
        yield p


@pytest.mark.parametrize("N", [16, 128])
def test_first_iteration_of_many_launches(plan, N):
    import paper_2009_07010_gb300 as psf

    cell, (ny, nx), (x, y) = 2.0 * obsgen.ARCSEC, (160, 192), (101, 77)
    img = torch.zeros((ny, nx), device="cuda")
    img[y, x] = 8.0
    lm = np.array([[(x - nx // 2) * cell, (y - ny // 2) * cell]])
    P = plan.approx_img_grid(psf.Batch(lm, N, cell))[:N * N].view(N, N).cpu().numpy().astype(np.float64)
    ref = img.cpu().numpy().astype(np.float64)
    h = N // 2
    win = (slice(max(0, y - h), min(ny, y - h + N)), slice(max(0, x - h), min(nx, x - h + N)))
    ref[win] -= 4.0 / P[h, h] * P[win[0].start - y + h:win[0].stop - y + h, win[1].start - x + h:win[1].stop - x + h]
    first = None
    for _ in range(200):
        res, _, pix, flux = plan.clean(img.clone(), cell, N, method="img_grid", gain=0.5, max_iter=1)
        assert pix.tolist() == [y * nx + x] and flux.tolist() == [4.0]
        if first is None:
            first = res
            # the PSF of the cluster and of the batched kernel: the same formulas in another order
            assert np.abs(res.cpu().numpy() - ref).max() <= 1e-5 * 8.0
        assert torch.equal(res, first)


@pytest.mark.parametrize("N,nl,nm,iters", [(2, 24, 4096, 2000), (16, 24, 4096, 2000), (16, 90, 2048, 2500)])
def test_given_psf_small_window_tall_image(plan, N, nl, nm, iters):
    """One PSF per image, row maxima of thousands of rows, small windows: every iteration the
    CTAs must see the same peak before any of them renews its rows.  The reference replays the
    loop in float32 with the device's rounding (one fused multiply-add per pixel, formed in
    float64), so it agrees to the last bits and a window around another pixel stands out."""
    import paper_2009_07010_gb300 as psf

    cell, gain, h = 2.0 * obsgen.ARCSEC, np.float32(0.3), N // 2
    g = np.random.default_rng(N + nl)
    img = (g.standard_normal((nm, nl)) + 20.0 * (g.random((nm, nl)) < 0.01)).astype(np.float32)
    centre = (0.004, -0.003)
    P = plan.approx_uv(psf.Batch(np.array([centre]), N, cell))[:N * N].view(N, N).cpu().numpy()
    res, model, pix, flux = plan.clean(torch.from_numpy(img.copy()).cuda(), cell, N, method="uv", gain=float(gain),
                                       max_iter=iters, centre=centre, facet_psf=True)
    ref, want = img.copy(), []
    for _ in range(iters):
        k = int(np.argmax(ref))
        y, x = divmod(k, nl)
        want.append(k)
        s = np.float32(gain * ref[y, x]) / P[h, h]
        ya, yb, xa, xb = max(0, y - h), min(nm, y - h + N), max(0, x - h), min(nl, x - h + N)
        w = P[ya - y + h:yb - y + h, xa - x + h:xb - x + h].astype(np.float64)
        ref[ya:yb, xa:xb] = (ref[ya:yb, xa:xb].astype(np.float64) - np.float64(s) * w).astype(np.float32)
    assert pix.cpu().tolist() == want
    assert np.abs(res.cpu().numpy() - ref).max() <= 1e-6 * np.abs(img).max()
