"""GPU: the CLEAN loop inside one kernel (row maxima, shared PSF, window rows) against the
same loop in numpy on the device's own PSF cutouts: image sizes that are no multiple of the
segments, windows clipped at every edge, equal maxima, several launches.

The choices are compared one by one (noise keeps candidates apart by far more than float32
rounding); residuals within 1e-5 of the brightest pixel (float32 subtractions)."""
import numpy as np
import pytest

import obsgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def plan():
    import paper_2009_07010_gb300 as psf

    obs = obsgen.tiny_obs(seed=31, nant=8, ntime=240, nchan=4, tavg=6, favg=2, radius_m=1200.0)
    with psf.Plan(obs, prec="fp32") as p:
        yield p


def _image(nl, nm, seed):
    g = np.random.default_rng(seed)
    img = 0.2 * g.standard_normal((nm, nl))
    for x, y in [(0, 0), (nl - 1, 0), (0, nm - 1), (nl - 1, nm - 1), (nl // 2, 1), (1, nm // 2), (nl // 2, nm // 2)]:
        img[y, x] += g.uniform(5.0, 20.0)
    return img.astype(np.float32)


def _numpy_clean(plan, img, cell, N, gain, iters, centre, facet):
    import paper_2009_07010_gb300 as psf

    res, (nm, nl) = img.copy(), img.shape
    pix, h = [], N // 2
    for _ in range(iters):
        k = int(np.argmax(res))
        y, x = divmod(k, nl)
        lm = np.array([centre]) if facet else np.array([[centre[0] + (x - nl // 2) * cell, centre[1] + (y - nm // 2) * cell]])
        P = plan.approx_img_grid(psf.Batch(lm, N, cell))[:N * N].view(N, N).cpu().numpy()
        s = np.float32(np.float32(gain) * res[y, x]) / P[h, h]
        ya, yb, xa, xb = max(0, y - h), min(nm, y - h + N), max(0, x - h), min(nl, x - h + N)
        res[ya:yb, xa:xb] -= s * P[ya - y + h:yb - y + h, xa - x + h:xb - x + h]
        pix.append(k)
    return res, pix


@pytest.mark.parametrize("N,nl,nm,facet", [(16, 50, 38, False), (32, 130, 66, False), (64, 64, 64, False),
                                           (128, 200, 258, False), (32, 130, 66, True), (128, 90, 40, True)])
def test_loop_matches_numpy(plan, N, nl, nm, facet):
    cell, centre, gain, iters = 2.0 * obsgen.ARCSEC, (0.004, -0.003), 0.3, 24
    img = _image(nl, nm, N + nl)
    ref, pix = _numpy_clean(plan, img, cell, N, gain, iters, centre, facet)
    res, model, cp, cf = plan.clean(torch.from_numpy(img.copy()).cuda(), cell, N, method="img_grid", gain=gain,
                                    max_iter=iters, centre=centre, facet_psf=facet)
    assert cp.cpu().tolist() == pix
    assert np.abs(res.cpu().numpy() - ref).max() <= 1e-5 * np.abs(img).max()
    m = np.zeros(nl * nm)
    np.add.at(m, cp.cpu().numpy(), cf.cpu().numpy().astype(np.float64))
    assert np.abs(model.cpu().numpy().ravel() - m).max() <= 1e-5 * np.abs(img).max()


def test_first_of_equal_maxima_and_several_launches(plan):
    cell = 2.0 * obsgen.ARCSEC
    img = np.zeros((96, 160), np.float32)
    img[70, 3] = img[20, 150] = img[20, 140] = 7.0
    _, _, cp, _ = plan.clean(torch.from_numpy(img.copy()).cuda(), cell, 16, gain=0.5, max_iter=3)
    assert cp.cpu().tolist() == [20 * 160 + 140, 20 * 160 + 150, 70 * 160 + 3]
    # more iterations than one launch runs: the same choices as in one shorter call, then on
    noise = _image(160, 96, 5)
    _, _, c1, _ = plan.clean(torch.from_numpy(noise.copy()).cuda(), cell, 16, gain=0.05, max_iter=2500)
    _, _, c2, _ = plan.clean(torch.from_numpy(noise.copy()).cuda(), cell, 16, gain=0.05, max_iter=900)
    assert len(c1) == 2500 and torch.equal(c1[:900], c2)
