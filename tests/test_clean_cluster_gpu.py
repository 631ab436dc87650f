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
