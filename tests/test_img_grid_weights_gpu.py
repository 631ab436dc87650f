"""GPU: the gridded form, its table and CLEAN with it follow psf_plan_set_weights: after the
weights were replaced they agree with a plan that had those weights from the start, and after
the natural weights came back with the first results.

The tables' sums over visibilities are float64 atomics (any order: 1e-15 relative), rounded to
float32 once; the transforms after that have a fixed order.  Tables may differ by one float32
rounding (1.2e-7 relative), cutouts by that in every term (1e-6 of the peak)."""
import numpy as np
import pytest

import obsgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", ["fp32", "tc_fp16"])
def test_gridded_form_follows_the_weights(prec):
    import paper_2009_07010_gb300 as psf

    obs = obsgen.tiny_obs(seed=47, nant=8, ntime=240, nchan=4, tavg=6, favg=2, radius_m=1200.0)
    cell, N = 2.0 * obsgen.ARCSEC, 32
    lm = np.array([[0.02, -0.01], [-0.005, 0.03]])
    b = psf.Batch(lm, N, cell)
    img = torch.zeros((96, 96), device="cuda")
    img[40, 50], img[60, 20] = 9.0, 5.0

    def results(plan):
        r = plan.clean(img.clone(), cell, N, gain=0.5, max_iter=4)[0]
        return plan.approx_img_grid(b).clone(), plan.img_grid_table(N, cell), r

    def same(got, want):
        assert (got[0] - want[0]).abs().max() <= 1e-6 * want[0].abs().max()
        assert ((got[1] - want[1]).abs() <= 2.4e-7 * want[1].abs().amax(dim=(0, 1))).all()
        assert (got[2] - want[2]).abs().max() <= 1e-5 * 9.0

    with psf.Plan(obs, prec=prec) as plan:
        natural = results(plan)
        g = torch.Generator(device="cuda").manual_seed(3)
        for _ in range(2):
            W = torch.rand(plan.nvis, generator=g, device="cuda") ** 4 * 10.0
            plan.set_weights(W)
            obs.weights = W.cpu().numpy()
            with psf.Plan(obs, prec=prec) as other:
                want = results(other)
            got = results(plan)
            same(got, want)
            # the weights matter: both the effective PSF and the cells' means have moved
            assert (got[0] - natural[0]).abs().max() > 1e-2 * natural[0].abs().max()
            assert (got[1][..., 2:] - natural[1][..., 2:]).abs().max() > 0
        plan.set_weights(None)
        same(results(plan), natural)
        assert plan.sync_status() == 0
