"""GPU: the batched form contracts a half plane of pixels and writes each pixel with its
point reflection.  Every cutout size (main rows, border row and border column, partial last
pixel tile) against the FP32 CUDA-core form, which evaluates every pixel."""
import numpy as np
import pytest

import obsgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def obs():
    # 55 baselines, bins of 5 samples, 4 output channels: 26 400 visibilities
    return obsgen.tiny_obs(seed=11, nant=11, ntime=600, nchan=8, tavg=5, favg=2, f0=1.3e9, df=1e6, dt=1.0,
                           radius_m=1500.0)


@pytest.mark.parametrize("npix", [32, 64, 96, 160, 224, 256])
@pytest.mark.parametrize("method", ["exact", "uv"])
def test_half_plane_matches_full_form(obs, npix, method):
    """250 positions (whole tiles are always batched, and a remainder this large).  The 16-bit
    operands leave at most a few 1e-5 of the peak on 2.6e4 visibilities (rounding of 2^-11
    per term, averaged, and the tensor core's accumulation); the path's stated bound is 1e-4."""
    import paper_2009_07010_gb300 as psf

    lm = np.random.default_rng(5).uniform(-0.02, 0.02, (250, 2))
    cell = 2.0 * obsgen.ARCSEC
    with psf.Plan(obs, prec="tc_fp16") as plan:
        got = plan.forward(method, psf.Batch(lm, npix, cell)).view(250, npix * npix)
        assert plan.sync_status() == 0
        check = [0, 63, 127, 128, 249]
        plan.set_opts(prec="fp32")
        ref = plan.forward(method, psf.Batch(lm[check], npix, cell)).view(len(check), npix * npix)
        err = ((got[check] - ref).abs().amax(dim=1) / ref.abs().amax(dim=1)).max().item()
    assert err <= 1e-4, err
