"""GPU: the FP32 adjoint takes one, two or four visibilities per thread by their number (edges
at 307 200 and 614 400), against the oracle's float64 vector-Jacobian product.  Bounds as for
the FP32 adjoint elsewhere: 2e-5 of max |dL/dW|, 2e-4 of max |dL/d(l0, m0)|."""
import numpy as np
import pytest

import obsgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("ntime", [698, 699, 1396, 1397])   # x 440 visibilities: both sides of each edge
def test_visibilities_per_thread(ntime):
    import paper_2009_07010_gb300 as psf

    obs = obsgen.tiny_obs(seed=21, nant=11, ntime=ntime, nchan=8, tavg=1, favg=1, f0=1.2e9, df=1e6, dt=2.0,
                          radius_m=1200.0, weights=True)
    batch = obsgen.Batch(np.array([[0.02, -0.01], [-0.015, 0.02]]), np.array([8, 6], np.int32), 4.0 * obsgen.ARCSEC)
    P = oracle.psf(obs, oracle.UV, batch)
    R = P + 0.1 * np.abs(P).max() * np.random.default_rng(4).standard_normal(P.size)
    g_lm_ref, g_W_ref = oracle.vjp(obs, oracle.UV, batch, R)
    with psf.Plan(obs, prec="fp32") as plan:
        g_lm, g_W = plan.adjoint("uv", psf.Batch.from_obsgen(batch), torch.tensor(R, dtype=torch.float32, device="cuda"))
        assert plan.sync_status() == 0
    assert np.max(np.abs(g_W.cpu().numpy() - g_W_ref)) <= 2e-5 * np.max(np.abs(g_W_ref))
    assert np.max(np.abs(g_lm.cpu().numpy() - g_lm_ref)) <= 2e-4 * np.max(np.abs(g_lm_ref))
