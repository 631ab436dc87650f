"""GPU: the FP32 contraction chooses among several tile shapes and splits small
observations over the whole chip; sizes at the shapes' edges, visibility counts around the
64-visibility chunks, against the float64 oracle within the path's 1e-6."""
import numpy as np
import pytest

import obsgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("npix", [2, 30, 32, 34, 40, 48, 50, 64, 80, 82, 96, 100, 130])
def test_tile_edges(npix):
    import paper_2009_07010_gb300 as psf

    obs = obsgen.tiny_obs(seed=21, nant=6, ntime=300, nchan=4, tavg=5, favg=2, weights=True)
    batch = obsgen.Batch(np.array([[0.01, -0.02], [0.0, 0.015]]), np.array([npix, npix], np.int32), 2.0 * obsgen.ARCSEC)
    with psf.Plan(obs, prec="fp32") as plan:
        got = plan.exact(psf.Batch.from_obsgen(batch)).cpu().numpy().astype(np.float64)
    ref = oracle.psf(obs, oracle.EXACT, batch)
    assert np.max(np.abs(got - ref)) <= 1e-6 * np.max(np.abs(ref))


@pytest.mark.parametrize("ntime", [5, 45, 320, 325, 5000])
def test_visibility_counts(ntime):
    """1, 9, 64, 65 and 1000 visibilities of one baseline (no partial chunk may be lost)."""
    import paper_2009_07010_gb300 as psf

    obs = obsgen.tiny_obs(seed=22, nant=2, ntime=ntime, nchan=1, tavg=5, favg=1, weights=True)
    batch = obsgen.Batch(np.array([[0.01, -0.02]]), np.array([48], np.int32), 2.0 * obsgen.ARCSEC)
    for prec, tol in (("fp32", 1e-6), ("tc_fp16", 2e-3)):   # 16-bit: a few unit roundoffs per term
        with psf.Plan(obs, prec=prec) as plan:
            got = plan.exact(psf.Batch.from_obsgen(batch)).cpu().numpy().astype(np.float64)
            assert plan.sync_status() == 0
        ref = oracle.psf(obs, oracle.EXACT, batch)
        assert np.max(np.abs(got - ref)) <= tol * np.max(np.abs(ref)), prec
