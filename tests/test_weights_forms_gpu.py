"""GPU: the 16-bit weight kernels share a bin's records, phasors and sincs among its output
channels; every channel count (groups of eight, partial groups, stages cut inside a bin)
against the FP32 CUDA-core form, whose weights are evaluated one by one.

2.6e4 visibilities or more: 16-bit rounding leaves a few 1e-5 of the peak; bound 1e-4, the
path's stated one."""
import numpy as np
import pytest

import obsgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _obs(nchan, favg):
    nout = nchan // favg
    ntime = 5 * max(40, -(-26400 // (55 * nout)))
    return obsgen.tiny_obs(seed=12, nant=11, ntime=ntime, nchan=nchan, tavg=5, favg=favg, f0=1.3e9, df=1e6, dt=1.0,
                           radius_m=1500.0, weights=True)


def _err(got, ref):
    return ((got - ref).abs().amax(dim=1) / ref.abs().amax(dim=1)).max().item()


@pytest.mark.parametrize("nchan,favg", [(9, 3), (12, 2), (16, 2), (7, 1), (20, 1), (24, 1)])
def test_batched_exact_weights(nchan, favg):
    import paper_2009_07010_gb300 as psf

    lm = np.random.default_rng(6).uniform(-0.03, 0.03, (130, 2))
    cell = 2.0 * obsgen.ARCSEC
    with psf.Plan(_obs(nchan, favg), prec="tc_fp16") as plan:
        got = plan.exact(psf.Batch(lm, 32, cell)).view(130, -1)
        assert plan.sync_status() == 0
        check = [0, 3, 4, 127, 128, 129]
        plan.set_opts(prec="fp32")
        assert _err(got[check], plan.exact(psf.Batch(lm[check], 32, cell)).view(len(check), -1)) <= 1e-4


@pytest.mark.parametrize("nchan,favg", [(8, 1), (16, 2), (12, 2)])
@pytest.mark.parametrize("method,literal", [("uv", False), ("img", False), ("img", True), ("exact", False)])
@pytest.mark.parametrize("npos", [1, 130])
def test_single_and_batched_weights(nchan, favg, method, literal, npos):
    import paper_2009_07010_gb300 as psf

    flags = 2 if literal else 0   # PSF_IMG_LITERAL_THETA
    lm = np.random.default_rng(7).uniform(-0.03, 0.03, (npos, 2))
    cell = 2.0 * obsgen.ARCSEC
    with psf.Plan(_obs(nchan, favg), prec="tc_fp16", flags=flags) as plan:
        got = plan.forward(method, psf.Batch(lm, 64, cell)).view(npos, -1)
        assert plan.sync_status() == 0
        check = sorted({0, npos // 2, npos - 1})
        plan.set_opts(prec="fp32")
        assert _err(got[check], plan.forward(method, psf.Batch(lm[check], 64, cell)).view(len(check), -1)) <= 1e-4


@pytest.mark.parametrize("df,dt,radius,tavg", [(1e6, 1.0, 0.03, 5), (1e6, 2.0, 0.03, 20), (2e7, 8.0, 0.4, 6)])
@pytest.mark.parametrize("favg", [1, 3])
def test_moment_and_general_sums(df, dt, radius, tavg, favg):
    """Exact weights (one position, a batch) and the adjoint's fold on both sides of the moment
    form's limit (wide channels and long bins far from the phase centre exceed it) and with
    more samples per bin than the fold caches.  Adjoint: 2e-3 of the largest component, the
    16-bit adjoint's bound on few visibilities."""
    import paper_2009_07010_gb300 as psf

    obs = obsgen.tiny_obs(seed=13, nant=11, ntime=60 * tavg, nchan=8 * favg, tavg=tavg, favg=favg, f0=1.0e9, df=df / favg,
                          dt=dt, radius_m=1500.0, weights=True)
    lm = np.random.default_rng(8).uniform(-radius, radius, (130, 2))
    cell = 2.0 * obsgen.ARCSEC
    with psf.Plan(obs, prec="tc_fp16") as plan:
        got = plan.exact(psf.Batch(lm, 32, cell)).view(130, -1)
        one = plan.exact(psf.Batch(lm[:1], 32, cell)).view(1, -1)
        check = [0, 65, 129]
        b = psf.Batch(lm[:5], 32, cell)
        g = torch.randn(b.total(), generator=torch.Generator("cuda").manual_seed(3), device="cuda")
        g_lm, g_W = plan.adjoint("exact", b, g)
        assert plan.sync_status() == 0
        plan.set_opts(prec="fp32")
        ref = plan.exact(psf.Batch(lm[check], 32, cell)).view(len(check), -1)
        r_lm, r_W = plan.adjoint("exact", b, g)
    scale = float(obs.weights.sum())   # the peak without decorrelation
    assert (got[check] - ref).abs().max().item() <= 1e-4 * scale
    assert (one - ref[:1]).abs().max().item() <= 1e-4 * scale
    assert (g_W - r_W).abs().max().item() <= 2e-3 * r_W.abs().max().item()
    assert (g_lm - r_lm).abs().max().item() <= 2e-3 * r_lm.abs().max().item()
