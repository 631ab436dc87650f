"""GPU: the batched form on calls of many short items, where every stage's inputs are refilled
soon after they were read: repeated calls agree.

The only freedom is the order in which a pixel's ranges (at most 20 here) are added: each
addition rounds by at most 2^-24 of the peak, twice for the two calls compared, so 2.4e-6 of it.
One 32-pixel run of one 64-visibility stage with foreign inputs is off by the sum of 64
unit phasors of random phase, about 8 of the 65 000 terms of the peak (1e-4)."""
import numpy as np
import pytest

import obsgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("method,N", [("exact", 64), ("exact", 256), ("uv", 64), ("uv", 256)])
def test_repeated_calls_agree(method, N):
    import paper_2009_07010_gb300 as psf

    obs = obsgen.tiny_obs(seed=67, nant=16, ntime=1088, nchan=8, tavg=16, favg=1, radius_m=1000.0)
    lm = np.random.default_rng(67).uniform(-0.02, 0.02, (128, 2))
    with psf.Plan(obs, prec="tc_fp16") as plan:
        assert 60_000 < plan.nvis < 70_000
        b = psf.Batch(lm, N, 2.0 * obsgen.ARCSEC)
        first = plan.forward(method, b).clone()
        peak = first.abs().max()
        out = torch.empty_like(first)
        worst = torch.zeros((), device="cuda")
        for _ in range(100):
            plan.forward(method, b, out=out)
            worst = torch.maximum(worst, (out - first).abs().max() / peak)
        assert plan.sync_status() == 0
        assert float(worst) <= 2.4e-6
