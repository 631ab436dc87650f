"""GPU: the partial sums of a call's visibility ranges stay bounded.

153 cutouts of 256 pixels make 306 tiles, two just incomplete waves and a few: without a bound
the last wave is bought with some 25 ranges, 1 GB of partial sums.  The plan's scratch is its
weights (8 bytes per position and visibility) and partials within half a gibibyte."""
import numpy as np
import pytest

import obsgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_partials_are_bounded():
    import paper_2009_07010_gb300 as psf

    obs = obsgen.tiny_obs(seed=53, nant=16, ntime=4200, nchan=4, tavg=1, favg=2, radius_m=1000.0)
    rng = np.random.default_rng(5)
    npos, N, cell = 153, 256, 1.5 * obsgen.ARCSEC
    lm = rng.uniform(-0.02, 0.02, (npos, 2))
    with psf.Plan(obs, prec="tc_fp16", algo=psf.PSF_ALGO_CUTOUT) as plan:
        assert plan.nvis > 1_000_000
        b = psf.Batch(lm, N, cell)
        out = torch.empty(b.total(), device="cuda")
        plan.exact(psf.Batch(lm[:1], 32, cell), out=out)   # kernels loaded
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        plan.exact(b, out=out)
        assert plan.sync_status() == 0
        used = free - torch.cuda.mem_get_info()[0]
        assert used <= npos * plan.nvis * 8 + (512 << 20) + (64 << 20), used
        # the same sums over other ranges (one cutout: many), FP32 additions in another order
        for p in (0, 77, 152):
            one = plan.exact(psf.Batch(lm[p:p + 1], N, cell))
            got = out[p * N * N:(p + 1) * N * N]
            assert (got - one).abs().max() <= 1e-5 * one.abs().max()
