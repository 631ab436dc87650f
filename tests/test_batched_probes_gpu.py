"""GPU: the batched form's autotuner on the first call of a plan.  Both forms are timed after an
untimed run, so the crossover does not depend on whether a kernel of the process was loaded by
the probe itself: the launches of the first call beyond those of the next are two of the batched
form and three of the per-cutout form per cutout size.  Options and profiling are as before it."""
import numpy as np
import pytest

import obsgen

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")


@pytest.mark.parametrize("method", ["exact", "uv"])
@pytest.mark.parametrize("sizes", [[64], [32, 96]])
def test_both_forms_are_probed_warm(method, sizes):
    import paper_2009_07010_gb300 as psf

    obs = obsgen.tiny_obs(seed=59, nant=16, ntime=1200, nchan=8, tavg=4, favg=1, radius_m=1000.0)
    rng = np.random.default_rng(59)
    npix = np.repeat(np.array(sizes, np.int32), 20)
    b = psf.Batch(rng.uniform(-0.02, 0.02, (len(npix), 2)), npix, 1.5 * obsgen.ARCSEC)
    with psf.Plan(obs, prec="tc_bf16") as plan:
        plan.profile_enable(True)
        plan.profile_read()
        launches, timed = [], []
        for _ in range(3):
            plan.forward(method, b)
            assert plan.sync_status() == 0
            ms, contractions, _ = plan.profile_read()
            launches.append(contractions)
            timed.append(ms > 0.0)   # profiling is still on after the probes
        assert launches[0] - launches[1] == 5 * len(sizes)
        assert launches[1] == launches[2] and all(timed)
