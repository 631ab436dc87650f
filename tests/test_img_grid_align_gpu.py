"""GPU: the gridded form into output buffers that start at any float and cutout offsets of
either parity: the same bits as into an aligned buffer, and nothing written between cutouts."""
import numpy as np
import pytest

import obsgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("N", [16, 32, 64, 128])
def test_output_alignment(N):
    import paper_2009_07010_gb300 as psf

    obs = obsgen.tiny_obs(seed=41, nant=8, ntime=120, nchan=4, tavg=6, favg=2, radius_m=1200.0)
    lm = np.array([[0.01, -0.02], [0.0, 0.0], [-0.03, 0.005]])
    cell = 2.0 * obsgen.ARCSEC
    with psf.Plan(obs, prec="fp32") as plan:
        ref = plan.approx_img_grid(psf.Batch(lm, N, cell))
        for gap in (0, 1):
            offs = np.arange(3, dtype=np.int64) * (N * N + gap)
            b = psf.Batch(lm, N, cell, out_offset=offs)
            for start in (0, 1, 2, 3):
                buf = torch.full((b.total() + 8,), 7.0, device="cuda")
                plan.approx_img_grid(b, out=buf[start:])
                want = torch.full_like(buf, 7.0)
                for p in range(3):
                    at = start + int(offs[p])
                    want[at:at + N * N] = ref[p * N * N:(p + 1) * N * N]
                assert torch.equal(buf, want)
