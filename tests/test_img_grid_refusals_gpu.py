"""GPU: the table of the gridded form is refused wherever the gridded form is (complex output:
its effective PSF would take twice the floats), in every precision, whether or not a table of
the size is kept already."""
import pytest

import obsgen

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")


@pytest.mark.parametrize("prec", ["fp32", "tc_fp16", "tc_bf16", "tc_fp16x3"])
@pytest.mark.parametrize("kept", [False, True])
def test_table_refused_with_complex_output(prec, kept):
    import torch

    import paper_2009_07010_gb300 as psf

    obs = obsgen.tiny_obs(seed=43, nant=6, ntime=60, nchan=4, tavg=6, favg=2, radius_m=1200.0)
    cell = 2.0 * obsgen.ARCSEC
    with psf.Plan(obs, prec=prec) as plan:
        before = plan.img_grid_table(32, cell) if kept else None
        plan.set_opts(flags=psf.PSF_COMPLEX_OUT)
        with pytest.raises(psf.PsfError):
            plan.img_grid_table(32, cell)
        with pytest.raises(psf.PsfError):
            plan.approx_img_grid(psf.Batch([[0.01, 0.0]], 32, cell))
        plan.set_opts(flags=0)
        t = plan.img_grid_table(32, cell)
        assert before is None or torch.equal(t, before)
        assert plan.sync_status() == 0
