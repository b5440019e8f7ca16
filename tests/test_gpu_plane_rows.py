"""Overlap-save planes whose rows are split over several CTAs per segment: the
planes of one trial, of a few and of many in one call (which are split into
different numbers of row ranges, or not at all) are the same bytes, for row
counts below, at and above the number of ranges, with and without remainders."""
import numpy as np
import pytest

from paper_1912_12807_gb300 import synth

pytestmark = pytest.mark.gpu

# (samples, zmax, dz): 5, 9, 17, 21, 65 and 201 rows
CASES = [(1 << 13, 2, 1.0), (1 << 14, 4, 1.0), (1 << 14, 16, 2.0), (1 << 13, 20, 2.0), (9001, 16, 0.5), (1 << 15, 200, 2.0)]


@pytest.mark.parametrize("nsamp,zmax,dz", CASES)
def test_planes_do_not_depend_on_the_row_ranges(nsamp, zmax, dz):
    import torch

    from paper_1912_12807_gb300 import pss
    wl = synth.workload_small(nsamp=nsamp)
    ctx = pss.Context(0)
    try:
        n = 160
        plan = pss.Plan(pss.FilDesc.of(wl.fil), [synth.Stage(20.0, 0.25, n, 1)])
        dev = torch.from_numpy(wl.fil.data).cuda()
        cfg = pss.search_cfg(zmax=zmax, dz=dz, numharm=2, whiten_block=256)
        per = pss.n_z(cfg) * plan.trial(0)["nfft"]
        whole = pss.pss_power_plane(ctx, plan, dev, cfg, 0, n)
        assert torch.isfinite(whole).all()
        for lo, hi in ((0, 1), (n - 1, n), (3, 5), (7, 14), (40, 71)):
            part = pss.pss_power_plane(ctx, plan, dev, cfg, lo, hi)
            assert torch.equal(part, whole[lo * per:hi * per]), (lo, hi)
    finally:
        ctx.close()
