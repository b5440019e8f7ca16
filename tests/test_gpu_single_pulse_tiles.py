"""Boxcar detection with both tile sizes: the events of a few trials searched
alone (small tiles) are those trials' events of a call with many (large tiles),
at a low threshold on data with many equal window sums and broad pulses, so with
detections, ties and long local-maximum windows at every tile edge; 32-bit and
64-bit prefix sums, the narrowest and the widest boxcars."""
import numpy as np
import pytest

from paper_1912_12807_gb300 import synth

pytestmark = pytest.mark.gpu

# (samples, channels, trials, ds, widths, threshold): the last one's window sums pass 2^31
CASES = [
    (16411, 16, 220, 1, (1, 2, 3, 150), 2.0),
    (16411, 16, 220, 1, (1, 1000, 1024), 1.0),
    (4099, 8, 640, 1, (7,), 2.0),
    (130001, 160, 640, 64, (1, 30, 1024), 1.5),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_events_do_not_depend_on_the_tiles(case):
    import torch

    from paper_1912_12807_gb300 import pss
    nsamp, nchan, ndm, ds, widths, thr = CASES[case]
    g = np.random.default_rng(case)
    d = g.integers(0, 4, (nsamp, nchan), dtype=np.uint8)
    for t in g.integers(0, nsamp - 1500 * ds if ds == 1 else nsamp // 2, 12):
        d[t:t + int(g.integers(2, 1400))] += np.uint8(g.integers(1, 3))
    if ds > 1:
        d *= 40
    foff = 64.0 / nchan
    plan = pss.Plan(pss.FilDesc(nchan, nsamp, 2e-4, 1400.0, foff, 8), [synth.Stage(0.0, 0.02, ndm, ds)])
    dev = torch.from_numpy(d).cuda()
    ctx = pss.Context(0)
    try:
        whole = pss.pss_single_pulse(ctx, plan, dev, 0, ndm, widths=widths, sigma_thr=thr)
        assert len(whole) > 2 * ndm
        for lo, hi in ((0, 1), (ndm // 2, ndm // 2 + 9), (ndm - 1, ndm)):
            part = pss.pss_single_pulse(ctx, plan, dev, lo, hi, widths=widths, sigma_thr=thr)
            at = whole[(whole["dm_idx"] >= lo) & (whole["dm_idx"] < hi)]
            assert part.tobytes() == np.ascontiguousarray(at).tobytes()
    finally:
        ctx.close()
