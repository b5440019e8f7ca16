"""Requests that change from call to call on one context (DM ranges walked in
steps that are no multiple of a group of trials, masks in turn, files whose
shared-sum tables are taken and files whose tables cost too much) give the
series and candidates of the same request on a context of its own."""
import numpy as np
import pytest

from paper_1912_12807_gb300 import synth

pytestmark = pytest.mark.gpu

# (channels, samples, bits, plan rows)
FILES = [(256, 20011, 8, [(0, 0.5, 150, 1)]), (64, 20011, 8, [(0, 1, 150, 1)]), (300, 9001, 8, [(10, 0.5, 80, 1), (50, 1, 40, 2)]),
         (96, 30003, 1, [(0, 0.5, 120, 1)])]


def test_changed_requests_equal_requests_alone():
    import torch

    from paper_1912_12807_gb300 import pss
    cfg = pss.search_cfg(numharm=2, sigma_thr=4.5)
    reqs = []
    for f, (nchan, nsamp, nbits, rows) in enumerate(FILES):
        g = np.random.default_rng(f)
        dev = torch.from_numpy(g.integers(0, 256, (nsamp, nchan * nbits // 8), dtype=np.uint8)).cuda()
        for masked in (0, nchan // 9, nchan // 5):
            mask = np.ones(nchan, dtype=np.uint8)
            mask[g.permutation(nchan)[:masked]] = 0
            plan = pss.Plan(pss.FilDesc(nchan, nsamp, 2e-4, 1230.0, 288.0 / nchan, nbits, chan_mask=mask if masked else None),
                            [synth.Stage(*r) for r in rows])
            for lo, hi in ((0, 8), (8, 41), (41, 111), (0, plan.ndm), (plan.ndm - 3, plan.ndm)):
                for k in ("dedisperse", "search", "pulses"):
                    reqs.append((plan, dev, k, lo, hi))

    def call(ctx, r):
        plan, dev, k, lo, hi = r
        if k == "dedisperse":
            out = pss.pss_dedisperse(ctx, plan, dev, lo, hi).cpu().numpy()
            pss.pss_ctx_check(ctx)
        elif k == "search":
            out = pss.pss_search_raw(ctx, plan, dev, cfg, lo, hi)
        else:
            out = pss.pss_single_pulse(ctx, plan, dev, lo, hi, sigma_thr=4.0)
        return out.tobytes()

    ref = []
    for r in reqs:
        ctx = pss.Context(0)
        ref.append(call(ctx, r))
        ctx.close()
    ctx = pss.Context(0)
    try:
        for i in np.random.default_rng(9).integers(0, len(reqs), 2 * len(reqs)):
            assert call(ctx, reqs[i]) == ref[i], reqs[i][2:]
    finally:
        ctx.close()
