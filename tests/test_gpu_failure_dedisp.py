"""Bounded waits of the shared-sum (8-bit) and bit-sliced (1-bit) dedispersion
kernels: a context whose waits give up after one non-blocking poll gets
PSS_ETIMEOUT from dedispersion, single pulses, folding and searches (the kernels
set the flag, drain their copies in flight and leave), and after the limit is
restored the same context gives the bytes of a context that never had it."""
import numpy as np
import pytest

from paper_1912_12807_gb300 import synth

pytestmark = pytest.mark.gpu

# (channels, samples, bits, trials): 257 and fewer kept channels, and more (sums written out part-way)
FILES = [(256, 40011, 8, 64), (400, 20011, 8, 64), (96, 100003, 1, 64)]


@pytest.mark.parametrize("nchan,nsamp,nbits,ndm", FILES)
def test_wait_runs_out_then_context_recovers(nchan, nsamp, nbits, ndm):
    import torch

    from paper_1912_12807_gb300 import pss
    dev = torch.from_numpy(np.random.default_rng(nchan).integers(0, 256, (nsamp, nchan * nbits // 8), dtype=np.uint8)).cuda()
    plan = pss.Plan(pss.FilDesc(nchan, nsamp, 2e-4, 1050.0, 400.0 / nchan, nbits), [synth.Stage(0.0, 0.5, ndm, 1)])
    cfg = pss.search_cfg(numharm=4, sigma_thr=5.0)
    calls = {
        "dedisperse": lambda c: pss.pss_dedisperse(c, plan, dev, 0, ndm).cpu().numpy().tobytes(),
        "pulses": lambda c: pss.pss_single_pulse(c, plan, dev, 0, ndm, sigma_thr=4.5).tobytes(),
        "search": lambda c: pss.pss_search_raw(c, plan, dev, cfg, 0, ndm).tobytes(),
        "sifted": lambda c: pss.pss_search_dm_batch(c, plan, dev, cfg, 0, ndm).tobytes(),
    }
    if nbits == 1:
        calls["fold"] = lambda c: pss.pss_fold(c, plan, dev, np.arange(0, ndm, 3), 7.0 + np.arange(0, ndm, 3), nbin=32)[0].tobytes()
    ref = {}
    for k, call in calls.items():
        ctx = pss.Context(0)
        ref[k] = call(ctx)
        ctx.close()
    ctx = pss.Context(0)
    try:
        for k, call in calls.items():
            assert call(ctx) == ref[k]
            pss.pss_ctx_set_wait_limit(ctx, 1)
            with pytest.raises(pss.PssError) as ei:
                call(ctx)
                pss.pss_ctx_check(ctx)  # (dedispersion alone is asynchronous)
            assert ei.value.status == pss.PSS_ETIMEOUT
            pss.pss_ctx_check(ctx)  # reported once, then clear
            pss.pss_ctx_set_wait_limit(ctx, 0)
            for again in calls:
                assert calls[again](ctx) == ref[again], (k, again)
            pss.pss_ctx_check(ctx)
        pss.pss_ctx_set_wait_limit(ctx, 1 << 24)  # long enough for any copy
        for k, call in calls.items():
            assert call(ctx) == ref[k]
        pss.pss_ctx_check(ctx)
    finally:
        ctx.close()
