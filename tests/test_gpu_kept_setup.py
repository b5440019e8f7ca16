"""Host set-ups that a context keeps between calls: requests of several kinds
and two plans in turn on one context, with a call among them that runs out of
device memory after it has replaced the delay tables, give the bytes that each
gives on a context of its own."""
import numpy as np
import pytest

from paper_1912_12807_gb300 import synth

pytestmark = pytest.mark.gpu


def test_requests_in_turn_equal_requests_alone():
    import torch

    from paper_1912_12807_gb300 import pss
    g = np.random.default_rng(5)
    files = []
    rows0 = [(0, 0.5, 40, 1), (20, 0.5, 20, 2)]
    # the third file has the delays of the first, and more samples
    for nchan, nsamp, rows in ((128, 20011, rows0), (200, 30011, [(5, 0.5, 64, 1)]), (128, 60011, rows0)):
        f0, foff = 1050.0, 400.0 / nchan
        plan = pss.Plan(pss.FilDesc(nchan, nsamp, 2e-4, f0, foff, 8), [synth.Stage(*r) for r in rows])
        files.append((plan, torch.from_numpy(g.integers(0, 256, (nsamp, nchan), dtype=np.uint8)).cuda()))
    cfg = pss.search_cfg(numharm=4, sigma_thr=4.0)
    acc = pss.search_cfg(numharm=2, zmax=20, sigma_thr=4.5)
    calls = {
        "dedisperse": lambda c, p, d: pss.pss_dedisperse(c, p, d, 0, p.ndm).cpu().numpy(),
        "part": lambda c, p, d: pss.pss_dedisperse(c, p, d, 7, p.ndm - 3).cpu().numpy(),
        "search": lambda c, p, d: pss.pss_search_raw(c, p, d, cfg, 0, p.ndm),
        "accel": lambda c, p, d: pss.pss_search_raw(c, p, d, acc, 0, p.ndm),
        "pulses": lambda c, p, d: pss.pss_single_pulse(c, p, d, 0, p.ndm),
        "fold": lambda c, p, d: pss.pss_fold(c, p, d, np.array([3, 30]), np.array([10.0, 7.5]), np.zeros(2), nbin=32)[0],
    }

    def alone(f, k):
        ctx = pss.Context(0)
        try:
            return np.asarray(calls[k](ctx, *files[f])).tobytes()
        finally:
            ctx.close()

    ref = {(f, k): alone(f, k) for f in (0, 1, 2) for k in calls}
    ctx = pss.Context(0)
    try:
        order = [(0, "search"), (0, "pulses"), (0, "search"), (0, "fold"), (0, "search"), (1, "dedisperse"), (0, "search"),
                 (0, "accel"), (0, "part"), (0, "accel"), (1, "search"), (1, "part"), (1, "search"), (1, "fold"),
                 (0, "fold"), (1, "pulses"), (0, "dedisperse"), (1, "pulses"), (1, "accel"), (0, "pulses"), (1, "accel")]
        for f, k in order:
            assert np.asarray(calls[k](ctx, *files[f])).tobytes() == ref[f, k], (f, k)
    finally:
        ctx.close()
    # a larger file's call fails at one of its allocations: the smaller one's kept set-up must not be taken for valid
    for other in (1, 2):
        for n in (1, 2, 3):
            for k in ("search", "dedisperse"):
                ctx = pss.Context(0)
                try:
                    assert np.asarray(calls[k](ctx, *files[0])).tobytes() == ref[0, k]
                    pss.pss_debug_fail_alloc(n)
                    try:
                        calls[k](ctx, *files[other])
                        assert n > 1  # (later than its last allocation)
                    except pss.PssError as e:
                        assert e.status == pss.PSS_ENOMEM
                    pss.pss_debug_fail_alloc(0)
                    assert np.asarray(calls[k](ctx, *files[0])).tobytes() == ref[0, k]
                    assert np.asarray(calls[k](ctx, *files[other])).tobytes() == ref[other, k]
                finally:
                    pss.pss_debug_fail_alloc(0)
                    ctx.close()
