"""Folding uploads the delays of the trials it folds from, and no others: calls
with few candidates of a long plan, with other candidates, masks and stages from
call to call, with searches and dedispersions between them and with calls that
run out of device memory, give the bytes of the same call on a context of its
own; and a fold leaves the device memory of a small request."""
import numpy as np
import pytest

from paper_1912_12807_gb300 import synth

pytestmark = pytest.mark.gpu


def _file(nbits, nchan, nsamp, rows, mask_seed=None):
    import torch

    from paper_1912_12807_gb300 import pss
    g = np.random.default_rng(nchan + nsamp)
    mask = None
    if mask_seed is not None:
        mask = np.ones(nchan, dtype=np.uint8)
        mask[np.random.default_rng(mask_seed).permutation(nchan)[:nchan // 8]] = 0
    plan = pss.Plan(pss.FilDesc(nchan, nsamp, 2e-4, 1230.0, 288.0 / nchan, nbits, chan_mask=mask),
                    [synth.Stage(*r) for r in rows])
    return plan, torch.from_numpy(g.integers(0, 256, (nsamp, nchan * nbits // 8), dtype=np.uint8)).cuda()


def test_candidates_masks_and_calls_in_turn():
    from paper_1912_12807_gb300 import pss
    rows = [(0, 0.5, 300, 1), (150, 1, 100, 2), (250, 2, 60, 8)]
    files = [_file(8, 96, 20011, rows, m) for m in (None, 1, 2)] + [_file(1, 96, 30011, rows[:2], m) for m in (None, 3)]
    files.append(_file(1, 248, 20011, [(0, 20, 60, 1)]))  # delay spreads that the bit-sliced kernel leaves to the bytes
    lists = [[5], [0, 459], [7, 8, 20, 310, 311, 405], list(range(0, 459, 2)), [301, 5, 5, 299], [12]]

    def fold(ctx, f, k):
        plan, dev = files[f]
        dm = np.minimum(np.array(lists[k]), plan.ndm - 1)
        p, c, r = pss.pss_fold(ctx, plan, dev, dm, 3.0 + 0.37 * np.arange(len(dm)), nbin=32, nfreq=3)
        return p.tobytes() + c.tobytes() + r.tobytes()

    ref = {}
    for f in range(len(files)):
        for k in range(len(lists)):
            ctx = pss.Context(0)
            ref[f, k] = fold(ctx, f, k)
            ctx.close()
    cfg = pss.search_cfg(numharm=2, sigma_thr=5.0)
    ctx = pss.Context(0)
    try:
        plan0, dev0 = files[0]
        series = pss.pss_dedisperse(ctx, plan0, dev0, 0, plan0.ndm).clone()
        raw = pss.pss_search_raw(ctx, plan0, dev0, cfg, 0, plan0.ndm).tobytes()
        for i, (f, k) in enumerate([(f, k) for k in range(len(lists)) for f in range(len(files))]):
            if i % 4 == 1:
                assert (pss.pss_dedisperse(ctx, plan0, dev0, 0, plan0.ndm) == series).all()
            if i % 5 == 2:
                assert pss.pss_search_raw(ctx, plan0, dev0, cfg, 0, plan0.ndm).tobytes() == raw
            assert fold(ctx, f, k) == ref[f, k], (f, k)
        # allocations refused in a fold of a larger file: the kept set-ups and tables are not taken for valid after it
        big = _file(8, 128, 60011, rows)
        for n in range(1, 8):
            pss.pss_debug_fail_alloc(n)
            try:
                pss.pss_fold(ctx, *big, np.array([3, 200]), np.array([4.0, 5.0]), nbin=32)
            except pss.PssError as e:
                assert e.status == pss.PSS_ENOMEM
            pss.pss_debug_fail_alloc(0)
            assert (pss.pss_dedisperse(ctx, plan0, dev0, 0, plan0.ndm) == series).all()
            assert pss.pss_search_raw(ctx, plan0, dev0, cfg, 0, plan0.ndm).tobytes() == raw
            assert fold(ctx, 0, 2) == ref[0, 2]
    finally:
        pss.pss_debug_fail_alloc(0)
        ctx.close()


def test_one_candidate_of_a_long_plan_takes_a_small_table():
    """The delays of 60 000 trials x 256 channels are 61 MB; one candidate's are 1 kB."""
    import torch

    from paper_1912_12807_gb300 import pss
    plan, dev = _file(8, 256, 4099, [(0, 0.001, 60000, 1)])
    ctx = pss.Context(0)
    try:
        pss.pss_fold(ctx, plan, dev, np.array([30000]), np.array([20.0]), nbin=32)
        ctx.close()
        torch.cuda.synchronize()
        ctx = pss.Context(0)
        free0 = torch.cuda.mem_get_info()[0]
        pss.pss_fold(ctx, plan, dev, np.array([30000]), np.array([20.0]), nbin=32)
        torch.cuda.synchronize()
        assert free0 - torch.cuda.mem_get_info()[0] < (40 << 20)
    finally:
        ctx.close()
