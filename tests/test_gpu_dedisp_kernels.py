"""The dedispersion kernels with shared partial sums (8-bit files) and with
bit-sliced counting (1-bit files) against plain integer sums over the plan's
delays: edges of their tiles, of the groups of trials that share a tile and of
the channel counts their accumulators hold, masks, both channel orders, every
downsampling, and files the kernels leave to the others."""
import numpy as np
import pytest

from oracle import dedisperse as OD
from paper_1912_12807_gb300 import synth

pytestmark = pytest.mark.gpu

# (channels, samples, bits, band lo, band hi, sampling time, plan rows, masked channels, descending)
CASES = {
    "8bit_tile_edge": (256, 512 * 20 + 4475, 8, 1050.0, 1450.0, 2e-4, [(0, 0.5, 33, 1)], 0, False),
    "8bit_groups": (128, 12345, 8, 1050.0, 1450.0, 2e-4, [(100, 0.25, 97, 1), (124, 0.5, 31, 2), (140, 0.5, 32, 4)], 0, True),
    "8bit_few_trials": (200, 9001, 8, 1050.0, 1450.0, 2e-4, [(50, 0.5, 8, 1)], 0, False),
    "8bit_257": (257, 8192, 8, 1050.0, 1450.0, 2e-4, [(0, 0.5, 40, 1)], 0, False),
    "8bit_258": (258, 8191, 8, 1050.0, 1450.0, 2e-4, [(0, 0.5, 40, 1)], 0, True),
    "8bit_wide_masked": (700, 7001, 8, 1050.0, 1450.0, 2e-4, [(0, 0.5, 40, 1), (20, 0.5, 20, 2)], 61, False),
    "8bit_odd_channels": (131, 9000, 8, 1050.0, 1450.0, 2e-4, [(10, 0.25, 64, 1)], 0, False),
    "8bit_large_spread": (24, 200001, 8, 400.0, 500.0, 1e-4, [(0, 3, 40, 1)], 0, False),
    "1bit_tile_edge": (96, 4096 * 3 + 188, 1, 1230.0, 1518.0, 2.5e-4, [(0, 0.5, 33, 1)], 0, False),
    "1bit_staged": (96, 30003, 1, 1230.0, 1518.0, 2.5e-4, [(0, 0.5, 17, 1), (8, 1, 16, 2), (24, 5, 15, 4), (99, 5, 7, 64), (134, 9, 3, 1024)], 5, True),
    "1bit_one_trial": (8, 5001, 1, 1230.0, 1518.0, 2.5e-4, [(3, 1, 1, 1)], 0, False),
    "1bit_255": (256, 9003, 1, 1230.0, 1518.0, 2.5e-4, [(0, 0.5, 20, 1)], 1, False),
    "1bit_256": (256, 9003, 1, 1230.0, 1518.0, 2.5e-4, [(0, 0.5, 20, 1)], 0, False),
    "1bit_large_spread": (248, 60001, 1, 300.0, 400.0, 2.5e-4, [(0, 5, 40, 1)], 0, False),
}


def _file(nchan, nsamp, nbits, seed):
    r = np.random.default_rng(seed)
    if nbits == 8:
        d = r.integers(0, 256, (nsamp, nchan), dtype=np.uint8)
        d[r.random((nsamp, nchan)) < 0.3] = 255  # large sums
        return d, d
    d = r.integers(0, 256, (nsamp, nchan // 8), dtype=np.uint8)
    d[r.random((nsamp, nchan // 8)) < 0.3] = 255
    return d, np.unpackbits(d, axis=1)


@pytest.mark.parametrize("name", sorted(CASES))
def test_series_are_the_plain_sums(name):
    import torch

    from paper_1912_12807_gb300 import pss
    nchan, nsamp, nbits, lo, hi, ts, rows, masked, desc = CASES[name]
    data, x = _file(nchan, nsamp, nbits, len(name))
    foff = (hi - lo) / nchan
    f0 = hi - 0.5 * foff if desc else lo + 0.5 * foff
    mask = np.ones(nchan, dtype=np.uint8)
    mask[np.random.default_rng(3).permutation(nchan)[:masked]] = 0
    plan = pss.Plan(pss.FilDesc(nchan, nsamp, ts, f0, -foff if desc else foff, nbits, chan_mask=mask if masked else None),
                    [synth.Stage(*r) for r in rows])
    xc = np.ascontiguousarray(x.T)[mask != 0]
    delays = plan.delays()[:, mask != 0]
    dev = torch.from_numpy(data).cuda()
    ctx = pss.Context(0)
    try:
        for lo_i, hi_i in ((0, plan.ndm), (plan.ndm // 3, plan.ndm)):
            out = pss.pss_dedisperse(ctx, plan, dev, lo_i, hi_i)
            pss.pss_ctx_check(ctx)
            out, off = out.cpu().numpy(), 0
            for i in range(lo_i, hi_i):
                t = plan.trial(i)
                if i < lo_i + 2 or i > hi_i - 3 or i % 16 in (0, 15):
                    ref = OD.dedisperse(xc, delays[i], plan.max_delay, t["ds"])
                    np.testing.assert_array_equal(out[off:off + t["nv"]], ref, err_msg="trial %d" % i)
                off += t["nv"]
        # the float series of the search path: candidates of the series equal those of a range of it
        cfg = pss.search_cfg(numharm=2, whiten_block=64, f_lo_hz=0.0)
        nmin = min(plan.trial(i)["nfft"] for i in range(plan.ndm))
        if nmin >= 128:
            a = pss.pss_spectrum(ctx, plan, dev, cfg, 0, plan.ndm).cpu().numpy()
            b = pss.pss_spectrum(ctx, plan, dev, cfg, plan.ndm // 3, plan.ndm).cpu().numpy()
            assert a[len(a) - len(b):].tobytes() == b.tobytes()
    finally:
        ctx.close()
