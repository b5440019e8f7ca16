"""The float series of the search path from the shared-sum and bit-sliced
dedispersion kernels: whitened spectra against FP64 spectra of the plain integer
series, so that the float epilogues, the partial sums that wait in the float rows
with more than 257 channels and the sums that form the mean are compared with
something other than themselves.  Powers within the relative bound of the
oracle comparisons."""
import numpy as np
import pytest

from _parity import check_powers
from oracle import dedisperse as OD
from oracle import spectrum as OS
from paper_1912_12807_gb300 import synth

pytestmark = pytest.mark.gpu

# (channels, samples, bits, plan rows, masked channels): one flush and several, tile edges, downsampled rows
CASES = {
    "8bit_256": (256, 512 * 20 + 4475, 8, [(0, 0.5, 33, 1)], 0),
    "8bit_258": (258, 8191, 8, [(0, 0.5, 40, 1)], 0),
    "8bit_wide_masked": (700, 9001, 8, [(0, 0.5, 40, 1), (20, 0.5, 20, 2)], 61),
    "8bit_staged": (256, 20003, 8, [(0, 0.5, 40, 1), (20, 0.5, 20, 2), (30, 0.5, 20, 4)], 3),
    "1bit_255": (256, 9003, 1, [(0, 0.5, 20, 1)], 1),
    "1bit_staged": (96, 30003, 1, [(0, 0.5, 17, 1), (8, 1, 16, 2), (24, 2, 15, 16)], 5),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_spectra_of_the_float_series(name):
    import torch

    from paper_1912_12807_gb300 import pss
    nchan, nsamp, nbits, rows, masked = CASES[name]
    g = np.random.default_rng(len(name))
    d = g.integers(0, 256, (nsamp, nchan * nbits // 8), dtype=np.uint8)
    x = d if nbits == 8 else np.unpackbits(d, axis=1)
    mask = np.ones(nchan, dtype=np.uint8)
    mask[g.permutation(nchan)[:masked]] = 0
    lo, hi = (1050.0, 1450.0) if nbits == 8 else (1230.0, 1518.0)
    foff = (hi - lo) / nchan
    plan = pss.Plan(pss.FilDesc(nchan, nsamp, 2e-4, lo + 0.5 * foff, foff, nbits, chan_mask=mask if masked else None),
                    [synth.Stage(*r) for r in rows])
    xc = np.ascontiguousarray(x.T)[mask != 0]
    delays = plan.delays()[:, mask != 0]
    W = 64
    cfg = pss.search_cfg(numharm=2, whiten_block=W)
    ctx = pss.Context(0)
    try:
        got = pss.pss_spectrum(ctx, plan, torch.from_numpy(d).cuda(), cfg, 0, plan.ndm).cpu().numpy()
        pss.pss_ctx_check(ctx)
    finally:
        ctx.close()
    off = first = 0
    for n, t in plan.stage_lengths():
        for i in range(first, first + n):
            if i in (first, first + 1, first + n // 2, first + n - 1):
                s = OD.dedisperse(xc, delays[i], plan.max_delay, t["ds"])
                ref = OS.whiten(OS.half_spectrum(OS.real_series(s, t["nfft"])), W)
                a = got[off:off + t["nfft"] // 2].astype(np.complex128)
                check_powers(np.abs(a) ** 2, np.abs(ref) ** 2, "%s trial %d" % (name, i))
            off += t["nfft"] // 2
        first += n
    assert off == len(got)
