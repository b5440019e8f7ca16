"""What admission charges for the dedispersion kernels' tables and for the
unpacked forms of a file: no more than such a batch can come to hold."""
import numpy as np
import pytest

from paper_1912_12807_gb300 import synth


@pytest.fixture(scope="module")
def L():
    from paper_1912_12807_gb300 import pss
    pss.lib()
    return pss


def _slack(n):
    return n + n // 8 + 256


def test_table_bytes_are_within_what_the_tables_can_take(L):
    # two plans that differ in the kept channels alone: unpacked rows, delays and shared-sum tables
    nchan, nsamp, ndm = 4096, 1 << 16, 60
    mask = np.zeros(nchan, dtype=np.uint8)
    mask[::2] = 1
    mask[-1] = 1  # the band's edges kept: the same largest delay, so the same series
    mask[0] = 1
    got = []
    for m in (None, mask):
        plan = L.Plan(L.FilDesc(nchan, nsamp, 2e-4, *synth.band(1050.0, 1450.0, nchan), chan_mask=m), [synth.Stage(0.0, 0.5, ndm, 1)])
        got.append((L.pss_search_footprint(plan, L.search_cfg(numharm=8)), nchan if m is None else int(m.sum())))
    dck = got[0][1] - got[1][1]
    pitch = (nsamp + 1024 + 256 + 63) // 64 * 64
    most = _slack(dck * pitch) + _slack(4 * dck * (ndm + 1)) + _slack(8 * ndm * dck)
    assert 0 < got[0][0] - got[1][0] <= most


def test_plans_of_many_trials_pay_nothing_for_tables(L):
    # more than 256 trials: a batch runs 30 % of them at once in buffers counted for up to 1024
    nchan, nsamp, nfft, ndm = 256, 1 << 18, 1 << 18, 1001
    plan = L.Plan(L.FilDesc(nchan, nsamp, 2e-4, *synth.band(1050.0, 1450.0, nchan)), [synth.Stage(0.0, 0.5, ndm, 1)])
    got = L.pss_search_footprint(plan, L.search_cfg(zmax=0, numharm=16))
    assert plan.trial(0)["nfft"] == nfft
    parts = [nchan * nsamp, nchan * ((nsamp + 1024 + 256 + 63) // 64 * 64) + 64, 4 * nchan * (ndm + 1), 4, 8, nfft // 2 * 8, nfft * 8,
             ndm * nfft * 4, ndm * 8, ndm * nfft * 4, 4 * 16 * 8, 5 * 4] + 3 * [ndm * nfft // 2 * 8]
    rest = got - sum(_slack(p) for p in parts)
    assert 0 < rest < _slack(32 << 20)  # the candidates


def test_bit_sliced_files_are_not_charged_for_bytes(L):
    nchan, nsamp = 96, 1 << 22
    desc = L.FilDesc(nchan, nsamp, 2.5e-4, *synth.band(1230.0, 1518.0, nchan), nbits=1)
    got = L.pss_search_footprint(L.Plan(desc, [synth.Stage(0.0, 0.5, 8, 1)]), L.search_cfg(numharm=8))
    nfft = 1 << 22
    others = _slack(nchan // 8 * nsamp) + 2 * _slack(8 * nfft * 4) + 3 * _slack(8 * nfft // 2 * 8) + _slack(nfft * 8) + _slack(nfft // 2 * 8)
    bits = _slack(nchan * (nsamp + 4096 + 1024) // 8 + 65536)
    assert got < others + bits + (64 << 20) < others + nchan * nsamp


@pytest.mark.gpu
def test_bit_sliced_files_take_no_rows_of_bytes(L):
    import torch
    nchan, nsamp = 96, 1 << 23  # 96 MiB in the file, 768 MiB as bytes
    dev = torch.randint(0, 256, (nsamp, nchan // 8), dtype=torch.uint8, device="cuda")
    desc = L.FilDesc(nchan, nsamp, 2.5e-4, *synth.band(1230.0, 1518.0, nchan), nbits=1)
    plan = L.Plan(desc, [synth.Stage(0.0, 0.5, 2, 1)])
    calls = [lambda c: L.pss_dedisperse(c, plan, dev, 0, 2), lambda c: L.pss_single_pulse(c, plan, dev, 0, 2, sigma_thr=30.0),
             lambda c: L.pss_fold(c, plan, dev, np.array([1]), np.array([20.0]), nbin=32)]
    for call in calls:
        ctx = L.Context(0)  # (kernels and allocator caches in place)
        call(ctx)
        ctx.close()
        torch.cuda.synchronize()
        ctx = L.Context(0)
        try:
            free0 = torch.cuda.mem_get_info()[0]
            call(ctx)
            torch.cuda.synchronize()
            taken = free0 - torch.cuda.mem_get_info()[0]
            series = 256 * 4 * nsamp if call is calls[2] else 4 * 4 * nsamp
            assert taken < _slack(nchan * nsamp // 8) + _slack(series) + (64 << 20)
        finally:
            ctx.close()
