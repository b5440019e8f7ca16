"""A prepared batch holds no more device memory than admission charges for its
shape, whatever its tuner tried: few and many trials, staged plans, 8 and 1 bit."""
import pytest

from paper_1912_12807_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1912_12807_gb300 import pss
    pss.lib()
    return pss


@pytest.mark.parametrize("shape", [(256, 1 << 15, 8, [(0, 0.5, 40, 1)]), (256, 1 << 15, 8, [(0, 0.5, 300, 1)]),
                                   (600, 20011, 8, [(0, 0.25, 70, 1), (17.5, 0.5, 100, 2), (67.5, 1, 30, 8)]),
                                   (96, 1 << 16, 1, [(0, 0.5, 300, 1), (150, 1, 40, 2)]), (96, 1 << 16, 1, [(0, 0.5, 20, 1)]),
                                   (248, 60001, 1, [(0, 5, 40, 1)])])
def test_footprint_covers_the_batch(L, shape):
    nchan, nsamp, nbits, rows = shape
    lo, hi = (300.0, 400.0) if nchan == 248 else (1230.0, 1518.0)
    plan = L.Plan(L.FilDesc(nchan, nsamp, 2.5e-4, *synth.band(lo, hi, nchan), nbits=nbits), [synth.Stage(*r) for r in rows])
    for zmax in (0, 20):
        cfg = L.search_cfg(zmax=zmax, numharm=4)
        b = L.Batch(plan, cfg)
        try:
            assert b.footprint <= L.pss_search_footprint(plan, cfg)
        finally:
            b.close()
