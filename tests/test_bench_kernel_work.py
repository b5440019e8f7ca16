"""The bench's rooflines divide by the kernels a search launches: which ones,
from the library's own choice, the bytes their unpacking writes, and ceilings
that no kernel can pass."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
ALU = {"channel_adds_per_s": 40.0e12, "smem_bound_adds_per_s": 40.0e12, "issue_bound_adds_per_s": 48.0e12,
       "logic_per_s": 20.0e12, "int32_adds_per_s": 40.0e12, "fp32_flops_per_s": 75.0e12}


@pytest.fixture(scope="module")
def B():
    sys.path.insert(0, ROOT)
    import bench
    from paper_1912_12807_gb300 import pss, synth
    pss.lib()
    return bench, pss, synth


def _forms(B, nchan, nsamp, nbits, rows, zmax=0):
    bench, pss, synth = B
    plan = pss.Plan(pss.FilDesc(nchan, nsamp, 2e-4, *synth.band(1050.0, 1450.0, nchan), nbits=nbits), [synth.Stage(*r) for r in rows])
    adds = sum(n * t["nv"] * t["ds"] for n, t in plan.stage_lengths()) * float(nchan)
    return pss.pss_dedisp_forms(plan, pss.search_cfg(zmax=zmax, numharm=8), 0, plan.ndm), adds, plan


def test_forms_count_every_addition_once(B):
    f, adds, _ = _forms(B, 256, 1 << 16, 8, [(0.0, 0.5, 300, 1)])
    assert f["shared"] == adds and f["direct"] == f["bits"] == f["boxcar"] == 0.0
    # less than a byte of shared memory per channel, trial and sample, which the direct kernel reads; more than a third
    assert adds / 3 < f["shared_bytes"] < 1.02 * adds
    f, adds, _ = _forms(B, 64, 1 << 16, 8, [(0.0, 3.0, 101, 1)])
    assert f["direct"] == adds and f["shared_bytes"] == 0.0
    f, adds, _ = _forms(B, 96, 1 << 16, 1, [(0.0, 0.5, 100, 1), (50.0, 1.0, 40, 2)])
    assert f["bits"] == adds and f["direct"] == f["shared"] == f["boxcar"] == 0.0
    f, adds, plan = _forms(B, 64, 1 << 17, 8, [(0.0, 0.5, 40, 8)])
    assert f["boxcar"] == adds / 8 and f["direct"] == f["shared"] == 0.0


def test_unpack_bytes_follow_the_forms(B):
    bench, pss, synth = B
    f1 = synth.make_1bit(96, 1 << 15, 2.5e-4, 1230.0, 1518.0, [], seed=1)
    wl = synth.Workload("one-bit", f1, [synth.Stage(0.0, 1.0, 8, 1)], synth.workload_small().cfg)
    plan = pss.Plan(pss.FilDesc.of(f1), wl.stages)
    forms = pss.pss_dedisp_forms(plan, pss.cfg_of(wl.cfg), 0, plan.ndm)
    w = bench.stage_work(plan, wl, f1.nbytes())
    got = bench.kernel_work(w, wl, f1.nbytes(), forms)
    assert got["unpack"] == ("hbm", 2.0 * f1.nbytes(), "bytes")
    assert {k: v for k, v in got.items() if k != "unpack"} == {k: v for k, v in w.items() if k != "unpack"}


def test_ceilings(B):
    bench = B[0]
    # 1081 trials of 96 x 10^6 1-bit samples in 1.17 ms: below its ceiling, far above the direct kernel's
    bits = {"direct": 0.0, "shared": 0.0, "bits": 96.0e6 * 1081, "boxcar": 0.0, "shared_bytes": 0.0}
    r = bench.roofline_of("dedisperse", "alu", bits["bits"], "channel-adds", 1.17, 1, {}, "measured", ALU, bits)
    assert r["kernels"] == ["k_dedisp_b1"] and 0.4 < r["frac"] < 1.0 and r["peak"] > 2 * 40.0
    # shared sums: the bytes of the tables over the shared-memory rate
    sh = {"direct": 0.0, "shared": 4.0e9, "bits": 0.0, "boxcar": 0.0, "shared_bytes": 3.0e9}
    r = bench.roofline_of("dedisperse", "alu", 4.0e9, "channel-adds", 0.1, 1, {}, "measured", ALU, sh)
    assert abs(r["frac"] - 3.0e9 / 40.0e12 / 1e-4) < 1e-9
    # the direct kernel as before
    d = {"direct": 4.0e9, "shared": 0.0, "bits": 0.0, "boxcar": 0.0, "shared_bytes": 0.0}
    assert bench.roofline_of("dedisperse", "alu", 4.0e9, "channel-adds", 0.2, 1, {}, "measured", ALU, d)["peak"] == 40.0
