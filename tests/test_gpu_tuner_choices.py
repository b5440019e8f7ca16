"""The tuner of a prepared batch times the choices that its kernels depend on
and leaves the others at their defaults: the staging budget only where trials
are dedispersed directly, the points per lane only where a plane is summed by
rows; the batch's candidates are those of the untuned search."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import sys, numpy as np
sys.path.insert(0, {root!r})
from paper_1912_12807_gb300 import pss, synth
nchan, nsamp, nbits, ndm, zmax = {shape!r}
d = np.random.default_rng(1).integers(0, 256, (nsamp, nchan * nbits // 8), dtype=np.uint8)
plan = pss.Plan(pss.FilDesc(nchan, nsamp, 2e-4, 1230.0, 288.0 / nchan, nbits), [synth.Stage(0.0, 0.5, ndm, 1)])
cfg = pss.search_cfg(zmax=zmax, numharm=4, sigma_thr=5.0)
b = pss.Batch(plan, cfg)
t = b.tuning
print("TUNED", t["dedisp_kb"], t["harm_run"], len(b.run(d)))
"""

# shape (channels, samples, bits, trials, zmax), is the staging budget timed, are the points per lane
CASES = [((64, 1 << 14, 8, 7, 0), True, True), ((256, 1 << 14, 8, 40, 0), False, True), ((96, 1 << 14, 1, 40, 0), False, True),
         ((96, 1 << 18, 1, 4, 200), False, False), ((96, 1 << 16, 1, 4, 200), False, True)]


@pytest.mark.parametrize("shape,kb,run", CASES)
def test_choices_without_effect_are_not_timed(shape, kb, run):
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, shape=shape)], capture_output=True, text=True, timeout=300,
                       env={**{k: v for k, v in os.environ.items() if not k.startswith("PSS_")}, "PSS_TIMING": "1"})
    assert r.returncode == 0, r.stderr[-2000:]
    assert ("tune dedisp kb" in r.stderr) == kb
    assert ("tune harm run" in r.stderr) == run
    got = r.stdout.split("TUNED")[1].split()
    assert kb or got[0] == "96"
    assert run or got[1] == "8"
