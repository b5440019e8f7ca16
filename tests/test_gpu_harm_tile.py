"""Harmonic sums of 2-D planes: the row-tile kernel (the default) gives the
bytes of the one-row kernel (PSS_HARM_ROWS=0) at a low threshold, so with
detections at every tile edge: centre rows and numbers of rows that are no
multiple of a tile, planes with fewer rows than a tile, every harmonic count
that the kernel takes and the next larger one, and short spectra."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# (zmax, dz, numharm, sigma)
CASES = [(2, 2.0, 8, 3.2), (14, 2.0, 8, 3.4), (16, 2.0, 16, 3.4), (30, 2.0, 16, 3.4), (7, 0.5, 4, 3.4), (20, 2.0, 2, 3.4),
         (18, 2.0, 1, 3.4), (34, 2.0, 32, 3.6), (64, 2.0, 8, 3.6)]

CHILD = r"""
import sys, numpy as np, torch
sys.path.insert(0, {root!r})
from paper_1912_12807_gb300 import pss, synth
out = []
for nsamp in (1 << 12, 1 << 14):
    wl = synth.workload_small(nsamp=nsamp)
    ctx = pss.Context(0)
    plan = pss.Plan(pss.FilDesc.of(wl.fil), [synth.Stage(45.0, 5.0, 3, 1)])
    d = torch.from_numpy(wl.fil.data).cuda()
    for zmax, dz, nh, sigma in {cases!r}:
        cfg = pss.search_cfg(zmax=zmax, dz=dz, numharm=nh, sigma_thr=sigma, f_lo_hz=2.0)
        raw = pss.pss_search_raw(ctx, plan, d, cfg, 0, plan.ndm)
        assert len(raw) > 50, (zmax, nh, len(raw))
        out.append(raw.view(np.uint8).ravel())
np.save({out!r}, np.concatenate(out))
"""


def test_row_tiles_give_the_bytes_of_single_rows(tmp_path):
    got = []
    for tag in ("1", "0"):
        out = str(tmp_path / ("raw_%s.npy" % tag))
        subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, cases=CASES, out=out)],
                       env=dict(os.environ, PSS_HARM_ROWS=tag), check=True, timeout=600)
        got.append(np.load(out))
    assert got[0].tobytes() == got[1].tobytes()
