"""The checked build (bounds-checked indices, NaN in the out-of-image lanes) through
every variant of the sweep kernel: which one runs goes by the tiles of a launch, so
ragged images and batches on each side of the limits, in every schedule. No flag may be
set, and the results are the plain build's."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# launches of tiles of 32 x 4 pixels: up to 114 by rows with more registers, up to 304 by
# rows, up to 608 by tiles, above with streamed stores (FP64: up to 76 by rows)
SINGLE = [(32, 609, 23, 120), (32, 609, 61, 320), (32, 671, 115, 609), (64, 127, 73, 76), (64, 129, 61, 80),
          (64, 609, 61, 320)]
BATCHES = [(32, [(609, 23), (70, 45)], 156), (32, [(609, 61), (33, 17)], 330), (32, [(609, 61), (610, 59)], 620),
           (64, [(129, 61), (33, 17)], 90)]

SCENARIOS = r'''
import json, sys
import numpy as np
import torch
sys.path.insert(0, ROOT)
import synth
import paper_2606_03989_gb300 as pv
dev = torch.device("cuda:0")
out = {"lib": pv.LIB_PATH}
cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)
for prec, w, h, _ in SINGLE:
    s = synth.realistic(11, 4, w, h, sweeps=3)
    t = pv.Tracker(s.cam.as_tuple(), pv.params(precision=prec, kf_interval=2, sigma_P=s.sigma_P), dev)
    poses = []
    for k in range(4):
        t.track(cu(s.frame(k)), cu(s.normals(k)) if k % 2 == 0 else None, 3)
        poses.append(t.pose().tolist())
    out["%dx%d FP%d" % (w, h, prec)] = {"flags": t.status(), "poses": poses}
for prec, sizes, tiles in BATCHES:
    seqs = [synth.realistic(40 + i, 3, w, h) for i, (w, h) in enumerate(sizes)]
    for sched, blocks in ((pv.SCHED_BATCHED, 4), (pv.SCHED_PERSISTENT, 4), (pv.SCHED_PERSISTENT, 1)):
        b = pv.Batch([s.cam.as_tuple() for s in seqs], pv.params(precision=prec, kf_interval=2, sigma_P=0.05), dev)
        b.set_schedule(sched, blocks)
        for k in range(3):
            b.set_inputs([cu(s.frame(k)) for s in seqs], [cu(s.normals(k)) for s in seqs])
            b.track(3)
        out["%d tiles FP%d schedule %d/%d" % (tiles, prec, sched, blocks)] = {"flags": b.status(),
                                                                            "poses": b.poses().tolist()}
print("RESULT " + json.dumps(out))
'''


def run(checked):
    env = dict(os.environ)
    if checked:
        env["PIXVOD_LIBRARY"] = "checked"
    else:
        env.pop("PIXVOD_LIBRARY", None)
    head = "ROOT, SINGLE, BATCHES = %r, %r, %r\n" % (ROOT, SINGLE, BATCHES)
    res = subprocess.run([sys.executable, "-c", head + SCENARIOS], env=env, capture_output=True, text=True, timeout=900)
    assert res.returncode == 0, res.stderr[-3000:]
    line = [l for l in res.stdout.splitlines() if l.startswith("RESULT ")][-1]
    return json.loads(line[len("RESULT "):])


def test_every_sweep_kernel_in_the_checked_build():
    tiles = lambda w, h: (w + 31) // 32 * ((h + 3) // 4)
    assert all(tiles(w, h) == n for _, w, h, n in SINGLE)
    assert all(sum(tiles(*s) for s in sizes) == n for _, sizes, n in BATCHES)
    checked, plain = run(True), run(False)
    assert checked.pop("lib").endswith("libpixvod_checked.so") and plain.pop("lib").endswith("libpixvod.so")
    assert len(checked) == len(SINGLE) + 3 * len(BATCHES)
    for key, r in checked.items():
        assert r["flags"] == 0, (key, r["flags"])
        a, b = np.array(r["poses"]), np.array(plain[key]["poses"])
        assert np.isfinite(a).all(), key
        assert np.abs(a - b).max() < (1e-9 if "FP64" in key else 1e-3), (key, np.abs(a - b).max())
