"""The sweep by rows (images of few tiles) and by tiles, on both sides of the rule
that chooses between them and at ragged sizes: one sweep against the oracle, and
batches swept by tiles or by rows against their sequences tracked alone, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import synth  # noqa: E402
import paper_2606_03989_gb300 as pv  # noqa: E402

from helpers import oracle_intrinsics, oracle_params, oracle_window, synthetic_state  # noqa: E402
from test_gpu_parity import one_sweep_check, sample_pixels  # noqa: E402

DEV = torch.device("cuda:0")


# tiles of 32 x 4: up to 304 (FP32; up to 114 with more registers) or 76 (FP64) are swept by rows
@pytest.mark.parametrize("prec,size,tiles", [(32, (31, 3), 1), (32, (608, 23), 114), (32, (609, 23), 120), (32, (608, 63), 304), (32, (609, 61), 320),
                                             (64, (33, 5), 4), (64, (127, 74), 76), (64, (129, 61), 80)])
def test_one_sweep_on_both_sides_of_the_rule(prec, size, tiles):
    w, h = size
    assert (w + 31) // 32 * ((h + 3) // 4) == tiles
    seq = synth.realistic(8, 2, w, h)
    p = oracle_params(sigma_P=seq.sigma_P)
    c = synthetic_state(h, w, p, seed=w, logz=np.log(seq.depth(0)))
    one_sweep_check(seq.cam, p, c, oracle_window(seq, oracle_intrinsics(seq.cam)), prec,
                    sample_pixels(h, w, min(60, w * h), prec))


@pytest.mark.parametrize("prec,sizes", [(32, [(608, 63), (609, 61), (70, 45)]), (32, [(70, 45), (320, 61), (31, 3)]),
                                         (64, [(127, 74), (129, 61), (33, 17)]), (64, [(33, 17), (65, 35)])])
def test_a_batch_matches_its_sequences(prec, sizes):
    seqs = [synth.realistic(60 + i, 3, w, h) for i, (w, h) in enumerate(sizes)]
    frames = [[torch.from_numpy(s.frame(k)).to(DEV) for k in range(3)] for s in seqs]
    normals = [torch.from_numpy(s.normals(0)).to(DEV) for s in seqs]
    par = pv.params(precision=prec, kf_interval=0, sigma_P=0.05)
    alone = []
    for s, f, n in zip(seqs, frames, normals):
        t = pv.Tracker(s.cam.as_tuple(), par, DEV)
        t.track(f[0], n)
        for k in (1, 2):
            t.track(f[k], n_iters=3)
        alone.append(t.save_state())
    for sched, blocks in ((pv.SCHED_PLAIN, 4), (pv.SCHED_BATCHED, 4), (pv.SCHED_PERSISTENT, 4), (pv.SCHED_PERSISTENT, 1)):
        b = pv.Batch([s.cam.as_tuple() for s in seqs], par, DEV)
        b.set_schedule(sched, blocks)
        for k in range(3):
            b.set_inputs([f[k] for f in frames], normals)
            b.track(3)
        assert b.status() == 0
        for i in range(len(seqs)):
            assert b.save_state(i) == alone[i], (sched, blocks, i)
