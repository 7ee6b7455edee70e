"""Sweeps captured in a CUDA graph before a checkpoint is loaded: the replayed sweeps
clear the values that the checkpoint holds in the identity slots that a quadtree pixel
does not use, as eager sweeps do."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import synth  # noqa: E402
import paper_2606_03989_gb300 as pv  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("sweeps", [2, 4])
def test_replayed_sweeps_clear_a_loaded_states_unused_slots(precision, sweeps):
    w, h = 70, 45
    seq = synth.realistic(5, 2, w, h)
    frames = [torch.from_numpy(seq.frame(k)).to(DEV) for k in range(2)]
    normals = torch.from_numpy(seq.normals(0)).to(DEV)
    s = torch.cuda.Stream(DEV)
    with torch.cuda.stream(s):
        t = pv.Tracker(seq.cam.as_tuple(), pv.params(precision=precision, kf_interval=0, topology=pv.TOPOLOGY_QUADTREE,
                                                      sigma_P=0.05), DEV, stream=s)
        t.track(frames[0], normals)
        t.track(frames[1], n_iters=2)
        clean = t.save_state()
        head = np.frombuffer(clean, np.int64, 32)
        plane = h * int(head[5]) * (precision // 8)
        lo, hi = int(head[8]) + 62 * plane, int(head[8]) + 143 * plane  # planes 62..142: slots 1..3
        dirty = bytearray(clean)
        np.frombuffer(dirty, np.float32 if precision == 32 else np.float64, (hi - lo) // (precision // 8),
                      lo).reshape(81, h, -1)[:, :, :w] = 3.0
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            t.sweep(sweeps)
        t.load_state(clean)
        t.sweep(sweeps)
        eager = t.save_state()
        t.load_state(bytes(dirty))
        assert t.save_state()[lo:hi] == dirty[lo:hi]  # what was loaded, until a sweep
        g.replay()
        s.synchronize()
        assert t.save_state() == eager
        for n in (1, 2):  # loads between single sweeps: both buffers have held values
            t.load_state(bytes(dirty))
            t.sweep(n)
            assert not any(t.save_state()[lo:hi])
        t.sweep(1)
        assert not any(t.save_state()[lo:hi])
    assert t.status() == 0
