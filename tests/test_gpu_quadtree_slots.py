"""The quadtree sweep does not write identity slots 1..3 of a pixel, which are
zero in both state buffers: a loaded checkpoint that holds values there must
give the same results as one that does not, and zeros from the first sweep on."""
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
@pytest.mark.parametrize("size", [(33, 17), (64, 48)])
def test_loaded_values_in_unused_slots(size, precision):
    w, h = size
    seq = synth.realistic(5, 2, w, h)
    frames = [torch.from_numpy(seq.frame(k)).to(DEV) for k in range(2)]
    normals = torch.from_numpy(seq.normals(0)).to(DEV)

    def tracker():
        t = pv.Tracker(seq.cam.as_tuple(), pv.params(precision=precision, kf_interval=0, topology=1, sigma_P=0.05), DEV)
        t.track(frames[0], normals)
        t.track(frames[1], n_iters=2)
        return t

    clean = tracker().save_state()
    head = np.frombuffer(clean, np.int64, 32)
    pitch, elt = int(head[5]), precision // 8
    dirty = bytearray(clean)
    plane = h * pitch * elt
    lo, hi = int(head[8]) + 62 * plane, int(head[8]) + 143 * plane   # planes 62..142: slots 1..3
    assert not any(clean[lo:hi])
    dirty[lo:hi] = np.full((hi - lo) // elt, 3.0, np.float32 if precision == 32 else np.float64).tobytes()
    for sweeps in (1, 2, 3):
        blobs = []
        for blob in (clean, bytes(dirty)):
            t = tracker()
            t.load_state(blob)
            for _ in range(sweeps):
                t.sweep(1)
            blobs.append(t.save_state())
        assert blobs[0] == blobs[1], sweeps
        assert not any(blobs[1][lo:hi])
