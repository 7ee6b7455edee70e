"""FP32 reverse sweeps whose adjoint grows by more than 2^58 a sweep. The frame is a
fixed point with a translation of 2^58: the derivative of a translation with respect
to the rotation is as large, and messages that couple the two hand it on from sweep to
sweep, while the depth's adjoint stays of order 1. So a pass that is scaled by what it
reads fits the float range, and two passes' growth together do not. With a constant
image and no pose prior the update is exactly zero and poses and depths do not mix, so
dL/dsigma_N is the depth's alone, and FP32 gives FP64's."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import synth  # noqa: E402
import paper_2606_03989_gb300 as pv  # noqa: E402

DEV = torch.device("cuda:0")
W, H, SWEEPS, RHO = 45, 13, 3, 2.0 ** 58
LOW = np.tril_indices(6)


def frame_state(blob, precision):
    """The blob of a keyframe with poses, depths and messages as described above."""
    out = bytearray(blob)
    head = np.frombuffer(blob, np.int64, 32)
    pitch, dt = int(head[5]), np.float32 if precision == 32 else np.float64
    px = np.frombuffer(out, dt, 151 * H * pitch, int(head[8])).reshape(151, H, pitch)[:, :, :W]
    msg = 0.3 * np.eye(6)
    msg[0, 4] = msg[4, 0] = msg[1, 3] = msg[3, 1] = 0.15  # rotations with the translations that they cause
    px[5] = RHO
    px[6] = np.random.default_rng(1).normal(size=(H, W)).astype(np.float32) * np.float32(0.1)
    px[7:28] = 0.0
    v, u = np.mgrid[:H, :W]
    for k, has in enumerate((u > 0, u < W - 1, v > 0, v < H - 1)):
        px[35 + 27 * k:35 + 27 * k + 21] = msg[LOW][:, None, None] * has
        px[7:28] += px[35 + 27 * k:35 + 27 * k + 21]
    return bytes(out)


@pytest.mark.parametrize("every", [1, 2])
def test_growth_of_two_sweeps_does_not_overflow(every):
    seq = synth.realistic(5, 2, W, H)
    flat = torch.full((H, W), 0.5, device=DEV)
    normals = torch.from_numpy(seq.normals(0)).to(DEV)
    g_inv = np.random.default_rng(2).normal(size=(H, W))
    out = {}
    for prec in (64, 32):
        t = pv.Tracker(seq.cam.as_tuple(), pv.params(precision=prec, kf_interval=0, sigma_D=1.0, sigma_P=2.0 ** 70,
                                                      sigma_R=1.0, sigma_N=1.0, sigma_Z=1.0), DEV)
        t.set_recording(SWEEPS, every)
        t.track(flat, normals)
        t.load_state(frame_state(t.save_state(), prec))
        t.track(flat, n_iters=SWEEPS)
        assert t.status() == 0
        # how much of the growth the sums keep depends on the order of their additions,
        # so several passes
        for _ in range(8):
            g = t.backward(np.ones(6), g_inv)
            assert g["status"] == pv.OK
            for k in ("sigma_D", "sigma_N", "I_s", "I_t"):
                assert bool(torch.isfinite(torch.as_tensor(g[k])).all()), (prec, k)
            out.setdefault(prec, []).append(float(g["sigma_N"]))
    # a fifth of the gradient is the last pass's, which reads the depth's adjoint some
    # 2^140 below its largest value: subnormal floats of 6 bits and more
    assert out[64][0] != 0 and out[32] == pytest.approx(out[64], rel=5e-3)
