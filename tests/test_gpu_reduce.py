"""The pose average over groups of tiles, around the sizes where a block takes one
tile or several and where its last group is short, against the mean of the state."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import synth  # noqa: E402
import paper_2606_03989_gb300 as pv  # noqa: E402

DEV = torch.device("cuda:0")


# tiles of 32 x 4: 1, 608 (a block each), 609 and 693 (two a block, the last alone), 1225 (three)
@pytest.mark.parametrize("prec", [32, 64])
@pytest.mark.parametrize("size,tiles", [((31, 3), 1), ((607, 126), 608), ((671, 115), 609), ((333, 251), 693),
                                        ((1117, 139), 1225)])
def test_the_pose_is_the_mean_over_the_pixels(prec, size, tiles):
    w, h = size
    assert (w + 31) // 32 * ((h + 3) // 4) == tiles
    seq = synth.realistic(12, 2, w, h)
    t = pv.Tracker(seq.cam.as_tuple(), pv.params(precision=prec, kf_interval=0, sigma_P=seq.sigma_P), DEV)
    t.track(torch.from_numpy(seq.frame(0)).to(DEV), torch.from_numpy(seq.normals(0)).to(DEV))
    t.track(torch.from_numpy(seq.frame(1)).to(DEV), n_iters=2)
    mu = np.asarray(t.state().mu[..., :6], dtype=np.float64).reshape(-1, 6)
    # a sum of n values in FP64, in any order: n 2^-53 sum |x|, on either side
    tol = 2 * len(mu) * 2.0 ** -53 * np.abs(mu).mean(axis=0)
    assert (np.abs(t.pose() - mu.mean(axis=0)) <= tol + 1e-300).all()
