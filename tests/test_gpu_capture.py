"""A frame step captured in a CUDA graph (programmatic dependent launches become
edges of the graph) replays to the same state as running it eagerly: the sweep by
rows, by tiles, and the quadtree's kernels, and the batched schedule."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import synth  # noqa: E402
import paper_2606_03989_gb300 as pv  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("prec,topology,batch", [(32, "GRID", False), (32, "QUADTREE", False), (64, "GRID", False),
                                                 (64, "QUADTREE", False), (32, "GRID", True), (32, "QUADTREE", True)])
@pytest.mark.parametrize("size", [(64, 48), (320, 243)])
def test_a_captured_step_replays_as_the_eager_one(prec, topology, batch, size):
    seq = synth.realistic(91, 3, *size)
    frames = [torch.from_numpy(seq.frame(k)).to(DEV) for k in range(3)]
    normals = torch.from_numpy(seq.normals(0)).to(DEV)
    par = pv.params(precision=prec, kf_interval=0, sigma_P=seq.sigma_P, topology=getattr(pv, "TOPOLOGY_" + topology))
    s = torch.cuda.Stream(DEV)
    outs = []
    for captured in (False, True):
        with torch.cuda.stream(s):
            frame, nrm = frames[0].clone(), normals.clone()
            if batch:
                t = pv.Batch([seq.cam.as_tuple()] * 2, par, DEV, stream=s)
                t.set_schedule(pv.SCHED_BATCHED, 4)
                t.set_inputs([frame, frame], [nrm, nrm])
                step = lambda n: t.track(n)
            else:
                t = pv.Tracker(seq.cam.as_tuple(), par, DEV, stream=s)
                step = lambda n: t.track(frame, nrm, n_iters=n)
            for k in range(2):
                frame.copy_(frames[k])
                step(4)
            frame.copy_(frames[2])
            if captured:
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=s):
                    step(4)
                g.replay()
            else:
                step(4)
            s.synchronize()
            outs.append([t.save_state(i)[256:] for i in range(2)] if batch else [t.save_state()[256:]])
            assert t.status() == 0
    assert outs[0] == outs[1]
