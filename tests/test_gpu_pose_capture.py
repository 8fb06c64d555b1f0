"""A captured pose: its arrays are read when the graph is replayed, whether
pageable, pinned or on the device."""
import numpy as np
import pytest

import scenegen as sg
from helpers import renderer, set_cam

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("memory", ["pageable", "pinned", "device"])
def test_replay_reads_the_pose_again(memory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    sc = sg.preset("mini")
    oc = sc.octree
    poses = [sg.random_pose(k) for k in (1, 2, 3)]
    hold = [torch.from_numpy(np.array(x, np.float32)) for x in (poses[0].axis_angle, poses[0].R, poses[0].T)]
    hold = [{"pageable": lambda t: t, "pinned": lambda t: t.pin_memory(), "device": lambda t: t.cuda()}[memory](t)
            for t in hold]
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        r = renderer(sc)
        set_cam(r, 0, sg.orbit_camera(sc.centroid, 64, 64, az_deg=40.0))
        F, A = torch.empty((64, 64, oc.C), device="cuda"), torch.empty((64, 64), device="cuda")

        def frame(p):
            r.set_pose(p[0], p[1], p[2])
            r.render_feature_maps(0, F, A)

        want = []
        for p in poses:
            frame((p.axis_angle, p.R, p.T))
            want.append((F.clone(), A.clone()))
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            frame(hold)
        for k in (0, 2, 1):
            for t, x in zip(hold, (poses[k].axis_angle, poses[k].R, poses[k].T)):
                t.copy_(torch.from_numpy(np.array(x, np.float32)))
            s.synchronize()
            g.replay()
            s.synchronize()
            assert torch.equal(F, want[k][0]) and torch.equal(A, want[k][1])
        r.sync_status()
