"""Calls captured into a program's own CUDA graph behind different predecessors: nothing, another kernel, a fill, a copy, and
two joined streams (where the first of the call's dependent launches has more than one predecessor).  Replays give the
plain call's outputs for new inputs."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("before", ["nothing", "kernel", "fill", "copy", "join"])
def test_capture_behind(tiny, tiny_rf, before):
    from paper_2511_21647_gb300 import _lib as L
    from paper_2511_21647_gb300 import rca
    from paper_2511_21647_gb300.pipeline import RcaSession
    F = 16
    src = tiny_rf.rf[:F].cuda().contiguous()
    prm = rca.make_ulm_params(d=5, sig_z=0.807, sig_lat=1.4495, alpha=0.1, ncc_min=0.5)
    with RcaSession(tiny.geom) as s:
        rf, y = src.clone(), torch.ones(1 << 22, device="cuda")
        planes = torch.empty((*s.planes_shape(F), 2), device="cuda")
        cap2, cap3 = 1 << 14, 1 << 12
        bufs = s.loc_buffers(cap2, cap3)
        motion = torch.empty((F, 3), device="cuda")
        slices = torch.randn((F, 2, tiny.geom.nzs, 32, 2), device="cuda")

        def call():
            s.beamform(rf, out=planes)
            s.localize(planes, prm, L.RCA_C32, cap2, cap3, bufs)
            rca.rca_motion_estimate(s.h, s.t, slices, F, motion)

        call()                                           # workspaces
        torch.cuda.synchronize()
        g, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(g):
            cur = torch.cuda.current_stream()
            rca.rca_set_stream(s.h, cur)
            if before == "kernel":
                rf.mul_(1.0)
            elif before == "fill":
                y.zero_()
            elif before == "copy":
                rf.copy_(src)
            elif before == "join":
                side.wait_stream(cur)
                motion.mul_(0.5)
                with torch.cuda.stream(side):
                    for _ in range(4):
                        y.mul_(1.0001)
                    rf[F // 2:].mul_(0.5)                # work that the call has to wait for
                cur.wait_stream(side)
            call()
        rca.rca_set_stream(s.h, torch.cuda.current_stream())
        for k in (1.0, 3.0):
            src.mul_(k)
            rf.copy_(src)
            planes.zero_()
            motion.zero_()
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            assert s.sync_status() == 0
            got = planes.clone(), motion.clone(), int(bufs[1].item()), int(bufs[3].item())
            call()                                       # on the inputs that the graph left
            torch.cuda.synchronize()
            assert torch.equal(planes, got[0]) and torch.equal(motion, got[1])
            assert (int(bufs[1].item()), int(bufs[3].item())) == got[2:] and got[2] > 0
            assert float(planes.abs().max()) > 0
