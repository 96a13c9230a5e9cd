"""Inference whose heatmap lies over its own input planes or their maxima gives the heatmap of separate buffers."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("at", ["start", "middle", "end", "maxima"])
def test_heatmap_over_the_input(at):
    from paper_2511_21647_gb300 import rca
    B, H, W = 700, 40, 32
    px = B * H * W
    h = rca.rca_create(0)
    rca.rca_set_stream(h, torch.cuda.current_stream())
    net = rca.ulm_cnn_create(h, max_pixels=px, seed=3)
    gen = torch.Generator(device="cuda").manual_seed(9)
    A = torch.rand((B, H, W), generator=gen, device="cuda")
    M = 0.5 + torch.rand(B // 4, generator=gen, device="cuda")
    ref = torch.empty((B, 4 * H, 4 * W), device="cuda")
    rca.ulm_cnn_infer(net, A, M, 4, B, H, W, ref)
    mem = torch.zeros(17 * px, device="cuda")
    a = {"start": 0, "middle": 7 * px, "end": 15 * px + 64, "maxima": 16 * px}[at]
    src = mem[a:a + px]
    src.copy_(A.view(-1))
    m = M
    if at == "maxima":
        m = mem[8 * px:8 * px + M.numel()]
        m.copy_(M)
    rca.ulm_cnn_infer(net, src, m, 4, B, H, W, mem)
    torch.cuda.synchronize()
    assert rca.rca_sync_status(h) == 0
    assert torch.equal(mem[:16 * px].view_as(ref), ref)
    rca.ulm_cnn_destroy(net)
    rca.rca_destroy(h)
