"""The streamed forward pass of the learned localiser at the sizes where its strips, windows and row runs begin and
end, against the FP64 oracle (rel-L2 <= 1e-2, the network's BF16 bound), and its activations through the gradients
(<= 2e-2)."""
import numpy as np
import pytest
import torch

from oracle import cnn as N

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


@pytest.fixture(scope="module")
def net():
    from paper_2511_21647_gb300 import rca
    h = rca.rca_create(0)
    rca.rca_set_stream(h, torch.cuda.current_stream())
    c = rca.ulm_cnn_create(h, max_pixels=1 << 17, seed=7)
    rng = np.random.default_rng(11)
    params = [p if p.ndim > 1 else 0.05 * rng.standard_normal(p.shape) for p in N.init_params(C=32, seed=5)]
    flat = N.flatten(params).astype(np.float32)
    rca.ulm_cnn_set_params(c, flat)
    yield h, c, N.unflatten(flat.astype(np.float64))
    rca.ulm_cnn_destroy(c)
    rca.rca_destroy(h)


# one pixel; one row; three, two and one planes per strip (W = 31, 32, 42, 63 / 64); a full strip and one column more;
# two and three windows; runs that cross many planes; planes longer than a run
SHAPES = [(1, 1, 1), (3, 2, 5), (5, 7, 31), (4, 9, 32), (3, 4, 42), (3, 5, 63), (2, 5, 64), (1, 6, 127), (2, 6, 128),
          (2, 5, 129), (1, 4, 240), (2, 3, 241), (700, 3, 16), (1, 1000, 20)]


@pytest.mark.parametrize("B,H,W", SHAPES)
def test_forward_shapes(net, B, H, W):
    from paper_2511_21647_gb300 import rca
    h, c, p = net
    rng = np.random.default_rng(B * 1000 + H * 10 + W)
    x = (rng.random((B, H, W)) ** 2).astype(np.float32)
    M = (0.5 + rng.random(B)).astype(np.float32)
    M[-1] = 0.0 if B > 2 else M[-1]                     # a frame without signal: the input counts as zero
    s = np.where(M > 0, np.float32(1) / np.where(M > 0, M, 1), 0).astype(np.float32)
    ref, _ = N.forward(p, (x * s[:, None, None]).astype(np.float64))
    A, Md = torch.from_numpy(x).cuda(), torch.from_numpy(M).cuda()
    buf = torch.full((B * 16 * H * W + 1,), float("nan"), device="cuda")
    for off in (0, 1):                                  # a heatmap that is not 16-byte aligned too
        heat = buf[off:off + B * 16 * H * W].view(B, 4 * H, 4 * W)
        rca.ulm_cnn_forward(c, A, Md, 1, B, H, W, heat)
        got = heat.cpu().numpy()
        assert rca.rca_sync_status(h) == 0
        assert rel(got, ref) < 1e-2


@pytest.mark.parametrize("B,H,W", [(5, 6, 31), (2, 5, 128), (2, 4, 130)])
def test_gradient_shapes(net, B, H, W):
    from paper_2511_21647_gb300 import rca
    h, c, p = net
    rng = np.random.default_rng(3)
    x = (rng.random((B, H, W)) ** 2).astype(np.float32)
    t = rng.random((B, 4 * H, 4 * W)).astype(np.float32)
    loss_o, grads_o = N.loss_and_grads(p, x.astype(np.float64), t.astype(np.float64))
    loss = torch.zeros(1, device="cuda")
    rca.ulm_cnn_train_step(c, torch.from_numpy(x).cuda(), None, 1, B, H, W, torch.from_numpy(t).cuda(), loss, False)
    got = N.unflatten(rca.ulm_cnn_get_grads(c))
    assert rca.rca_sync_status(h) == 0
    assert abs(float(loss.item()) - loss_o) < 1e-2 * loss_o
    assert all(rel(a, b) < 2e-2 for a, b in zip(got, grads_o))
