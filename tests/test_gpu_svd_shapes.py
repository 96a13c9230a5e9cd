"""The clutter filter at the sizes where its kernels change: frame tiles of the covariance (n = 16 .. 128 columns in
the last), rows per cluster block (also none), warps that own one to three columns, the basis kernel's limits of 320
and 512 frames, and every padded rank of the projection; exact-SVD scenes against the FP64 oracle (1e-5 of the
input, the filter's FP32 bound)."""
import numpy as np
import pytest

from test_gpu_svd import check, exact_svd_scene, run

pytestmark = pytest.mark.gpu

SIZES = [(2, 1), (9, 3), (16, 7), (48, 9), (65, 13), (127, 17), (128, 21), (129, 32), (144, 25), (256, 4), (257, 31),
         (320, 32), (321, 20), (400, 12), (512, 16), (513, 3), (640, 18)]


@pytest.mark.parametrize("F,rank", SIZES)
def test_filter_sizes(tiny, F, rank):
    from paper_2511_21647_gb300.pipeline import RcaSession
    g = tiny.geom
    rng = np.random.default_rng(F)
    tissue, blood = exact_svd_scene(rng, F, 2 * len(g.ang_rc), g.nzs, g.n_el, rank=rank, amp=100.0)
    sl32 = (tissue + blood).astype(np.complex64)
    with RcaSession(g) as s:
        out = run(s, sl32, F, rank)
    check(out, sl32, blood, rank, 1e-5)
