"""Motion estimation at every transform length of either axis (32 to 256 columns; 2 to 512 padded rows, of which up to
16 are one thread's) and with frames in more than one chunk, against the oracle on moving speckle; the bounds of
test_gpu_motion."""
from dataclasses import replace

import numpy as np
import pytest

from test_gpu_motion import c_tensor, compare, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,nz,us,F", [(64, 2, 1, 3), (128, 2, 2, 3), (256, 4, 2, 3), (32, 8, 2, 3),
                                       (64, 9, 2, 4), (128, 17, 2, 3), (256, 33, 2, 3), (32, 128, 1, 5), (64, 129, 1, 3),
                                       (256, 256, 2, 3), (32, 512, 1, 4), (128, 250, 2, 20)])
def test_motion_sizes(tiny, N, nz, us, F):
    from paper_2511_21647_gb300.pipeline import RcaSession
    g = replace(tiny.geom, n_el=N, nz=nz, us=us)
    nzs, nt = g.nzs, 2 * len(g.ang_rc)
    rng = np.random.default_rng(N + nz)
    base = rng.normal(size=(nt, nzs, N)) + 1j * rng.normal(size=(nt, nzs, N))
    base = base + 0.6 * (np.roll(base, 1, -1) + np.roll(base, 1, -2))        # a peak wider than one pixel
    sl = np.empty((F, nt, nzs, N), dtype=np.complex64)
    for f in range(F):
        dz, dx = (0, 0) if f == 0 else (int(rng.integers(-nzs // 4, nzs // 4 + 1)), int(rng.integers(-N // 4, N // 4)))
        moved = np.roll(base, (dz, dx), (1, 2))
        sl[f] = moved + 0.05 * (rng.normal(size=base.shape) + 1j * rng.normal(size=base.shape))
    with RcaSession(g) as s:
        motion, shifts, peaks = run_gpu(s, c_tensor(sl), F, nt)
        again = run_gpu(s, c_tensor(sl), F, nt)
    assert all(np.array_equal(a, b) for a, b in zip((motion, shifts, peaks), again))
    frames = sorted({0, 1, F // 2, F - 1})
    compare(g, sl.astype(np.complex128), frames, motion, shifts, peaks)
