"""Stage 1 where the pixel pairs share their warps with a second run of rows (32, 96, 160 and 224 elements), row counts
that end inside a tile and inside a run, against the sum over elements in FP64 on the library's own delay and weight
tables (which test_gpu_beamform compares with the oracle): what is left is the kernel's FP32 rounding of at most 448
products, far below 1e-5; 2e-3 for FP16 samples and weights."""
from dataclasses import replace

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _slices(s, g, iq):
    """iq [F][2K][ns][N] complex -> slices [F][2K][nzs][N]"""
    from paper_2511_21647_gb300 import _lib as L
    from paper_2511_21647_gb300 import rca
    tx, rx, W, dmax = (rca.rca_tables_download(s.t, t) for t in (L.RCA_TAB_TX_Q16, L.RCA_TAB_RX_Q16, L.RCA_TAB_W,
                                                                 L.RCA_TAB_DMAX))
    F, nt, ns, N = iq.shape
    out = np.zeros((F, nt, g.nzs, N), dtype=np.complex128)
    for k in range(nt):
        for r in range(g.nzs):
            for d in range(int(dmax[r]) + 1):
                q = int(tx[k, r]) + int(rx[r, d])
                if d >= N or q < 0 or q > (ns - 1) << 16:
                    continue
                n, fr = q >> 16, (q & 0xffff) / 65536.0
                v = iq[:, k, n] * (1 - fr) + (iq[:, k, n + 1] * fr if fr else 0)
                v = v * complex(W[r, d])
                out[:, k, r, d:] += v[:, :N - d]
                if d:
                    out[:, k, r, :N - d] += v[:, d:]
    return out


@pytest.mark.parametrize("iq_name,tdt,tol", [("C32", torch.float32, 1e-5), ("C16F", torch.float16, 2e-3),
                                             ("C16BF", torch.bfloat16, 1e-5)])
@pytest.mark.parametrize("ns", [256, 500])                             # the deepest rows past the last sample, or within
@pytest.mark.parametrize("N,nz,z0", [(32, 80, 5e-3), (32, 10, 2e-3), (96, 20, 12e-3), (96, 23, 18e-3), (160, 9, 30e-3),
                                     (224, 14, 40e-3)])
def test_split_stage1(tiny, N, nz, z0, ns, iq_name, tdt, tol):
    from paper_2511_21647_gb300 import _lib as L
    from paper_2511_21647_gb300.pipeline import RcaSession
    g = replace(tiny.geom, n_el=N, nz=nz, z0=z0, ns=ns)
    F, nt = 2, 2 * len(g.ang_rc)
    rng = np.random.default_rng(N + nz)
    iq = torch.from_numpy(rng.standard_normal((F, nt, g.ns, N, 2)).astype(np.float32)).to(tdt).cuda()
    r = iq.float().cpu().numpy().astype(np.float64)
    with RcaSession(g) as s:
        ref = _slices(s, g, r[..., 0] + 1j * r[..., 1])
        got = s.stage1(iq, iq_dtype=getattr(L, "RCA_" + iq_name)).cpu().numpy().astype(np.float64)
        assert s.sync_status() == 0
    got = got[..., 0] + 1j * got[..., 1]
    for rows in (slice(None), slice(-3, None)):                          # and the last rows by themselves; nothing adds up to zero
        assert np.linalg.norm(got[:, :, rows] - ref[:, :, rows]) <= tol * np.linalg.norm(ref[:, :, rows])
