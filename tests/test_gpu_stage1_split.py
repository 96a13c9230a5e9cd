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


@pytest.mark.parametrize("tuned", [(False, False), (True, True), (True, False)])
def test_split_batch_equals_single_calls(tiny, tiny_rf, tuned):
    """32 elements in a batch with a row per thread (the default tiles), two (the tuned tiles) or both, in each launch mode:
    the planes of the single calls bit for bit"""
    from paper_2511_21647_gb300 import _lib as L
    from paper_2511_21647_gb300 import rca
    from paper_2511_21647_gb300.pipeline import complex_buffer
    h = rca.rca_create(0)
    rca.rca_set_stream(h, torch.cuda.current_stream())
    g, items, keep = tiny.geom, [], []
    for tune, F in zip(tuned, (9, 30)):
        geo = rca.rca_geometry_create(h, g)
        t = rca.rca_delay_tables(h, geo)
        rf = tiny_rf.rf[:F].contiguous().cuda()
        if tune:
            iq = complex_buffer((F, 2 * len(g.ang_rc), g.ns, g.n_el), L.RCA_C32, "cuda")
            rca.rca_ingest(h, t, rf, L.RCA_F32, None, F, L.RCA_CLUTTER_MEAN, iq, L.RCA_C32)
            rca.rca_autotune(h, t, iq, L.RCA_C32, F)
        items.append(dict(tables=t, rf=rf, n_frames=F, planes=complex_buffer((F, 2, 2, g.n_slab, g.nz, g.n_el), L.RCA_C32, "cuda")))
        keep.append(geo)
    ref = []
    for it in items:
        p = torch.zeros_like(it["planes"])
        rca.rca_beamform_projections(h, it["tables"], it["rf"], L.RCA_F32, None, it["n_frames"], rca.bf_params(), p,
                                     L.RCA_C32)
        ref.append(p)
    b = rca.rca_batch_create(h, items, L.RCA_F32, L.RCA_C32, L.RCA_C32)
    for mode in (L.RCA_BATCH_PERSISTENT, L.RCA_BATCH_STAGED):
        rca.rca_batch_set_mode(b, mode)
        for it in items:
            it["planes"].zero_()
        rca.rca_batch_run(b, use_graph=False, h=h)
        assert rca.rca_sync_status(h) == L.RCA_OK
        assert all(torch.equal(it["planes"], p) for it, p in zip(items, ref))
    rca.rca_batch_destroy(b)
    for it, geo in zip(items, keep):
        rca.rca_tables_destroy(it["tables"])
        rca.rca_geometry_destroy(geo)
    rca.rca_destroy(h)
