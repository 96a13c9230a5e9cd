"""Separation at every frame count of the two-pass kernel (plans 12, 16 and 20 times 4 .. 16), against the oracle: windows
of a quarter and of half of the bins at every start (1 band, 4 uneven bands with a low cut, one of them empty at the
shorter counts), a lateral count that is no multiple of the pixel group.  Bounds as for the other plans: subsets 1e-5 of
the input, amplitudes and maxima 2e-5 in FP32 from the same planes."""
from dataclasses import replace

import numpy as np
import pytest
import torch

import oracle as O
from oracle import separation as OSep

pytestmark = pytest.mark.gpu
COUNTS = [48, 60, 64, 72, 80, 96, 100, 120, 128, 144, 160, 180, 192, 200, 240, 256, 300, 320]


@pytest.mark.parametrize("edges", [[0.0, 200.0], [3.0, 6.0, 70.0, 110.0, 200.0]])
@pytest.mark.parametrize("F", COUNTS)
def test_two_pass_plans(tiny, F, edges):
    from paper_2511_21647_gb300 import _lib as L, rca
    from paper_2511_21647_gb300.pipeline import RcaSession
    g = replace(tiny.geom, n_el=36, P=4, nz=3)
    rng = np.random.default_rng(F)
    with RcaSession(g) as s:
        shape = s.planes_shape(F)
        x32 = torch.from_numpy(rng.standard_normal(shape + (2,)).astype(np.float32))
        prm = rca.make_sep_params(400.0, len(edges) - 1, edges)
        for dt, tdt in ((L.RCA_C32, torch.float32), (L.RCA_C16BF, torch.bfloat16), (L.RCA_C16F, torch.float16)):
            xd = x32.to(tdt)
            xr = xd.double().numpy()
            x = xr[..., 0] + 1j * xr[..., 1]
            ref = OSep.separate(x, 400.0, np.array(edges))
            got = s.separate(xd.cuda(), prm, dt).cpu().double().numpy()
            got = got[..., 0] + 1j * got[..., 1]
            for k in range(len(ref)):
                assert np.linalg.norm(got[k] - ref[k]) <= 1e-5 * np.linalg.norm(x), (k, dt)
            for enh in (L.ULM_ENH_XDOPPLER, L.ULM_ENH_COHERENT):
                A, M = s.separate_enhance(xd.cuda(), prm, planes_dtype=dt, enh=enh)
                A, M = A.cpu().numpy(), M.cpu().numpy()
                for k in range(len(ref)):
                    if enh == L.ULM_ENH_XDOPPLER:
                        A_o, M_o = O.xdoppler(ref[k])
                    else:
                        A_o = np.abs(ref[k][:, :, 0] + ref[k][:, :, 1])
                        M_o = A_o.reshape(F, -1).max(axis=1)
                    assert np.linalg.norm(A[k] - A_o) <= 2e-5 * np.linalg.norm(A_o), (k, dt, enh)
                    assert np.allclose(M[k], M_o, rtol=2e-5, atol=0), (k, dt, enh)
        assert s.sync_status() == 0


@pytest.mark.parametrize("enh", [0, 1])
def test_nan_pixels_and_maxima(tiny, enh):
    """a NaN pixel has NaN amplitudes and no part in the maxima, as in k_separate (90 frames)"""
    from paper_2511_21647_gb300 import rca
    from paper_2511_21647_gb300.pipeline import RcaSession
    g = replace(tiny.geom, n_el=36, P=4, nz=3)
    with RcaSession(g) as s:
        for F in (90, 100):
            x = torch.randn(s.planes_shape(F) + (2,), generator=torch.Generator().manual_seed(1)).cuda()
            x[7, 0, 0, 0, 1, 5, 0] = float("nan")
            A, M = s.separate_enhance(x, rca.make_sep_params(400.0, 2), enh=enh)
            assert torch.isnan(A[:, :, 0, 0, 1, 5]).all() and int(torch.isnan(A).sum()) == 4 * F
            assert torch.equal(M, torch.nan_to_num(A).flatten(2).amax(2))
