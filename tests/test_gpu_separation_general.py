"""Separation at frame counts without a two-pass plan, over the three forms of the general kernel (up to 128, 304 and 512
frames; packed arithmetic in the first two, scalar in the last), against the oracle: every radix from 2 to 20, one to
five passes, a lateral count that is no multiple of the pixel group.  Bounds as for the other plans: subsets 1e-5 of the
input, amplitudes and maxima 2e-5 in FP32 from the same planes."""
from dataclasses import replace

import numpy as np
import pytest
import torch

import oracle as O
from oracle import separation as OSep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("F", [2, 8, 15, 50, 125, 135, 243, 288, 324, 375, 384, 400, 405, 486, 500, 512])
def test_general_plans(tiny, F):
    from paper_2511_21647_gb300 import _lib as L, rca
    from paper_2511_21647_gb300.pipeline import RcaSession
    g = replace(tiny.geom, n_el=36, P=4, nz=3)
    edges = [0.0, 60.0, 200.0]
    with RcaSession(g) as s:
        x32 = torch.randn(s.planes_shape(F) + (2,), generator=torch.Generator().manual_seed(F))
        x = x32.double().numpy()
        x = x[..., 0] + 1j * x[..., 1]
        prm = rca.make_sep_params(400.0, 2, edges)
        ref = OSep.separate(x, 400.0, np.array(edges))
        got = s.separate(x32.cuda(), prm, L.RCA_C32).cpu().double().numpy()
        got = got[..., 0] + 1j * got[..., 1]
        for k in range(len(ref)):
            assert np.linalg.norm(got[k] - ref[k]) <= 1e-5 * np.linalg.norm(x), k
        for enh in (L.ULM_ENH_XDOPPLER, L.ULM_ENH_COHERENT):
            A, M = s.separate_enhance(x32.cuda(), prm, planes_dtype=L.RCA_C32, enh=enh)
            A, M = A.cpu().numpy(), M.cpu().numpy()
            for k in range(len(ref)):
                if enh == L.ULM_ENH_XDOPPLER:
                    A_o, M_o = O.xdoppler(ref[k])
                else:
                    A_o = np.abs(ref[k][:, :, 0] + ref[k][:, :, 1])
                    M_o = A_o.reshape(F, -1).max(axis=1)
                assert np.linalg.norm(A[k] - A_o) <= 2e-5 * np.linalg.norm(A_o), (k, enh)
                assert np.allclose(M[k], M_o, rtol=2e-5, atol=0), (k, enh)
        assert s.sync_status() == 0
