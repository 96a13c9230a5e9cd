"""Detections with more peaks in a strip than its slot keeps (white-noise amplitudes, low NCC threshold): the status word
says so, the count is the true one, and the list stays in order over it, with entries of frame n_frames behind those
kept, whatever the buffer held.  Pairing that list gives the oracle's pairs of the entries kept, from ulm_localize as
from ulm_detect2d and ulm_pair3d."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fill", [0, -1, 7])
def test_list_with_dropped_candidates_stays_in_order(fill):
    import dataclasses
    from paper_2511_21647_gb300 import _lib as L
    from paper_2511_21647_gb300 import rca
    from paper_2511_21647_gb300.pipeline import RcaSession, list2d_numpy, list3d_numpy
    from synth.rca_sim import _tiny_geom
    g = dataclasses.replace(_tiny_geom(1), n_el=64, nz=64)
    F, S = 3, 64 // g.P
    gen = torch.Generator(device="cuda").manual_seed(5)
    planes = torch.randn((F, 2, 2, S, g.nz, 64, 2), generator=gen, device="cuda")
    prm = rca.make_ulm_params(d=3, sig_z=0.8, sig_lat=1.4, alpha=0.01, ncc_min=0.2)
    cap2, cap3 = 1 << 15, 1 << 14
    with RcaSession(g) as s:
        out = [torch.full((c, 10), fill, dtype=torch.int32, device="cuda") for c in (cap2, cap3, cap2, cap3)]
        n2, n3, m2, m3 = (torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(4))
        poff = torch.zeros(F * 2 * S + 1, dtype=torch.int32, device="cuda")
        s.localize(planes, prm, L.RCA_C32, cap2, cap3, (out[0], n2, out[1], n3))
        assert s.sync_status() == L.RCA_ERR_CAPACITY
        A, M = s.enhance(planes)
        rca.ulm_detect2d(s.h, s.t, A, M, F, prm, out[2], cap2, m2, None, poff)
        assert s.sync_status() == L.RCA_ERR_CAPACITY
        rca.ulm_pair3d(s.h, s.t, out[2], m2, cap2, F, out[3], cap3, m3)
        assert s.sync_status() == L.RCA_OK
        n, p = int(n2.item()), int(n3.item())
        kept = int(poff[-1].item())
        assert 0 < kept < n <= cap2 and 0 < p <= cap3
        assert (int(m2.item()), int(m3.item())) == (n, p)
        assert torch.equal(out[0][:n], out[2][:n]) and torch.equal(out[1][:p], out[3][:p])
        a = list2d_numpy(out[0], n)
        pairs = list3d_numpy(out[1], p)
    key = (a["frame"] * 2 + a["axis"]) * S + a["slab"]
    assert np.all(np.diff(key) >= 0) and np.all(key[:kept] < F * 2 * S)
    assert np.all(a["frame"][kept:] == F)
    ref = np.zeros(kept, dtype=O.LOC2D)
    for name in O.LOC2D.names:
        ref[name] = a[name][:kept]
    want = [(int(r["i_xz"]), int(r["i_yz"])) for r in O.pair3d(ref, g.P)]
    assert [(int(r["i_xz"]), int(r["i_yz"])) for r in pairs] == want
