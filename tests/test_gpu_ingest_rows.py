"""Ingest of records whose rows begin off 16 bytes (sample counts that are no multiple of 4), tiles of 128 samples and 32
elements that end anywhere, the record's last tile holding 1 to 4 samples, against the oracle's demodulation: FP32 rounding
of the mean, the mixer and 17 filter products, 1e-5 as for the aligned records."""
from dataclasses import replace

import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rf", ["f32", "f16", "i16"])
@pytest.mark.parametrize("n_el,P,ns,F", [(32, 8, 257, 3), (36, 4, 258, 2), (40, 8, 387, 9), (96, 8, 255, 2), (72, 8, 130, 2)])
def test_ingest_rows(tiny, n_el, P, ns, F, rf):
    from paper_2511_21647_gb300 import _lib as L
    from paper_2511_21647_gb300.pipeline import RcaSession
    g = replace(tiny.geom, n_el=n_el, P=P, ns=ns)
    nt = 2 * len(g.ang_rc)
    rng = np.random.default_rng(ns + n_el)
    x = 100.0 * rng.standard_normal((F, nt, n_el, ns)) + 30.0
    kw = {}
    if rf == "i16":
        d = torch.from_numpy(np.round(x).astype(np.int16))
        sc = torch.from_numpy(rng.uniform(0.5, 2.0, (nt, n_el)).astype(np.float32))
        ref = d.numpy().astype(np.float64) * sc.numpy().astype(np.float64)[None, :, :, None]
        kw = dict(rf_dtype=L.RCA_I16, scale=sc.cuda())
    else:
        d = torch.from_numpy(x).to(torch.float16 if rf == "f16" else torch.float32)
        ref = d.double().numpy()
        kw = dict(rf_dtype=L.RCA_F16 if rf == "f16" else L.RCA_F32)
    with RcaSession(g) as s:
        got = s.ingest(d.cuda(), **kw).cpu().double().numpy()
        assert s.sync_status() == 0
    got = (got[..., 0] + 1j * got[..., 1]).transpose(0, 1, 3, 2)
    ref = O.demod(g, ref)
    for part in (slice(None), slice(-4, None)):                          # and the last samples by themselves
        assert np.linalg.norm(got[..., part] - ref[..., part]) < 1e-5 * np.linalg.norm(ref[..., part])
