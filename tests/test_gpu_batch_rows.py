"""Batched beamforming of records that begin off 16 bytes (ns not a multiple of 4), whose demodulation reads rows and
clutter mean element by element: both launch modes give the planes of single calls bit for bit, run after run.  In the
persistent launch the mean comes from other blocks of the same launch."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns,rf", [(258, "f32"), (257, "f16"), (255, "i16"), (256, "f32")])
def test_batch_of_unaligned_records_equals_single_calls(ns, rf):
    import dataclasses
    from paper_2511_21647_gb300 import _lib as L
    from paper_2511_21647_gb300 import rca
    from paper_2511_21647_gb300.pipeline import complex_buffer
    from synth.rca_sim import _tiny_geom
    rf_t = {"f32": L.RCA_F32, "f16": L.RCA_F16, "i16": L.RCA_I16}[rf]
    gen = torch.Generator(device="cuda").manual_seed(ns)
    h = rca.rca_create(0)
    rca.rca_set_stream(h, torch.cuda.current_stream())
    items, keep, single = [], [], []
    for F, K in ((9, 1), (30, 2), (17, 4)):
        g = dataclasses.replace(_tiny_geom(K), ns=ns)
        geo = rca.rca_geometry_create(h, g)
        t = rca.rca_delay_tables(h, geo)
        keep.append((geo, t))
        x = torch.randn((F, 2 * K, g.n_el, ns), generator=gen, device="cuda") + 3.0
        scale = None
        if rf == "i16":
            x, scale = (x * 1000).to(torch.int16), torch.full((2 * K, g.n_el), 1e-3, device="cuda")
        elif rf == "f16":
            x = x.half()
        pl = complex_buffer((F, 2, 2, g.n_slab, g.nz, g.n_el), L.RCA_C32, "cuda")
        items.append(dict(tables=t, rf=x, scale=scale, n_frames=F, planes=pl))
        one = torch.empty_like(pl)
        rca.rca_beamform_projections(h, t, x, rf_t, scale, F, rca.bf_params(), one, L.RCA_C32)
        single.append(one)
    b = rca.rca_batch_create(h, items, rf_t, L.RCA_C32, L.RCA_C32)
    try:
        for mode in (L.RCA_BATCH_PERSISTENT, L.RCA_BATCH_STAGED):
            rca.rca_batch_set_mode(b, mode)
            for _ in range(3):
                for it in items:
                    it["planes"].zero_()
                rca.rca_batch_run(b, use_graph=False, h=h)
                assert rca.rca_sync_status(h) == L.RCA_OK
                for it, one in zip(items, single):
                    assert torch.equal(it["planes"], one), mode
        assert all(float(one.abs().max()) > 0 for one in single)
    finally:
        rca.rca_batch_destroy(b)
        for geo, t in keep:
            rca.rca_tables_destroy(t)
            rca.rca_geometry_destroy(geo)
        rca.rca_destroy(h)
