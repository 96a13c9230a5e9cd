"""Batches of wider arrays and of mixed widths, whose Stage 1 runs the unpaired row loop while single calls run the paired
or split one: the sums have the same order, so the planes agree bit for bit, in both launch modes and IQ precisions."""
import dataclasses

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths,iq", [((96,), "c32"), ((32, 96), "c32"), ((64, 128), "c32"), ((160, 36), "c32"), ((96, 64), "c16f")])
def test_batch_widths_equal_single_calls(widths, iq):
    from paper_2511_21647_gb300 import _lib as L
    from paper_2511_21647_gb300 import rca
    from paper_2511_21647_gb300.pipeline import complex_buffer
    from synth.rca_sim import _tiny_geom
    iq_t = {"c32": L.RCA_C32, "c16f": L.RCA_C16F}[iq]
    gen = torch.Generator(device="cuda").manual_seed(sum(widths))
    h = rca.rca_create(0)
    rca.rca_set_stream(h, torch.cuda.current_stream())
    items, keep, single = [], [], []
    for q, n_el in enumerate(widths):
        g = dataclasses.replace(_tiny_geom(2 - q), n_el=n_el, P=4, nz=45)
        geo = rca.rca_geometry_create(h, g)
        t = rca.rca_delay_tables(h, geo)
        keep.append((geo, t))
        F, nt = 6 + 5 * q, 2 * (2 - q)
        x = torch.randn((F, nt, n_el, g.ns), generator=gen, device="cuda") + 1.0
        pl = complex_buffer((F, 2, 2, g.n_slab, g.nz, n_el), L.RCA_C32, "cuda")
        items.append(dict(tables=t, rf=x, n_frames=F, planes=pl))
        one = torch.empty_like(pl)
        rca.rca_beamform_projections(h, t, x, L.RCA_F32, None, F, rca.bf_params(iq_dtype=iq_t), one, L.RCA_C32)
        single.append(one)
    b = rca.rca_batch_create(h, items, L.RCA_F32, iq_t, L.RCA_C32)
    try:
        for mode in (L.RCA_BATCH_PERSISTENT, L.RCA_BATCH_STAGED):
            rca.rca_batch_set_mode(b, mode)
            for it in items:
                it["planes"].zero_()
            rca.rca_batch_run(b, use_graph=False, h=h)
            assert rca.rca_sync_status(h) == L.RCA_OK
            for it, one in zip(items, single):
                assert float(one.abs().max()) > 0 and torch.equal(it["planes"], one), mode
    finally:
        rca.rca_batch_destroy(b)
        for geo, t in keep:
            rca.rca_tables_destroy(t)
            rca.rca_geometry_destroy(geo)
        rca.rca_destroy(h)
