"""Pairing of lists on either side of the length from which on two lanes share an entry instead of sixteen: the pairs of a
long list are those of its halves (frames do not interact), which the oracle checks on a part.  Amplitudes from few
values, so that costs tie; planes without entries among them."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu

WIDE = 1 << 18


def make_list(rng, F, S, P, n, z_max):
    a = np.zeros(n, dtype=O.LOC2D)
    pl = np.sort(rng.integers(0, F * 2 * S, n))
    pl[(pl % 7) == 3] -= 1                                    # some planes have none
    a["frame"], a["axis"], a["slab"] = pl // (2 * S), pl // S % 2, pl % S
    a["iz"], a["ilat"] = rng.integers(1, z_max, n), rng.integers(0, S * P, n)
    o = np.lexsort((a["ilat"], a["iz"], pl))
    a = a[o]
    a["z"] = a["iz"] + rng.integers(-2, 3, n) * 0.25
    a["lat"] = a["ilat"]
    a["amp"] = 1.0 + 0.05 * rng.integers(0, 12, n)
    return a


@pytest.mark.parametrize("n,F", [(WIDE - 1, 60), (WIDE, 60), (WIDE + 77, 400), (3 * WIDE // 2, 12)])
def test_pairs_of_a_long_list_are_those_of_its_parts(n, F):
    import dataclasses
    from paper_2511_21647_gb300 import rca
    from paper_2511_21647_gb300._lib import LOC2D
    from paper_2511_21647_gb300.pipeline import RcaSession, list3d_numpy
    from synth.rca_sim import _tiny_geom
    g = dataclasses.replace(_tiny_geom(1), nz=200, ns=900)
    P, S = g.P, g.n_slab
    rng = np.random.default_rng(n)
    a = make_list(rng, F, S, P, n, 199)
    rec = np.zeros(n, dtype=LOC2D)
    for f in O.LOC2D.names:
        rec[f] = a[f]
    L2 = torch.from_numpy(rec.view(np.int32).reshape(n, 10)).cuda()
    with RcaSession(g) as s:
        def pair(lo, hi):
            out = torch.empty((hi - lo, 10), dtype=torch.int32, device="cuda")
            n3 = torch.zeros(1, dtype=torch.int32, device="cuda")
            n2 = torch.tensor([hi - lo], dtype=torch.int32, device="cuda")
            rca.ulm_pair3d(s.h, s.t, L2[lo:hi].contiguous(), n2, hi - lo, F, out, hi - lo, n3)
            assert s.sync_status() == 0
            p = list3d_numpy(out, int(n3.item()))
            return [(int(r["i_xz"]) + lo, int(r["i_yz"]) + lo) for r in p]

        cuts = [int(np.searchsorted(a["frame"], f)) for f in (F // 3, 2 * F // 3)]
        whole = pair(0, n)
        parts = [pair(lo, hi) for lo, hi in zip([0] + cuts, cuts + [n])]
    assert len(whole) > 500 and whole == sum(parts, [])
    m = int(np.searchsorted(a["frame"], 1))
    want = [(int(r["i_xz"]), int(r["i_yz"])) for r in O.pair3d(a[:m], P)]
    assert want == [q for q in whole if q[0] < m]
