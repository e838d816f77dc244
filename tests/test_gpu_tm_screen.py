"""The maximum over a degenerate site's variants under salt methods 6 and 7, where variants are screened in single precision:
buffers from next to no salt to far above saturation and strand concentrations over twelve decades, so that temperatures
and corrections leave the range the screen is used in.  Against the oracle's evaluation of every variant.  Needs a GPU."""
import math

import pytest

import oracle
import synth
from tests import compare
from tests.test_gpu_tm_group_enum import ctx  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu

PRIMERS = ["RYBDHVNACGTTGCA", "NACGTTGCAAGCTAGN", "ANNNNNGRTTGCAAGC", "WSWSWSWSWSGCTA", "NNNNN", "ACN", "RGCRGCRGCYGCYGCYGC"]
SALTS = [dict(saltcorr=6, Na=na) for na in (1e-6, 1e-2, 50.0, 1e4, 1e7)] + \
        [dict(saltcorr=7, Na=0.0, Mg=mg) for mg in (1e-9, 1e-3, 1.5, 1e3, 1e6)] + \
        [dict(saltcorr=7, Na=na, Mg=mg) for na, mg in ((50.0, 1.5), (1e-5, 1e-5), (800.0, 20.0), (1e4, 1e6))]


@pytest.mark.parametrize("dnac", [1e-6, 25.0, 1e6])
@pytest.mark.parametrize("salt", SALTS, ids=str)
def test_extreme_buffers(ctx, salt, dnac):  # noqa: F811
    from paper_2511_00170_gb300 import ah

    st = synth.Stream(synth.make_key(17, int(dnac), salt["saltcorr"]))
    prims, sites, ks = [], [], []
    for p in PRIMERS:
        for k in (0, 1, 2, 15):
            prims.append(p)
            sites.append(synth.substitute(st, synth.concrete_variant(st, p), min(k, len(p) - 1)))
            ks.append(k)
    prm = dict(dnac1=dnac, dnac2=dnac / 2, **salt)
    got = ah.ah_tm_sites(ctx, prims, sites, ah.tm_params(**prm), k=ks, clamp=[0] * len(ks))
    defined = 0
    for p, s, k, g in zip(prims, sites, ks, got):
        r = oracle.tm_site(p, s, synth.TmParams(**prm), k=k, clamp=0)
        if r is None:
            assert math.isnan(g), (p, s, k, g)
        else:
            defined += 1
            # TM_TOL at 100 C; further out rounding grows with T^2 (T = 1 / (1 / T0 + c))
            assert abs(g - r) <= compare.TM_TOL * max(1.0, (abs(r) / 300.0) ** 2), (p, s, k, g, r)
    assert defined > 10
