"""Tm over the variants that match the site within the budget (variants = 1, ah_tm_sites) for primers without a branch
position, or with one elsewhere, when mismatches up to the whole budget include the first base: it is counted once.
Against the oracle.  Needs a GPU."""
import itertools
import math

import pytest

import oracle
import synth
from tests import compare
from tests.test_gpu_tm_group_enum import ctx  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("salt", [dict(saltcorr=s) for s in range(6)] + [dict(saltcorr=6), dict(saltcorr=7, Mg=1.5)])
def test_mismatch_at_the_first_base(ctx, salt):  # noqa: F811
    from paper_2511_00170_gb300 import ah

    prims, sites, ks = [], [], []
    for p, k in itertools.product(["ACGTTGCAAGCTAGGT", "GCATTGCCAAGTC", "CACG", "TCGTTGCNAGCTAGGT", "GCGTTGCAAGCTAGGR"],
                                  (0, 1, 2, 3)):
        v = p.replace("N", "A").replace("R", "A")
        for first in "ACGT":
            s = first + v[1:]
            for at, b in list(zip((6, 2), "GA"))[:max(0, k - 1)]:  # the rest of the budget
                if at < len(s) - 1:
                    s = s[:at] + ("C" if s[at] == b else b) + s[at + 1:]
            prims.append(p), sites.append(s), ks.append(k)
    prm = dict(Na=50.0, **salt)
    got = ah.ah_tm_sites(ctx, prims, sites, ah.tm_params(variants=1, **prm), k=ks, clamp=[0] * len(ks))
    spent = 0
    for p, s, k, g in zip(prims, sites, ks, got):
        r = oracle.tm_site(p, s, synth.TmParams(**prm), k=k, clamp=0)
        if r is None:
            assert math.isnan(g), (p, s, k, g)
        else:
            spent += k > 0 and s[0] != p[0]
            assert abs(g - r) <= compare.TM_TOL, (p, s, k, g, r)
    assert spent > 10
