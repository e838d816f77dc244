"""Degenerate-site Tm under salt methods 6 and 7, enumerated by a group of lanes over the combinations of
the branch positions' codes: no branch position, every number of choices, the largest number of
combinations it takes and the first it leaves to the pruning walk, mismatch budgets and clamps,
every nearest-neighbour set, against the oracle's enumeration of every variant.  Needs a GPU."""
import math

import pytest

import oracle
import synth
from tests import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2511_00170_gb300 import ah

    c = ah.ah_ctx_create(0)
    yield c
    ah.ah_ctx_destroy(c)


PRIMERS = ["ACGTTGCAAGCTAGGT",                 # one combination
           "NACGTTGCAAGCTAGN", "RYBDHVNACGTTGCA",  # ends; 2 x 2 x 3^4 x 4 combinations
           "ANNNNNGRTTGCAAGC", "ANNNNNGBTTGCAAGC",  # 2,048, then 3,072
           "BBBBBBGTTGCAAGCH", "WWWWWWWWWWWTTAAT",  # 2,187; 2,048 without G or C in many
           "ACG", "ACN"]


@pytest.mark.parametrize("nn_table", [0, 1, 2, 4, 5, 8])
@pytest.mark.parametrize("salt", [dict(saltcorr=6), dict(saltcorr=7, Mg=1.5, dNTPs=0.8)])
def test_group_enumeration(ctx, nn_table, salt):
    from paper_2511_00170_gb300 import ah

    st = synth.Stream(synth.make_key(91, nn_table, salt["saltcorr"]))
    prims, sites, ks, clamps = [], [], [], []
    for p in PRIMERS:
        for k in (0, 1, 2, 5, 15):
            v = synth.concrete_variant(st, p)
            prims.append(p)
            sites.append(synth.substitute(st, v, min(st.randint(0, 3), len(p))))
            ks.append(k)
            clamps.append(st.randint(0, 2))
    prm = dict(Na=50.0, nn_table=nn_table, **salt)
    got = ah.ah_tm_sites(ctx, prims, sites, ah.tm_params(**prm), k=ks, clamp=clamps)
    defined = 0
    for p, s, k, c, g in zip(prims, sites, ks, clamps, got):
        r = oracle.tm_site(p, s, synth.TmParams(**prm), k=k, clamp=c)
        if r is None:
            assert math.isnan(g), (p, s, k, c, g)
        else:
            defined += 1
            assert abs(g - r) <= compare.TM_TOL, (p, s, k, c, g, r)
    assert defined > 10
