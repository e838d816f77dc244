"""Under salt methods 6 and 7 the thread-per-site Tm kernels list every site for the enumeration, in windows of their full
size whatever the capacity: a plan's results are the oracle's.  Needs a GPU."""
import pytest

import oracle
import synth
from tests import compare
from tests.test_gpu_one_block_tail import _run_plan
from tests.test_gpu_parity import engine  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("salt", [6, 7])
@pytest.mark.parametrize("hit_capacity", [4000, 400_000])
def test_windows(engine, hit_capacity, salt):  # noqa: F811
    wl = synth.random_small(21, n_records=8, len_lo=500, len_hi=6000, n_pairs=3, plant=6, n_deg=3, k_max=2)
    wl.orient_mask = 15
    wl.tm.min_tm, wl.tm.saltcorr, wl.tm.Mg = None, salt, 1.5
    ref = oracle.run(wl)
    assert len(ref.hits) <= 4000 and len(ref.amps) > 20
    out, info = _run_plan(engine, wl, hit_capacity=hit_capacity)
    assert info["hit_capacity"] == hit_capacity
    compare.assert_same_hits(out, ref)
    compare.assert_same_amplicons(out, ref, filtered=False)
