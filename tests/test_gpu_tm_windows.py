"""The thread-per-site Tm kernels take windows of 128 to 1,024 site slots by the slots there are: a plan's results are
the oracle's whatever its capacity, degenerate primers (generated and built-in kernel) included."""
import pytest

import oracle
import synth
from tests import compare
from tests.test_gpu_one_block_tail import _run_plan
from tests.test_gpu_parity import engine  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel_mode", [0, 1])
@pytest.mark.parametrize("hit_capacity", [4000, 311_295, 311_296, 622_592, 1_245_184, 2_490_369])
def test_windows(engine, hit_capacity, kernel_mode):  # noqa: F811
    from paper_2511_00170_gb300 import ah

    wl = synth.random_small(21, n_records=8, len_lo=500, len_hi=6000, n_pairs=3, plant=6, n_deg=3, k_max=2)
    wl.orient_mask = 15
    wl.tm.min_tm = None  # every amplicon, with its Tm
    ref = oracle.run(wl)
    assert len(ref.hits) <= 4000 and len(ref.amps) > 20
    ah.ah_ctx_set_tm_kernel(engine.ctx, kernel_mode)
    try:
        out, info = _run_plan(engine, wl, hit_capacity=hit_capacity)
    finally:
        ah.ah_ctx_set_tm_kernel(engine.ctx, 0)
    assert info["hit_capacity"] == hit_capacity
    compare.assert_same_hits(out, ref)
    compare.assert_same_amplicons(out, ref, filtered=False)
    compare.assert_same_sequences(out, ref)
