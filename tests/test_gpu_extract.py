"""Extraction builds 16-byte units of the arena, across field borders and from reversed fields: fields from
empty to longer than many units, clipped at the records' ends, with invalid bases, all orientations, on the
regular path and in a plan, against the oracle's strings exactly."""
import pytest

import synth
from tests import compare
from tests.test_gpu_parity import _run_both, engine  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu


def _workload(fb, rb, trim, max_len):
    wl = synth.random_small(77 + fb + 3 * rb + max_len, n_records=9, len_lo=40, len_hi=3000, n_pairs=2, plen_lo=6,
                            plen_hi=9, k_max=1, clamp=2, n_frac=0.02, plant=6, min_len=1, max_len=max_len, fb=fb, rb=rb,
                            trim=trim)
    wl.orient_mask = 15
    wl.tm.min_tm = None
    return wl


CASES = [(fb, rb, trim, mx) for fb, rb in ((0, 0), (1, 0), (15, 16), (17, 33), (64, 5), (700, 300)) for trim, mx in
         ((False, 1200), (True, 30))]


@pytest.mark.parametrize("fb,rb,trim,max_len", CASES)
def test_fields(engine, fb, rb, trim, max_len):  # noqa: F811
    out, ref = _run_both(engine, _workload(fb, rb, trim, max_len))
    assert ref.keep.any()


@pytest.mark.parametrize("fb,rb,trim,max_len", CASES[::3])
def test_fields_in_a_plan(engine, fb, rb, trim, max_len):  # noqa: F811
    import oracle
    from paper_2511_00170_gb300 import ah
    from paper_2511_00170_gb300.pipeline import Params

    wl = _workload(fb, rb, trim, max_len)
    ref = oracle.run(wl)
    batch = engine.pack(wl.seq, wl.offsets, wl.genome_ids)
    plan = engine.plan(batch, Params.from_workload(wl), with_seqs=True)
    try:
        ah.ah_plan_run(plan, engine.ctx)
        compare.assert_same_sequences(engine.plan_output(plan), ref)
    finally:
        ah.ah_plan_free(plan)
        ah.ah_batch_free(batch)
