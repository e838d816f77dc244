"""Batches of 65,536 tiles and more whose tiles hold many sites are sorted and emitted a tile to a warp, in plans and in
the emission of single scans; the sites equal those of a tile shape with fewer tiles, on both sides of eight sites per
tile on average.  Needs a GPU."""
import numpy as np
import pytest

import synth
from tests.test_gpu_parity import engine  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("primer,dense", [("ACGTCA", True), ("ACGTCATGC", False)])
def test_a_tile_to_a_warp(engine, primer, dense):  # noqa: F811
    from paper_2511_00170_gb300 import ah
    from paper_2511_00170_gb300.pipeline import Params

    n_tiles = 65_543
    n = n_tiles * 2048 - 700   # tiles of 64 groups: one record, the last tile short
    seq = np.frombuffer(b"ACGT", np.uint8)[np.random.default_rng(len(primer)).integers(0, 4, n, dtype=np.uint8)]
    seq[2048 * 17 + 5:2048 * 17 + 1405] = np.resize(np.frombuffer(primer.encode(), np.uint8), 1400)
    wl = synth.random_small(3, n_records=1, len_lo=10, len_hi=10, n_pairs=1, plant=0)
    wl.fwd, wl.rev, wl.k, wl.clamp = [primer], ["GGATCCTTAGC"], [1], 1
    wl.min_len, wl.max_len, wl.tm.min_tm = 20, 400, None
    p = Params.from_workload(wl)
    batch = engine.pack(seq, np.array([0, n], dtype=np.int64), np.zeros(1, dtype=np.uint32))
    try:
        want = engine.step(batch, p, with_seqs=False)
        ah.ah_ctx_set_scan_config(engine.ctx, 64, 1, 64, 0)
        try:
            got = [engine.step(batch, p, with_seqs=False)]
            plan = engine.plan(batch, p, with_seqs=False)
            try:
                ah.ah_plan_run(plan, engine.ctx)
                assert ah.ah_plan_info_get(plan)["threads"] == 64
                got.append(engine.plan_output(plan, with_seqs=False))
            finally:
                ah.ah_plan_free(plan)
        finally:
            ah.ah_ctx_set_scan_config(engine.ctx, 256, 4, 256, 0)
    finally:
        ah.ah_batch_free(batch)
    assert (len(want.hits) > 10 * n_tiles) == dense and len(want.hits) > 1000
    for g in got:
        assert np.array_equal(g.hits, want.hits) and g.amps.tobytes() == want.amps.tobytes()
