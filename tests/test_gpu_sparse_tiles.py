"""Batches of 65,536 tiles and more are sorted and emitted eight tiles to a warp: the sites equal those of a tile shape
with fewer tiles (a warp each), with a tile that overflows a warp's sort, empty tiles and a last warp that is cut off."""
import numpy as np
import pytest

from tests.test_gpu_parity import engine  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tiles", [65535, 65536, 65543])
def test_eight_tiles_per_warp(engine, n_tiles):  # noqa: F811
    from paper_2511_00170_gb300 import ah
    from paper_2511_00170_gb300.pipeline import Params

    import synth

    rng = np.random.default_rng(n_tiles)
    n = n_tiles * 2048 - 700   # tiles of 64 groups: one record, the last tile short
    seq = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, n, dtype=np.uint8)]
    seq[2048 * 17 + 5:2048 * 17 + 405] = ord("A")           # more sites in a tile than a warp sorts
    seq[n - 60:n - 30] = ord("A")
    wl = synth.random_small(3, n_records=1, len_lo=10, len_hi=10, n_pairs=2, plant=0)
    wl.fwd, wl.rev, wl.k, wl.clamp = ["AAAAAAAAAA", "ACGTCATGC"], ["GGATCCTTAGC", "CCCATTGGAC"], [0, 1], 2
    wl.min_len, wl.max_len, wl.tm.min_tm = 20, 400, None
    p = Params.from_workload(wl)
    batch = engine.pack(seq, np.array([0, n], dtype=np.int64), np.zeros(1, dtype=np.uint32))
    try:
        want = engine.step(batch, p, with_seqs=False)
        ah.ah_ctx_set_scan_config(engine.ctx, 64, 1, 16, 0)
        try:
            got = engine.step(batch, p, with_seqs=False)
        finally:
            ah.ah_ctx_set_scan_config(engine.ctx, 256, 4, 256, 0)
    finally:
        ah.ah_batch_free(batch)
    assert len(want.hits) > 2000
    assert np.array_equal(got.hits, want.hits) and got.amps.tobytes() == want.amps.tobytes()
