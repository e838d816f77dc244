"""Plans with few sites or amplicons run the pairing and the steps after the Tm stage in one block each, larger ones
over many; prefix sums switch at 8,192 counts.  The same workload with capacities on either side of the limit (4,096)
gives the oracle's results, overflowing capacities are reported alike, and sites around the block's strides (1,023 to
4,096) are paired as the regular path pairs them."""
import numpy as np
import pytest

import oracle
import synth
from tests import compare
from tests.test_gpu_parity import engine  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu


def _run_plan(engine, wl, with_seqs=True, **caps):
    from paper_2511_00170_gb300 import ah
    from paper_2511_00170_gb300.pipeline import Params

    batch = engine.pack(wl.seq, wl.offsets, wl.genome_ids)
    plan = engine.plan(batch, Params.from_workload(wl), with_seqs=with_seqs, **caps)
    try:
        ah.ah_plan_run(plan, engine.ctx)
        return engine.plan_output(plan, with_seqs=with_seqs), ah.ah_plan_info_get(plan)
    finally:
        ah.ah_plan_free(plan)
        ah.ah_batch_free(batch)


@pytest.mark.parametrize("filtered", [False, True])
@pytest.mark.parametrize("hit_cap,amp_cap", [(4096, 4096), (4097, 4096), (4096, 4097), (4097, 4097)])
def test_both_sides_of_the_limit(engine, hit_cap, amp_cap, filtered):  # noqa: F811
    wl = synth.random_small(5, n_records=6, len_lo=500, len_hi=4000, n_pairs=3, plant=4, trim=True)
    wl.orient_mask = 15
    wl.tm.min_tm = 35.0 if filtered else None
    ref = oracle.run(wl)
    out, info = _run_plan(engine, wl, hit_capacity=hit_cap, amp_capacity=amp_cap)
    assert info["hit_capacity"] == hit_cap and info["amp_capacity"] == amp_cap and len(ref.amps) > 10
    compare.assert_same_hits(out, ref)
    compare.assert_same_amplicons(out, ref, filtered=filtered)
    compare.assert_same_sequences(out, ref)


@pytest.mark.parametrize("n_sites", [1, 31, 1023, 1024, 1025, 2048, 3000, 4096])
def test_sites_around_the_strides(engine, n_sites):  # noqa: F811
    """n_sites planted sites in alternating senses on a neutral background, every + site with partners that lie
    in other warps and strides."""
    from paper_2511_00170_gb300.pipeline import Params

    wl = synth.random_small(9, n_records=1, len_lo=10, len_hi=10, n_pairs=1, plant=0)
    wl.fwd, wl.rev, wl.k, wl.clamp = ["ACGTCATGCA"], ["GGATCCTTAG"], [0], 0
    rc = {"A": "T", "C": "G", "G": "C", "T": "A"}
    back = "".join(rc[c] for c in reversed(wl.rev[0]))
    parts = [wl.fwd[0] if i % 7 < 2 else back for i in range(n_sites)]
    g = "TTTTT".join(parts)
    wl.seq = np.frombuffer(g.encode(), dtype=np.uint8).copy()
    wl.offsets = np.array([0, len(g)], dtype=np.int64)
    wl.genome_ids = np.zeros(1, dtype=np.uint32)
    wl.min_len, wl.max_len, wl.orient_mask, wl.fb_len, wl.rb_len, wl.trim = 1, 2000, 15, 3, 3, False
    wl.tm.min_tm = None
    batch = engine.pack(wl.seq, wl.offsets, wl.genome_ids)
    try:
        from paper_2511_00170_gb300 import ah

        want = engine.step(batch, Params.from_workload(wl))
    finally:
        ah.ah_batch_free(batch)
    out, info = _run_plan(engine, wl, hit_capacity=4096)
    assert info["n_hits"] == n_sites == len(want.hits)
    assert np.array_equal(out.hits, want.hits)
    assert out.amps.tobytes() == want.amps.tobytes()
    assert bytes(out.arena) == bytes(want.arena) and np.array_equal(out.field_off, want.field_off)


@pytest.mark.parametrize("n_records", [4096, 4097, 8191, 8192, 8193, 12289])
def test_prefix_sums_around_their_limit(engine, n_records):  # noqa: F811
    """The group offsets of n_records reads, scanned on the device, against packing them with known lengths."""
    from paper_2511_00170_gb300 import ah
    from tests.test_gpu_fasta import _batch_bytes

    rng = np.random.default_rng(n_records)
    lens = rng.integers(0, 90, n_records)
    seq = np.frombuffer(b"ACGTN", np.uint8)[rng.integers(0, 5, int(lens.sum()))]
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    text = b"".join(b"@\n" + seq[a:b].tobytes() + b"\n+\n" + b"I" * int(b - a) + b"\n" for a, b in zip(off[:-1], off[1:]))
    got, quals, _ = ah.ah_fastq_pack(engine.ctx, text, names=False)
    want = ah.ah_pack_batch(engine.ctx, seq, off)
    try:
        assert _batch_bytes(ah, got) == _batch_bytes(ah, want)
    finally:
        ah.ah_quals_free(quals)
        ah.ah_batch_free(got)
        ah.ah_batch_free(want)
