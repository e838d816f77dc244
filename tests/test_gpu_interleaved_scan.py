"""The interleaved scan form of plans against the regular path's shifted form (which the parity tests pin
to the oracle), at the sizes and primers where it can go wrong: tile (32,768-base) and group edges,
windows that run from one lane's word into the next, 2- to 32-base primers with every kind of code,
candidate queues that overflow, more patterns than it takes, slices, and ranges scanned as an upload
lands.  Plans of few tiles keep the shifted form, so a record of invalid bases fills the batches up.
Needs a GPU."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def engine():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2511_00170_gb300.pipeline import Engine

    e = Engine(0)  # no scan shape is set on this context, so its plans choose the form themselves
    yield e
    e.close()


FILLER = np.full(17 << 20, ord("N"), dtype=np.uint8)  # 544 tiles


def _filled(wl):
    """The workload with the filler as its last record."""
    wl.seq = np.concatenate([wl.seq, FILLER])
    wl.offsets = np.append(wl.offsets, wl.offsets[-1] + len(FILLER))
    wl.genome_ids = np.arange(len(wl.offsets) - 1, dtype=np.uint32)
    return wl


def _workload(records, fwd, rev, k, clamp):
    wl = synth.random_small(5, n_records=1, len_lo=8, len_hi=8, n_pairs=1, plant=0)
    wl.seq = np.frombuffer("".join(records).encode(), dtype=np.uint8).copy()
    wl.offsets = np.cumsum([0] + [len(r) for r in records]).astype(np.int64)
    wl.genome_ids = np.arange(len(records), dtype=np.uint32)
    wl.fwd, wl.rev, wl.k, wl.clamp = fwd, rev, k, clamp
    wl.min_len, wl.max_len, wl.trim, wl.fb_len, wl.rb_len = 20, 400, True, 5, 4
    return _filled(wl)


def _random(n, seed, alphabet="ACGT"):
    return "".join(np.array(list(alphabet))[np.random.default_rng(seed).integers(0, len(alphabet), n)])


def _check(engine, wl, interleaved=None, slice_from=None):
    """The plan's sites, amplicons and sequences equal the regular path's; returns the sites."""
    from paper_2511_00170_gb300 import ah
    from paper_2511_00170_gb300.pipeline import Params

    p = Params.from_workload(wl)
    db = batch = engine.pack(wl.seq, wl.offsets)
    try:
        if slice_from is not None:
            batch = ah.ah_batch_slice(engine.ctx, db, slice_from, wl.n_records - slice_from)
        ref = engine.step(batch, p)
        plan = engine.plan(batch, p)
        try:
            if interleaved is not None:
                info = ah.ah_plan_info_get(plan)
                assert (info["threads"] == 64 and info["groups_per_thread"] == 32) == interleaved, info
            ah.ah_plan_run(plan, engine.ctx)
            out = engine.plan_output(plan)
        finally:
            ah.ah_plan_free(plan)
    finally:
        if batch is not db:
            ah.ah_batch_free(batch)
        ah.ah_batch_free(db)
    assert out.hits.tobytes() == ref.hits.tobytes()
    assert out.amps.tobytes() == ref.amps.tobytes()
    assert out.arena == ref.arena and np.array_equal(out.field_off, ref.field_off)
    return out.hits


TILE = 32768


@pytest.mark.parametrize("n", [1, 9, 31, 32, 33, 63, 64, 65, 1000, TILE - 64, TILE - 1, TILE, TILE + 1, TILE + 33,
                               2 * TILE - 65, 2 * TILE + 31, 5 * TILE + 7])
def test_sizes(engine, n):
    wl = _workload([_random(n, n), _random(77, n + 1), _random(n // 2 + 1, n + 2)], ["ACGTTGCAAG"], ["TTGACRSTAG"], [2], 2)
    hits = _check(engine, wl, interleaved=True)
    assert n < 5 * TILE or len(hits) > 100


@pytest.mark.parametrize("at", [0, 1, 20, 31, 1023, 1024, TILE - 33, TILE - 32, TILE - 19, TILE - 1, TILE])
@pytest.mark.parametrize("length", [18, 32])
def test_windows_across_edges(engine, at, length):
    """One exact copy of a primer at every kind of edge: a group's, a lane's and a tile's."""
    primer = _random(length, 3)
    text = _random(2 * TILE + 500, 4)
    text = text[:at] + primer + text[at + length:]
    wl = _workload([text], [primer], [_random(length, 5)], [1], 3)
    hits = _check(engine, wl, interleaved=True)
    assert (hits["pos"][hits["pattern"] == 0] == at).sum() == 1


@pytest.mark.parametrize("fwd,rev,k,clamp", [
    ("ACGTACGTACGTACGTACGTACGTACGTACGT", "TTTTGGGGCCCCAAAATTTTGGGGCCCCAAAA", 5, 4),
    ("ACRYSWKMBDHVNGTACC", "VVHHDDBBACGTTGCAGT", 1, 3), ("ACGTTGCAAGCT", "ACGTTGCAAGCT", 0, 0),
    ("NNNNACGTTGCANNNNACGT", "ACGTNNNNNNACGTTGCA", 2, 2), ("ACGTAGCTAGCTAG", "GATCGATCGATCCA", 0, 13),
    ("AC", "GT", 0, 1), ("ACGTA", "TTGAC", 1, 2), ("ACGTAGCTAGCTAGGT", "GATCGATCGATCCATT", 15, 2),
    ("RRRRRRRRRRYYYYYYYYYY", "SWSWSWSWSWSWSWSWSW", 3, 5)])
def test_primer_kinds(engine, fwd, rev, k, clamp):
    """Lengths, codes, budgets and clamps of every kind; the sets that let too many windows through
    keep the shifted form."""
    n = 3000 if len(fwd) < 6 or k > 6 else 30000  # a plan's tile holds at most 4,096 sites
    _check(engine, _workload([_random(n, 6), "N" * 40 + _random(n // 3, 7) + "N"], [fwd], [rev], [k], clamp))


@pytest.mark.parametrize("period", [9, 11, 16, 31])
def test_queue_overflow(engine, period):
    """A tandem repeat of the primer's own bases: thousands of sites per tile, far more words than the
    candidate queue holds, so tiles are run again with care and iterations a few lanes at a time."""
    unit = _random(period, 40 + period)
    text = _random(20000, 8) + unit * (70000 // period) + _random(9000, 9)
    primer = (unit * 4)[:20]
    wl = _workload([text, _random(500, 10)], [primer], [_random(20, 11)], [3], 3)
    wl.max_len = 30
    hits = _check(engine, wl, interleaved=True)
    assert len(hits) > 60000 // period


@pytest.mark.parametrize("pairs,interleaved", [(2, True), (3, True), (8, True), (9, True), (32, True), (33, False)])
def test_pattern_counts(engine, pairs, interleaved):
    wl = synth.batched(n_genomes=12, len_lo=2e3, len_hi=2e5, n_pairs=pairs)
    wl.k = [i % 3 for i in range(pairs)]
    _check(engine, _filled(wl), interleaved=interleaved)


def test_few_tiles(engine):
    """A batch of fewer tiles than fill the GPU keeps the shifted form."""
    _check(engine, synth.batched(n_genomes=12, len_lo=2e3, len_hi=2e5, n_pairs=2), interleaved=False)


def test_low_complexity_and_invalid(engine):
    """Composition far from the uniform one the filters are drawn for, lower case and invalid bases."""
    recs = [_random(40000, 12, "AAAAAAAC"), _random(40000, 13, "ATatN"), "A" * 3000 + "N" * 100 + _random(5000, 14, "GGGC")]
    wl = _workload(recs, ["AAAAATAATAAAACAAAT"], ["GGGGCGGGGGGCGGGCGG"], [3], 3)
    _check(engine, wl, interleaved=True)


def test_slice(engine):
    wl = synth.batched(n_genomes=9, len_lo=2e3, len_hi=2e5, n_pairs=2)
    _check(engine, _filled(wl), interleaved=True, slice_from=4)


def test_ranges_of_an_upload(engine):
    """Tile ranges scanned chunk by chunk as the genomes cross the link, over two staged chunks."""
    import torch

    from paper_2511_00170_gb300 import ah
    from paper_2511_00170_gb300.pipeline import Params

    wl = synth.batched(n_genomes=200, n_pairs=2)
    assert wl.total_bp > (256 << 20)
    p = Params.from_workload(wl)
    text = torch.empty(wl.total_bp, dtype=torch.uint8, pin_memory=True)
    text.numpy()[:] = wl.seq
    other = torch.full((wl.total_bp,), ord("A"), dtype=torch.uint8, pin_memory=True)  # the batch's bases before
    batch = engine.pack(wl.seq, wl.offsets)
    try:
        ref = engine.step(batch, p)
        plan = engine.plan(batch, p)
        try:
            assert ah.ah_plan_info_get(plan)["threads"] == 64
            ah.ah_batch_pack_range(engine.ctx, batch, 0, other.data_ptr(), wl.offsets)
            ah.ah_plan_launch_host(plan, text.data_ptr(), wl.offsets, engine.ctx)
            ah.ah_plan_check(plan, engine.ctx)
            out = engine.plan_output(plan)
        finally:
            ah.ah_plan_free(plan)
    finally:
        ah.ah_batch_free(batch)
    assert out.hits.tobytes() == ref.hits.tobytes() and out.amps.tobytes() == ref.amps.tobytes()
