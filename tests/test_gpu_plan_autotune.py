"""The autotuned plan on dense sites keeps the faster of the interleaved form and the best shifted one, and gives the same
results as the regular path: genomes where tandem repeats of the primers' bases make a warp of the interleaved form check
a whole repeat, and random ones, where the interleaved form is far ahead.  Needs a GPU."""
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


@pytest.mark.parametrize("n,repeats", [(40_000_000, 60), (40_000_000, 0), (400_000_000, 0)])
def test_form_and_results(engine, n, repeats):
    from paper_2511_00170_gb300 import ah
    from paper_2511_00170_gb300.pipeline import Params

    rng = np.random.default_rng(repeats + 1)
    seq = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, n, dtype=np.uint8)]
    for at in rng.integers(0, n - 5_000, repeats):
        seq[at:at + 5_000] = np.resize(np.frombuffer(b"ACG", np.uint8), 5_000)
    wl = synth.random_small(3, n_records=1, len_lo=10, len_hi=10, n_pairs=1, plant=0)
    wl.fwd, wl.rev, wl.k, wl.clamp = ["RCGRCGRCGRCGRCGACG"], ["TTSGTTAACCWTGGATCC"], [2], 3
    wl.min_len, wl.max_len, wl.tm.min_tm = 50, 2000, None
    p = Params.from_workload(wl)
    batch = engine.pack(seq, np.array([0, n], dtype=np.int64), np.zeros(1, dtype=np.uint32))
    try:
        ref = engine.step(batch, p, with_seqs=False)
        plan = engine.plan(batch, p, with_seqs=False, autotune=True)
        try:
            ah.ah_plan_run(plan, engine.ctx)
            out, info = engine.plan_output(plan, with_seqs=False), ah.ah_plan_info_get(plan)
        finally:
            ah.ah_plan_free(plan)
    finally:
        ah.ah_batch_free(batch)
    assert out.hits.tobytes() == ref.hits.tobytes() and out.amps.tobytes() == ref.amps.tobytes()
    interleaved = (info["threads"], info["groups_per_thread"]) == (64, 32)
    if repeats:
        assert len(ref.hits) > 50_000
    elif n > 100_000_000:
        assert interleaved, info


@pytest.mark.parametrize("mode", [1, 2, 3])
def test_interleaved_plan_on_a_context_with_the_generic_scan(engine, mode):
    """Contexts that scan with the generic kernel, first or throughout: a plan of the interleaved form is sized over that
    form's tiles by it, and finds what the regular path finds."""
    from paper_2511_00170_gb300 import ah
    from paper_2511_00170_gb300.pipeline import Engine, Params

    n = 20_000_000
    seq = np.frombuffer(b"ACGT", np.uint8)[np.random.default_rng(mode).integers(0, 4, n, dtype=np.uint8)]
    wl = synth.random_small(3, n_records=1, len_lo=10, len_hi=10, n_pairs=1, plant=0)
    wl.fwd, wl.rev, wl.k, wl.clamp = ["ACGTTGCAAG" + "ACG"[mode - 1]], ["TTGACRSTAGC"], [1], 2
    wl.min_len, wl.max_len, wl.tm.min_tm = 20, 4000, None
    p = Params.from_workload(wl)
    off = np.array([0, n], dtype=np.int64)
    batch = engine.pack(seq, off)
    e = Engine(0)
    try:
        ref = engine.step(batch, p)
        ah.ah_ctx_set_generic_scan(e.ctx, mode)
        mine = e.pack(seq, off)
        plan = e.plan(mine, p)
        try:
            info = ah.ah_plan_info_get(plan)
            assert (info["threads"], info["groups_per_thread"]) == (64, 32)
            ah.ah_plan_run(plan, e.ctx)
            out = e.plan_output(plan)
        finally:
            ah.ah_plan_free(plan)
            ah.ah_batch_free(mine)
    finally:
        e.close()
        ah.ah_batch_free(batch)
    assert len(ref.hits) > 100
    assert out.hits.tobytes() == ref.hits.tobytes() and out.amps.tobytes() == ref.amps.tobytes() and out.arena == ref.arena
