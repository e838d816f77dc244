"""FASTA and FASTQ text from host memory in several chunks, with every kind of byte on both sides of the first and the
second chunk's border (computed by the rule the library uses), from pageable memory, where a chunk's copy is staged
before the next is enqueued, and from page-locked memory, where all copies and passes are in flight together; the same
for text scanned by a plan as it lands.  Against the line-by-line reference, exactly.  Needs a GPU."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_fasta import _batch_bytes, ah_ctx  # noqa: F401 (the fixture)
from tests.test_gpu_parity import engine  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu

TILE, LEAST, LEAST_HOOK, MOST = 16384, 12 << 20, 32 << 20, 256 << 20


def borders(n_bytes, least):
    """The chunks' ends before the text's: half of the rest in whole tiles, at least `least`, at most 256 MiB."""
    n, least, most, at, out = -(-n_bytes // TILE), least // TILE, MOST // TILE, 0, []
    while n - at > least + least // 2:
        at += min(most, max(least, (n - at) // 8 * 4))
        out.append(at * TILE)
    return out


def parse_fasta(text):
    """oracle.parse_fasta with the bytes of a line dropped by a table."""
    names, seqs = [], []
    for line in text.split(b"\n"):
        if line.startswith(b">"):
            names.append(line[1:].rstrip(b"\r").decode("latin-1"))
            seqs.append([])
        elif seqs:
            seqs[-1].append(line.translate(None, b"\r \t"))
    return names, [b"".join(s) for s in seqs]


class _Memory:
    """The text as the program holds it."""

    def __init__(self, text, kind):
        import torch

        self.keep = torch.empty(len(text), dtype=torch.uint8, pin_memory=kind == "pinned")
        self.keep.numpy()[:] = np.frombuffer(text, dtype=np.uint8)
        self.ptr, self.n = self.keep.data_ptr(), len(text)


def _check(ah, ctx, batch, seqs):
    lens = np.array([len(s) for s in seqs], dtype=np.uint64)
    want = ah.ah_pack_batch(ctx, np.frombuffer(b"".join(seqs) or b"\0", dtype=np.uint8),
                            np.concatenate([[0], np.cumsum(lens)]).astype(np.int64))
    try:
        assert _batch_bytes(ah, batch) == _batch_bytes(ah, want)
    finally:
        ah.ah_batch_free(want)


# what lies across a border: the bytes before it and after it
ACROSS = {"header line": (b"ACGT\n>a header of", b" more than a few words\nACGTACGT"),
          "first byte of a header": (b"ACGT\n", b">header\nACGT"),
          "last byte a header's first": (b"ACGT\n>", b"header\nACGT"),
          "break after a header": (b"\n>header", b"\nACGT"),
          "break before a header": (b"ACGT", b"\n>header\nAC"),
          "sequence line": (b"\nACGTNAC", b"GTT>ACG ACGT\nAC"),
          "carriage return": (b"\n>header\r", b"\nACGT\r\nAC"),
          "blank": (b"ACGT ", b"\tACGT")}


def _fasta(n_bytes, ends, across, seed, record=5000):
    rng = np.random.default_rng(seed)
    text = np.frombuffer(b"ACGTN", np.uint8)[rng.integers(0, 5, n_bytes, dtype=np.uint8)]
    text[80::81] = ord("\n")
    heads = np.arange(0, n_bytes - 100, record // 81 * 81)   # line starts
    text[heads] = ord(">")
    text = bytearray(text.tobytes())
    for end, (before, after) in zip(ends, across):
        text[end - len(before):end] = before
        text[end:end + len(after)] = after
    return bytes(text)


KINDS = list(ACROSS)


def test_borders():
    assert len(borders(60 << 20, LEAST)) == 2 and len(borders(110 << 20, LEAST_HOOK)) == 2
    text = _fasta(2 << 20, [500_000, 1_000_000], [ACROSS["blank"], ACROSS["carriage return"]], 1)
    names, seqs = oracle.parse_fasta(text)
    assert parse_fasta(text) == (names, seqs) and len(names) > 300


@pytest.mark.parametrize("memory", ["pageable", "pinned"])
@pytest.mark.parametrize("k", range(len(KINDS)))
def test_fasta_across_chunks(ah_ctx, k, memory):
    ah, ctx = ah_ctx
    n = (60 << 20) + 7 * k
    text = _fasta(n, borders(n, LEAST), [ACROSS[KINDS[k]], ACROSS[KINDS[(k + 3) % len(KINDS)]]], k)
    names, seqs = parse_fasta(text)
    m = _Memory(text, memory)
    for _ in range(2):
        batch, got = ah.ah_fasta_pack(ctx, m.ptr, n_bytes=m.n)
        try:
            assert got == names
            _check(ah, ctx, batch, seqs)
        finally:
            ah.ah_batch_free(batch)


@pytest.mark.parametrize("memory", ["pageable", "pinned"])
def test_fasta_more_records_than_the_first_room(ah_ctx, memory):
    ah, ctx = ah_ctx
    n = 30 << 20
    text = _fasta(n, borders(n, LEAST), [ACROSS["header line"]], 9, record=81)
    names, seqs = parse_fasta(text)
    assert len(borders(n, LEAST)) >= 1 and len(names) > 4096 + n // 128
    m = _Memory(text, memory)
    batch, got = ah.ah_fasta_pack(ctx, m.ptr, n_bytes=m.n)
    try:
        assert got == names
        _check(ah, ctx, batch, seqs)
    finally:
        ah.ah_batch_free(batch)


@pytest.mark.parametrize("memory", ["pageable", "pinned"])
@pytest.mark.parametrize("k", [0, 1, 4, 5])
def test_plan_launch_fasta_across_chunks(engine, k, memory):  # noqa: F811
    from paper_2511_00170_gb300 import ah
    from paper_2511_00170_gb300.pipeline import Params

    import synth

    n = (110 << 20) + 11 * k
    text = _fasta(n, borders(n, LEAST_HOOK), [ACROSS[KINDS[k]], ACROSS[KINDS[(k + 3) % len(KINDS)]]], 20 + k, 50_000)
    _, seqs = parse_fasta(text)
    wl = synth.random_small(3, n_records=1, len_lo=10, len_hi=10, n_pairs=1, plant=0)
    wl.fwd, wl.rev, wl.k, wl.clamp = ["ACGTTGCA"], ["GGATCCTA"], [1], 2
    wl.min_len, wl.max_len, wl.tm.min_tm = 20, 4000, None
    p = Params.from_workload(wl)
    offs = np.concatenate([[0], np.cumsum([len(s) for s in seqs])])
    m = _Memory(text, memory)
    batch = engine.pack(np.frombuffer(b"".join(seqs), np.uint8), offs.astype(np.int64))
    other = np.full(int(offs[-1]), ord("G"), np.uint8)
    try:
        plan = engine.plan(batch, p)
        try:
            ah.ah_plan_run(plan, engine.ctx)
            ref = engine.plan_output(plan)
            want = _batch_bytes(ah, batch)
            assert len(ref.hits) > 100
            for _ in range(2):
                ah.ah_batch_pack_range(engine.ctx, batch, 0, other.ctypes.data, offs.astype(np.uint64))
                ah.ah_plan_launch_fasta(plan, m.ptr, m.n, engine.ctx)
                out = engine.plan_output(plan)
                assert out.hits.tobytes() == ref.hits.tobytes() and out.amps.tobytes() == ref.amps.tobytes()
                assert _batch_bytes(ah, batch) == want
        finally:
            ah.ah_plan_free(plan)
    finally:
        ah.ah_batch_free(batch)


def _fastq_record(rng, name, length):
    return (b"@" + name + b"\n" + np.frombuffer(b"ACGTN", np.uint8)[rng.integers(0, 5, length)].tobytes() + b"\n+\n" +
            rng.integers(33, 127, length, dtype=np.uint8).tobytes() + b"\n")   # 2 length + len(name) + 6 bytes


FASTQ_KINDS = {"first byte of a header": 0, "header": 20, "break after a header": 41, "first base": 42, "bases": 142,
               "break after the bases": 242, "plus": 243, "qualities": 345, "last break": 445}  # offsets in a record


def _fastq(n_bytes, ends, offsets, seed, read=251):
    """FASTQ text of n_bytes; a record of a 40-byte name and 200 bases lies with its byte offsets[i] at ends[i]."""
    rng = np.random.default_rng(seed)
    out, pos = [], 0

    def add(rec):
        nonlocal pos
        out.append(rec)
        pos += len(rec)

    def fill(upto):
        while upto - pos > 4 * read + 200:
            add(_fastq_record(rng, b"r", read))
        rest = upto - pos - 6
        name = b"n" if rest % 2 else b"nn"
        add(_fastq_record(rng, name, (rest - len(name)) // 2))
        assert pos == upto

    for end, off in zip(ends, offsets):
        fill(end - off)
        add(_fastq_record(rng, b"x" * 40, 200))
    fill(n_bytes)
    return b"".join(out)


@pytest.mark.parametrize("memory", ["pageable", "pinned"])
@pytest.mark.parametrize("k", range(len(FASTQ_KINDS)))
def test_fastq_across_chunks(ah_ctx, k, memory):
    ah, ctx = ah_ctx
    n = (44 << 20) + 13 * k
    at = list(FASTQ_KINDS.values())
    ends = borders(n, LEAST)
    assert len(ends) == 2
    text = _fastq(n, ends, [at[k], at[(k + 4) % len(at)]], 50 + k, 20_000)
    names, seqs, quals = oracle.parse_fastq(text)
    m = _Memory(text, memory)
    for _ in range(2):
        batch, q, got = ah.ah_fastq_pack(ctx, m.ptr, n_bytes=m.n)
        try:
            assert got == names
            _check(ah, ctx, batch, seqs)
            raw, off = ah.ah_quals_copy(q)
            assert raw == b"".join(quals)
            assert off.tolist() == np.concatenate([[0], np.cumsum([len(x) for x in quals])]).tolist()
        finally:
            ah.ah_quals_free(q)
            ah.ah_batch_free(batch)


@pytest.mark.parametrize("memory", ["pageable", "pinned"])
def test_fastq_more_records_than_the_first_room(ah_ctx, memory):
    ah, ctx = ah_ctx
    n = 20 << 20
    text = _fastq(n, borders(n, LEAST), [142], 70, 15)
    names, seqs, quals = oracle.parse_fastq(text)
    assert len(borders(n, LEAST)) >= 1 and len(names) > 4096 + n // 64
    m = _Memory(text, memory)
    batch, q, got = ah.ah_fastq_pack(ctx, m.ptr, n_bytes=m.n)
    try:
        assert got == names
        _check(ah, ctx, batch, seqs)
        assert ah.ah_quals_copy(q)[0] == b"".join(quals)
    finally:
        ah.ah_quals_free(q)
        ah.ah_batch_free(batch)


@pytest.mark.parametrize("memory", ["pageable", "pinned"])
@pytest.mark.parametrize("share", [0.1, 0.6, 0.99])
def test_fastq_refused_in_a_later_chunk(ah_ctx, share, memory):
    """A base more than qualities in a record of the first, the second or the last chunk; then good text is taken."""
    ah, ctx = ah_ctx
    n = 44 << 20
    text = _fastq(n, [], [], 80, 5_000)
    at = text.index(b"\n+\n", int(n * share))
    m, good = _Memory(text[:at] + b"A" + text[at:], memory), _fastq(100_000, [], [], 81)
    with pytest.raises(ah.AhError) as e:
        ah.ah_fastq_pack(ctx, m.ptr, n_bytes=m.n)
    assert e.value.status == ah.AH_EINVAL
    batch, q, got = ah.ah_fastq_pack(ctx, good)
    _check(ah, ctx, batch, oracle.parse_fastq(good)[1])
    ah.ah_quals_free(q)
    ah.ah_batch_free(batch)
