"""FASTA and FASTQ parsed in one pass per chunk: the tiles' counts are taken for every line state that a tile
may be entered in, chained on the device, and records past the first room for them are listed again.  The
text is laid so that 16 KiB tiles and the chunks (an eighth of the text, at least 4 MiB) are entered inside
headers, bases, qualities and line breaks; results equal the line-by-line oracle exactly."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_fasta import _batch_bytes, ah_ctx  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu

TILE = 16384


def _check(ah, ctx, batch, seqs):
    lens = np.array([len(s) for s in seqs], dtype=np.uint64)
    want = ah.ah_pack_batch(ctx, np.frombuffer(b"".join(seqs) or b"\0", dtype=np.uint8),
                            np.concatenate([[0], np.cumsum(lens)]).astype(np.int64))
    try:
        assert _batch_bytes(ah, batch) == _batch_bytes(ah, want)
    finally:
        ah.ah_batch_free(want)


def _fasta(rng, n_bytes, header, line, empty):
    """Records whose headers, lines and blanks drift over the tile borders."""
    out, size = [], 0
    while size < n_bytes:
        h = b">" + bytes(rng.integers(33, 127, rng.integers(0, header), dtype=np.uint8))
        rows = [] if rng.random() < empty else \
            [np.frombuffer(b"ACGTN acgt", np.uint8)[rng.integers(0, 10, rng.integers(1, line))].tobytes()
             for _ in range(rng.integers(1, 6))]
        rec = b"\n".join([h] + rows) + (b"\r\n" if rng.random() < 0.2 else b"\n")
        out.append(rec)
        size += len(rec)
    return b"".join(out)


@pytest.mark.parametrize("on_device", [False, True])
@pytest.mark.parametrize("n_bytes,header,line,empty", [
    (3 * TILE, 40, 80, 0.1),                 # a few tiles
    (2 * TILE + 5, 3 * TILE, 90, 0.0),       # headers that span whole tiles ('>' and blanks inside them)
    (400_000, 3, 2, 0.9),                    # a record per few bytes: more than the first room for records
    (TILE * 300, 60, 3 * TILE, 0.0),         # more tiles than the chain's threads, lines longer than a tile
    (5 << 20, 60, 200, 0.05),                # a whole chunk and a rest
])
def test_fasta_tiles(ah_ctx, n_bytes, header, line, empty, on_device):
    import torch

    ah, ctx = ah_ctx
    rng = np.random.default_rng(n_bytes + header)
    text = _fasta(rng, n_bytes, header, line, empty)
    names, seqs = oracle.parse_fasta(text)
    d = torch.frombuffer(bytearray(text), dtype=torch.uint8).cuda() if on_device else None
    if on_device:
        batch, got = ah.ah_fasta_pack(ctx, d.data_ptr(), n_bytes=len(text))
    else:
        batch, got = ah.ah_fasta_pack(ctx, text)
    try:
        assert got == names
        _check(ah, ctx, batch, seqs)
    finally:
        ah.ah_batch_free(batch)


def _fastq(rng, n_records, header, read):
    out = []
    for _ in range(n_records):
        n = int(rng.integers(0, read))
        s = np.frombuffer(b"ACGTN", np.uint8)[rng.integers(0, 5, n)].tobytes()
        q = bytes(rng.integers(33, 127, n, dtype=np.uint8))  # qualities may start with '@' and '+'
        out.append(b"@" + bytes(rng.integers(33, 127, rng.integers(0, header), dtype=np.uint8)) + b"\n" + s + b"\n+\n" + q +
                   b"\n")
    return b"".join(out)


@pytest.mark.parametrize("on_device", [False, True])
@pytest.mark.parametrize("n_records,header,read", [
    (700, 60, 300),
    (9, 3 * TILE, 2 * TILE),                 # every line class spans whole tiles
    (40_000, 2, 2),                          # a record per 6 bytes: more than the first room for records
    (600, 30, 2 * TILE),                     # several chunks, more tiles than the chain's threads
])
def test_fastq_tiles(ah_ctx, n_records, header, read, on_device):
    import torch

    ah, ctx = ah_ctx
    rng = np.random.default_rng(n_records + read)
    text = _fastq(rng, n_records, header, read)
    names, seqs, quals = oracle.parse_fastq(text)
    d = torch.frombuffer(bytearray(text), dtype=torch.uint8).cuda() if on_device else None
    if on_device:
        batch, q, got = ah.ah_fastq_pack(ctx, d.data_ptr(), n_bytes=len(text))
    else:
        batch, q, got = ah.ah_fastq_pack(ctx, text)
    try:
        assert got == names
        _check(ah, ctx, batch, seqs)
        raw, off = ah.ah_quals_copy(q)
        assert raw == b"".join(quals)
        assert off.tolist() == np.concatenate([[0], np.cumsum([len(x) for x in quals])]).tolist()
    finally:
        ah.ah_quals_free(q)
        ah.ah_batch_free(batch)


@pytest.mark.parametrize("break_at", [0, 1, 3, 7000, 9000])
def test_fastq_refused_in_any_chunk(ah_ctx, break_at):
    """A record whose bases outnumber its qualities, and a text that is nearly all bases: refused."""
    ah, ctx = ah_ctx
    rng = np.random.default_rng(break_at)
    recs = _fastq(rng, 10_000, 40, 600).split(b"\n")
    recs[4 * break_at + 1] += b"A" * 5
    for text in (b"\n".join(recs), b"@r\n" + b"ACGT" * (3 * TILE + break_at) + b"\n+\nI\n"):
        with pytest.raises(ah.AhError) as e:
            ah.ah_fastq_pack(ctx, text)
        assert e.value.status == ah.AH_EINVAL
