"""Packing against a plain numpy packing of the same bytes: record lengths around the words, groups and
windows of the kernels, every source alignment, all 256 byte values, few long records and many short
ones, from device memory (whole batches and ranges of one) and from host memory.  Needs a GPU."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def engine():
    import __graft_entry__

    __graft_entry__.build()
    from paper_2511_00170_gb300.pipeline import Engine

    e = Engine(0)
    yield e
    e.close()


CODE = np.full(256, 255, dtype=np.uint8)
for letter, code in zip(b"ACTG", range(4)):
    CODE[letter] = CODE[letter + 32] = code


def _expected(seq, off):
    """(planes, invalid) of the batch's groups as the layout defines them."""
    lens = np.diff(off)
    groups = (lens // 64 + 1) * 2
    start = np.concatenate([[0], np.cumsum(groups)])
    code = np.full(int(start[-1]) * 32, 255, dtype=np.uint8)
    for r in range(len(lens)):
        code[start[r] * 32:start[r] * 32 + lens[r]] = CODE[seq[off[r]:off[r + 1]]]
    bad = code == 255
    code[bad] = 0
    bits = lambda x: np.packbits(x.reshape(-1, 32), axis=1, bitorder="little").view("<u4").ravel()
    return np.stack([bits(code & 1), bits(code >> 1)], axis=1), bits(bad.astype(np.uint8))


def _arrays(batch):
    from paper_2511_00170_gb300 import ah

    planes, groups, words = ah.ah_batch_export(batch)
    invalid = np.zeros(len(planes), dtype=np.uint32)
    invalid[groups.astype(np.int64)] = words
    return planes, invalid


def _text(n, seed):
    rng = np.random.default_rng(seed)
    s = np.frombuffer(b"ACGTacgt", dtype=np.uint8)[rng.integers(0, 8, n)].copy()
    at = rng.integers(0, max(1, n), n // 40 + 1)
    s[at[at < n]] = rng.integers(0, 256, len(at))[at < n]
    return s


CASES = {"edges": [0, 1, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 500, 511, 512, 1023, 1024, 1025],
         "reads": [251] * 3001 + [0, 1, 64, 600], "short": [7] * 5000, "one": [1_000_003], "word": [16],
         "windows": [32 * 1024 - 64, 32 * 1024 - 1, 32 * 1024, 70_001, 64, 2_100_000],
         "mixed": [300 + 97 * (i % 800) for i in range(700)]}


@pytest.mark.parametrize("lead", [0, 1, 7, 15])
@pytest.mark.parametrize("name", sorted(CASES))
def test_pack(engine, name, lead):
    import torch

    from paper_2511_00170_gb300 import ah

    lens = np.array(CASES[name], dtype=np.int64)
    off = np.concatenate([[0], np.cumsum(lens)]) + lead
    seq = _text(int(off[-1]), 100 + lead)
    planes, invalid = _expected(seq, off)
    d = torch.from_numpy(seq).cuda()
    for how in ("device", "range", "host"):
        if how == "device":
            b = engine.pack_device(d.data_ptr(), off)
        elif how == "range":
            b = ah.ah_batch_create(engine.ctx, lens)
            cut = len(lens) // 2
            if cut:
                ah.ah_batch_pack_range(engine.ctx, b, 0, d.data_ptr() + int(off[0]), (off[:cut + 1] - off[0]).astype(np.uint64))
            ah.ah_batch_pack_range(engine.ctx, b, cut, d.data_ptr() + int(off[cut]), (off[cut:] - off[cut]).astype(np.uint64))
        else:
            b = ah.ah_pack_batch(engine.ctx, seq, off.astype(np.uint64))
        try:
            p, v = _arrays(b)
        finally:
            ah.ah_batch_free(b)
        assert np.array_equal(p, planes), how
        assert np.array_equal(v, invalid), how
