"""Records packed from host memory, one address each, and into ranges of a batch: windows of consecutive groups over a
list of pieces.  Many short records, empty ones, a long one among short ones, records scattered in memory, ranges that
start inside the batch, and totals around the narrow form's and the windows' limits; the batch equals the one packed
from the whole text on the device.  Needs a GPU."""
import ctypes

import numpy as np
import pytest

from tests.test_gpu_fasta import _batch_bytes, ah_ctx  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu


def _lengths(kind, n, rng):
    if kind == "reads":
        return rng.integers(0, 300, n)
    if kind == "tiny":
        return rng.integers(0, 3, n)
    if kind == "one long":     # a record of several pieces among reads
        lens = rng.integers(1, 300, n)
        lens[n // 3] = 1_100_003
        return lens
    if kind == "contigs":
        return rng.integers(480, 560, n)  # 16 groups a record on average: the narrow form's limit
    return np.full(n, 0)


@pytest.mark.parametrize("n", [1, 7, 33, 4097, 20_000])
@pytest.mark.parametrize("kind", ["reads", "tiny", "one long", "contigs", "empty"])
def test_pieces(ah_ctx, kind, n):
    import torch

    ah, ctx = ah_ctx
    lib = ah.load()
    rng = np.random.default_rng(n)
    lens = _lengths(kind, n, rng).astype(np.uint64)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    seq = np.frombuffer(b"ACGTNacgt-", np.uint8)[rng.integers(0, 10, max(1, off[-1]), dtype=np.uint8)]
    d = torch.from_numpy(seq.copy()).cuda()
    want = ah.ah_pack_batch_device(ctx, d.data_ptr(), off)
    # records scattered in host memory: a gap after each, the odd ones in another array, every second run contiguous
    gap = np.where(np.arange(n) % 4 == 1, 0, rng.integers(0, 40, n))
    at = np.concatenate([[0], np.cumsum(lens.astype(np.int64) + gap)])
    host = np.full(int(at[-1]) + 1, ord("G"), np.uint8)
    for r in range(n):
        host[at[r]:at[r] + int(lens[r])] = seq[off[r]:off[r + 1]]
    addr = (host.ctypes.data + at[:-1]).astype(np.uint64)
    out = ctypes.c_void_p()
    try:
        expect = _batch_bytes(ah, want)
        assert lib.ah_pack_batch(ctx, n, ctypes.c_void_p(addr.ctypes.data), ctypes.c_void_p(lens.ctypes.data), None,
                                 ctypes.byref(out)) == ah.AH_OK
        assert _batch_bytes(ah, out) == expect
        # ranges, from host and from device memory (at an odd address), over other contents
        other = np.full(max(1, int(off[-1])), ord("T"), np.uint8)
        d1 = torch.cat([torch.zeros(3, dtype=torch.uint8, device="cuda"), d])
        torch.cuda.synchronize()
        for base in (seq.ctypes.data, d1.data_ptr() + 3):
            ah.ah_batch_pack_range(ctx, out, 0, other.ctypes.data, off.astype(np.uint64))
            cut = sorted({0, n // 3, n // 2, n})
            for a, b in zip(cut, cut[1:]):
                ah.ah_batch_pack_range(ctx, out, a, base + int(off[a]), (off[a:b + 1] - off[a]).astype(np.uint64))
            assert _batch_bytes(ah, out) == expect
    finally:
        ah.ah_batch_free(want)
        if out:
            ah.ah_batch_free(out)
