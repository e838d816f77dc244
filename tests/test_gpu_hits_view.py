"""The sites' device view is complete when ah_hits_device returns: a copy and a pairing on other streams, with no
synchronisation in between, see every site.  Needs a GPU."""
import numpy as np
import pytest

import synth
from tests.test_gpu_parity import engine  # noqa: F401 (the fixture)

pytestmark = pytest.mark.gpu


class _View:
    def __init__(self, ptr, n, typestr):
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": (n,), "typestr": typestr, "version": 3}


@pytest.mark.parametrize("n,per_record", [(3_000, False), (2_000_000, False), (200_000, True)])
def test_sites_read_on_another_stream(engine, n, per_record):  # noqa: F811
    import torch

    from paper_2511_00170_gb300 import ah
    from paper_2511_00170_gb300.pipeline import Params

    wl = synth.random_small(3, n_records=1, len_lo=10, len_hi=10, n_pairs=1, plant=0)
    wl.fwd, wl.rev, wl.k, wl.clamp = ["ACAC"], ["GGTT"], [1], 1   # a site every few bases
    p = Params.from_workload(wl)
    seq = np.frombuffer(b"ACGT", np.uint8)[np.random.default_rng(n).integers(0, 4, n, dtype=np.uint8)]
    batch = engine.pack(seq, np.array([0, n], dtype=np.int64), np.zeros(1, dtype=np.uint32))
    primers = ah.ah_primers_create(engine.ctx, p.fwd, p.rev, p.k, p.clamp)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    plen = torch.tensor([4, 4, 4, 4], dtype=torch.uint8, device="cuda")
    out = torch.empty(n * ah.AMP_DTYPE.itemsize, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    try:
        for _ in range(3):
            hits = (ah.ah_scan_primers_per_record if per_record else ah.ah_scan_primers)(engine.ctx, batch, primers)
            d_hits, d_off = ah.ah_hits_device(hits)
            n_hits = ah.ah_hits_count(hits)
            with torch.cuda.stream(streams[0]):
                view = torch.as_tensor(_View(d_hits, n_hits * ah.HIT_DTYPE.itemsize, "|u1"), device="cuda").clone()
            n_pairs = ah.ah_pair_amplicons_noalloc(streams[1].cuda_stream, d_hits, min(n_hits, 1 << 20), d_off,
                                                   plen.data_ptr(), 20, 400, 15, out.data_ptr(), n) if n_hits <= 1 << 20 else 0
            torch.cuda.synchronize()
            want = ah.ah_hits_copy(hits)
            assert len(want) > n // 100
            assert view.cpu().numpy().tobytes() == want.tobytes()
            if n_hits <= 1 << 20:
                amps = ah.ah_pair_amplicons(engine.ctx, batch, primers, hits, 20, 400, 15)
                ref = ah.ah_amplicons_copy(amps)
                ah.ah_amplicons_free(amps)
                assert out[:n_pairs * ah.AMP_DTYPE.itemsize].cpu().numpy().tobytes() == ref.tobytes()
            ah.ah_hits_free(hits)
    finally:
        ah.ah_primers_free(primers)
        ah.ah_batch_free(batch)
