"""The work a user of the in-silico PCR engine has it do, as cases that can be timed.

Each case goes through the public entry points (``paper_2511_00170_gb300.ah`` and ``.pipeline``):

  step_*   one call of ``Engine.step`` on a batch that is already packed: scan, pairing, Tm,
           extraction, results copied to the host.  One contig with exact primers (the smallest
           call a user makes), a set of genomes, and contigs under PCR buffer conditions with
           several primer pairs.
  plan_*   one replay of a graph-captured plan over a resident batch, results copied out:
           a small set of genomes, the 2,000-genome database, eight primer pairs over genomes of
           very different lengths, and degenerate primers over tandem repeats (many sites).
  upload   a plan's step on genomes that lie in page-locked host memory as ASCII.
  pack     contigs in device memory to 2-bit planes.
  fasta    a draft assembly as FASTA text in page-locked host memory, parsed and packed.
  fastq    amplicon reads as FASTQ text, parsed, packed and run through the whole step.
  serve    requests of different primer sets and genome subsets against a resident database.

Genomes, primers and parameters follow the workloads that ``synth`` and ``bench.py`` draw; the
primers below are the ones drawn there for the default seed.
"""
import math

import numpy as np
import torch

from paper_2511_00170_gb300 import ah
from paper_2511_00170_gb300.pipeline import Engine, Params

# the pair of the plain workloads (19 nt with 2 codes, 20 nt with 3), the eight pairs of the batched
# one (17-26 nt, 0-6 codes) and the pair of the dense one (18 nt, 9 codes)
PLAIN = (["AGATACCKWCAACAACTGC"], ["CTCCTCGTATAWTMTCRACC"])
BATCHED = (["CGATANRNCGCGCCRCATMGTA", "MYGTGCTGYCACAACRCGA", "GTYAGCAAWGCACTCGMAAC", "GGCGMCGCGGGTYACRGTTGA",
            "CNGRRTATATSARCWGTATC", "CTAACCGGTAAACACTCACGA", "AGCGCTCAGTACAGCTAT", "TGCARTGAATCCTCWGCAGCCT"],
           ["GTRTGGGAGTGGTRAGTCGNTTACA", "CAGCAGTTCGGRTGCTCTGG", "CCGGCGTGTAGATCCTGTGATTA",
            "GGGCGTKTAGTGTSTGTTGTACACT", "AGGGSMGMAAGARARCMCGA", "TTAGCACWGATTTSGAACCAG", "CACKANCRKACCRCCCACA",
            "SGKGAATAGTTTARWTGTAG"])
DENSE = (["SRNNAWCRWYAAGTSACC"], ["ATCWKSRANTMRRNATAA"])
# the plain pair's variant without codes, for exact-match checks
EXACT = (["AGATACCTACAACAACTGC"], ["CTCCTCGTATAATATCGACC"])

CODES = {"A": "A", "C": "C", "G": "G", "T": "T", "R": "AG", "Y": "CT", "S": "CG", "W": "AT", "K": "GT", "M": "AC",
         "B": "CGT", "D": "AGT", "H": "ACT", "V": "ACG", "N": "ACGT"}
COMPLEMENT = {"A": "T", "C": "G", "G": "C", "T": "A"}


def listed():
    return [
        # is this product unique on this plasmid: exact primers, one contig, answer at once
        {"name": "step_contig", "kind": "step", "records": 1, "lo": 48502, "hi": 48502, "primers": "exact", "k": 0,
         "planted": 6},
        # an ordinary interactive run: 16 genomes of 1-3 Mbp, k = 2, products below 45 C dropped
        {"name": "step_genomes", "kind": "step", "records": 16, "lo": 1000000, "hi": 3000000, "primers": "plain", "k": 2,
         "planted": 3, "min_tm": 45.0},
        # a panel of four pairs against a draft assembly's contigs under PCR buffer conditions
        # (Owczarzy's Mg correction, variants that match the site only, trimmed, 12-base barcodes)
        {"name": "step_panel", "kind": "step", "records": 3001, "lo": 300, "hi": 120000, "primers": "panel4", "k": 2,
         "planted": 2, "buffer": True, "trim": True, "barcode": 12},
        # the same 16 genomes screened again and again: one graph replay and its results
        {"name": "plan_genomes", "kind": "plan", "records": 16, "lo": 1000000, "hi": 3000000, "primers": "plain", "k": 2,
         "planted": 3, "min_tm": 45.0},
        # the 2,000-genome database (7.6 Gbp), trimmed amplicons with 16-base barcodes
        {"name": "plan_database", "kind": "plan", "records": 2000, "median": 3500000, "primers": "plain", "k": 3,
         "planted": 8, "trim": True, "barcode": 16, "autotune": True},
        # eight pairs at once over genomes from plasmids to 12 Mbp
        {"name": "plan_eight_pairs", "kind": "plan", "records": 2003, "lo": 10000, "hi": 12000000, "primers": "batched",
         "k": -1, "planted": 2, "autotune": True},
        # degenerate primers over genomes with tandem repeats: many sites, Tm of every paired one
        {"name": "plan_repeats", "kind": "plan", "records": 400, "median": 3500000, "primers": "dense", "k": 4,
         "planted": 0, "repeats": True, "max_len": 5000, "extract": False, "autotune": True},
        # genomes read from disk into page-locked memory, scanned as they cross the link
        {"name": "upload_genomes", "kind": "upload", "records": 57, "median": 3500000, "primers": "plain", "k": 2,
         "planted": 3},
        # a downloaded assembly collection already on the device, packed to 2 bits
        {"name": "pack_contigs", "kind": "pack", "records": 20011, "lo": 500, "hi": 400000},
        # draft assemblies as 80-column FASTA, as they come from a download
        {"name": "fasta_contigs", "kind": "fasta", "records": 1501, "lo": 500, "hi": 400000},
        # an amplicon sequencing run: 251-base reads, whole step, sequences back on the host
        {"name": "fastq_reads", "kind": "fastq", "records": 200003, "read": 251, "primers": "plain", "k": 2},
        # a shared database serving six users' panels, one to four pairs each
        {"name": "serve_panels", "kind": "serve", "records": 240, "median": 3500000, "requests": 6},
    ]


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["step", "step", "plan", "plan", "repeats", "upload", "pack", "fasta", "fastq", "serve"])
    primers = rng.choice(["plain", "panel2", "panel4"])
    if kind == "step":
        n = log(1, 3000)
        hi = min(3000000, max(3000, 60000000 // n))
        return {"kind": "step", "records": n, "lo": max(300, hi // rng.choice([2, 20, 100])), "hi": hi, "primers": primers,
                "k": rng.randint(0, 3), "planted": rng.randint(0, 4), "trim": rng.random() < 0.5,
                "barcode": rng.choice([0, 8, 16]), "buffer": rng.random() < 0.3}
    if kind == "plan":
        n = log(4, 1500)
        return {"kind": "plan", "records": n, "lo": 10000 + rng.randint(0, 999), "hi": log(100000, 6000000),
                "primers": rng.choice([primers, "batched"]), "k": rng.randint(1, 3), "planted": rng.randint(0, 6),
                "trim": rng.random() < 0.5, "barcode": rng.choice([0, 16])}
    if kind == "repeats":
        n = log(5, 300)
        return {"kind": "plan", "records": n, "median": log(500000, 3500000), "primers": "dense", "k": rng.randint(3, 4),
                "planted": 0, "repeats": True, "max_len": rng.choice([2000, 5000]),
                "extract": n <= 12 and rng.random() < 0.5}
    if kind == "upload":
        return {"kind": "upload", "records": log(3, 60), "median": log(300000, 3500000), "primers": primers,
                "k": rng.randint(1, 3), "planted": rng.randint(0, 4)}
    if kind == "pack":
        return {"kind": "pack", "records": log(1, 20000), "lo": 500, "hi": log(1000, 400000)}
    if kind == "fasta":
        return {"kind": "fasta", "records": log(1, 1500), "lo": 500, "hi": log(5000, 400000)}
    if kind == "fastq":
        return {"kind": "fastq", "records": log(2000, 200000), "read": rng.choice([150, 251, 300]), "primers": "plain",
                "k": rng.randint(1, 3)}
    return {"kind": "serve", "records": log(20, 240), "median": log(500000, 3500000), "requests": rng.randint(2, 8)}


# ---------------------------------------------------------------------------------------------- inputs
def _lengths(case):
    """Record lengths: the same for every seed of a case."""
    rng = np.random.default_rng(case["records"] * 7919 + case.get("lo", 0) + case.get("hi", 0) + case.get("median", 0))
    n = case["records"]
    if "median" in case:
        return np.maximum(1000, np.rint(case["median"] * np.exp(0.4 * rng.standard_normal(n)))).astype(np.int64)
    lo, hi = case["lo"], case["hi"]
    if hi > 10 * lo:
        return np.exp(rng.uniform(np.log(lo), np.log(hi), n)).astype(np.int64)
    return rng.integers(lo, hi + 1, n)


def _primers(case, which=None):
    which = which or case["primers"]
    if which in ("panel2", "panel4"):
        n = int(which[-1])
        fwd, rev = BATCHED[0][:n], BATCHED[1][:n]
    else:
        fwd, rev = {"plain": PLAIN, "batched": BATCHED, "dense": DENSE, "exact": EXACT}[which]
    k = case.get("k", 2)
    return list(fwd), list(rev), [i % 4 for i in range(len(fwd))] if k < 0 else [k] * len(fwd)


def _reverse_complement_choices(c):
    return [[COMPLEMENT[b] for b in s] for s in reversed(c)]


def _genomes(lengths, seed, gen, n_fraction=0.005):
    """Random genomes of G/C content 30-70 % with runs of N, back to back on the GPU."""
    off = np.zeros(len(lengths) + 1, dtype=np.int64)
    off[1:] = np.cumsum(lengths)
    total = int(off[-1])
    seq = torch.empty(total, dtype=torch.uint8, device="cuda")
    rng = np.random.default_rng(seed)
    # genomes of one G/C class are drawn together, in pieces: letter = table[random byte]
    classes = np.linspace(0.30, 0.70, 9)
    tables = []
    for gc in classes:
        at = int(round(256 * (1 - gc) / 2))
        cg = 128 - at
        tables.append(np.frombuffer(b"A" * at + b"C" * cg + b"G" * cg + b"T" * at, dtype=np.uint8).copy())
    tables = torch.from_numpy(np.stack(tables)).cuda()
    cls = rng.integers(0, 9, len(lengths))
    r, piece = 0, 1 << 25
    while r < len(lengths):
        e = r + 1  # short records share a class, so that a draft assembly's contigs do
        while e < len(lengths) and off[e + 1] - off[r] <= 1 << 20:
            e += 1
        for a in range(int(off[r]), int(off[e]), piece):
            b = min(int(off[e]), a + piece)
            x = torch.randint(0, 256, (b - a,), dtype=torch.uint8, device="cuda", generator=gen)
            seq[a:b] = tables[cls[r]][x.int()]
        r = e
    if n_fraction:
        runs = int(total * n_fraction / 25.5)
        for a in range(0, runs, 1 << 20):
            m = min(1 << 20, runs - a)
            start = torch.randint(0, max(1, total - 50), (m,), device="cuda", generator=gen)
            length = torch.randint(1, 51, (m,), device="cuda", generator=gen)
            at = start[:, None] + torch.arange(50, device="cuda")
            seq[at[torch.arange(50, device="cuda") < length[:, None]].clamp_(max=total - 1)] = ord("N")
    return seq, off


def _variants(choices, n, subs, gen):
    """n concrete variants of a primer (lists of allowed letters) with each base replaced at rate subs."""
    L = len(choices)
    table = np.empty((L, 12), dtype=np.uint8)
    for j, c in enumerate(choices):
        for i in range(12):
            table[j, i] = ord(c[i % len(c)])
    table = torch.from_numpy(table).cuda()
    pick = torch.randint(0, 12, (n, L), device="cuda", generator=gen)
    v = table.gather(1, pick.t()).t().contiguous()
    letters = torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device="cuda")
    other = letters[torch.randint(0, 4, (n, L), device="cuda", generator=gen)]
    return torch.where(torch.rand((n, L), device="cuda", generator=gen) < subs, other, v)


def _plant(seq, off, fwd, rev, per_record, subs, gen, lo=200, hi=1500):
    """Product templates in every record that has room: a forward primer's variant, then the other
    primer's reverse complement lo-hi bases on, half of them on the other strand; never overlapping."""
    if per_record <= 0:
        return
    lens = np.diff(off)
    room = hi + 80
    counts = np.minimum(per_record, lens // room)
    rec = np.repeat(np.arange(len(lens)), counts)
    if not len(rec):
        return
    slot = np.arange(len(rec)) - np.repeat(np.cumsum(counts) - counts, counts)
    seg = lens[rec] // np.maximum(1, counts[rec])
    seg_t, first = torch.from_numpy(seg).cuda(), torch.from_numpy(off[:-1][rec] + slot * seg).cuda()
    n = len(rec)
    start = first + (torch.rand(n, device="cuda", generator=gen, dtype=torch.float64) * (seg_t - room)).long()
    gap = torch.randint(lo, hi + 1, (n,), device="cuda", generator=gen)
    pair = torch.randint(0, len(fwd), (n,), device="cuda", generator=gen)
    strand = torch.randint(0, 2, (n,), device="cuda", generator=gen)
    for p in range(len(fwd)):
        f, r = [CODES[c] for c in fwd[p]], [CODES[c] for c in rev[p]]
        for s, (a, b) in enumerate(((f, _reverse_complement_choices(r)), (r, _reverse_complement_choices(f)))):
            m = torch.nonzero((pair == p) & (strand == s)).flatten()
            if not len(m):
                continue
            for choices, at in ((a, start[m]), (b, start[m] + gap[m])):
                seq[at[:, None] + torch.arange(len(choices), device="cuda")] = _variants(choices, len(m), subs, gen)


def _repeats(seq, off, seed, gen):
    """Tandem repeats (period 2-12, 1-20 kbp) in 30 % of the records."""
    rng = np.random.default_rng(seed + 1)
    letters = torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device="cuda")
    for g in range(len(off) - 1):
        if rng.random() >= 0.30:
            continue
        for _ in range(int(rng.integers(1, 6))):
            n = int(min(off[g + 1] - off[g], rng.integers(1000, 20001)))
            period = int(rng.integers(2, 13))
            a = int(off[g] + rng.integers(0, max(1, off[g + 1] - off[g] - n)))
            unit = letters[torch.randint(0, 4, (period,), device="cuda", generator=gen)]
            seq[a:a + n] = unit.repeat(n // period + 1)[:n]


def _sequences(case, seed, fwd, rev):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    seq, off = _genomes(_lengths(case), seed, gen, 0.0 if case.get("primers") == "exact" else 0.005)
    _plant(seq, off, fwd, rev, case.get("planted", 0), 0.0 if case.get("primers") == "exact" else 0.08, gen)
    if case.get("repeats"):
        _repeats(seq, off, seed, gen)
    torch.cuda.synchronize()
    return seq, off


def _params(case):
    fwd, rev, k = _primers(case)
    more = {}
    if case.get("buffer"):
        more = {"K": 50.0, "Na": 0.0, "Tris": 10.0, "Mg": 1.5, "dNTPs": 0.8, "dnac1": 250.0, "dnac2": 0.0, "saltcorr": 7,
                "variants": 1}
    return Params(fwd, rev, k, 3, 50, case.get("max_len", 2000), min_tm=case.get("min_tm"), trim=bool(case.get("trim")),
                  fb_len=case.get("barcode", 0), rb_len=case.get("barcode", 0), **more)


# ----------------------------------------------------------------------------------------------- states
_ENGINE = []


def _engine():
    """The one engine a program keeps."""
    if not _ENGINE:
        _ENGINE.append(Engine(0))
    return _ENGINE[0]


class _State:
    """What the program holds for one case; its native objects are released with it."""

    def __init__(self, case):
        self.case = case
        self.batch = self.primers = self.plan = self.server = None

    def __del__(self):
        if self.server is not None:
            ah.ah_server_destroy(self.server)
        if self.plan is not None:
            ah.ah_plan_free(self.plan)
        if self.primers is not None:
            ah.ah_primers_free(self.primers)
        if self.batch is not None:
            ah.ah_batch_free(self.batch)


class _DeviceArray:
    """A library buffer as an object torch can view; the view keeps the buffer's owner."""

    def __init__(self, owner, ptr, shape, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = {"data": (int(ptr), False), "shape": shape, "typestr": typestr, "version": 3}


class _Batch:
    """A packed batch, freed when neither the state nor a view of it is left."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        ah.ah_batch_free(self.handle)

    def arrays(self):
        v = ah.ah_batch_view_get(self.handle)
        n, r = v["n_groups"], v["n_records"]
        return [torch.as_tensor(_DeviceArray(self, v[name], shape, kind), device="cuda") for name, shape, kind in
                (("planes", (n, 2), "<i4"), ("invalid", (n,), "<i4"), ("rec_group", (r,), "<i8"), ("rec_len", (r,), "<i4"))]


def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h


def prepare(case, seed):
    st = _State(case)
    eng = _engine()
    kind = case["kind"]
    if kind == "fastq":
        return _prepare_fastq(st, case, seed)
    fwd, rev = _primers(case)[:2] if "primers" in case else ([], [])
    seq, off = _sequences(case, seed, fwd, rev)
    st.offsets = off.astype(np.uint64)
    if kind in ("step", "plan", "upload"):
        st.params = _params(case)
        st.out = _Results(*_room(case), bool(case.get("extract", True)))
        st.batch = eng.pack_device(seq.data_ptr(), off)
        ah.ah_ctx_synchronize(eng.ctx)
    if kind in ("plan", "upload"):
        p = st.params
        st.with_seqs = bool(case.get("extract", True))
        st.primers = ah.ah_primers_create(eng.ctx, p.fwd, p.rev, p.k, p.clamp)
        st.plan = ah.ah_plan_create(eng.ctx, st.batch, st.primers, ah.plan_params(
            p.min_len, p.max_len, p.orient_mask, p.tm_params(), st.with_seqs, p.trim, p.fb_len, p.rb_len,
            autotune=bool(case.get("autotune"))))
    if kind == "upload":
        st.text = _pinned(seq)
    elif kind == "pack":
        st.seq = seq
    elif kind == "fasta":
        st.text = _pinned(_fasta_text(seq, off))
    elif kind == "serve":
        st.batch = eng.pack_device(seq.data_ptr(), off)
        ah.ah_ctx_synchronize(eng.ctx)
        st.server = ah.ah_server_create(st.batch, 4)
        st.requests = _requests(case)
        st.outs = [_Results(*_room(case, len(r["fwd"]))) for r in st.requests]
    del seq
    torch.cuda.synchronize()
    return st


def _room(case, pairs=None):
    """Sites and amplicons a program keeps room for, and bytes of their sequences."""
    if case["kind"] == "fastq":
        n = 2 * case["records"]
        return 2 * n, n, n * (case["read"] + 80)
    bases = int(_lengths(case).sum())
    if case.get("primers") == "dense":
        n = 200000 + bases // 300
        return n, n, (3 * bases if case.get("extract", True) else 1)
    pairs = pairs or len(_primers(case)[0])
    planted = 2 * case.get("planted", 0) * case["records"]
    amps = 256 + planted + bases * pairs // 500000
    return 2048 + 2 * planted + bases * pairs // 50000, amps, 1700 * amps


class _Results:
    """A program's own page-locked result buffers."""

    def __init__(self, hits, amps, arena, with_seqs=True):
        def room(n, dtype):
            return torch.zeros(n * np.dtype(dtype).itemsize, dtype=torch.uint8, pin_memory=True).numpy().view(dtype)

        self.hits, self.amps = room(hits, ah.HIT_DTYPE), room(amps, ah.AMP_DTYPE)
        self.arena = room(arena, np.uint8) if with_seqs else None
        self.field_off = room(5 * amps + 1, np.uint64) if with_seqs else None

    def take(self, hits, amps, arena, field_off):
        """Results that came as arrays of their own."""
        for mine, theirs in ((self.hits, hits), (self.amps, amps), (self.arena, np.frombuffer(arena, dtype=np.uint8)),
                             (self.field_off, field_off)):
            mine[:len(theirs)] = theirs
        return self.arrays(len(hits), len(amps))

    def arrays(self, n_hits, n_amps):
        out = [n_hits, n_amps, self.hits.view(np.int32).reshape(-1, 3), self.amps.view(np.int32).reshape(-1, 8)[:, :6],
               self.amps["tm"]]
        return out if self.arena is None else out + [self.arena, self.field_off.view(np.int64)]


def _requests(case):
    """One to four pairs each over a contiguous part of the database."""
    rng = np.random.default_rng(case["requests"] * 31 + case["records"])
    out = []
    for i in range(case["requests"]):
        n = int(rng.integers(1, 5))
        first = int(rng.integers(0, 8 - n + 1))
        count = max(1, int(round(case["records"] * math.exp(rng.uniform(math.log(0.03), 0.0)))))
        out.append(dict(fwd=BATCHED[0][first:first + n], rev=BATCHED[1][first:first + n],
                        k=[int(x) for x in rng.integers(1, 4, n)], clamp=3,
                        first_record=int(rng.integers(0, case["records"] - count + 1)), n_records=count, min_len=50,
                        max_len=2000))
    return out


def _fasta_text(seq, off):
    """80-column FASTA of the records."""
    heads = [(">contig_%06d length=%d" % (i, off[i + 1] - off[i])).encode() + b"\n" for i in range(len(off) - 1)]
    lens = np.diff(off)
    size = np.array([len(h) for h in heads]) + lens + (lens + 79) // 80
    at = np.zeros(len(size) + 1, dtype=np.int64)
    at[1:] = np.cumsum(size)
    text = torch.full((int(at[-1]),), 10, dtype=torch.uint8, device="cuda")
    blob = torch.from_numpy(np.frombuffer(b"".join(heads), dtype=np.uint8).copy()).cuda()
    h0 = 0
    for i, h in enumerate(heads):
        a, n = int(at[i]) + len(h), int(lens[i])
        text[int(at[i]):a] = blob[h0:h0 + len(h)]
        h0 += len(h)
        full = n // 80
        text[a:a + 81 * full].view(full, 81)[:, :80] = seq[int(off[i]):int(off[i]) + 80 * full].view(full, 80)
        if n % 80:
            text[a + 81 * full:a + 81 * full + n % 80] = seq[int(off[i]) + 80 * full:int(off[i]) + n]
    return text


def _prepare_fastq(st, case, seed):
    """Reads that hold a variant of the forward primer 0-10 bases in and of the reverse primer 0-10
    bases before the end, a tenth of them random, 1 % errors; qualities '!' to 'J'."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, L = case["records"], case["read"]
    st.params = _params(case)
    st.out = _Results(*_room(case))
    p = st.params
    letters = torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device="cuda")
    reads = letters[torch.randint(0, 4, (n, L), device="cuda", generator=gen)]
    keep = torch.rand(n, device="cuda", generator=gen) >= 0.1
    for choices, end in (([CODES[c] for c in p.fwd[0]], False), (_reverse_complement_choices([CODES[c] for c in p.rev[0]]), True)):
        m = len(choices)
        at = torch.randint(0, 11, (n,), device="cuda", generator=gen)
        at = (L - m - at if end else at)[:, None] + torch.arange(m, device="cuda")
        reads.scatter_(1, at, torch.where(keep[:, None], _variants(choices, n, 0.01, gen), reads.gather(1, at)))
    quals = torch.randint(33, 75, (n, L), dtype=torch.uint8, device="cuda", generator=gen)
    digits = 10
    text = torch.empty((n, 1 + digits + 1 + L + 3 + L + 1), dtype=torch.uint8, device="cuda")
    text[:, 0] = ord("@")
    index = torch.arange(n, device="cuda")
    for d in range(digits):
        text[:, 1 + d] = (48 + index // 10 ** (digits - 1 - d) % 10).to(torch.uint8)
    c = 1 + digits
    text[:, c] = 10
    text[:, c + 1:c + 1 + L] = reads
    c += 1 + L
    text[:, c] = 10
    text[:, c + 1] = ord("+")
    text[:, c + 2] = 10
    text[:, c + 3:c + 3 + L] = quals
    text[:, -1] = 10
    st.text = _pinned(text.view(-1))
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------------------------------------- runs
def run(st):
    return _RUN[st.case["kind"]](st)


def _run_step(st):
    o = _engine().step(st.batch, st.params)
    return st.out.take(o.hits, o.amps, o.arena, o.field_off)


def _copy_plan(st):
    o = st.out
    ah.ah_plan_copy_results(st.plan, _engine().ctx, o.hits, o.amps, o.arena, o.field_off)
    i = ah.ah_plan_info_get(st.plan)
    return o.arrays(i["n_hits"], i["n_kept"])


def _run_plan(st):
    ah.ah_plan_launch(st.plan, _engine().ctx)
    return _copy_plan(st)


def _run_upload(st):
    ah.ah_plan_launch_host(st.plan, st.text.data_ptr(), st.offsets, _engine().ctx)
    return _copy_plan(st)


def _run_pack(st):
    return _Batch(_engine().pack_device(st.seq.data_ptr(), st.offsets)).arrays()


def _run_fasta(st):
    batch, names = ah.ah_fasta_pack(_engine().ctx, st.text.data_ptr(), n_bytes=st.text.numel())
    return _Batch(batch).arrays() + [len(names)]


def _run_fastq(st):
    eng, lib, o = _engine(), ah.load(), st.out
    batch, quals, _ = ah.ah_fastq_pack(eng.ctx, st.text.data_ptr(), n_bytes=st.text.numel(), names=False)
    hits, amps = eng.step(batch, st.params, copy_out=False)
    try:
        n_hits, n_amps = ah.ah_hits_count(hits), ah.ah_amplicons_count(amps)
        for status in (lib.ah_hits_copy(hits, o.hits.ctypes.data, len(o.hits)),
                       lib.ah_amplicons_copy(amps, o.amps.ctypes.data, len(o.amps)),
                       lib.ah_amplicons_seq_copy(amps, o.arena.ctypes.data, len(o.arena), o.field_off.ctypes.data,
                                                 len(o.field_off))):
            if status != ah.AH_OK:
                raise ah.AhError(status, ah.ah_last_error(eng.ctx))
    finally:
        ah.ah_hits_free(hits)
        ah.ah_amplicons_free(amps)
        ah.ah_quals_free(quals)
        ah.ah_batch_free(batch)
    return o.arrays(n_hits, n_amps)


def _run_serve(st):
    tickets = [ah.ah_server_submit(st.server, **r) for r in st.requests]
    out = []
    for t, o in zip(tickets, st.outs):
        r = ah.ah_server_wait(st.server, t)
        out.append(o.take(r["hits"], r["amps"], r["arena"], r["field_off"]))
    return out


_RUN = {"step": _run_step, "plan": _run_plan, "upload": _run_upload, "pack": _run_pack, "fasta": _run_fasta,
        "fastq": _run_fastq, "serve": _run_serve}


# ------------------------------------------------------------------------------------------------- work
def work(case):
    """Bytes: a scan reads two code bits and one validity bit per base, a parser its text once, and
    packing writes three bits per base; a shown site is about 12 bytes and an amplicon 32 beside its
    letters, both small.  Operations: three per compared pattern position, 32 positions at a time."""
    kind = case["kind"]
    if kind == "fastq":
        n, L = case["records"], case["read"]
        return {"bytes": n * (2 * L + 16) + 0.375 * n * L + n * (L + 110), "flops": 4 * 60 * n * L / 32}
    bases = float(_lengths(case).sum())
    if kind == "pack":
        return {"bytes": 1.375 * bases, "flops": 0.0}
    if kind == "fasta":
        return {"bytes": bases * (1 + 1 / 80) + 0.375 * bases, "flops": 0.0}
    if kind == "serve":
        b = f = 0.0
        lens = _lengths(case)
        for r in _requests(case):
            part = float(lens[r["first_record"]:r["first_record"] + r["n_records"]].sum())
            b += 0.25 * part
            f += 4 * len(r["fwd"]) * 60 * part / 32
        return {"bytes": b, "flops": f}
    pairs = len(_primers(case)[0])
    text = bases if kind == "upload" else 0.0
    return {"bytes": 0.25 * bases + text, "flops": 4 * pairs * 60 * bases / 32}


# ------------------------------------------------------------------------------------------------ exact
# Allawi & SantaLucia 1997: kcal/mol and cal/(K mol) of a stack, read 5'-3' over its complement
_STACK = {"AA": (-7.9, -22.2), "AT": (-7.2, -20.4), "TA": (-7.2, -21.3), "CA": (-8.5, -22.7), "GT": (-8.4, -22.4),
          "CT": (-7.8, -21.0), "GA": (-8.2, -22.2), "CG": (-10.6, -27.2), "GC": (-9.8, -24.4), "GG": (-8.0, -19.9)}


def _tm_of(s):
    """Tm of a perfectly matched duplex at 50 mM Na+ and 25 nM of each strand, in 64 bits."""
    h = s_ = 0.0
    for a, b in zip(s, s[1:]):
        dh, ds = _STACK.get(a + b) or _STACK[COMPLEMENT[b] + COMPLEMENT[a]]
        h, s_ = h + dh, s_ + ds
    for e in (s[0], s[-1]):
        dh, ds = (2.3, 4.1) if e in "AT" else (0.1, -2.8)
        h, s_ = h + dh, s_ + ds
    s_ += 0.368 * (len(s) - 1) * math.log(50e-3)
    return 1000 * h / (s_ + 1.987 * math.log((25 - 25 / 2.0) * 1e-9)) - 273.15


def _find(text, word):
    at, i = [], text.find(word)
    while i >= 0:
        at.append(i)
        i = text.find(word, i + 1)
    return at


def exact(case, seed):
    """The melting temperatures of an exact-match check; sites and letters are whole numbers."""
    if case["kind"] != "step" or case["primers"] != "exact" or case["records"] != 1:
        return None
    fwd, rev = EXACT[0][0], EXACT[1][0]
    seq, _ = _sequences(case, seed, [fwd], [rev])
    text = seq.cpu().numpy().tobytes().decode("ascii")
    sites = []
    for primer, s in enumerate((fwd, rev)):
        rc = "".join(COMPLEMENT[c] for c in reversed(s))
        sites += [(i, 0, primer, len(s)) for i in _find(text, s)] + [(i, 1, primer, len(s)) for i in _find(text, rc)]
    sites.sort(key=lambda x: (x[0], 2 * x[1] + x[2]))
    tms = []
    for i, a in enumerate(sites):
        if a[1]:
            continue
        for b in sites[i + 1:]:
            if not b[1] or b[0] + b[3] - a[0] > 2000:
                break
            if b[0] + b[3] - a[0] >= 50:
                tms.append(min(_tm_of((fwd, rev)[a[2]]), _tm_of((fwd, rev)[b[2]])))
    tm = np.zeros(_room(case)[1])
    tm[:len(tms)] = tms
    return [None, None, None, None, tm, None, None]
