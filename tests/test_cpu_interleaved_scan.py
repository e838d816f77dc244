"""The interleaved scan form on the CPU: the generated kernel's own text, compiled for the host and run a warp at a
time with every lane as a fiber (warp_emulator.h), finds exactly the windows that a per-position count and clamp check
finds.  It runs with its lanes in several orders between two warp-wide operations, so that a result that rests on a
warp staying converged shows.  It also compiles for sm_103a (NVRTC on the host).  No GPU is needed."""
import os
import re
import subprocess

import numpy as np
import pytest

import synth
from tests.scan_emulator import CODE, COMP, SETS

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BUILD = os.path.join(ROOT, "paper_2511_00170_gb300", "_build")
TESTS = os.path.join(ROOT, "tests")

EIGHT = ["CGATANRNCGCGCCRCATMGTA", "MYGTGCTGYCACAACRCGA", "GTYAGCAAWGCACTCGMAAC", "GGCGMCGCGGGTYACRGTTGA",
         "CNGRRTATATSARCWGTATC", "CTAACCGGTAAACACTCACGA", "AGCGCTCAGTACAGCTAT", "TGCARTGAATCCTCWGCAGCCT",
         "GTRTGGGAGTGGTRAGTCGNTTACA", "CAGCAGTTCGGRTGCTCTGG", "CCGGCGTGTAGATCCTGTGATTA",
         "GGGCGTKTAGTGTSTGTTGTACACT", "AGGGSMGMAAGARARCMCGA", "TTAGCACWGATTTSGAACCAG", "CACKANCRKACCRCCCACA",
         "SGKGAATAGTTTARWTGTAG"]
PLAIN = ["AGATACCKWCAACAACTGC", "CTCCTCGTATAWTMTCRACC"]


@pytest.fixture(scope="module")
def dump():
    import __graft_entry__

    __graft_entry__.build()
    exe, lib = os.path.join(BUILD, "il_dump"), os.path.join(ROOT, "paper_2511_00170_gb300")
    sources = [os.path.join(TESTS, "il_dump.cpp"), os.path.join(TESTS, "jit_dump.cpp")]
    if not os.path.exists(exe) or os.path.getmtime(exe) < max(map(os.path.getmtime, sources + [f"{lib}/libah.so"])):
        subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", "/usr/local/cuda/include", sources[0], "-o", exe,
                               "-L", lib, "-lah", f"-Wl,-rpath,{lib}"])

    def run(what, k, clamp, primers, windows=1024):
        return subprocess.run([exe, what, f"windows={windows}", str(k), str(clamp)] + primers, text=True,
                              capture_output=True, check=what != "compile").stdout

    return run


def host_source(src):
    """The generated text as C++ for warp_emulator.h."""
    src = re.sub(r'asm\("lop3\.b32 %0, %1, %2, %3, (0x[0-9a-f]+);" : "=r"\((\w+)\) : "r"\(([\w.]+)\), "r"\(([\w.]+)\), '
                 r'"r"\(([\w.]+)\)\);', r"\2 = lop3(\3, \4, \5, \1);", src)
    src = re.sub(r'asm volatile\("prefetch[^;]*;"[^;]*;', ";", src)
    assert 'asm("' not in src
    with open(os.path.join(TESTS, "il_run.cpp")) as f:
        return '#include "warp_emulator.h"\n' + src + f.read()


def build(tmp, src):
    cpp, exe = os.path.join(tmp, "kernel.cpp"), os.path.join(tmp, "kernel")
    with open(cpp, "w") as f:
        f.write(host_source(src))
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-w", "-I", TESTS, cpp, "-o", exe])
    return exe


def planes_of(text):
    """Text (ACGT, anything else invalid) to plane and invalid words of whole groups, and 64 groups after them."""
    b = np.frombuffer(text.encode(), dtype=np.uint8)
    n = (len(b) + 31) // 32
    code, bad = np.zeros(n * 32, np.uint8), np.ones(n * 32, bool)
    for c, v in CODE.items():
        m = np.flatnonzero(b == ord(c))
        code[m], bad[m] = v, False
    word = lambda bits: np.packbits(bits.astype(np.uint8), bitorder="little").view(np.uint32)
    planes = np.zeros((n + 64, 2), np.uint32)
    invalid = np.full(n + 64, 0xFFFFFFFF, np.uint32)
    planes[:n, 0], planes[:n, 1], invalid[:n] = word(code & 1), word(code >> 1), word(bad)
    return n, planes, invalid, code, bad


def run(exe, tmp, text, cap=1 << 17, order=0, first=0, count=None):
    """(returncode, status, tile counts, sorted sites (tile, key))"""
    n, planes, invalid, _, _ = planes_of(text)
    count = n - first if count is None else count
    a, b = os.path.join(tmp, "in"), os.path.join(tmp, "out")
    with open(a, "wb") as f:
        f.write(np.array([n, first, count, cap], np.uint32).tobytes() + planes.tobytes() + invalid.tobytes())
    r = subprocess.run([exe, a, b, str(order)], capture_output=True, text=True, timeout=300)
    if r.returncode:
        return r.returncode, r.stderr, None, None
    raw = np.fromfile(b, np.uint8)
    tiles = (n + 1023) // 1024
    status = int(raw[:4].view(np.uint32)[0])
    counts = raw[4:4 + 4 * tiles].view(np.uint32)
    slots = raw[4 + 4 * tiles:].view(np.uint64).reshape(tiles, cap)
    sites = sorted((t, int(s)) for t in range(tiles) for s in slots[t, :min(cap, counts[t])])
    return 0, status, counts, sites


def expected(text, primers, k, clamp):
    n, _, _, code, bad = planes_of(text)
    code, bad = np.pad(code, (0, 64)), np.pad(bad, (0, 64), constant_values=True)
    out, x = [], np.arange(n * 32)
    q = 0
    for p in primers:
        p, kk = (p.split(":")[0], int(p.split(":")[1])) if ":" in p else (p, k)
        rc = "".join(COMP[c] for c in reversed(p))
        for pat, cl in ((p, range(len(p) - clamp, len(p))), (rc, range(0, clamp))):
            mism, ok = np.zeros(n * 32, int), np.ones(n * 32, bool)
            for j, ch in enumerate(pat):
                match = np.isin(code[x + j], [CODE[c] for c in SETS[ch]])
                mism += ~match
                ok &= ~bad[x + j]
                if j in cl:
                    ok &= match
            for pos in np.flatnonzero(ok & (mism <= kk)):
                t = int(pos) // 32768
                out.append((t, (q // 4) << 48 | (int(pos) - t * 32768) << 16 | (q % 4) << 8 | int(mism[pos])))
            q += 1
    return sorted(out)


def _random(n, seed):
    return "".join(np.array(list("ACGT"))[np.random.default_rng(seed).integers(0, 4, n)])


def _repeats(n, seed, primers, share):
    """Random bases with tandem repeats of a primer's concrete bases in `share` of them, and some Ns."""
    rng = np.random.default_rng(seed)
    out = list(_random(n, seed))
    while share > 0:
        p = primers[int(rng.integers(len(primers)))].split(":")[0]
        if rng.random() < 0.5:
            p = "".join(COMP[c] for c in reversed(p))
        unit = "".join(SETS[c][0] for c in p)
        m = int(min(n, rng.integers(200, 3000)))
        at = int(rng.integers(0, n - m + 1))
        out[at:at + m] = (unit * (m // len(unit) + 1))[:m]
        share -= m / n
    for at in rng.integers(0, n, 5):
        out[at] = "N"
    return "".join(out)


@pytest.mark.parametrize("order", [0, 1, 2, 3])
@pytest.mark.parametrize("k,primers", [(3, PLAIN), (2, EIGHT[:8]), (0, ["ACGTACGT"])])
def test_queue_overflow_with_lanes_in_any_order(dump, tmp_path, k, primers, order):
    """Tiles whose surviving windows overflow the warp's queue many times over: the careful mode, in which the queue's
    length is read after every iteration and decides for the whole warp how it goes on."""
    exe = build(str(tmp_path), dump("source", k, 3, primers))
    text = _repeats(50_000, 7 + k, primers, 0.4)
    rc, status, counts, sites = run(exe, str(tmp_path), text, order=order)
    assert rc == 0, status
    want = expected(text, primers, k, 3)
    assert len(want) > 4 * 96 and sites == want  # the queue holds 96, the text is two tiles


@pytest.mark.parametrize("clamp", [0, 2])
@pytest.mark.parametrize("k,primers", [(3, PLAIN), (0, ["ACGTACGT", "NNACGTAC"]), (1, EIGHT[:4]), (5, EIGHT[4:8])])
def test_self_check(dump, tmp_path, k, primers, clamp):
    """Windows that a filter lets through by design set no status; with the circuit's verdict altered in one place of
    the text (one more position let through for every window) the check reports it, and the sites are still right."""
    src = dump("source", k, clamp, primers)
    text = _random(33_000, k) + "N" * 7 + _random(500, k + 1)
    want = expected(text, primers, k, clamp)
    rc, status, _, sites = run(build(str(tmp_path), src), str(tmp_path), text)
    assert (rc, status) == (0, 0) and sites == want
    m = re.search(r"const u32 f1_1 = (\S+);", src)
    rc, status, _, sites = run(build(str(tmp_path), src.replace(m.group(0), f"const u32 f1_1 = {m.group(1)} & ~2u;")),
                               str(tmp_path), text)
    assert (rc, status) == (0, 1) and sites == want


def test_more_patterns_than_an_iteration_may_queue(dump, tmp_path):
    """Sets far above what plans give the form (128 patterns): the iteration shrinks so that the queue holds one lane's
    words at least, and a set that cannot fit is refused when the kernel is built, not left to spin."""
    many = [synth.random_primer(synth.Stream(synth.make_key(5, i, 0)), 12, 2, 0) for i in range(100)]   # 200 patterns
    text = _repeats(33_000, 3, many[:2], 0.1)
    rc, status, _, sites = run(build(str(tmp_path), dump("source", 0, 1, many)), str(tmp_path), text, order=2)
    assert (rc, status) == (0, 0) and sites == expected(text, many, 0, 1) and len(sites) > 100
    assert dump("compile", 0, 1, many * 2).startswith("error")   # 400 patterns


@pytest.mark.parametrize("threads,groups", [(32, 1), (64, 4), (128, 8), (256, 4), (256, 8), (1024, 16), (96, 5)])
def test_generic_kernel_covers_the_forms_tiles(dump, threads, groups):
    """The generic kernel, which scans first on contexts that compile in the background, has blocks enough for every
    group of the interleaved form's tiles whatever the context's scan shape, and grids within the limit."""
    exe = os.path.join(BUILD, "il_dump")
    for tiles in (1, 2, 511, 100_003):
        covered, most, blocks = map(int, subprocess.check_output([exe, "generic", str(threads), str(groups), str(tiles)]).split())
        assert tiles * 1024 <= covered < tiles * 1024 + threads * groups
        assert most >= 1 and blocks <= 0x7fffffff


TILE = 32768


@pytest.mark.parametrize("k,clamp,primers", [
    (2, 3, PLAIN), (0, 0, ["ACGTACGT"]), (1, 2, ["ACGRYSWKMBDHVN"]), (3, 3, ["NNNNACGTNNNNACGTAC"]),
    (5, 1, ["ACGTAGCTAGCTAGCATCGATCGATCGATCGA"]), (7, 0, ["AGCTTGACCGTAGGCATTAC"]), (2, 20, ["AGCTTGACCGTAGGCATTAC"]),
    (6, 3, ["RRRRRRRRRRYYYYYYYYYY"]), (0, 2, ["AC"]), (0, 0, EIGHT), (1, 3, [f"{p}:{i % 4}" for i, p in enumerate(EIGHT)]),
    (3, 3, EIGHT + PLAIN + [p[::-1] for p in EIGHT])])
def test_sites_equal_the_exact_count(dump, tmp_path, k, clamp, primers):
    """Every set's sites on random bases with planted copies, invalid bases, and windows over every kind of edge: a
    group's, a lane's (the next lane's words), a tile's and the batch's."""
    exe = build(str(tmp_path), dump("source", k, clamp, primers))
    rng = np.random.default_rng(len(primers) + k)
    text = list(_random(2 * TILE + 77, k))
    first = primers[0].split(":")[0]
    for at in (0, 31, 1000, 1023, 1024, TILE - 40, TILE - 32, TILE - 19, TILE - 1, TILE, 2 * TILE - 5, 2 * TILE + 77 - len(first)):
        p = primers[int(rng.integers(len(primers)))].split(":")[0] if at % 2 else first
        if at + len(p) <= len(text):
            text[at:at + len(p)] = [SETS[c][int(rng.integers(len(SETS[c])))] for c in p]
    for at in rng.integers(0, len(text), 40):
        text[at] = "N"
    text = "".join(text)
    want = expected(text, primers, k, clamp)
    for order in (0, 2):
        rc, status, counts, sites = run(exe, str(tmp_path), text, order=order)
        assert (rc, status) == (0, 0) and sites == want
    # a range of tiles, as an upload scans it: what starts in it, and nothing else
    rc, status, _, sites = run(exe, str(tmp_path), text, first=1024, count=1024)
    assert (rc, status) == (0, 0) and sites == [s for s in want if s[0] == 1]
    # slot lists shorter than a tile's sites: counted in full, the lists hold what fits
    rc, _, counts, _ = run(exe, str(tmp_path), text, cap=1)
    assert rc == 0 and counts.sum() == len(want)


@pytest.mark.parametrize("n", [1, 9, 31, 32, 33, 63, 65, 1000, TILE - 1, TILE, TILE + 1, TILE + 33])
def test_sizes(dump, tmp_path, n):
    exe = build(str(tmp_path), dump("source", 1, 1, ["ACGT", "GGA"]))
    text = _random(n, n)
    rc, status, _, sites = run(exe, str(tmp_path), text, order=3)
    assert (rc, status) == (0, 0) and sites == expected(text, ["ACGT", "GGA"], 1, 1)


@pytest.mark.parametrize("windows", [1024, 4096])
@pytest.mark.parametrize("primers", [PLAIN, EIGHT, EIGHT * 4], ids=["one pair", "eight", "thirty-two"])
def test_compiles(dump, primers, windows):
    """For sm_103a, with NVRTC on the host: the smallest and the largest set that plans give the form, at the phase splits
    that the autotuner tries."""
    out = dump("compile", 2, 3, primers, windows=windows)
    assert out.startswith("compiled "), out[:2000]


def test_which_sets_suit(dump):
    """Plans choose the form for sets whose filters leave few windows, of at most 32 pairs."""
    assert dump("suits", 3, 3, PLAIN).strip() == "1" and dump("suits", 2, 3, EIGHT * 4).strip() == "1"
    assert dump("suits", 0, 0, ["AC"]).strip() == "0" and dump("suits", 1, 0, ["NN"]).strip() == "0"
    assert dump("suits", 2, 3, EIGHT * 4 + PLAIN).strip() == "0"


def test_bench_tables_describe_the_generated_circuits(dump):
    """bench.py keys its measured ALU-pipe and DRAM figures of this form by circuit size: the bench pair's 71 instructions
    per 32 positions and the 8-pair batched set's 324, k = i mod 4."""
    import bench

    assert int(dump("ops", 3, 3, PLAIN)) == 71
    wl = synth.batched(n_genomes=3)
    batched = [f"{p}:{k}" for f, r, k in zip(wl.fwd, wl.rev, wl.k) for p in (f, r)]
    assert int(dump("ops", 0, wl.clamp, batched)) == 324
    for ops in (71, 324):
        assert ops in bench.SCAN_PIPE and (ops, 64, 32, 0, 0) in bench.SCAN_TRAFFIC
