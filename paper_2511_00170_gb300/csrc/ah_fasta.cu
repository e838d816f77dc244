// FASTA input on the device (Abstract and Section "Implementations": the pipeline packs FASTA into
// 2-bit batches).  Raw FASTA text, a '>' header line per record followed by sequence lines, is
// parsed where it lies in HBM: a pass over 16 KiB tiles that gives each tile's line-state function and
// its counts from every entry state, a block that chains the tiles, and an emitting pass that
// compacts the sequence bytes (line breaks and blanks dropped) and records every header.  Nothing is
// read back in between, so host text is parsed chunk by chunk while it crosses the link.  The compacted
// sequences are packed like any other device source.
//
// Line state: LS at the start of a line, H inside a header line, S inside a sequence line.  A line
// whose first byte is '>' is a header and starts a record; '\n' ends a line; '\r', ' ' and '\t' in a
// sequence line are not bases.  Bytes before the first header belong to no record.
#include <algorithm>
#include <cstring>

#include "ah_internal.h"

struct ah_fasta {
  std::vector<std::string> names;  // header lines without '>' (or '@') and trailing '\r'
};

namespace ah {
namespace {

constexpr int kFaThreads = 256, kFaBytes = 64, kFaTile = kFaThreads * kFaBytes;
// a thread takes 64 consecutive bytes, its masks are 64-bit words; a tile (one CTA) is 16 KiB
enum : uint32_t { FS_LS = 0, FS_H = 1, FS_S = 2 };
// a transfer function over the three states: bits 2s..2s+1 hold the state after, from state s
constexpr uint32_t kIdentity = FS_LS | (FS_H << 2) | (FS_S << 4);

__device__ __forceinline__ uint32_t apply(uint32_t f, uint32_t s) { return (f >> (2 * s)) & 3u; }
// first a, then b
__device__ __forceinline__ uint32_t compose(uint32_t a, uint32_t b) {
  return apply(b, apply(a, FS_LS)) | (apply(b, apply(a, FS_H)) << 2) | (apply(b, apply(a, FS_S)) << 4);
}
// A thread's bytes (little-endian words, in registers) and their classes, bit j for byte j: within the text;
// line breaks; '>' (FASTA only); blanks (FASTA: carriage returns, spaces and tabs; FASTQ: carriage returns).
struct Text {
  uint32_t w[16];
  uint64_t valid, nl, gt, blank;
};

__device__ __forceinline__ uint64_t below(int bit) { return bit >= 64 ? ~0ull : (1ull << bit) - 1ull; }

// bits 7, 15, 23, 31 of m to bits 0-3 (the four partial products land on distinct bits below 28)
__device__ __forceinline__ uint32_t bit7_mask(uint32_t m) { return ((m & 0x80808080u) * 0x00204081u) >> 28; }

// bit j: byte j of w equals the byte in ch4 (exact per byte: no borrow crosses bytes)
__device__ __forceinline__ uint32_t bytes_eq(uint32_t w, uint32_t ch4) {
  const uint32_t y = w ^ ch4;
  return bit7_mask(~(((y & 0x7f7f7f7fu) + 0x7f7f7f7fu) | y));
}

// The thread's bytes [p, p + 64) of the text's n: whole and 16-byte aligned, four vector loads issued
// together; otherwise byte loads up to the end.  A 16-byte segment of letters alone (FASTA: bit 7 clear and
// bit 6 set, which line breaks, '>' and blanks don't have) or without control characters (FASTQ) has no class
// to find, so most skip the exact tests.
template <bool fastq>
__device__ __forceinline__ void load_text(const uint8_t* __restrict__ t, uint64_t n, uint64_t p, Text* x) {
  if (p + kFaBytes <= n && (((uint64_t)(uintptr_t)t) & 15) == 0) {
    const uint4* v = reinterpret_cast<const uint4*>(t + p);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 y = __ldg(v + q);
      x->w[4 * q] = y.x, x->w[4 * q + 1] = y.y, x->w[4 * q + 2] = y.z, x->w[4 * q + 3] = y.w;
    }
    x->valid = ~0ull;
  } else {
    const int len = p >= n ? 0 : (int)min((uint64_t)kFaBytes, n - p);
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      x->w[k] = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (4 * k + j < len) x->w[k] |= (uint32_t)t[p + 4 * k + j] << (8 * j);
    }
    x->valid = below(len);
  }
  x->nl = x->gt = x->blank = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t other = 0;
#pragma unroll
    for (int k = 4 * q; k < 4 * q + 4; ++k) {
      const uint32_t v = x->w[k];
      other |= (fastq ? (v - 0x20202020u) & ~v : ~(~v & (v << 1))) & 0x80808080u;
    }
    if (!other) continue;
    uint32_t nl = 0, gt = 0, blank = 0, rest = 0;
#pragma unroll
    for (int k = 4 * q; k < 4 * q + 4; ++k) {
      const uint32_t v = x->w[k];
      nl |= bytes_eq(v, 0x0a0a0a0au) << (4 * (k & 3));
      if (fastq) blank |= bytes_eq(v, 0x0d0d0d0du) << (4 * (k & 3));
      else rest |= bit7_mask(~(~v & (v << 1))) << (4 * (k & 3));
    }
    if (!fastq && rest != nl) {
#pragma unroll
      for (int k = 4 * q; k < 4 * q + 4; ++k) {
        const uint32_t v = x->w[k];
        gt |= bytes_eq(v, 0x3e3e3e3eu) << (4 * (k & 3));
        blank |= (bytes_eq(v, 0x0d0d0d0du) | bytes_eq(v, 0x20202020u) | bytes_eq(v, 0x09090909u)) << (4 * (k & 3));
      }
    }
    x->nl |= (uint64_t)nl << (16 * q);
    x->gt |= (uint64_t)gt << (16 * q);
    x->blank |= (uint64_t)blank << (16 * q);
  }
  x->nl &= x->valid, x->gt &= x->valid, x->blank &= x->valid;
}

// the thread's transfer function
__device__ __forceinline__ uint32_t text_function(const Text& x) {
  if (!x.valid) return kIdentity;
  if (x.nl) {
    const uint64_t after = ~below(64 - __clzll((long long)x.nl)) & x.valid;  // the bytes of the last line
    const uint32_t e = !after ? FS_LS : (x.gt & after & (0ull - after)) ? FS_H : FS_S;
    return e | (e << 2) | (e << 4);
  }
  return ((x.gt & 1) ? FS_H : FS_S) | (FS_H << 2) | (FS_S << 4);
}

// The thread's bytes from entry state s: its headers' '>', its sequence bytes, its header lines' breaks.
// A header line's bytes are those that a carry from its '>' (or, entered inside one, from the first byte) runs
// through until the line break.
struct FaMasks {
  uint64_t heads, seq, ends;
};
__device__ __forceinline__ FaMasks fa_masks(const Text& x, uint32_t s) {
  const uint64_t in = s == FS_H ? 1 : 0;
  const uint64_t line = x.valid & ~x.nl;
  FaMasks m;
  m.heads = x.gt & ((x.nl << 1) | (s == FS_LS ? 1 : 0));
  const uint64_t header = line & ~(line + ((m.heads | in) & line));
  m.seq = line & ~header & ~x.blank;
  m.ends = x.nl & ((header << 1) | in);
  return m;
}

// The bytes of mask, in order, to the staging buffer from offset `at` on: compacted word by word (lut: the byte
// permutation of each mask of four), collected in 64 bits and stored as whole words; the first and the last word,
// which may be shared with other threads, byte by byte.  The buffer keeps a word free after every 64 bytes
// (padded()), so that threads 64 bytes apart store to different banks: without it 16 lanes share one.
__device__ __forceinline__ uint32_t padded(uint32_t a) { return a + ((a >> 6) << 2); }
constexpr uint32_t kStage = (kFaTile + 64) / 64 * 68;
__device__ __forceinline__ void make_lut(uint32_t* lut) {
  if (threadIdx.x < 16) {
    uint32_t sel = 0x4444u, k = 0;  // selector 4: a byte of the zero operand
    for (uint32_t b = 0; b < 4; ++b)
      if (threadIdx.x >> b & 1) sel = (sel & ~(15u << (4 * k))) | (b << (4 * k)), ++k;
    lut[threadIdx.x] = sel;
  }
}
__device__ __forceinline__ void stage_bytes(const Text& x, uint64_t mask, uint32_t at, uint8_t* staged,
                                            const uint32_t* lut) {
  const uint32_t lead = at & 3u, first = at & ~3u;
  uint32_t fill = lead, wp = first, head = 0;
  uint64_t acc = 0;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const uint32_t m = (uint32_t)(mask >> (4 * k)) & 15u;
    acc |= (uint64_t)__byte_perm(x.w[k], 0u, lut[m]) << (8 * fill);
    fill += __popc(m);
    if (fill >= 4) {
      if (wp == first) head = (uint32_t)acc;
      else *reinterpret_cast<uint32_t*>(staged + padded(wp)) = (uint32_t)acc;
      wp += 4, fill -= 4, acc >>= 32;
    }
  }
  if (wp != first)
    for (uint32_t b = lead; b < 4; ++b) staged[padded(first + b)] = (uint8_t)(head >> (8 * b));
  for (uint32_t b = wp == first ? lead : 0; b < fill; ++b) staged[padded(wp + b)] = (uint8_t)(acc >> (8 * b));
}

// out[base, base + count) from the staging buffer's [lead, lead + count), lead = base modulo 16 after a multiple
// of 16: whole aligned 16-byte units as uint4, the partial first and last units byte by byte (their other bytes
// belong to the next tiles)
__device__ __forceinline__ void copy_staged(uint8_t* __restrict__ out, uint64_t base, const uint8_t* staged, uint32_t lead,
                                            uint32_t count) {
  const uint32_t end = lead + count, full_lo = (lead + 15u) & ~15u, full_hi = end & ~15u;
  uint8_t* dst = out + base - lead;
  for (uint32_t u = full_lo + 16u * threadIdx.x; u < full_hi; u += 16u * kFaThreads) {
    const uint32_t* v = reinterpret_cast<const uint32_t*>(staged + padded(u));
    *reinterpret_cast<uint4*>(dst + u) = make_uint4(v[0], v[1], v[2], v[3]);
  }
  if (threadIdx.x < 32) {
    for (uint32_t i = lead + threadIdx.x; i < min(full_lo, end); i += 32) dst[i] = staged[padded(i)];
    for (uint32_t i = max(full_hi, full_lo) + threadIdx.x; i < end; i += 32) dst[i] = staged[padded(i)];
  }
}

// exclusive composition of the block's thread functions (thread order) and the block's total
__device__ uint32_t block_exclusive_function(uint32_t f, uint32_t* total) {
  __shared__ uint32_t warp_f[kFaThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = f;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t other = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc = compose(other, inc);
  }
  uint32_t exc = __shfl_up_sync(0xffffffffu, inc, 1);
  if (lane == 0) exc = kIdentity;
  if (lane == 31) warp_f[warp] = inc;
  __syncthreads();
  uint32_t before = kIdentity;
  for (int w = 0; w < warp; ++w) before = compose(before, warp_f[w]);
  if (total) {
    uint32_t all = kIdentity;
    for (int w = 0; w < kFaThreads / 32; ++w) all = compose(all, warp_f[w]);
    *total = all;
  }
  __syncthreads();
  return compose(before, exc);
}

// exclusive sums of two per-thread counts over the block, and their totals
__device__ void block_exclusive_sums(uint32_t a, uint32_t b, uint32_t* ea, uint32_t* eb, uint32_t* ta, uint32_t* tb) {
  __shared__ uint32_t wa[kFaThreads / 32], wb[kFaThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t ia = a, ib = b;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t xa = __shfl_up_sync(0xffffffffu, ia, o), xb = __shfl_up_sync(0xffffffffu, ib, o);
    if (lane >= o) ia += xa, ib += xb;
  }
  if (lane == 31) wa[warp] = ia, wb[warp] = ib;
  __syncthreads();
  uint32_t ba = 0, bb = 0, sa = 0, sb = 0;
  for (int w = 0; w < kFaThreads / 32; ++w) {
    if (w < warp) ba += wa[w], bb += wb[w];
    sa += wa[w], sb += wb[w];
  }
  __syncthreads();
  *ea = ba + ia - a;
  *eb = bb + ib - b;
  *ta = sa;
  *tb = sb;
}

// Pass 1: each tile's transfer function (x) and, for each entry state (LS, H, S: y, z, w), its sequence
// bytes (low 16 bits) and headers.  Only the bytes before a tile's first line break depend on the entry
// state, so few threads count more than once.  One read of the text, bound by the masks' integer work: 49 MB in
// 21 us (a walk byte by byte from each state took 70; a function pass and a counting pass before it 46).
__global__ void __launch_bounds__(kFaThreads) k_fa_tiles(const uint8_t* __restrict__ t, uint64_t n,
                                                         uint4* __restrict__ info) {
  Text x;
  load_text<false>(t, n, (uint64_t)blockIdx.x * kFaTile + threadIdx.x * kFaBytes, &x);
  uint32_t total;
  const uint32_t before = block_exclusive_function(text_function(x), &total);
  auto count = [&](uint32_t s) {
    const FaMasks m = fa_masks(x, s);
    return (uint32_t)__popcll(m.seq) | ((uint32_t)__popcll(m.heads) << 16);  // 16,384 and 8,192 at most over the tile
  };
  const uint32_t s_ls = apply(before, FS_LS), s_h = apply(before, FS_H), s_s = apply(before, FS_S);
  uint32_t c[3];
  c[0] = count(s_ls);
  c[1] = s_h == s_ls ? c[0] : count(s_h);
  c[2] = s_s == s_ls ? c[0] : s_s == s_h ? c[1] : count(s_s);
  __shared__ uint32_t sums[3][kFaThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const uint32_t sum = __reduce_add_sync(0xffffffffu, c[e]);
    if (lane == 0) sums[e][warp] = sum;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint4 out = make_uint4(total, 0u, 0u, 0u);
    for (int w = 0; w < kFaThreads / 32; ++w) out.y += sums[0][w], out.z += sums[1][w], out.w += sums[2][w];
    info[blockIdx.x] = out;
  }
}

// The line state and the totals after the tiles chained so far, in device memory.
struct FaState {
  uint64_t seq, hdr;
  uint32_t state;
};

// exclusive sums of two 64-bit counts over a block of kFaThreads, and their totals
__device__ void block_exclusive_sums64(uint64_t a, uint64_t b, uint64_t* ea, uint64_t* eb, uint64_t* ta, uint64_t* tb) {
  __shared__ uint64_t wa[kFaThreads / 32], wb[kFaThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint64_t ia = a, ib = b;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t xa = __shfl_up_sync(0xffffffffu, ia, o), xb = __shfl_up_sync(0xffffffffu, ib, o);
    if (lane >= o) ia += xa, ib += xb;
  }
  if (lane == 31) wa[warp] = ia, wb[warp] = ib;
  __syncthreads();
  uint64_t ba = 0, bb = 0, sa = 0, sb = 0;
  for (int w = 0; w < kFaThreads / 32; ++w) {
    if (w < warp) ba += wa[w], bb += wb[w];
    sa += wa[w], sb += wb[w];
  }
  __syncthreads();
  *ea = ba + ia - a;
  *eb = bb + ib - b;
  *ta = sa;
  *tb = sb;
}

// One block chains n_tiles tiles after those before (st): each tile's entry state and its first sequence
// byte's and header's number in the text.  A thread takes consecutive tiles: their composed function, the
// block's scan of those, the counts from the now known entry states, the scan of those, the results.
// host (page-locked, optional): the totals after the chunk.
__global__ void __launch_bounds__(kFaThreads) k_fa_chain(const uint4* __restrict__ info, uint64_t n_tiles,
                                                         FaState* __restrict__ st, uint8_t* __restrict__ tile_entry,
                                                         uint64_t* __restrict__ seq_base, uint64_t* __restrict__ hdr_base,
                                                         uint64_t* __restrict__ host) {
  const uint64_t per = (n_tiles + kFaThreads - 1) / kFaThreads;
  const uint64_t i0 = min(n_tiles, per * threadIdx.x), i1 = min(n_tiles, i0 + per);
  const FaState s0 = *st;
  uint32_t f = kIdentity;
#pragma unroll 8
  for (uint64_t i = i0; i < i1; ++i) f = compose(f, info[i].x);
  uint32_t all;
  const uint32_t entry = apply(block_exclusive_function(f, &all), s0.state);
  auto counts = [](const uint4& v, uint32_t s) { return s == FS_LS ? v.y : s == FS_H ? v.z : v.w; };
  uint64_t seq = 0, hdr = 0;
  uint32_t s = entry;
#pragma unroll 4
  for (uint64_t i = i0; i < i1; ++i) {
    const uint4 v = info[i];
    const uint32_t c = counts(v, s);
    seq += c & 0xFFFFu, hdr += c >> 16;
    s = apply(v.x, s);
  }
  uint64_t e_seq, e_hdr, t_seq, t_hdr;
  block_exclusive_sums64(seq, hdr, &e_seq, &e_hdr, &t_seq, &t_hdr);
  e_seq += s0.seq, e_hdr += s0.hdr;
  s = entry;
#pragma unroll 4
  for (uint64_t i = i0; i < i1; ++i) {
    const uint4 v = info[i];
    const uint32_t c = counts(v, s);
    tile_entry[i] = (uint8_t)s;
    seq_base[i] = e_seq, hdr_base[i] = e_hdr;
    e_seq += c & 0xFFFFu, e_hdr += c >> 16;
    s = apply(v.x, s);
  }
  if (threadIdx.x == 0) {
    *st = FaState{s0.seq + t_seq, s0.hdr + t_hdr, apply(all, s0.state)};
    if (host) host[0] = s0.seq + t_seq, host[1] = s0.hdr + t_hdr;
  }
}

// Pass 2: the bytes classified again from the tiles' entry states; sequence bytes to out[rank], and per
// header (record r < hdr_cap) hdr_pos[r] (first byte after '>'), seq_rank[r] (sequence bytes before it)
// and hdr_end[r] (its '\n').  pos_off: the text's bytes before t.  49 MB in 42 us (83 with bytes staged one at a
// time, 16 lanes to a bank); what is left is the compaction's instructions, 15 per four bytes.
__global__ void __launch_bounds__(kFaThreads) k_fa_emit(const uint8_t* __restrict__ t, uint64_t n,
                                                        const uint8_t* __restrict__ tile_entry,
                                                        const uint64_t* __restrict__ seq_base,
                                                        const uint64_t* __restrict__ hdr_base, uint8_t* __restrict__ out,
                                                        uint64_t* __restrict__ hdr_pos, uint64_t* __restrict__ hdr_end,
                                                        uint64_t* __restrict__ seq_rank, uint64_t pos_off,
                                                        uint64_t hdr_cap) {
  __shared__ __align__(16) uint8_t staged[kStage];  // the tile's sequence bytes, compacted
  __shared__ uint32_t lut[16];
  make_lut(lut);
  Text x;
  const uint64_t p = (uint64_t)blockIdx.x * kFaTile + threadIdx.x * kFaBytes;
  load_text<false>(t, n, p, &x);
  const uint32_t before = block_exclusive_function(text_function(x), nullptr);
  const FaMasks m = fa_masks(x, apply(before, tile_entry[blockIdx.x]));
  uint32_t e_seq, e_hdr, t_seq, t_hdr;
  block_exclusive_sums((uint32_t)__popcll(m.seq), (uint32_t)__popcll(m.heads), &e_seq, &e_hdr, &t_seq, &t_hdr);
  const uint64_t base = seq_base[blockIdx.x];
  const uint32_t lead = (uint32_t)(base & 15);                // staged[lead + i] goes to out[base + i]
  const uint64_t rec = hdr_base[blockIdx.x] + e_hdr;          // headers started before this thread's bytes
  for (uint64_t h = m.heads; h; h &= h - 1) {
    const int j = __ffsll((long long)h) - 1;
    const uint64_t r = rec + __popcll(m.heads & below(j));
    if (r < hdr_cap) hdr_pos[r] = pos_off + p + j + 1, seq_rank[r] = base + e_seq + __popcll(m.seq & below(j));
  }
  for (uint64_t h = m.ends; h; h &= h - 1) {
    const int j = __ffsll((long long)h) - 1;
    const uint64_t r = rec + __popcll(m.heads & below(j));    // a header line is open: r >= 1
    if (r <= hdr_cap) hdr_end[r - 1] = pos_off + p + j;
  }
  stage_bytes(x, m.seq, lead + e_seq, staged, lut);
  __syncthreads();
  copy_staged(out, base, staged, lead, t_seq);
}

// names of records [0, n_rec) into one buffer: name r is text[hdr_pos[r], hdr_pos[r] + len[r])
__global__ void k_fa_names(const uint8_t* __restrict__ t, const uint64_t* __restrict__ hdr_pos,
                           const uint64_t* __restrict__ name_off, uint32_t n_rec, uint8_t* __restrict__ names) {
  const uint32_t r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (r >= n_rec) return;
  const uint64_t len = name_off[r + 1] - name_off[r];
  for (uint64_t i = threadIdx.x & 31; i < len; i += 32) names[name_off[r] + i] = t[hdr_pos[r] + i];
}

// ------------------------------------------------------------------------------------------
// FASTQ (four lines per record: '@' header, bases, '+' line, qualities).  The line of a byte is the
// number of line breaks before it, so a tile needs only the line breaks before it (an exclusive
// sum) and no state machine; line 4r is record r's header, 4r + 1 its bases, 4r + 3 its qualities
// ('\r' dropped from all three).

// One walk over a thread's runs between line breaks.  line: the number of the line that its first byte lies
// in (any count that is right modulo 4 where only line & 3 matters); start: that byte starts the line.
// run(line, mask): the non-blank bytes of a line; head(line, j): the line's first byte, if it has one;
// brk(line, j): its line break.
template <class Run, class Head, class Brk>
__device__ __forceinline__ void fq_walk(const Text& x, uint64_t line, bool start, Run&& run, Head&& head, Brk&& brk) {
  uint64_t rest = x.nl, left = x.valid;  // left: the bytes from the line on
  for (;;) {
    const int stop = rest ? __ffsll((long long)rest) - 1 : 64;
    const uint64_t bytes = left & below(stop);
    if (bytes) {
      run(line, bytes & ~x.blank);
      if (start) head(line, __ffsll((long long)bytes) - 1);
    }
    if (!rest) break;
    brk(line, stop);
    rest &= rest - 1;
    left &= ~below(stop + 1);
    ++line;
    start = true;
  }
}

__device__ __forceinline__ bool fq_starts_line(const uint8_t* __restrict__ t, uint64_t n, uint64_t p) {
  return p == 0 || (p < n && t[p - 1] == '\n');
}

// What a tile holds, its lines numbered from the tile's first byte (a line's class is its number modulo 4, a
// 16-bit field each): non-blank bytes, lines that start with '@', with something else, and the line breaks.
// A tile's line of class (0 - phase) & 3 is a header, (1 - phase) & 3 bases, (3 - phase) & 3 qualities, where
// phase is the number of lines before the tile modulo 4.
struct FqTile {
  uint64_t bytes, at, other, breaks;
};

// Pass 1, which needs nothing of the tiles before: one read of the text gives every count (52 MB in 21 us; line
// breaks alone and then a counting pass from the known lines took 34 and a round of prefix sums between them).
__global__ void __launch_bounds__(kFaThreads) k_fq_tiles(const uint8_t* __restrict__ t, uint64_t n, uint64_t tile0,
                                                         FqTile* __restrict__ info) {
  const uint64_t tile = tile0 + blockIdx.x, p = tile * kFaTile + threadIdx.x * kFaBytes;
  Text x;
  load_text<true>(t, n, p, &x);
  uint32_t e_nl, e_x, t_nl, t_x;
  block_exclusive_sums((uint32_t)__popcll(x.nl), 0, &e_nl, &e_x, &t_nl, &t_x);
  uint64_t v[3] = {0, 0, 0};
  auto field = [](uint64_t line) { return (uint32_t)(line & 3) * 16u; };
  fq_walk(x, e_nl, fq_starts_line(t, n, p),
          [&](uint64_t line, uint64_t m) { v[0] += (uint64_t)__popcll(m) << field(line); },
          [&](uint64_t line, int j) {
            const bool at = t[p + j] == '@';
            v[1] += (at ? 1ull : 0ull) << field(line), v[2] += (at ? 0ull : 1ull) << field(line);
          }, [](uint64_t, int) {});
  __shared__ uint64_t sums[3][kFaThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    uint64_t sum = v[k];
#pragma unroll
    for (int o = 16; o; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
    if (lane == 0) sums[k][warp] = sum;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    FqTile out = {0, 0, 0, t_nl};
    for (int w = 0; w < kFaThreads / 32; ++w) out.bytes += sums[0][w], out.at += sums[1][w], out.other += sums[2][w];
    info[tile] = out;
  }
}

// The totals of the tiles chained so far, in device memory.
struct FqState {
  uint64_t lines, seq, qual, hdr, bad;
};

// One block chains n_tiles tiles after those before (st), as k_fa_chain does: the lines, bases and qualities
// before each; host: the totals after the chunk (page-locked).
__global__ void __launch_bounds__(kFaThreads) k_fq_chain(const FqTile* __restrict__ info, uint64_t n_tiles,
                                                         FqState* __restrict__ st, uint64_t* __restrict__ line_base,
                                                         uint64_t* __restrict__ seq_base, uint64_t* __restrict__ qual_base,
                                                         uint64_t* __restrict__ host) {
  const uint64_t per = (n_tiles + kFaThreads - 1) / kFaThreads;
  const uint64_t i0 = min(n_tiles, per * threadIdx.x), i1 = min(n_tiles, i0 + per);
  const FqState s0 = *st;
  uint64_t breaks = 0;
#pragma unroll 4
  for (uint64_t i = i0; i < i1; ++i) breaks += info[i].breaks;
  uint64_t e_lines, e_x, t_lines, t_x;
  block_exclusive_sums64(breaks, 0, &e_lines, &e_x, &t_lines, &t_x);
  auto field = [](uint64_t v, uint64_t cls) { return (uint32_t)(v >> (16 * (cls & 3))) & 0xFFFFu; };
  const uint64_t line0 = s0.lines + e_lines;
  uint64_t line = line0, seq = 0, qual = 0, hdr = 0, bad = 0;
#pragma unroll 4
  for (uint64_t i = i0; i < i1; ++i) {
    const FqTile v = info[i];
    seq += field(v.bytes, 1 - line), qual += field(v.bytes, 3 - line);
    hdr += field(v.at, 0 - line), bad += field(v.other, 0 - line);
    line += v.breaks;
  }
  uint64_t e_seq, e_qual, t_seq, t_qual, e_h, e_b, t_h, t_b;
  block_exclusive_sums64(seq, qual, &e_seq, &e_qual, &t_seq, &t_qual);
  block_exclusive_sums64(hdr, bad, &e_h, &e_b, &t_h, &t_b);
  line = line0, seq = s0.seq + e_seq, qual = s0.qual + e_qual;
#pragma unroll 4
  for (uint64_t i = i0; i < i1; ++i) {
    const FqTile v = info[i];
    line_base[i] = line, seq_base[i] = seq, qual_base[i] = qual;
    seq += field(v.bytes, 1 - line), qual += field(v.bytes, 3 - line);
    line += v.breaks;
  }
  if (threadIdx.x == 0) {
    const FqState x = {s0.lines + t_lines, s0.seq + t_seq, s0.qual + t_qual, s0.hdr + t_h, s0.bad + t_b};
    *st = x;
    host[0] = x.seq, host[1] = x.qual, host[2] = x.hdr, host[3] = x.bad;
  }
}

// Pass 2: the bases and qualities compacted (those of a tile that would pass byte_cap are left out: the text is
// refused) and per record r < rec_cap hdr_pos[r] (after '@'), hdr_end[r] (its line break), seq_rank[r] and
// qual_rank[r] (bases and qualities before the record).  Tiles tile0 .. tile0 + gridDim.x - 1 of the text.
// 52 MB in 62 us (119 with bytes staged one at a time).
__global__ void __launch_bounds__(kFaThreads) k_fq_emit(const uint8_t* __restrict__ t, uint64_t n, uint64_t tile0,
                                                        const uint64_t* __restrict__ line_base,
                                                        const uint64_t* __restrict__ seq_base,
                                                        const uint64_t* __restrict__ qual_base, uint8_t* __restrict__ seq_out,
                                                        uint8_t* __restrict__ qual_out, uint64_t byte_cap,
                                                        uint64_t* __restrict__ hdr_pos, uint64_t* __restrict__ hdr_end,
                                                        uint64_t* __restrict__ seq_rank, uint64_t* __restrict__ qual_rank,
                                                        uint64_t rec_cap) {
  __shared__ __align__(16) uint8_t staged[kStage];  // the tile's bases, then its qualities
  __shared__ uint32_t lut[16];
  make_lut(lut);
  const uint64_t tile = tile0 + blockIdx.x, p = tile * kFaTile + threadIdx.x * kFaBytes;
  Text x;
  load_text<true>(t, n, p, &x);
  uint32_t e_nl, e_x, t_nl, t_x;
  block_exclusive_sums((uint32_t)__popcll(x.nl), 0, &e_nl, &e_x, &t_nl, &t_x);
  const uint64_t line0 = line_base[tile] + e_nl;
  const bool start = fq_starts_line(t, n, p);
  uint64_t m_seq = 0, m_qual = 0;
  fq_walk(x, line0, start,
          [&](uint64_t line, uint64_t m) {
            if ((line & 3) == 1) m_seq |= m;
            if ((line & 3) == 3) m_qual |= m;
          },
          [](uint64_t, int) {}, [](uint64_t, int) {});
  uint32_t e_seq, e_qual, t_seq, t_qual;
  block_exclusive_sums((uint32_t)__popcll(m_seq), (uint32_t)__popcll(m_qual), &e_seq, &e_qual, &t_seq, &t_qual);
  const uint64_t sbase = seq_base[tile], qbase = qual_base[tile];
  const uint32_t slead = (uint32_t)(sbase & 15);
  const uint32_t qlead = ((slead + t_seq + 15u) & ~15u) + (uint32_t)(qbase & 15);
  fq_walk(x, line0, start, [](uint64_t, uint64_t) {},
          [&](uint64_t line, int j) {
            const uint64_t r = line >> 2;
            if ((line & 3) == 0 && r < rec_cap && t[p + j] == '@')  // more records are listed by a second pass
              hdr_pos[r] = p + j + 1, seq_rank[r] = sbase + e_seq + __popcll(m_seq & below(j)),
              qual_rank[r] = qbase + e_qual + __popcll(m_qual & below(j));
          },
          [&](uint64_t line, int j) {
            if ((line & 3) == 0 && (line >> 2) < rec_cap) hdr_end[line >> 2] = p + j;
          });
  if (m_seq) stage_bytes(x, m_seq, slead + e_seq, staged, lut);
  if (m_qual) stage_bytes(x, m_qual, qlead + e_qual, staged, lut);
  __syncthreads();
  if (sbase + t_seq <= byte_cap) copy_staged(seq_out, sbase, staged, slead, t_seq);
  if (qbase + t_qual <= byte_cap) copy_staged(qual_out, qbase, staged, qlead, t_qual);
}

// hdr_end[r] = the text's end before the emitting pass (a record whose header line ends the text)
__global__ void k_fill_u64(uint64_t* __restrict__ p, uint64_t n, uint64_t v) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    p[i] = v;
}

// every record listed has its header (its rank was written), fewer than 2^32 bases and as many qualities
// as bases; *bad = 1 if not (page-locked; nothing is said of more records than rec_cap)
__global__ void k_fq_check(const uint64_t* __restrict__ seq_rank, const uint64_t* __restrict__ qual_rank,
                           const FqState* __restrict__ st, uint64_t rec_cap, uint64_t* bad) {
  const uint64_t n = st->hdr;
  if (n > rec_cap) return;
  for (uint64_t r = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; r < n; r += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t s0 = seq_rank[r], s1 = r + 1 < n ? seq_rank[r + 1] : st->seq;
    const uint64_t q0 = qual_rank[r], q1 = r + 1 < n ? qual_rank[r + 1] : st->qual;
    if (s0 == ~0ull || s1 < s0 || q1 < q0 || s1 - s0 != q1 - q0 || s1 - s0 > 0xffffffffull) *bad = 1;
  }
}

// off[r] = rank[r] - rank[0] for r < n, off[n] = total - rank[0]
__global__ void k_rank_offsets(const uint64_t* __restrict__ rank, uint64_t n, uint64_t total, uint64_t* __restrict__ off) {
  const uint64_t r = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  if (r <= n) off[r] = (r < n ? rank[r] : total) - rank[0];
}

// Tiles of the next chunk of host text when rest are left: half of it (98 MB of FASTA took 614 us in four equal chunks,
// 699 in eight, 980 in sixteen, 530 this way; three quarters and 8 MiB at least 30 more; the copy alone 487).
constexpr uint64_t kLeastChunk = 12ull << 20, kLeastHookChunk = 32ull << 20;  // (a hook waits for each chunk)
uint64_t next_tiles(uint64_t rest, uint64_t least) { return next_chunk(rest, least / kFaTile, kChunkBases / kFaTile, 4); }

}  // namespace
}  // namespace ah

using namespace ah;

namespace ah {
namespace {

// Parse and pack: into a new batch (*batch_out) or, with `into`, into an existing batch whose record
// lengths must equal the text's.
// hook (into mode only): after each chunk, the compacted record bases so far (the first record's first
// base at d_concat, `avail` of them, last = false), and once all are in and the records checked
// against the batch (last = true); it then packs them instead of the final pack
ah_status fasta_pack(ah_ctx* ctx, const char* text, uint64_t n_bytes, const uint32_t* genome_ids, ah_batch* into,
                     ah_batch** batch_out, ah_fasta** names_out, const FastaChunkHook* hook = nullptr) {
  cudaSetDevice(ctx->device);
  cudaPointerAttributes pa;
  const bool known = cudaPointerGetAttributes(&pa, text) == cudaSuccess;
  cudaGetLastError();
  const bool on_device = known && (pa.type == cudaMemoryTypeDevice || pa.type == cudaMemoryTypeManaged);
  const bool page_locked = known && pa.type == cudaMemoryTypeHost;
  ah_status st = AH_OK;
  const uint8_t* t = (const uint8_t*)text;
  uint8_t* staged = nullptr;
  const uint64_t n_tiles = (n_bytes + kFaTile - 1) / kFaTile;
  // host text is parsed in chunks as it lands: a copy stream moves chunk c + 1 while the passes run on
  // chunk c, each chunk continuing from the state the one before left in device memory
  uint8_t *tile_entry = nullptr, *compact = nullptr;
  uint4* info = nullptr;
  FaState* state = nullptr;
  uint64_t *seq_base = nullptr, *hdr_base = nullptr, *hdr_pos = nullptr, *hdr_end = nullptr, *seq_rank = nullptr;
  uint64_t hdr_cap = 0;
  cudaStream_t cs = nullptr;
  std::vector<cudaEvent_t> landed;
  uint64_t total_seq = 0, total_hdr = 0;
  uint64_t rank0 = ~0ull;  // the first record's first base in the compacted text (hook only)
  auto cleanup = [&] {
    if (cs) {
      cudaStreamSynchronize(cs);
      cudaStreamDestroy(cs);
    }
    for (cudaEvent_t e : landed) cudaEventDestroy(e);
    for (void* p : {(void*)staged, (void*)info, (void*)tile_entry, (void*)compact, (void*)state, (void*)seq_base,
                    (void*)hdr_base, (void*)hdr_pos, (void*)hdr_end, (void*)seq_rank})
      dfree(ctx, p);
  };
  // record arrays with room for `need` records, contents kept, a missing header end read as the end
  // of the text
  auto grow = [&](uint64_t need) -> ah_status {
    if (need <= hdr_cap) return AH_OK;
    const uint64_t cap = std::max<uint64_t>(need, 2 * hdr_cap);
    uint64_t *np = nullptr, *ne = nullptr, *nr = nullptr;
    ah_status e = AH_OK;
    if ((e = dalloc(ctx, &np, cap)) || (e = dalloc(ctx, &ne, cap)) || (e = dalloc(ctx, &nr, cap + 1))) {
      dfree(ctx, np), dfree(ctx, ne), dfree(ctx, nr);
      return e;
    }
    k_fill_u64<<<(unsigned)std::min<uint64_t>((cap - hdr_cap + 255) / 256, 4096), 256, 0, ctx->stream>>>(
        ne + hdr_cap, cap - hdr_cap, n_bytes);
    launched(ctx);
    if (hdr_cap) {
      cudaMemcpyAsync(np, hdr_pos, hdr_cap * 8, cudaMemcpyDeviceToDevice, ctx->stream);
      cudaMemcpyAsync(ne, hdr_end, hdr_cap * 8, cudaMemcpyDeviceToDevice, ctx->stream);
      cudaMemcpyAsync(nr, seq_rank, hdr_cap * 8, cudaMemcpyDeviceToDevice, ctx->stream);
    }
    dfree(ctx, hdr_pos), dfree(ctx, hdr_end), dfree(ctx, seq_rank);
    hdr_pos = np, hdr_end = ne, seq_rank = nr, hdr_cap = cap;
    return cudaGetLastError() == cudaSuccess ? AH_OK : fail(ctx, AH_ECUDA, "ah_fasta_pack: record arrays");
  };
  auto emit = [&](uint64_t t0, uint64_t nt) {
    const uint64_t b0 = t0 * kFaTile, nb = std::min(n_bytes, b0 + nt * kFaTile) - b0;
    k_fa_emit<<<(unsigned)nt, kFaThreads, 0, ctx->stream>>>(t + b0, nb, tile_entry + t0, seq_base + t0, hdr_base + t0,
                                                            compact, hdr_pos, hdr_end, seq_rank, b0, hdr_cap);
    launched(ctx);
  };
  do {
    // room for a record per 128 bytes of text; a text of more has them listed by a second pass
    if ((st = dalloc(ctx, &info, n_tiles)) || (st = dalloc(ctx, &tile_entry, n_tiles)) ||
        (st = dalloc(ctx, &seq_base, n_tiles)) || (st = dalloc(ctx, &hdr_base, n_tiles)) ||
        (st = dalloc(ctx, &state, 1)) || (st = dalloc(ctx, &compact, n_bytes + 16)) || (st = grow(4096 + n_bytes / 128)))
      break;
    static_assert(FS_LS == 0, "a cleared state is the start of a line");
    cudaMemsetAsync(state, 0, sizeof(FaState), ctx->stream);
    if (!on_device) {
      if ((st = dalloc(ctx, &staged, n_bytes + 16))) break;
      cudaEvent_t ready;
      if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess ||
          cudaEventCreateWithFlags(&ready, cudaEventDisableTiming) != cudaSuccess) {
        st = fail(ctx, AH_ECUDA, "ah_fasta_pack: copy stream");
        break;
      }
      landed.push_back(ready);  // the buffer was allocated in the context stream's order
      cudaEventRecord(ready, ctx->stream);
      cudaStreamWaitEvent(cs, ready, 0);
      t = staged;
    }
    // Copies run ahead of the passes by as many chunks as the call has enqueued.  Nothing is waited for without a
    // hook.  With one each chunk's totals are: from page-locked memory all copies are enqueued before, so that the link
    // never waits for a pass or a hook; from pageable memory, where a copy returns once it is staged, the next
    // chunk's.  (7.6 GB of FASTA into a plan 36.6 ms; 42.3 with a chunk's copy enqueued after the hook of the one
    // before.)
    std::vector<uint64_t> chunk{0};  // first tiles, and the end
    while (chunk.back() < n_tiles)
      chunk.push_back(on_device ? n_tiles
                                : chunk.back() + next_tiles(n_tiles - chunk.back(), hook ? kLeastHookChunk : kLeastChunk));
    const size_t n_chunks = chunk.size() - 1;
    std::vector<cudaEvent_t> arrived;
    auto copy_upto = [&](size_t n) -> ah_status {
      for (size_t c = arrived.size(); !on_device && c < std::min(n, n_chunks); ++c) {
        const uint64_t b0 = chunk[c] * kFaTile, b1 = std::min(n_bytes, chunk[c + 1] * kFaTile);
        cudaEvent_t e = nullptr;
        if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess)
          return fail(ctx, AH_ECUDA, "ah_fasta_pack: copy");
        landed.push_back(e), arrived.push_back(e);
        if (cudaMemcpyAsync(staged + b0, text + b0, b1 - b0, cudaMemcpyHostToDevice, cs) != cudaSuccess ||
            cudaEventRecord(e, cs) != cudaSuccess)
          return fail(ctx, AH_ECUDA, "ah_fasta_pack: copy");
      }
      return AH_OK;
    };
    for (size_t c = 0; c < n_chunks; ++c) {
      const uint64_t t0 = chunk[c], nt = chunk[c + 1] - t0;
      const uint64_t b0 = t0 * kFaTile, nb = std::min(n_bytes, b0 + nt * kFaTile) - b0;
      if ((st = copy_upto(hook && page_locked ? n_chunks : c + 1))) break;
      if (!on_device && cudaStreamWaitEvent(ctx->stream, arrived[c], 0) != cudaSuccess) {
        st = fail(ctx, AH_ECUDA, "ah_fasta_pack: copy");
        break;
      }
      k_fa_tiles<<<(unsigned)nt, kFaThreads, 0, ctx->stream>>>(t + b0, nb, info + t0);
      k_fa_chain<<<1, kFaThreads, 0, ctx->stream>>>(info + t0, nt, state, tile_entry + t0, seq_base + t0, hdr_base + t0,
                                                    ctx->h_read);
      launched(ctx, 2);
      if (hook) {  // the chunk's totals before its bases are handed on
        if ((st = copy_upto(c + 2))) break;
        if (cudaStreamSynchronize(ctx->stream) != cudaSuccess) st = fail(ctx, AH_ECUDA, "ah_fasta_pack: parsing failed");
        if (st || (st = grow(ctx->h_read[1]))) break;
        total_seq = ctx->h_read[0], total_hdr = ctx->h_read[1];
      }
      emit(t0, nt);
      if (hook && total_hdr) {
        if (rank0 == ~0ull && (st = read_u64(ctx, seq_rank, &rank0))) break;
        if ((st = (*hook)(compact + rank0, total_seq - rank0, false))) break;
      }
    }
    if (st) break;
    if (!hook) {
      if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
        st = fail(ctx, AH_ECUDA, "ah_fasta_pack: parsing failed");
        break;
      }
      total_seq = ctx->h_read[0], total_hdr = ctx->h_read[1];
      if (total_hdr > hdr_cap) {
        if ((st = grow(total_hdr))) break;
        emit(0, n_tiles);
      }
    }
    if (total_hdr == 0) {
      st = fail(ctx, AH_EINVAL, "ah_fasta_pack: no record (no line starts with '>')");
      break;
    }
    if (total_hdr > 0xffffffffull) {
      st = fail(ctx, AH_EINVAL, "ah_fasta_pack: more than 2^32 - 1 records");
      break;
    }
    std::vector<uint64_t> h_pos(total_hdr), h_end(total_hdr), h_rank(total_hdr + 1);
    if (3 * total_hdr * 8 <= kBounceBytes) {  // through the page-locked buffer in one round trip
      if ((st = stage_buffer(ctx))) break;
      uint64_t* h = (uint64_t*)ctx->bounce[0];
      cudaMemcpyAsync(h, hdr_pos, total_hdr * 8, cudaMemcpyDeviceToHost, ctx->stream);
      cudaMemcpyAsync(h + total_hdr, hdr_end, total_hdr * 8, cudaMemcpyDeviceToHost, ctx->stream);
      cudaMemcpyAsync(h + 2 * total_hdr, seq_rank, total_hdr * 8, cudaMemcpyDeviceToHost, ctx->stream);
      if (cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
        st = fail(ctx, AH_ECUDA, "ah_fasta_pack: record table");
        break;
      }
      std::copy(h, h + total_hdr, h_pos.begin());
      std::copy(h + total_hdr, h + 2 * total_hdr, h_end.begin());
      std::copy(h + 2 * total_hdr, h + 3 * total_hdr, h_rank.begin());
    } else if ((st = copy_to_host(ctx, h_pos.data(), hdr_pos, total_hdr * 8)) ||
               (st = copy_to_host(ctx, h_end.data(), hdr_end, total_hdr * 8)) ||
               (st = copy_to_host(ctx, h_rank.data(), seq_rank, total_hdr * 8))) {
      break;
    }
    h_rank[total_hdr] = total_seq;
    const uint32_t n_rec = (uint32_t)total_hdr;
    // records: sequence offsets relative to the first record's first base
    std::vector<uint64_t> offs(n_rec + 1);
    for (uint32_t r = 0; r <= n_rec; ++r) offs[r] = h_rank[r] - h_rank[0];
    if (into) {
      bool same = into->n_records == n_rec;
      for (uint32_t r = 0; same && r < n_rec; ++r) same = into->h_rec_len[r] == offs[r + 1] - offs[r];
      if (!same) {
        st = fail(ctx, AH_EINVAL, "ah_fasta_pack_into: the text's records differ from the batch's in number or length");
        break;
      }
      st = hook ? (*hook)(compact + h_rank[0], offs[n_rec], true)
                : ah_batch_pack_range(ctx, into, 0, n_rec, compact + h_rank[0], offs.data());
    } else {
      // not waited for before the names are made
      st = pack_device_records(ctx, n_rec, compact + h_rank[0], offs.data(), genome_ids, batch_out);
    }
    if (st) break;
    if (names_out) {
      ah_fasta* f = new ah_fasta();
      f->names.resize(n_rec);
      std::vector<uint64_t> name_off(n_rec + 1, 0);
      for (uint32_t r = 0; r < n_rec; ++r) name_off[r + 1] = name_off[r] + (h_end[r] - h_pos[r]);
      std::vector<char> all(name_off[n_rec] + 1);
      if (on_device) {
        uint64_t* d_off = nullptr;
        uint8_t* d_names = nullptr;
        st = dalloc(ctx, &d_off, n_rec + 1);
        if (!st) st = dalloc(ctx, &d_names, name_off[n_rec] + 1);
        if (!st) {
          cudaMemcpyAsync(d_off, name_off.data(), (n_rec + 1) * 8, cudaMemcpyHostToDevice, ctx->stream);
          k_fa_names<<<(n_rec + 7) / 8, 256, 0, ctx->stream>>>(t, hdr_pos, d_off, n_rec, d_names);
          launched(ctx);
          cudaMemcpyAsync(all.data(), d_names, name_off[n_rec], cudaMemcpyDeviceToHost, ctx->stream);
          if (cudaStreamSynchronize(ctx->stream) != cudaSuccess) st = fail(ctx, AH_ECUDA, "ah_fasta_pack: names");
        }
        dfree(ctx, d_off);
        dfree(ctx, d_names);
      } else {
        for (uint32_t r = 0; r < n_rec; ++r) memcpy(all.data() + name_off[r], text + h_pos[r], h_end[r] - h_pos[r]);
      }
      for (uint32_t r = 0; r < n_rec && !st; ++r) {
        std::string nm(all.data() + name_off[r], name_off[r + 1] - name_off[r]);
        while (!nm.empty() && nm.back() == '\r') nm.pop_back();
        f->names[r] = std::move(nm);
      }
      if (st) {
        delete f;
        if (!into) {
          ah_batch_free(*batch_out);
          *batch_out = nullptr;
        }
        break;
      }
      *names_out = f;
    }
    if (!into && cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
      st = fail(ctx, AH_ECUDA, "ah_fasta_pack: packing failed");
      ah_batch_free(*batch_out);
      *batch_out = nullptr;
      if (names_out) {
        delete *names_out;
        *names_out = nullptr;
      }
    }
  } while (false);
  cleanup();
  return st;
}

}  // namespace

ah_status fasta_pack_hooked(ah_ctx* ctx, const char* text, uint64_t n_bytes, ah_batch* into, const FastaChunkHook& hook) {
  return fasta_pack(ctx, text, n_bytes, nullptr, into, nullptr, nullptr, &hook);
}
}  // namespace ah

extern "C" {

ah_status ah_fasta_pack(ah_ctx* ctx, const char* text, uint64_t n_bytes, const uint32_t* genome_ids,
                        ah_batch** batch_out, ah_fasta** names_out) {
  if (!ctx || !text || !batch_out || n_bytes == 0) return fail(ctx, AH_EINVAL, "ah_fasta_pack: bad arguments");
  *batch_out = nullptr;
  if (names_out) *names_out = nullptr;
  return fasta_pack(ctx, text, n_bytes, genome_ids, nullptr, batch_out, names_out);
}

ah_status ah_fasta_pack_into(ah_ctx* ctx, const char* text, uint64_t n_bytes, ah_batch* batch, ah_fasta** names_out) {
  if (!ctx || !text || !batch || n_bytes == 0 || batch->view)
    return fail(ctx, AH_EINVAL, "ah_fasta_pack_into: bad arguments");
  if (names_out) *names_out = nullptr;
  return fasta_pack(ctx, text, n_bytes, nullptr, batch, nullptr, names_out);
}

ah_status ah_fastq_pack(ah_ctx* ctx, const char* text, uint64_t n_bytes, const uint32_t* genome_ids,
                        ah_batch** batch_out, ah_quals** quals_out, ah_fasta** names_out) {
  if (!ctx || !text || !batch_out || !quals_out || n_bytes == 0) return fail(ctx, AH_EINVAL, "ah_fastq_pack: bad arguments");
  *batch_out = nullptr;
  *quals_out = nullptr;
  if (names_out) *names_out = nullptr;
  cudaSetDevice(ctx->device);
  cudaPointerAttributes pa;
  const bool on_device = cudaPointerGetAttributes(&pa, text) == cudaSuccess &&
                         (pa.type == cudaMemoryTypeDevice || pa.type == cudaMemoryTypeManaged);
  cudaGetLastError();
  ah_status st = AH_OK;
  const uint8_t* t = (const uint8_t*)text;
  uint8_t *staged = nullptr, *seq = nullptr, *qual = nullptr;
  const uint64_t n_tiles = (n_bytes + kFaTile - 1) / kFaTile;
  // host text is parsed in chunks as it lands, as FASTA is: a copy stream moves chunk c + 1 while the
  // passes run on chunk c, which continue from the totals the chunks before it left in device memory
  FqTile* info = nullptr;
  FqState* state = nullptr;
  uint64_t *line_base = nullptr, *seq_base = nullptr, *qual_base = nullptr;
  uint64_t *hdr_pos = nullptr, *hdr_end = nullptr, *seq_rank = nullptr, *qual_rank = nullptr;
  uint64_t rec_cap = 0;
  ah_quals* q = nullptr;
  cudaStream_t cs = nullptr;
  std::vector<cudaEvent_t> landed;
  auto cleanup = [&] {
    if (cs) {
      cudaStreamSynchronize(cs);
      cudaStreamDestroy(cs);
    }
    for (cudaEvent_t e : landed) cudaEventDestroy(e);
    for (void* x : {(void*)staged, (void*)seq, (void*)info, (void*)state, (void*)line_base, (void*)seq_base,
                    (void*)qual_base, (void*)hdr_pos, (void*)hdr_end, (void*)seq_rank, (void*)qual_rank})
      dfree(ctx, x);
  };
  auto fill = [&](uint64_t* p, uint64_t n, uint64_t v) {
    k_fill_u64<<<(unsigned)std::min<uint64_t>((n + 255) / 256, 4096), 256, 0, ctx->stream>>>(p, n, v);
    launched(ctx);
  };
  // record arrays with room for `need` records; a record's header end reads as the end of the text and
  // its rank as missing (~0) until its header is seen
  auto grow = [&](uint64_t need) -> ah_status {
    for (uint64_t** a : {&hdr_pos, &hdr_end, &seq_rank, &qual_rank}) {
      dfree(ctx, *a);
      *a = nullptr;
      const ah_status e = dalloc(ctx, a, need);
      if (e) return e;
    }
    fill(hdr_end, need, n_bytes);
    fill(seq_rank, need, ~0ull);
    rec_cap = need;
    return cudaGetLastError() == cudaSuccess ? AH_OK : fail(ctx, AH_ECUDA, "ah_fastq_pack: record arrays");
  };
  // Valid FASTQ has as many qualities as bases, at most half the text each: other text is refused, and
  // what goes past that isn't kept.
  const uint64_t byte_cap = n_bytes / 2;
  auto emit = [&](uint64_t t0, uint64_t nt) {
    k_fq_emit<<<(unsigned)nt, kFaThreads, 0, ctx->stream>>>(t, n_bytes, t0, line_base, seq_base, qual_base, seq, qual,
                                                            byte_cap, hdr_pos, hdr_end, seq_rank, qual_rank, rec_cap);
    launched(ctx);
  };
  auto check = [&] {
    ctx->h_read[4] = 0;  // nothing in flight writes it
    k_fq_check<<<(unsigned)std::min<uint64_t>((rec_cap + 255) / 256, 1216), 256, 0, ctx->stream>>>(
        seq_rank, qual_rank, state, rec_cap, ctx->h_read + 4);
    launched(ctx);
  };
  do {
    // Room for a record per 64 bytes of text, as far as 16 Mi records go (0.5 GB of arrays), and one per 256 bytes
    // beyond; a text of more has them listed by a second pass.  (One per 256 throughout: 1,000,000 reads of 75 bases from
    // page-locked text 3.58 ms, 3.31 without the second pass; 3,000,000 of 40 bases, on the device, 9.59 ms, 9.27
    // before there were two passes.)
    if ((st = dalloc(ctx, &info, n_tiles)) || (st = dalloc(ctx, &state, 1)) || (st = dalloc(ctx, &line_base, n_tiles)) ||
        (st = dalloc(ctx, &seq_base, n_tiles)) || (st = dalloc(ctx, &qual_base, n_tiles)) ||
        (st = dalloc(ctx, &seq, byte_cap + 16)) || (st = dalloc(ctx, &qual, byte_cap + 16)) ||
        (st = grow(4096 + std::max(n_bytes / 256, std::min<uint64_t>(n_bytes / 64, 16ull << 20)))))
      break;
    if (cudaMemsetAsync(state, 0, sizeof(FqState), ctx->stream) != cudaSuccess) {
      st = fail(ctx, AH_ECUDA, "ah_fastq_pack: memset failed");
      break;
    }
    if (!on_device) {
      if ((st = dalloc(ctx, &staged, n_bytes + 16))) break;
      cudaEvent_t ready;
      if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess ||
          cudaEventCreateWithFlags(&ready, cudaEventDisableTiming) != cudaSuccess) {
        st = fail(ctx, AH_ECUDA, "ah_fastq_pack: copy stream");
        break;
      }
      landed.push_back(ready);  // the buffer was allocated in the context stream's order
      cudaEventRecord(ready, ctx->stream);
      cudaStreamWaitEvent(cs, ready, 0);
      t = staged;
    }
    for (uint64_t t0 = 0, nt; t0 < n_tiles && !st; t0 += nt) {
      nt = on_device ? n_tiles : next_tiles(n_tiles - t0, kLeastChunk);
      if (!on_device) {
        const uint64_t b0 = t0 * kFaTile, nb = std::min(n_bytes, b0 + nt * kFaTile) - b0;
        cudaEvent_t e = nullptr;
        if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess ||
            cudaMemcpyAsync(staged + b0, text + b0, nb, cudaMemcpyHostToDevice, cs) != cudaSuccess ||
            cudaEventRecord(e, cs) != cudaSuccess || cudaStreamWaitEvent(ctx->stream, e, 0) != cudaSuccess)
          st = fail(ctx, AH_ECUDA, "ah_fastq_pack: copy");
        if (e) landed.push_back(e);
        if (st) break;
      }
      k_fq_tiles<<<(unsigned)nt, kFaThreads, 0, ctx->stream>>>(t, n_bytes, t0, info);
      k_fq_chain<<<1, kFaThreads, 0, ctx->stream>>>(info + t0, nt, state, line_base + t0, seq_base + t0, qual_base + t0,
                                                    ctx->h_read);
      launched(ctx, 2);
      emit(t0, nt);
    }
    if (st) break;
    check();
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
      st = fail(ctx, AH_ECUDA, "ah_fastq_pack: parsing failed");
      break;
    }
    const uint64_t total_seq = ctx->h_read[0], total_qual = ctx->h_read[1], n_rec = ctx->h_read[2];
    if (n_rec == 0 || ctx->h_read[3] || n_rec > 0xffffffffull) {
      st = fail(ctx, AH_EINVAL, "ah_fastq_pack: not FASTQ (every record is four lines, the first starting with '@')");
      break;
    }
    if (n_rec > rec_cap) {
      if ((st = grow(n_rec))) break;
      emit(0, n_tiles);
      check();
      if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(ctx->stream) != cudaSuccess) {
        st = fail(ctx, AH_ECUDA, "ah_fastq_pack: parsing failed");
        break;
      }
    }
    if (ctx->h_read[4]) {
      st = fail(ctx, AH_EINVAL, "ah_fastq_pack: a record lacks its header line or its qualities differ in length from its bases");
      break;
    }
    // the sequence ranks come back for the batch's host record table (the quality offsets equal the
    // sequence offsets), header positions only for the names.  Through the page-locked buffer they ride
    // on the packing's own round trip, and the tables are filled from there.
    const uint32_t R = (uint32_t)n_rec;
    std::vector<uint64_t> h_pos(names_out ? n_rec : 0), h_end(names_out ? n_rec : 0), ranks;
    if (names_out && ((st = copy_to_host(ctx, h_pos.data(), hdr_pos, n_rec * 8)) ||
                      (st = copy_to_host(ctx, h_end.data(), hdr_end, n_rec * 8))))
      break;
    uint64_t* h_srank;
    if ((n_rec + 1) * 8 <= kBounceBytes) {
      if ((st = stage_buffer(ctx))) break;
      h_srank = (uint64_t*)ctx->bounce[0];
      if (cudaMemcpyAsync(h_srank, seq_rank, n_rec * 8, cudaMemcpyDeviceToHost, ctx->stream) != cudaSuccess) {
        st = fail(ctx, AH_ECUDA, "ah_fastq_pack: record table");
        break;
      }
    } else {
      ranks.resize(n_rec + 1);
      h_srank = ranks.data();
      if ((st = copy_to_host(ctx, h_srank, seq_rank, n_rec * 8))) break;
    }
    h_srank[n_rec] = total_seq;
    if ((st = pack_batch_ranked(ctx, R, seq, seq_rank, h_srank, genome_ids, batch_out))) break;
    q = new ah_quals();
    q->ctx = ctx;
    q->n_records = R;
    if ((st = dalloc(ctx, &q->d_off, R + 1))) break;
    k_rank_offsets<<<(unsigned)((R + 256) / 256), 256, 0, ctx->stream>>>(qual_rank, R, total_qual, q->d_off);
    launched(ctx);
    // the qualities into a buffer of their own size: none come before the first record (line 0 is its
    // header), and their offsets are the bases' (the lengths match)
    if ((st = dalloc(ctx, &q->d_qual, total_qual + 16))) break;
    AH_CUDA(ctx, cudaMemcpyAsync(q->d_qual, qual, total_qual, cudaMemcpyDeviceToDevice, ctx->stream));
    q->h_off.resize(R + 1);
    for (uint32_t r = 0; r <= R; ++r) q->h_off[r] = h_srank[r] - h_srank[0];
    if (names_out) {
      ah_fasta* f = new ah_fasta();
      f->names.resize(R);
      std::vector<uint64_t> name_off(R + 1, 0);
      for (uint32_t r = 0; r < R; ++r) name_off[r + 1] = name_off[r] + (h_end[r] - h_pos[r]);
      std::vector<char> all(name_off[R] + 1);
      if (on_device) {
        uint64_t* d_off = nullptr;
        uint8_t* d_names = nullptr;
        st = dalloc(ctx, &d_off, R + 1);
        if (!st) st = dalloc(ctx, &d_names, name_off[R] + 1);
        if (!st) {
          cudaMemcpyAsync(d_off, name_off.data(), (R + 1) * 8, cudaMemcpyHostToDevice, ctx->stream);
          k_fa_names<<<(R + 7) / 8, 256, 0, ctx->stream>>>(t, hdr_pos, d_off, R, d_names);
          launched(ctx);
          cudaMemcpyAsync(all.data(), d_names, name_off[R], cudaMemcpyDeviceToHost, ctx->stream);
          if (cudaStreamSynchronize(ctx->stream) != cudaSuccess) st = fail(ctx, AH_ECUDA, "ah_fastq_pack: names");
        }
        dfree(ctx, d_off);
        dfree(ctx, d_names);
      } else {
        for (uint32_t r = 0; r < R; ++r) memcpy(all.data() + name_off[r], text + h_pos[r], h_end[r] - h_pos[r]);
      }
      for (uint32_t r = 0; r < R; ++r) {
        std::string nm(all.data() + name_off[r], name_off[r + 1] - name_off[r]);
        while (!nm.empty() && nm.back() == '\r') nm.pop_back();
        f->names[r] = std::move(nm);
      }
      if (st) {
        delete f;
        break;
      }
      *names_out = f;
    }
  } while (false);
  if (!st && cudaStreamSynchronize(ctx->stream) != cudaSuccess) st = fail(ctx, AH_ECUDA, "ah_fastq_pack: copies failed");
  if (qual) dfree(ctx, qual);
  cleanup();
  if (st) {
    if (*batch_out) ah_batch_free(*batch_out);
    *batch_out = nullptr;
    ah_quals_free(q);
    return st;
  }
  *quals_out = q;
  return AH_OK;
}

uint32_t ah_quals_count(const ah_quals* q) { return q ? q->n_records : 0; }

ah_status ah_quals_copy(const ah_quals* q, char* out, uint64_t cap, uint64_t* offsets_out) {
  if (!q || !offsets_out) return AH_EINVAL;
  memcpy(offsets_out, q->h_off.data(), q->h_off.size() * sizeof(uint64_t));
  if (!out) return AH_OK;
  if (cap < q->h_off.back()) return fail(q->ctx, AH_EOVERFLOW, "ah_quals_copy: need %llu bytes",
                                         (unsigned long long)q->h_off.back());
  return copy_to_host(q->ctx, out, q->d_qual, q->h_off.back());
}

void ah_quals_free(ah_quals* q) {
  if (!q) return;
  if (q->ctx) {
    dfree(q->ctx, q->d_qual);
    dfree(q->ctx, q->d_off);
  }
  delete q;
}

uint32_t ah_fasta_count(const ah_fasta* f) { return f ? (uint32_t)f->names.size() : 0; }

const char* ah_fasta_name(const ah_fasta* f, uint32_t i) {
  return f && i < f->names.size() ? f->names[i].c_str() : nullptr;
}

ah_status ah_fasta_names_copy(const ah_fasta* f, char* out, uint64_t cap, uint64_t* offsets_out) {
  if (!f || !offsets_out) return AH_EINVAL;
  uint64_t total = 0;
  offsets_out[0] = 0;
  for (size_t i = 0; i < f->names.size(); ++i) offsets_out[i + 1] = total += f->names[i].size();
  if (!out) return AH_OK;
  if (cap < total) return AH_EOVERFLOW;
  for (size_t i = 0; i < f->names.size(); ++i) memcpy(out + offsets_out[i], f->names[i].data(), f->names[i].size());
  return AH_OK;
}

void ah_fasta_free(ah_fasta* f) { delete f; }

}  // extern "C"
