// Extraction stage (Supplementary, "Primer trimming and barcode extraction", "Headers and
// outputs"; "Amplicon calling and orientation": RF amplicons are reverse-complemented).
//
// Per amplicon five fields go into one byte arena: amplicon (or trimmed interior), forward barcode,
// reverse barcode, site i and site j in primer orientation.  A length pass and an exclusive scan
// place every amplicon; then blocks decode the fields of consecutive amplicons from the 2-bit planes,
// an aligned 16-byte unit of the arena per thread.
#include "ah_amps.cuh"
#include "ah_internal.h"

namespace ah {
namespace {

struct Fields {
  int64_t a[5], b[5];  // top-strand ranges [a, b) per field, clipped
  bool rc[5];          // write the range reverse-complemented
};

__device__ __forceinline__ int64_t clip(int64_t x, int64_t len) { return x < 0 ? 0 : (x > len ? len : x); }

__device__ Fields fields_of(const ah_amplicon& m, const ah_hit& hi, const ah_hit& hj, const uint8_t* plen,
                            int64_t len, int trim, int64_t fb, int64_t rb) {
  Fields f;
  const int64_t s_i = hi.pos, e_i = hi.pos + plen[hi.pattern], s_j = hj.pos, e_j = hj.pos + plen[hj.pattern];
  const bool rc = m.orient == 1;
  if (trim) {
    f.a[0] = e_i;
    f.b[0] = s_j < e_i ? e_i : s_j;
  } else {
    f.a[0] = s_i;
    f.b[0] = e_j;
  }
  f.rc[0] = rc;
  if (!rc) {
    f.a[1] = clip(s_i - fb, len), f.b[1] = clip(s_i, len);
    f.a[2] = clip(e_j, len), f.b[2] = clip(e_j + rb, len);
  } else {
    f.a[1] = clip(e_j, len), f.b[1] = clip(e_j + fb, len);
    f.a[2] = clip(s_i - rb, len), f.b[2] = clip(s_i, len);
  }
  f.rc[1] = f.rc[2] = rc;
  f.a[3] = s_i, f.b[3] = e_i, f.rc[3] = ((hi.pattern >> 1) & 1u) != 0;
  f.a[4] = s_j, f.b[4] = e_j, f.rc[4] = ((hj.pattern >> 1) & 1u) != 0;
  return f;
}

__global__ void k_extract_len(const ah_amplicon* __restrict__ amps, uint64_t n, const ah_hit* __restrict__ hits,
                              const uint32_t* __restrict__ rec_len, const uint8_t* __restrict__ plen, int trim,
                              int64_t fb, int64_t rb, uint64_t* __restrict__ total,
                              const uint64_t* __restrict__ d_n = nullptr) {
  const uint64_t m = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= n) return;
  if (d_n && m >= *d_n) {
    total[m] = 0;
    return;
  }
  const ah_amplicon A = amps[m];
  const Fields f = fields_of(A, hits[A.hit_i], hits[A.hit_j], plen, rec_len[A.record], trim, fb, rb);
  uint64_t t = 0;
  for (int q = 0; q < 5; ++q) t += (uint64_t)(f.b[q] - f.a[q]);
  total[m] = t;
}

// bit k of the low byte to bit 4k
__device__ __forceinline__ uint32_t to_nibbles(uint32_t x) {
  x = (x | (x << 12)) & 0x000F000Fu;
  x = (x | (x << 6)) & 0x03030303u;
  return (x | (x << 3)) & 0x11111111u;
}

// A field as the units see it.  Bases are counted from the batch's first group (planes): output byte o of the
// amplicons' bytes is base o + x of a forward field, base x - o of a reverse one (x taken 15 back, so that it is the
// lowest of the unit's sixteen).
struct FieldSpan {
  int64_t from;              // its first byte, from the amplicons' first 16-byte boundary
  int64_t x;
  uint64_t group;            // its first base's group
  uint32_t more, rc;         // groups after that one; reverse
};

// Sixteen output bytes in the bit domain: each byte's two code bits and its invalid bit.
struct UnitBits {
  uint32_t p, q, v;
};

// Bytes u16 .. u16 + 15 as far as they lie in the field, which ends at `to` (at least one does): the sixteen bases
// are a shift of two neighbouring groups, reversed and complemented for a reverse field.
__device__ __forceinline__ void add_field(const uint2* __restrict__ planes, const uint32_t* __restrict__ invalid,
                                          const FieldSpan& f, int64_t to, int64_t u16, UnitBits* out) {
  const uint64_t x0 = (uint64_t)(f.rc ? f.x - u16 : f.x + u16);
  const uint32_t sh = (uint32_t)x0 & 31u;
  const int g = (int)((uint32_t)(x0 >> 5) - (uint32_t)f.group);  // from the field's first: -1 to more + 1
  const uint64_t gA = f.group + (uint32_t)min((int)f.more, max(0, g));  // groups without a base of the field aren't read
  const uint2 A = planes[gA];
  const uint32_t iA = invalid[gA];
  uint2 B = A;
  uint32_t iB = iA;
  if (sh > 16) {
    const uint64_t gB = f.group + (uint32_t)min((int)f.more, max(0, g + 1));
    B = planes[gB], iB = invalid[gB];
  }
  uint32_t p = __funnelshift_r(A.x, B.x, sh), q = __funnelshift_r(A.y, B.y, sh), v = __funnelshift_r(iA, iB, sh);
  if (f.rc) p = __brev(p) >> 16, q = ~__brev(q) >> 16, v = __brev(v) >> 16;
  const int64_t before = f.from - u16, left = to - u16;  // before < 16, left > 0
  const uint32_t lo = before > 0 ? (uint32_t)before : 0u, hi = left < 16 ? (uint32_t)left : 16u;
  const uint32_t m = ((1u << hi) - 1u) & ~((1u << lo) - 1u);
  out->p |= p & m, out->q |= q & m, out->v |= v & m;
}

// the bits' letters: a byte permute selects four at a time
__device__ __forceinline__ uint4 unit_letters(const UnitBits& x) {
  const uint32_t letters = 'A' | ('C' << 8) | ('T' << 16) | ('G' << 24), none = 0x4E4E4E4Eu;  // 'N'
  uint32_t s0 = to_nibbles(x.p & 0xFFu) | (to_nibbles(x.q & 0xFFu) << 1);
  uint32_t s1 = to_nibbles(x.p >> 8) | (to_nibbles(x.q >> 8) << 1);
  if (x.v) s0 |= to_nibbles(x.v & 0xFFu) << 2, s1 |= to_nibbles(x.v >> 8) << 2;
  return make_uint4(__byte_perm(letters, none, s0), __byte_perm(letters, none, s0 >> 16),
                    __byte_perm(letters, none, s1), __byte_perm(letters, none, s1 >> 16));
}

// A block takes consecutive amplicons, whose fields lie end to end in the arena, in batches of up to kExAmps: a
// thread per amplicon works out its fields, then every thread builds whole aligned 16-byte units of the batch's
// bytes, from each field that a unit touches (found by halving), and stores them at once, neighbours to neighbouring
// addresses whatever the fields' lengths.  The batch's first and last unit, which other blocks may share, are stored
// byte by byte.  An amplicon that would pass the arena (they are the last ones) is left out.
// Bound by integer work: 171,776 reads' amplicons and barcodes in 72 us; a warp per amplicon and a byte per
// lane and step took 147, sixteen lanes per amplicon and a unit per lane 107 (most of it spent on the fields, once
// per lane).
constexpr int kExThreads = 128, kExAmps = 32, kExMinAmps = 4;
constexpr uint64_t kExBlocksPerSm = 16;

__global__ void __launch_bounds__(kExThreads) k_extract_write(
    const ah_amplicon* __restrict__ amps, uint64_t n, const ah_hit* __restrict__ hits, const uint2* __restrict__ planes,
    const uint32_t* __restrict__ invalid, const uint64_t* __restrict__ rec_group, const uint32_t* __restrict__ rec_len,
    const uint8_t* __restrict__ plen, int trim, int64_t fb, int64_t rb, const uint64_t* __restrict__ base,
    char* __restrict__ arena, uint64_t* __restrict__ field_off, const uint64_t* __restrict__ d_n = nullptr,
    uint64_t arena_cap = ~0ull, uint32_t* __restrict__ overflow = nullptr) {
  __shared__ FieldSpan spans[5 * kExAmps];
  __shared__ int64_t ends[5 * kExAmps];
  if (d_n) {
    const uint64_t live = min(*d_n, n);
    if (blockIdx.x == 0 && threadIdx.x == 0 && live == 0) field_off[0] = 0;
    n = live;
  }
  const uint64_t share = max((uint64_t)kExMinAmps, (n + gridDim.x - 1) / gridDim.x);
  const uint64_t batches = (share + kExAmps - 1) / kExAmps, batch = (share + batches - 1) / batches;
  const uint64_t stop = min(n, (blockIdx.x + 1) * share);
  for (uint64_t m0 = blockIdx.x * share; m0 < stop; m0 += batch) {
    const int count = (int)min(batch, stop - m0);
    const uint64_t w0 = base[m0];
    const int64_t lead = (int64_t)((uintptr_t)(arena + w0) & 15);
    if (threadIdx.x < count) {
      const uint64_t m = m0 + threadIdx.x;
      const ah_amplicon A = amps[m];
      const uint64_t g0 = rec_group[A.record], w = base[m], w_end = base[m + 1];
      const bool fits = w_end <= arena_cap;
      const Fields f = fields_of(A, hits[A.hit_i], hits[A.hit_j], plen, rec_len[A.record], trim, fb, rb);
      uint64_t at = w;
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const int64_t len = f.b[q] - f.a[q], from = (int64_t)(at - w0) + lead;
        if (fits) field_off[5 * m + q] = at;
        at += (uint64_t)len;
        FieldSpan& sp = spans[5 * threadIdx.x + q];
        const int64_t x = 32 * (int64_t)g0 + (f.rc[q] ? f.b[q] - 16 + from : f.a[q] - from);
        sp = FieldSpan{from, x, g0 + (uint64_t)(f.a[q] >> 5), len ? (uint32_t)(((f.b[q] - 1) >> 5) - (f.a[q] >> 5)) : 0u,
                       f.rc[q] ? 1u : 0u};
        ends[5 * threadIdx.x + q] = from + len;
      }
      if (m == n - 1) field_off[5 * n] = w_end;
      if (!fits && overflow) atomicOr(overflow, 8u);
    }
    // the amplicons that fit, and their bytes
    const int live = __syncthreads_count(threadIdx.x < count && base[m0 + threadIdx.x + 1] <= arena_cap);
    const int64_t total = live ? ends[5 * live - 1] : 0;
    char* const dst = arena + w0 - lead;
    for (int64_t u16 = 16 * (int64_t)threadIdx.x; u16 < total; u16 += 16 * kExThreads) {
      int lo = 0;  // the amplicon that u16 lies in: the first that ends past it
#pragma unroll
      for (int step = kExAmps / 2; step; step >>= 1)
        if (lo + step <= live && ends[5 * (lo + step) - 1] <= u16) lo += step;
      lo *= 5;
      while (ends[lo] <= u16) ++lo;  // and its field
      UnitBits bits = {0, 0, 0};
      for (; lo < 5 * live && spans[lo].from < u16 + 16; ++lo)
        if (ends[lo] > spans[lo].from) add_field(planes, invalid, spans[lo], ends[lo], u16, &bits);
      const uint4 v = unit_letters(bits);
      if (u16 >= lead && u16 + 16 <= total) {
        *reinterpret_cast<uint4*>(dst + u16) = v;
      } else {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 16; ++k)
          if (u16 + k >= lead && u16 + k < total) dst[u16 + k] = (char)(w[k >> 2] >> (8 * (k & 3)));
      }
    }
    __syncthreads();
  }
}

unsigned extract_blocks(uint64_t n, int sm_count) {
  const uint64_t most = kExBlocksPerSm * (uint64_t)std::max(1, sm_count);
  return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(most, (n + kExMinAmps - 1) / kExMinAmps));
}

// What follows the Tm stage in one block for up to kOneBlockItems amplicons: threshold, compaction (with the filter) and,
// with ebase, the bytes of each kept amplicon and their offsets.  4 kept of 26 amplicons took 36 us in nine kernels, 7.4
// here.
constexpr int kOneThreads = 1024;
__global__ void __launch_bounds__(kOneThreads) k_finish_one(
    ah_amplicon* __restrict__ amps, uint64_t cap, const uint64_t* __restrict__ d_n, const double* __restrict__ hit_tm,
    int filter, double min_tm, ah_amplicon* __restrict__ kept, uint64_t* __restrict__ n_kept,
    const ah_hit* __restrict__ hits, const uint32_t* __restrict__ rec_len, const uint8_t* __restrict__ plen, int trim,
    int64_t fb, int64_t rb, uint64_t* __restrict__ ebase) {
  __shared__ uint64_t bytes_of[kOneThreads / 32];
  __shared__ uint32_t kept_of[kOneThreads / 32];
  const uint64_t n = min(*d_n, cap);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint64_t n_out = 0, n_bytes = 0;
  for (uint64_t base = 0; base < n; base += kOneThreads) {
    const uint64_t i = base + threadIdx.x;
    ah_amplicon m{};
    bool keep = false;
    uint64_t len = 0;
    if (i < n) {
      m = amps[i];
      keep = decide_amplicon(&m, hit_tm[m.hit_i], hit_tm[m.hit_j], min_tm) || !filter;
      amps[i] = m;
      if (keep && ebase) {
        const Fields f = fields_of(m, hits[m.hit_i], hits[m.hit_j], plen, rec_len[m.record], trim, fb, rb);
        for (int q = 0; q < 5; ++q) len += (uint64_t)(f.b[q] - f.a[q]);
      }
    }
    const uint32_t votes = __ballot_sync(0xffffffffu, keep);
    uint64_t inc = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) bytes_of[warp] = inc, kept_of[warp] = __popc(votes);
    __syncthreads();
    uint64_t at = n_bytes + inc - len, k = n_out + __popc(votes & ((1u << lane) - 1u));
    for (int w = 0; w < kOneThreads / 32; ++w) {
      if (w < warp) at += bytes_of[w], k += kept_of[w];
      n_bytes += bytes_of[w], n_out += kept_of[w];
    }
    if (keep) {
      if (filter) kept[k] = m;
      if (ebase) ebase[k] = at;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (filter) *n_kept = n_out;
    if (ebase) ebase[n_out] = ebase[cap] = n_bytes;
  }
}

// qualities of field 0 (the amplicon or its trimmed interior) at the field's arena offset, reversed
// for RF like the bases (qualities are not complemented); one warp per amplicon
__global__ void k_extract_qual(const ah_amplicon* __restrict__ amps, uint64_t n, const ah_hit* __restrict__ hits,
                               const uint32_t* __restrict__ rec_len, const uint8_t* __restrict__ plen, int trim,
                               const uint8_t* __restrict__ qual, const uint64_t* __restrict__ qoff,
                               const uint64_t* __restrict__ field_off, char* __restrict__ qarena) {
  const int lane = threadIdx.x & 31;
  const uint64_t m = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (m >= n) return;
  const ah_amplicon A = amps[m];
  const Fields f = fields_of(A, hits[A.hit_i], hits[A.hit_j], plen, rec_len[A.record], trim, 0, 0);
  const uint8_t* q = qual + qoff[A.record];
  const uint64_t w = field_off[5 * m];
  const int64_t len = f.b[0] - f.a[0];
  for (int64_t i = lane; i < len; i += 32) qarena[w + i] = (char)(f.rc[0] ? q[f.b[0] - 1 - i] : q[f.a[0] + i]);
}

}  // namespace

void launch_finish_one(cudaStream_t s, ah_amplicon* amps, uint64_t cap, const uint64_t* d_n, const double* hit_tm,
                       int filter, double min_tm, ah_amplicon* kept, uint64_t* n_kept, const ah_hit* hits,
                       const uint32_t* rec_len, const uint8_t* plen, int trim, uint32_t fb, uint32_t rb, uint64_t* ebase) {
  k_finish_one<<<1, kOneThreads, 0, s>>>(amps, cap, d_n, hit_tm, filter, min_tm, kept, n_kept, hits, rec_len, plen, trim,
                                         (int64_t)fb, (int64_t)rb, ebase);
}

void launch_extract(cudaStream_t s, bool write, const ah_amplicon* amps, uint64_t cap, const uint64_t* d_n,
                    const ah_hit* hits, const uint2* planes, const uint32_t* invalid, const uint64_t* rec_group,
                    const uint32_t* rec_len, const uint8_t* plen, int trim, uint32_t fb, uint32_t rb, uint64_t* len_or_base,
                    char* arena, uint64_t* field_off, uint64_t arena_cap, uint32_t* overflow, int sm_count) {
  if (!write)
    k_extract_len<<<(unsigned)std::max<uint64_t>(1, (cap + 255) / 256), 256, 0, s>>>(amps, cap, hits, rec_len, plen, trim,
                                                                                    (int64_t)fb, (int64_t)rb,
                                                                                    len_or_base, d_n);
  else
    k_extract_write<<<extract_blocks(cap, sm_count), kExThreads, 0, s>>>(
        amps, cap, hits, planes, invalid, rec_group, rec_len, plen, trim, (int64_t)fb, (int64_t)rb, len_or_base, arena,
        field_off, d_n, arena_cap, overflow);
}

ah_status extract(ah_ctx* ctx, const ah_batch* b, const ah_primers* p, const ah_hits* h, ah_amplicons* a, int trim,
                  uint32_t fb, uint32_t rb) {
  ah_status st;
  dfree(ctx, a->d_arena);
  dfree(ctx, a->d_field_off);
  a->d_arena = nullptr;
  a->d_field_off = nullptr;
  a->arena_bytes = 0;
  const uint64_t n = a->n;
  uint64_t *tot = nullptr, *base = nullptr;
  if ((st = dalloc(ctx, &tot, n)) || (st = dalloc(ctx, &base, n + 1))) return st;
  if (n)
    k_extract_len<<<(unsigned)((n + 255) / 256), 256, 0, ctx->stream>>>(a->d, n, h->d, b->rec_len, p->d_plen, trim,
                                                                       (int64_t)fb, (int64_t)rb, tot);
  if (n) launched(ctx);
  if ((st = exclusive_scan_u64(ctx, tot, base, n, ctx->h_read))) return st;
  AH_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  const uint64_t bytes = ctx->h_read[0];
  if ((st = dalloc(ctx, &a->d_arena, bytes)) || (st = dalloc(ctx, &a->d_field_off, 5 * n + 1))) return st;
  if (n) {
    k_extract_write<<<extract_blocks(n, ctx->sm_count), kExThreads, 0, ctx->stream>>>(a->d, n, h->d, b->planes, b->invalid, b->rec_group,
                                                                     b->rec_len, p->d_plen, trim, (int64_t)fb,
                                                                     (int64_t)rb, base, a->d_arena, a->d_field_off);
    launched(ctx);
  } else {
    AH_CUDA(ctx, cudaMemsetAsync(a->d_field_off, 0, sizeof(uint64_t), ctx->stream));
  }
  AH_CUDA(ctx, cudaGetLastError());
  a->arena_bytes = bytes;
  a->trim = trim;
  dfree(ctx, a->d_qarena);
  a->d_qarena = nullptr;
  dfree(ctx, tot);
  dfree(ctx, base);
  return AH_OK;
}

}  // namespace ah

using namespace ah;

extern "C" {

ah_status ah_extract_qualities(ah_ctx* ctx, const ah_quals* q, const ah_batch* b, const ah_primers* p,
                               const ah_hits* h, ah_amplicons* a) {
  if (!ctx || !q || !b || !p || !h || !a) return fail(ctx, AH_EINVAL, "ah_extract_qualities: NULL argument");
  if (!a->d_field_off) return fail(ctx, AH_EINVAL, "ah_extract_qualities: run ah_extract_barcodes first");
  bool same = q->n_records == b->n_records;
  for (uint32_t r = 0; same && r < b->n_records; ++r) same = q->h_off[r + 1] - q->h_off[r] == b->h_rec_len[r];
  if (!same) return fail(ctx, AH_EINVAL, "ah_extract_qualities: the qualities do not belong to this batch");
  cudaSetDevice(ctx->device);
  dfree(ctx, a->d_qarena);
  a->d_qarena = nullptr;
  ah_status st = dalloc(ctx, &a->d_qarena, a->arena_bytes + 1);
  if (st) return st;
  if (a->n) {
    k_extract_qual<<<(unsigned)((a->n + 7) / 8), 256, 0, ctx->stream>>>(a->d, a->n, h->d, b->rec_len, p->d_plen, a->trim,
                                                                        q->d_qual, q->d_off, a->d_field_off, a->d_qarena);
    launched(ctx);
  }
  AH_CUDA(ctx, cudaGetLastError());
  return AH_OK;
}

ah_status ah_amplicons_qual_copy(const ah_amplicons* a, char* out, uint64_t cap) {
  if (!a) return AH_EINVAL;
  if (!a->d_qarena) return fail(a->ctx, AH_EINVAL, "ah_amplicons_qual_copy: no qualities extracted");
  if (cap < a->arena_bytes) return fail(a->ctx, AH_EOVERFLOW, "ah_amplicons_qual_copy: need %llu bytes",
                                        (unsigned long long)a->arena_bytes);
  return copy_to_host(a->ctx, out, a->d_qarena, a->arena_bytes);
}

}  // extern "C"
