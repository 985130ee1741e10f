// Decompression kernels of cszp (sm_103a).
//
//   dec_setup_kernel       codec / block-size validation and payload offsets (scan),
//                          decode tables + 14-bit lookup table per book, record
//                          validation and each block's first record
//   stream_decode_kernel   one warp per interleaved 32-lane stream (Huffman code
//                          streams, RLE+Huffman value and length streams)
//   reconstruct_kernel<ND> one CTA per listed block (runs, or cut by the field's edge):
//                          runs to codes, fuse outliers (q' = q - r, or delta), N-D
//                          partial sums per chunk (Alg. 1, Sec. IV-B2), scale by 2eb,
//                          verbatim patches
//   dec_status_kernel      the status word of an asynchronous decompression
// and their batch forms (per-field tables in device memory, headers read and checked
// on the device by dec_header_batch_kernel).
#include "common.cuh"
#include "host.h"
#include "kernels.h"

namespace cszp {

__device__ __forceinline__ void flag(DevState* st, uint32_t bits) { atomicOr(&st->status, bits); }

// A field whose set-up found it corrupt, or whose set-up gave up a wait, has no payload
// offsets, block lists or run codes that may be used as such: the launches that follow leave
// its output alone.
__device__ __forceinline__ bool undecodable(uint32_t status) { return (status & (ERR_CORRUPT | ERR_TIMEOUT)) != 0; }

// =================================================================================
// archive validation and offsets
// =================================================================================
// Single-field set-up, one CTA per 1024 codec blocks (chunks taken by ticket and
// chained by decoupled look-back, so no CTA scans the whole block list): codec and
// block-size validation, payload offsets, the lists of run blocks and of the blocks
// the reconstruction kernel takes, per-codec counts.  The chunk counted last checks
// the totals against the header.
__device__ void dec_prep_chunk_body(const DecodeArgs& a, uint32_t nchunks) {
  if (a.dead) return;  // (a batch field whose header failed: all its chunks leave)
  __shared__ uint64_t s_scan[33];
  __shared__ uint32_t s_scan32[33];
  __shared__ uint32_t s_nc[3];
  __shared__ uint32_t s_chunk;
  __shared__ unsigned long long s_cp, s_cc;
  __shared__ bool s_last;
  const int tid = threadIdx.x;
  if (tid == 0) s_chunk = atomicAdd(&a.st->ticket_encode, 1u);
  if (tid < 3) s_nc[tid] = 0;
  __syncthreads();
  const uint32_t chunk = s_chunk;
  if (chunk == 0 && a.check_hdr && tid < 32) {
    // the launch was set up from a host copy of the header: it must be this archive's
    const uint8_t* h = a.ar + 4 * tid;
    const uint32_t v = (uint32_t)h[0] | ((uint32_t)h[1] << 8) | ((uint32_t)h[2] << 16) | ((uint32_t)h[3] << 24);
    if (__any_sync(~0u, v != a.hdr[tid]) && tid == 0) flag(a.st, ERR_CORRUPT);
  }
  const uint32_t b = chunk * 1024u + tid;
  uint64_t bb = 0;
  bool run = false, slow = false, bad = false;
  if (b < a.g.nblk) {
    const uint32_t c = a.ar[a.off_codec + b];
    bb = reinterpret_cast<const uint32_t*>(a.ar + a.off_bb)[b];
    if (c > 2 || (bb & 3)) bad = true;
    else atomicAdd(&s_nc[c], 1u);
    run = c == CODEC_RLE || c == CODEC_RLE_HUFF;
    slow = !(a.fuse && c == CODEC_HUFF && block_is_full(a.g, b));
  }
  uint64_t tot_pay;
  const uint64_t ex_pay = block_excl_scan<uint64_t>(bb, s_scan, &tot_pay);
  uint32_t tot_cnt;  // (slow << 16) | run, at most 1024 each in a chunk
  const uint32_t ex_cnt = block_excl_scan<uint32_t>(((uint32_t)slow << 16) | (uint32_t)run, s_scan32, &tot_cnt);
  if (tid < 32) {
    // chunk totals: payload bytes; (slow blocks << 32) | run blocks (each below 2^19)
    const uint64_t cnt = ((uint64_t)(tot_cnt >> 16) << 32) | (tot_cnt & 0xffffu);
    if (tid == 0) {
      lookback_publish(a.prep_lb, chunk, tot_pay);
      lookback_publish(a.prep_lb + nchunks, chunk, cnt);
    }
    const uint64_t cp = lookback_warp(a.prep_lb, chunk, tot_pay, &a.st->status, kSpinLimit);
    const uint64_t cc = lookback_warp(a.prep_lb + nchunks, chunk, cnt, &a.st->status, kSpinLimit);
    if (tid == 0) {
      s_cp = cp;
      s_cc = cc;
    }
  }
  __syncthreads();
  const uint64_t cp = s_cp, cc = s_cc;
  if (b < a.g.nblk) a.blk_off[b] = cp + ex_pay;
  if (run && a.runblk) a.runblk[(uint32_t)cc + (ex_cnt & 0xffffu)] = b;
  if (slow && a.slowblk) a.slowblk[(uint32_t)(cc >> 32) + (ex_cnt >> 16)] = b;
  if (tid == 0) {
    if (chunk == nchunks - 1) {
      a.blk_off[a.g.nblk] = cp + tot_pay;
      a.st->n_slow = (uint32_t)(cc >> 32) + (tot_cnt >> 16);
      if (cp + tot_pay != a.payload) bad = true;
    }
    for (int c = 0; c < 3; c++)
      if (s_nc[c]) atomicAdd(&a.st->ncodec[c], s_nc[c]);
    __threadfence();
    s_last = atomicAdd(&a.st->encode_done, 1u) == nchunks - 1;
  }
  if (bad) flag(a.st, ERR_CORRUPT);
  __syncthreads();
  if (s_last && tid == 0) {
    __threadfence();
    uint32_t nc[3];
    for (int c = 0; c < 3; c++) nc[c] = atomicAdd(&a.st->ncodec[c], 0u);
    bool wrong = (nc[CODEC_HUFF] && !(a.flags & 1u)) || (nc[CODEC_RLE_HUFF] && !(a.flags & 2u));
    for (int c = 0; c < 3; c++)
      if (nc[c] != a.n_codec[c]) wrong = true;  // the header's counts decide which kernels run
    if (wrong) flag(a.st, ERR_CORRUPT);
  }
}

__device__ void dec_records_body(const DecodeArgs& a, uint32_t cta, uint32_t nctas) {
  if (a.dead) return;
  const uint32_t* rec = reinterpret_cast<const uint32_t*>(a.ar + a.off_rec);
  const uint64_t nslots = (uint64_t)a.g.nblk * kSlots;
  const uint64_t n = a.n_rec > (uint64_t)a.g.nblk + 1 ? a.n_rec : (uint64_t)a.g.nblk + 1;
  for (uint64_t i = cta * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)nctas * blockDim.x) {
    if (i < a.n_rec) {
      const uint32_t key = rec[2 * i];
      bool bad = ((i + 1 < a.n_rec) && key >= rec[2 * (i + 1)]) || (a.f64 && (key & 1u));
      const uint64_t slot = key >> 1;
      if (slot >= nslots) {
        bad = true;
      } else {
        uint32_t org[3], w[3];
        block_box(a.g, (uint32_t)(slot / kSlots), org, w);
        if (slot % kSlots >= (uint64_t)w[0] * w[1] * w[2]) bad = true;
      }
      if (bad) flag(a.st, ERR_CORRUPT);
    }
    if (i <= a.g.nblk) {
      const uint64_t target = i * (uint64_t)kSlots * 2;
      uint64_t lo = 0, hi = a.n_rec;
      while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        if ((uint64_t)rec[2 * mid] < target) lo = mid + 1;
        else hi = mid;
      }
      a.rec_start[i] = (uint32_t)lo;
    }
  }
}

// One CTA per book: lengths from the archive, Kraft check, canonical tables, the
// kLutBits-bit lookup table (16-bit entries) and the second-level table of longer codes.
// Bound by latency (one CTA per book, ahead of the whole decoding), so nothing here runs
// serially over the 64 lengths or searches per table entry: lengths map to lanes, and a
// thread fills eight lookup entries at a time, at one store where they share a code.
__device__ void dec_tables_body(const DecodeArgs& a, int book) {
  if (a.dead) return;
  __shared__ uint8_t s_len[kNsymLen];
  __shared__ uint16_t s_wcnt[(kNsymLen / 32) * (kMaxLen + 1)];
  __shared__ uint16_t s_sorted[kNsymLen];
  __shared__ CanonSmem cs;
  __shared__ uint32_t s_cnt[kMaxLen + 2];
  // the limits' upper words, all ones once the code space is full (a limit of at most 31
  // bits that is not full never reads all ones; longer ones are not looked up here)
  __shared__ uint32_t s_lim[kMaxLen + 1];
  __shared__ uint32_t s_bad, s_full[2];
  const int tid = threadIdx.x;
  const int nsym = book == 2 ? kNsymLen : kNsymCode;
  DecTab* t = &a.tabs[book];
  const bool present = book == 0 ? (a.flags & 1u) : (a.flags & 2u);
  if (!present) {
    if (tid == 0) t->present = 0;
    return;
  }
  uint64_t off = a.off_books;
  if (book >= 1 && (a.flags & 1u)) off += kNsymCode;
  if (book == 2) off += kNsymCode;
  if (tid == 0) s_bad = 0;
  for (int l = tid; l < kMaxLen + 2; l += blockDim.x) s_cnt[l] = 0;
  __syncthreads();
  for (int s = tid; s < nsym; s += blockDim.x) {
    const uint8_t l = a.ar[off + s];
    s_len[s] = l;
    if (l > kMaxLen || (book < 2 && s >= (int)(2 * a.radius) && l)) s_bad = 1;
    else if (l) atomicAdd(&s_cnt[l], 1u);
  }
  __syncthreads();
  if (tid < 32) {
    // Kraft sum in 2^-64 steps, exactly: whole parts, and the fractions' upper and lower
    // words (no sum of 64 such words overflows 64 bits)
    uint64_t whole = 0, fh = 0, fl = 0;
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const int l = 2 * tid + 1 + k;
      const uint64_t c = s_cnt[l], f = c << (64 - l);
      whole += l < 64 ? c >> l : 0ull;
      fh += f >> 32;
      fl += f & 0xffffffffull;
    }
    whole = warp_sum(whole);
    fh = warp_sum(fh);
    fl = warp_sum(fl);
    fh += fl >> 32;
    whole += fh >> 32;
    const bool frac = (fh & 0xffffffffull) != 0 || (fl & 0xffffffffull) != 0;
    if (tid == 0 && (whole > 1 || (whole == 1 && frac))) s_bad = 1;
  }
  __syncthreads();
  if (s_bad) {
    if (tid == 0) {
      flag(a.st, ERR_CORRUPT);
      t->present = 0;
    }
    return;
  }
  canonical_build(s_len, nsym, &cs, s_wcnt, nullptr, nullptr, s_sorted);
  if (tid == 0) s_bad = s_full[0] = s_full[1] = 0;  // s_bad: now the largest length
  __syncthreads();
  if (tid <= kMaxLen) {
    // canonical codes of length l, left-justified to 64 bits, end at
    // (first_l + count_l) << (64-l); these ends never decrease, and wrap to 0 where the
    // code space is exhausted
    const int l = tid;
    const unsigned long long end = cs.first[l] + cs.cnt[l];
    const unsigned long long lim = l == 0 ? 0ull : end << (64 - l);
    const bool full = l > 0 && lim == 0 && cs.off[l] + cs.cnt[l] > 0;
    t->first[l] = cs.first[l];
    t->count[l] = cs.cnt[l];
    t->off[l] = cs.off[l];
    t->limit[l] = lim;
    s_lim[l] = full ? ~0u : (uint32_t)(lim >> 32);
    if (l > 0 && cs.cnt[l]) atomicMax(&s_bad, (uint32_t)l);
    if (full && l < 64) atomicOr(&s_full[l >> 5], 1u << (l & 31));
  }
  for (int s = tid; s < nsym; s += blockDim.x) t->sorted[s] = s_sorted[s];
  __syncthreads();
  const int maxlen = (int)s_bad;
  // the second level: cells of 2^s2 in the code space above the codes of kLutBits bits
  const uint32_t top = s_lim[kLutBits];
  const uint32_t rest = 0u - top;  // 0 when the table holds every code (top all ones: 1)
  int s2 = 0;
  while (s2 < 32 && ((rest - 1u) >> s2) >= (uint32_t)kLut2Size) s2++;
  if (tid == 0) {
    t->fullmask = ((unsigned long long)s_full[1] << 32) | s_full[0];
    t->maxlen = (uint32_t)maxlen;
    t->present = 1;
    t->lut2_base = top;
    t->lut2_shift = (uint32_t)s2;
  }
  uint32_t lim[kLutBits + 1];
#pragma unroll
  for (int l = 1; l <= kLutBits; l++) lim[l] = s_lim[l];
  // length of the code that prefix v starts with: the smallest whose codes end above it
  auto entry = [&](uint32_t v) -> uint32_t {
    const uint32_t x = v << (32 - kLutBits);
    int l = 1;
#pragma unroll
    for (int k = 1; k <= kLutBits; k++) l += x >= lim[k] ? 1 : 0;
    if (l > kLutBits) return 0u;
    return lut_entry(s_sorted[cs.off[l] + (v >> (kLutBits - l)) - (uint32_t)cs.first[l]], (uint32_t)l);
  };
  for (uint32_t g = tid; g < (1u << kLutBits) / 8; g += blockDim.x) {
    uint32_t e[8];
    e[0] = entry(8 * g);
    if (e[0] && lut_len(e[0]) <= kLutBits - 3) {
#pragma unroll
      for (int k = 1; k < 8; k++) e[k] = e[0];
    } else {
#pragma unroll 1
      for (int k = 1; k < 8; k++) {
        const uint32_t v = entry(8 * g + k);
#pragma unroll
        for (int j = 1; j < 8; j++) e[j] = j == k ? v : e[j];
      }
    }
    reinterpret_cast<uint4*>(t->lut)[g] =
        make_uint4(e[0] | e[1] << 16, e[2] | e[3] << 16, e[4] | e[5] << 16, e[6] | e[7] << 16);
  }
  for (uint32_t c = tid; book < 2 && c < (uint32_t)kLut2Size; c += blockDim.x) {
    const uint64_t x = (uint64_t)top + ((uint64_t)c << s2);
    uint32_t e = 0;
    if (x < ~0u && rest > 1u) {
      int l = kLutBits + 1;
      while (l <= kLut2Max && l <= maxlen && (uint32_t)x >= s_lim[l]) l++;
      // a cell inside one code (its 2^(32-l) values) resolves it
      if (l <= kLut2Max && l <= maxlen && 32 - l >= s2) {
        const uint64_t code = x >> (32 - l);
        if (code - cs.first[l] < cs.cnt[l])
          e = lut2_entry(s_sorted[cs.off[l] + (uint32_t)(code - cs.first[l])], (uint32_t)l);
      }
    }
    t->lut2()[c] = (uint16_t)e;
  }
}

// One launch for archive set-up: the first `nchunks` CTAs validate codecs and scan
// block sizes (one chunk of 1024 blocks each), the next three build the decode tables
// of the three books, the rest validate records and find each block's first record.
__global__ __launch_bounds__(1024) void dec_setup_kernel(DecodeArgs a, uint32_t nchunks) {
  chained_begin();
  if (blockIdx.x < nchunks) {
    dec_prep_chunk_body(a, nchunks);
  } else if (blockIdx.x < nchunks + 3) {
    dec_tables_body(a, (int)(blockIdx.x - nchunks));
  } else {
    dec_records_body(a, blockIdx.x - nchunks - 3, gridDim.x - nchunks - 3);
  }
}

// =================================================================================
// interleaved Huffman streams: one warp decodes one stream (see common.cuh)
// =================================================================================
struct BookView {
  const LutEntry* lut;  // 1 << kLutBits entries
  const unsigned long long* first;
  const unsigned long long* limit;
  const uint32_t* count;
  const uint32_t* off;
  const uint16_t* sorted;
  const uint16_t* lut2;  // second-level table (codes just longer than kLutBits), lut2_n cells
  uint32_t lut2_n, lut2_base, lut2_shift;
  int maxlen;
  unsigned long long fullmask;
};

// Matching the next codeword among the nb valid top bits of bb, for a code longer than
// the lookup table's: its length is the smallest one whose left-justified codes end
// above bb (a binary search over the canonical limits), the true length whenever it is
// <= nb (zero bits below nb cannot complete a shorter codeword), checked to be a codeword.
// Returns that length (0 if none fits in nb bits) and sets sym.
__device__ __forceinline__ int ihs_match_long(uint64_t bb, int nb, const BookView& bk, int& sym) {
  int lo = kLutBits + 1, hi = bk.maxlen + 1;  // smallest k whose codes end above bb
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (((bk.fullmask >> mid) & 1ull) || bb < bk.limit[mid]) hi = mid;
    else lo = mid + 1;
  }
  if (lo > bk.maxlen || lo > nb) return 0;
  const uint64_t c = bb >> (64 - lo);
  if (c < bk.first[lo] || c - bk.first[lo] >= bk.count[lo]) return 0;  // not a codeword
  sym = (int)bk.sorted[bk.off[lo] + (uint32_t)(c - bk.first[lo])];
  return lo;
}

// A warp's reader of one interleaved stream in[0..avail).
//
// Bound by instruction issue (it is the decoder's inner loop), so the step rests on two
// facts of the unit order.  A lane takes units only until its next code is complete, so
// it enters every step with at most 15 bits: its state is one 32-bit word.  And whether
// nb bits hold a whole code needs no table: exactly when, zero-padded, they lie below the
// end of the canonical codes of up to nb bits -- 16 words, one per lane, read by a
// shuffle.  So a step is one compare, one ballot, one unit and one table lookup; a code
// of up to 16 bits is complete after one unit, and the lookup misses only for codes
// longer than the table (a second-level table, then a search).  The step this replaces
// looked up twice and kept 64-bit windows: 159 warp instructions per 32 symbols with the
// reconstruction, 693 us at 3-D 512^3 (rel 1e-4; 941 us when one block's run codec put
// the other books' tables beside the code book's and halved the occupancy).  This one:
// 415 us either way, 2-D 1800x3600 61 -> 33 us.
//
// The stream's next 128 units wait in a ring in shared memory; each half is refilled
// from registers loaded one half ahead, so no load sits on the step's path.
struct IhsReader {
  const uint16_t* __restrict__ in;
  uint32_t avail;
  uint32_t ring;   // shared-memory address of the warp's 128 units, 256-byte aligned
  uint32_t lim;    // lane 16 - k: the end of the codes of up to k bits, upper word
  uint32_t p0, p1; // this lane's units of the half after the ring's
  uint32_t cur;    // units taken so far by the warp
  uint32_t half;   // cur reaching this refills the half before it
  uint32_t bb;     // this lane's bits, left-aligned
  int sh;          // 16 - (number of bits): 1..16 between steps
  bool bad;        // this lane met a damaged stream

  __device__ __forceinline__ uint32_t fetch(uint32_t i) const { return i < avail ? (uint32_t)__ldg(&in[i]) : 0u; }
  __device__ __forceinline__ uint32_t unit(uint32_t i) const {
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(((2u * i) & 254u) | ring) : "memory");
    return v;
  }
  __device__ __forceinline__ void put(uint32_t i, uint32_t v) const {
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(((2u * i) & 254u) | ring), "h"((uint16_t)v) : "memory");
  }

  __device__ __forceinline__ void init(const uint16_t* p, uint32_t n, const BookView& bk, uint32_t ring_addr) {
    const uint32_t lane = threadIdx.x & 31;
    in = p;
    avail = n;
    ring = ring_addr;
    uint32_t v[4];
#pragma unroll
    for (int k = 0; k < 4; k++) v[k] = fetch(32 * k + lane);
    p0 = fetch(128 + lane);
    p1 = fetch(160 + lane);
    const int k = 16 - (int)lane;  // (lanes 0 and 17 to 31 are never read)
    lim = k >= 0 && k < 16 ? (((bk.fullmask >> k) & 1ull) ? ~0u : (uint32_t)(bk.limit[k] >> 32)) : 0u;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 4; i++) put(32 * i + lane, v[i]);
    __syncwarp();
    cur = 0;
    half = 64;
    bb = 0;
    sh = 16;
    bad = false;
  }

  __device__ __forceinline__ void advance(uint32_t taken) {
    cur += taken;
    if (cur >= half) {
      const uint32_t lane = threadIdx.x & 31;
      __syncwarp();
      put(half + lane + 64, p0);
      put(half + lane + 96, p1);
      __syncwarp();
      p0 = fetch(half + 128 + lane);
      p1 = fetch(half + 160 + lane);
      half += 64;
    }
  }

  // Lanes with `open`: the code is longer than the tables resolve, or incomplete.  They
  // search, and take further units in rounds until it is complete (at most 48 bits are
  // held before a unit: more marks the stream damaged).  Returns the symbol and leaves
  // the state past the code.
  __device__ __forceinline__ int step_long(bool open, const BookView& bk) {
    const uint32_t lt = (1u << (threadIdx.x & 31)) - 1u;
    uint64_t w = (uint64_t)bb << 32;
    int nb = 16 - sh, ml = 0, sym = 0;
    const bool mine = open;
    while (true) {
      if (open) ml = ihs_match_long(w, nb, bk, sym);
      const bool need = open && ml == 0;
      const uint32_t ballot = __ballot_sync(~0u, need);
      if (ballot == 0u) break;
      const bool over = nb > 48;
      bad = bad || (need && over);
      const uint64_t u = unit(cur + __popc(ballot & lt));
      open = need && !over;
      if (open) {
        w |= u << (48 - nb);
        nb += 16;
      }
      advance(__popc(ballot));
    }
    if (mine) {
      w = ml > 0 && ml < 64 && !bad ? w << ml : 0ull;
      bb = (uint32_t)(w >> 32);
      sh = bad ? 16 : 16 - (nb - ml);
    }
    return sym;
  }

  // One decoding step of the 32 lanes (every lane calls): each active lane whose bits
  // hold no whole code takes the next unit, then consumes its code.  Returns the
  // symbol, meaningful where the lane was active and is not bad.
  __device__ __forceinline__ int step(bool active, const BookView& bk) {
    const uint32_t lt = (1u << (threadIdx.x & 31)) - 1u;
    const uint32_t end = __shfl_sync(~0u, lim, sh);  // (by every lane, active or not)
    const bool need = active && bb >= end;
    const uint32_t ballot = __ballot_sync(~0u, need);
    const uint32_t u = unit(cur + __popc(ballot & lt));
    if (need) {
      bb |= u << sh;
      sh -= 16;
    }
    advance(__popc(ballot));
    const uint32_t e = bk.lut[bb >> (32 - kLutBits)];
    int l = lut_len(e), sym = lut_sym(e);
    const bool miss = active && e == 0u;
    if (__builtin_expect(__any_sync(~0u, miss), 0)) {
      bool open = miss;
      if (miss) {
        // (bb lies at or above the second level's base: the lookup missed.  A damaged
        // stream can point past its cells.)
        const uint32_t c = (bb - bk.lut2_base) >> bk.lut2_shift;
        const uint32_t e2 = c < bk.lut2_n ? (uint32_t)bk.lut2[c] : 0u;
        const int l2 = lut2_len(e2);
        if (e2 != 0u && l2 <= 16 - sh) {
          l = l2;
          sym = lut2_sym(e2);
          open = false;
        }
      }
      if (__any_sync(~0u, open)) {
        const int s3 = step_long(open, bk);
        if (open) {
          sym = s3;
          l = 0;
        }
      }
    }
    if (active) {
      bb <<= l;
      sh += l;
    }
    return sym;
  }

  // After the last step: the warp's verdict on the stream (uniform).
  __device__ __forceinline__ bool sound() const { return !__any_sync(~0u, bad) && cur <= avail; }
};

// One warp decodes N symbols (+add) from in[0..avail) into out[].  Returns false
// (warp-uniform) if the stream is damaged; *used gets the units read.
__device__ bool ihs_decode_warp(const uint16_t* __restrict__ in, uint32_t avail, uint32_t N,
                                const BookView& bk, uint16_t* out, int add, uint32_t* used, uint32_t ring) {
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t T = (N + 31) / 32;
  IhsReader rd;
  rd.init(in, avail, bk, ring);
#pragma unroll 1
  for (uint32_t t = 0; t < T; t++) {
    const bool active = 32 * t + lane < N;
    const int sym = rd.step(active, bk);
    if (active && !rd.bad) out[32 * t + lane] = (uint16_t)(sym + add);
  }
  *used = rd.cur;
  return rd.sound();
}

__device__ __forceinline__ float scale(int32_t k, float ebx2) { return __fmul_rn(__int2float_rn(k), ebx2); }

// The reconstruction's output by element type: x' = fl32(k * 2eb_f) for FP32 fields,
// x' = fl64(k * step) for double fields (which have no verbatim patches).
template <typename E>
struct Out;
template <>
struct Out<float> {
  float* __restrict__ p;
  float ebx2;
  __device__ explicit Out(const DecodeArgs& a) : p(a.out), ebx2(a.ebx2_f) {}
  __device__ __forceinline__ float value(int32_t k) const { return scale(k, ebx2); }
  __device__ __forceinline__ void put(uint64_t i, int32_t k) const { __stcs(&p[i], scale(k, ebx2)); }
  // four consecutive elements, i a multiple of four elements from x0: vec4(x0) must hold
  __device__ __forceinline__ bool vec4(uint64_t x0) const { return ((uintptr_t)(p + x0) & 15) == 0; }
  __device__ __forceinline__ void put4(uint64_t i, int4 k) const {
    __stcs(reinterpret_cast<float4*>(&p[i]),
           make_float4(scale(k.x, ebx2), scale(k.y, ebx2), scale(k.z, ebx2), scale(k.w, ebx2)));
  }
  __device__ __forceinline__ void patch(uint64_t i, uint32_t bits) const { p[i] = __uint_as_float(bits); }
};
template <>
struct Out<double> {
  double* __restrict__ p;
  double step;
  __device__ explicit Out(const DecodeArgs& a) : p(a.out64), step(a.step_d) {}
  // (double)k built from bits: the conversion instruction would take the FP64 pipe, 2
  // results a cycle and SM, once more beside the product (3-D 256^3: 107 -> 97 us)
  __device__ __forceinline__ static double to_double(int32_t k) {
    const uint32_t m = (uint32_t)abs(k), z = (uint32_t)__clz((int)m), t = m << (z & 31u);
    const uint32_t hi = m ? ((1053u - z) << 20) + (t >> 11) : 0u;
    return __hiloint2double((int)(hi | ((uint32_t)k & 0x80000000u)), (int)(t << 21));
  }
  __device__ __forceinline__ void put(uint64_t i, int32_t k) const { __stcs(&p[i], __dmul_rn(to_double(k), step)); }
  __device__ __forceinline__ bool vec4(uint64_t x0) const { return ((uintptr_t)(p + x0) & 15) == 0; }
  __device__ __forceinline__ void put4(uint64_t i, int4 k) const {
    __stcs(reinterpret_cast<double2*>(&p[i]), make_double2(__dmul_rn(to_double(k.x), step), __dmul_rn(to_double(k.y), step)));
    __stcs(reinterpret_cast<double2*>(&p[i + 2]),
           make_double2(__dmul_rn(to_double(k.z), step), __dmul_rn(to_double(k.w), step)));
  }
  __device__ __forceinline__ void patch(uint64_t, uint32_t) const {}
};

// =================================================================================
// fused decoding and reconstruction of full Huffman blocks (Alg. 1 decompression,
// Sec. IV-B "Partial-Sum Lorenzo Reconstruction")
//
// A full block's stream A holds its first 2048 codes and stream B the rest, and
// 2048 codes end on a Lorenzo-chunk boundary in every dimensionality: 8 chunks of
// 256 (1-D), rows 0-31 / 32-63 (2-D, 16x16 chunks), z 0-7 / 8-15 (3-D, 8^3 chunks).
// So the warp that decodes a stream owns whole chunks, and at step t lane l holds
// code 32t + l, which is already where the partial sums want it:
//   1-D  element 32t + l: the x sum is a warp scan plus a carry within each chunk
//        of 8 steps;
//   2-D  row t/2, column 32(t&1) + l: x sums over 16-lane groups by shuffles, y sums
//        in a register per column half, restarting every 16 rows;
//   3-D  plane t/8, row 2(t%8) + l/16, column l%16: x sums over 8-lane groups, y sums
//        across the lane pair (l, l^16) by one shuffle and a running pair sum that
//        restarts every 4 steps, z sums in a register per step of the plane.
// Each step then scales the exact integers and stores them: the codes never leave
// the registers.  Outliers (code 0) take their delta from the block's records, found
// by binary search (records are sorted by slot); verbatim patches overwrite their
// elements after the warp's own stores.
// =================================================================================

// The block's outlier records, merged into the decode order.  Records are sorted by
// key (slot * 2 + kind), and step t of a stream covers 32 consecutive slots, so the
// warp keeps the key of its next record in a register; only a step that reaches it
// loads the step's records (at most 64: an outlier and a patch per slot) and hands
// each outlier's delta to the lane of its slot through a 32-word per-warp table in
// shared memory (the fused code q' of Alg. 1).  The step's outlier records must match
// its code-0 slots one for one; anything else marks the stream corrupt.  Patches are
// applied after the stream (they only overwrite output values).
struct RecordCursor {
  const uint2* __restrict__ rec;
  uint32_t ptr, end;  // next record, end of the block's records
  uint32_t next;      // key of rec[ptr] (0xffffffff when none is left)

  // Positions the cursor at the first record with key >= key_lo among rec[rs..re).
  __device__ __forceinline__ void init(const uint2* r, uint32_t rs, uint32_t re, uint32_t key_lo) {
    rec = r;
    end = re;
    uint32_t lo = rs, hi = re;
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if (rec[mid].x < key_lo) lo = mid + 1;
      else hi = mid;
    }
    ptr = lo;
    next = ptr < end ? rec[ptr].x : 0xffffffffu;
  }

  // The step whose first slot has key key0 (the calling lane's slot has key key0 +
  // 2 lane): where sym == 0, q becomes the outlier's delta.  All lanes call
  // (warp-uniform control flow).  s_tab: this warp's 32 words of shared memory.
  __device__ __forceinline__ void step(uint32_t key0, int sym, int32_t& q, bool& bad, uint32_t* s_tab) {
    const uint32_t lane = threadIdx.x & 31;
    if (next >= key0 + 64u) {  // no record in this step (the common case)
      bad |= sym == 0;
      return;
    }
    uint32_t omask = 0;
#pragma unroll
    for (int half = 0; half < 2; half++) {
      const uint32_t i = ptr + lane;  // ptr has moved past the first half's records
      const uint2 kv = i < end ? rec[i] : make_uint2(0xffffffffu, 0u);
      const bool here = kv.x < key0 + 64u;
      const uint32_t l = ((kv.x >> 1) - (key0 >> 1)) & 31u;  // the record's lane
      const bool outlier = here && !(kv.x & 1u);
      if (outlier) s_tab[l] = kv.y;
      omask |= __reduce_or_sync(~0u, outlier ? 1u << l : 0u);
      const uint32_t hb = __ballot_sync(~0u, here);
      ptr += __popc(hb);
      if (hb != ~0u) break;
    }
    __syncwarp();
    if ((omask >> lane) & 1u) q = (int32_t)s_tab[lane];
    bad |= __ballot_sync(~0u, sym == 0) != omask;
    next = ptr < end ? rec[ptr].x : 0xffffffffu;
    __syncwarp();  // the table is free again
  }
};

// Decodes stream `which` (0: A, 1: B) of full Huffman block b from u[0..avail) and
// writes its 2048 reconstructed elements.  The warp decodes 8 steps into a register
// window, then runs their 8 prefix chains together (independent shuffles overlap)
// and stores them.  Returns false (warp-uniform) if the stream is damaged or its records do not
// match its outlier slots; *used gets the units read.  s_tab: this warp's 32 words of
// shared memory (the record table), ring: its ring of units.
template <int ND, typename E>
__device__ bool fused_decode_reconstruct(const DecodeArgs& a, uint32_t b, uint32_t which, const uint16_t* u,
                                         uint32_t avail, const BookView& bk, uint32_t* used, uint32_t* s_tab,
                                         uint32_t ring) {
  const uint32_t lane = threadIdx.x & 31;
  const int32_t r = (int32_t)a.radius;
  const Out<E> out(a);
  const uint32_t key0 = (b * (uint32_t)kSlots + 2048u * which) * 2u;  // record key of the stream's first slot
  uint32_t org[3], w[3];
  block_box(a.g, b, org, w);
  const uint64_t ny = a.g.n[1], nx = a.g.n[2];
  const uint2* rec = reinterpret_cast<const uint2*>(a.ar + a.off_rec);
  const uint32_t rs = a.rec_start[b], re = a.rec_start[b + 1];
  IhsReader rd;
  rd.init(u, avail, bk, ring);
  RecordCursor rc;
  rc.init(rec, rs, re, key0);
  bool bad = false;
  int32_t carry = 0, ysum0 = 0, ysum1 = 0;
  int32_t zs[8];  // 3-D: the running z sum of each of the lane's 8 rows of a plane
#pragma unroll
  for (int s = 0; s < 8; s++) zs[s] = 0;
#pragma unroll 1
  for (uint32_t t0 = 0; t0 < 64; t0 += 8) {
    // four copies of the step per iteration (eight overflow the instruction cache: 507
    // against 415 us at 3-D 512^3; two: 426)
    int32_t q[8];
#pragma unroll 1
    for (int s0 = 0; s0 < 8; s0 += 4) {
#pragma unroll
      for (int s = 0; s < 4; s++) q[s] = q[s + 4];
#pragma unroll
      for (int s = 0; s < 4; s++) q[4 + s] = rd.step(true, bk) - r;
    }
    // the window's outlier records, if it reaches any (a code 0 without one is damage)
    if (rc.next < key0 + 64u * (t0 + 8)) {
#pragma unroll
      for (int s = 0; s < 8; s++) {
        const int sym = q[s] + r;
        rc.step(key0 + 64u * (t0 + s), sym, q[s], bad, s_tab);
      }
    } else {
#pragma unroll
      for (int s = 0; s < 8; s++) bad |= q[s] == -r;
    }
    if (ND == 1) {
      // 8 steps = one 256-element chunk: per-step warp scans, then the carries
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
        for (int s = 0; s < 8; s++) {
          const int32_t up = __shfl_up_sync(~0u, q[s], o);
          if (lane >= (uint32_t)o) q[s] += up;
        }
      }
      carry = 0;
      const uint64_t base = (uint64_t)org[2] + 2048u * which + 32u * t0 + lane;
#pragma unroll
      for (int s = 0; s < 8; s++) {
        const int32_t v = q[s] + carry;
        carry += __shfl_sync(~0u, q[s], 31);
        out.put(base + 32u * s, v);
      }
    } else if (ND == 2) {
      // rows t/2, columns 32 (t&1) + lane: x sums over 16-lane groups, y sums down
      // each column half, restarting every 16 rows (32 steps)
#pragma unroll
      for (int o = 1; o < 16; o <<= 1) {
#pragma unroll
        for (int s = 0; s < 8; s++) {
          const int32_t up = __shfl_up_sync(~0u, q[s], o);
          if ((lane & 15) >= (uint32_t)o) q[s] += up;
        }
      }
      if ((t0 & 31) == 0) ysum0 = ysum1 = 0;
      const uint64_t base = ((uint64_t)org[1] + 32u * which + (t0 >> 1)) * nx + org[2] + lane;
#pragma unroll
      for (int s = 0; s < 8; s++) {
        int32_t& ys = (s & 1) ? ysum1 : ysum0;
        ys += q[s];
        out.put(base + (uint64_t)(s >> 1) * nx + 32u * (s & 1), ys);
      }
    } else {
      // plane t/8 of the stream's z chunk, rows 2s + lane/16, column lane%16: x sums
      // over 8-lane groups, y sums across the lane pair (l, l^16) within each 8-row
      // chunk, z sums in registers
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
#pragma unroll
        for (int s = 0; s < 8; s++) {
          const int32_t up = __shfl_up_sync(~0u, q[s], o);
          if ((lane & 7) >= (uint32_t)o) q[s] += up;
        }
      }
      const uint32_t p = lane >> 4;
      const uint32_t zp = t0 >> 3;
      const uint64_t base = ((uint64_t)(org[0] + 8u * which + zp) * ny + org[1] + p) * nx + org[2] + (lane & 15);
      int32_t pair = 0;
#pragma unroll
      for (int s = 0; s < 8; s++) {
        const int32_t other = __shfl_xor_sync(~0u, q[s], 16);
        if (s == 4) pair = 0;  // rows 8-15: the second y chunk
        zs[s] += pair + q[s] + (p ? other : 0);
        pair += q[s] + other;
        out.put(base + (uint64_t)(2 * s) * nx, zs[s]);
      }
    }
  }
  *used = rd.cur;
  const bool ok = !__any_sync(~0u, bad) & rd.sound();
  // verbatim patches of this stream's slots overwrite their elements (after the
  // warp's own stores: __syncwarp orders them)
  __syncwarp();
  for (uint32_t i = rs + lane; i < re; i += 32) {
    const uint2 kv = rec[i];
    const uint32_t j = (kv.x >> 1) % kSlots;
    if ((kv.x & 1u) && (j >> 11) == which) {
      uint64_t e;
      if (ND == 1) e = (uint64_t)org[2] + j;
      else if (ND == 2) e = (uint64_t)(org[1] + (j >> 6)) * nx + org[2] + (j & 63);
      else e = ((uint64_t)(org[0] + (j >> 8)) * ny + org[1] + ((j >> 4) & 15)) * nx + org[2] + (j & 15);
      out.patch(e, kv.y);
    }
  }
  return ok;
}

constexpr int kStreamWarps = kStreamWarpsPerCta;
// per decoding warp: its ring of 128 units (64 words, 256-byte aligned) and, for fused
// streams, its record table (32 words); 64 words of slack align the rings
constexpr int kRingWords = 64, kRecTabWords = 32;
static size_t stream_smem_bytes(int nluts, int warps) {
  return (size_t)nluts * (1u << kLutBits) * sizeof(LutEntry) + 4u * (size_t)(kRingWords * (warps + 1) + kRecTabWords * warps);
}

// Entropy decoding, persistent: each CTA stages the lookup tables of the books the
// archive uses in shared memory once, then its warps take (block, stream) slots from
// a ticket; a warp decodes one stream of a Huffman block, or the value or the length
// stream of an RLE+Huffman block (runs go to the workspace run arrays).  With fusion
// (ND != 0 and a.fuse), a stream of a full Huffman block is reconstructed by the
// warp as it is decoded (fused_decode_reconstruct); other Huffman streams leave
// their codes in the workspace for the reconstruction kernel.
// Streams come from the field's ticket (b_end == 0) or, in batches, from the CTA's
// chunk of blocks [b_begin, b_end): each warp draws the chunk's next stream from a
// shared counter until none is left.
template <int ND, typename E>
__device__ void stream_decode_body(const DecodeArgs& a, uint32_t b_begin, uint32_t b_end) {
  extern __shared__ __align__(16) uint32_t s_dyn[];  // the present books' tables, then record tables
  __shared__ unsigned long long s_first[kMaxLen + 1], s_limit[kMaxLen + 1];
  __shared__ uint32_t s_off[kMaxLen + 1], s_count[kMaxLen + 1];
  __shared__ int s_go;
  if (a.dead) return;
  // the status is read once, by thread 0, and acted on after the staging barrier, so
  // that a corruption flagged by another CTA meanwhile cannot split this CTA
  __shared__ uint32_t s_next;  // batches: the chunk's next stream slot
  if (threadIdx.x == 0) {
    s_go = !undecodable(a.st->status);
    s_next = 0;
  }
  const bool huff = (a.flags & 1u) != 0, rle = (a.flags & 2u) != 0;
  LutEntry* s_luts = reinterpret_cast<LutEntry*>(s_dyn);
  LutEntry* lut_code = s_luts;
  LutEntry* lut_val = s_luts + (huff ? (1 << kLutBits) : 0);
  LutEntry* lut_len = lut_val + (1 << kLutBits);
  // after the tables, the warps' rings and record tables (stream_smem_bytes)
  uint32_t* s_tail =
      reinterpret_cast<uint32_t*>(s_luts + (huff ? (1 << kLutBits) : 0) + (rle ? 2 * (1 << kLutBits) : 0));
  const uint32_t ring0 = (smem_u32(s_tail) + 255u) & ~255u;
  const uint32_t wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const uint32_t ring = ring0 + 4u * kRingWords * wid;
  uint32_t* s_rectab = s_tail + (ring0 - smem_u32(s_tail)) / 4 + kRingWords * nwarps + kRecTabWords * wid;
  // a chunk of blocks (batches) copies only the tables its own blocks use
  bool need_code = huff, need_runs = rle;
  if (b_end != 0) {
    const uint32_t b = b_begin + threadIdx.x;
    const int c = (b < b_end) ? a.ar[a.off_codec + b] : -1;
    need_code = __syncthreads_or(huff && c == CODEC_HUFF) != 0;
    need_runs = __syncthreads_or(rle && c == CODEC_RLE_HUFF) != 0;
  }
  constexpr int kLutVec = (1 << kLutBits) * (int)sizeof(LutEntry) / 16;  // 16-byte pieces per table
  for (int i = threadIdx.x; i < kLutVec; i += blockDim.x) {
    if (need_code) reinterpret_cast<uint4*>(lut_code)[i] = reinterpret_cast<const uint4*>(a.tabs[0].lut)[i];
    if (need_runs) {
      reinterpret_cast<uint4*>(lut_val)[i] = reinterpret_cast<const uint4*>(a.tabs[1].lut)[i];
      reinterpret_cast<uint4*>(lut_len)[i] = reinterpret_cast<const uint4*>(a.tabs[2].lut)[i];
    }
  }
  for (int i = threadIdx.x; i <= kMaxLen; i += blockDim.x) {
    s_first[i] = a.tabs[0].first[i];
    s_limit[i] = a.tabs[0].limit[i];
    s_off[i] = a.tabs[0].off[i];
    s_count[i] = a.tabs[0].count[i];
  }
  __syncthreads();
  if (!s_go) return;
  const bool lane0 = (threadIdx.x & 31) == 0;
  const bool ticketed = b_end == 0;
  // work items are (block, stream) slots: a Huffman block's streams A and B, an
  // RLE+Huffman block's value and length streams
  for (;;) {
    uint32_t slot = 0;
    if (ticketed) {
      if (lane0) slot = atomicAdd(&a.st->ticket_decode, 1u);
      slot = __shfl_sync(~0u, slot, 0);
      if (slot >= 2 * a.g.nblk) break;
    } else {
      // the chunk's streams, drawn one at a time by whichever warp is free
      if (lane0) slot = atomicAdd(&s_next, 1u);
      slot = 2 * b_begin + __shfl_sync(~0u, slot, 0);
      if (slot >= 2 * b_end) break;
    }
    const uint32_t b = slot >> 1, which = slot & 1;
    const int codec = a.ar[a.off_codec + b];
    if (codec == CODEC_RLE) continue;
    uint32_t org[3], w[3];
    block_box(a.g, b, org, w);
    const uint32_t m = w[0] * w[1] * w[2];
    const uint64_t bytes = a.blk_off[b + 1] - a.blk_off[b];
    const uint8_t* pay = a.ar + a.off_pay + a.blk_off[b];
    uint32_t used = 0;
    bool ok;
    if (codec == CODEC_HUFF) {
      const DecTab* t = &a.tabs[0];
      const uint16_t* u = reinterpret_cast<const uint16_t*>(pay);
      const uint32_t nu = (uint32_t)(bytes / 2);
      const uint32_t na = nu >= 1 ? u[0] : 0u;
      if (!t->present || nu < 1 || na > nu - 1) {
        if (lane0) flag(a.st, ERR_CORRUPT);
        continue;
      }
      const uint32_t h = huff_split(m);
      const BookView bk{lut_code, s_first, s_limit, s_count, s_off, t->sorted, t->sorted + kNsymCode,
                        (uint32_t)kLut2Size, t->lut2_base, t->lut2_shift, (int)t->maxlen, t->fullmask};
      const uint16_t* us = which == 0 ? u + 1 : u + 1 + na;
      const uint32_t nus = which == 0 ? na : nu - 1 - na;
      if (ND != 0 && a.fuse && m == (uint32_t)kSlots) {
        ok = fused_decode_reconstruct<ND, E>(a, b, which, us, nus, bk, &used, s_rectab, ring);
      } else {
        ok = ihs_decode_warp(us, nus, which == 0 ? h : m - h, bk, a.codes + (uint64_t)b * kSlots + (which == 0 ? 0u : h),
                             0, &used, ring);
      }
      ok = ok && (which == 0 ? used == na : ((2ull * (1ull + na + used) + 3) & ~3ull) == bytes);
    } else {
      const DecTab* tv = &a.tabs[1];
      const DecTab* tl = &a.tabs[2];
      if (!tv->present || !tl->present) {
        if (lane0) flag(a.st, ERR_CORRUPT);
        continue;
      }
      const uint32_t* p32 = reinterpret_cast<const uint32_t*>(pay);
      const uint32_t nr = bytes >= 8 ? p32[0] : 0u, vu = bytes >= 8 ? p32[1] : 0u;
      if (bytes < 8 || nr > m || 8ull + 2ull * vu > bytes) {
        if (lane0) flag(a.st, ERR_CORRUPT);
        continue;
      }
      const uint32_t lavail = (uint32_t)((bytes - 8) / 2 - vu);
      const uint16_t* p16 = reinterpret_cast<const uint16_t*>(pay) + 4;
      const DecTab* tb = which == 0 ? tv : tl;
      const BookView bk{which == 0 ? lut_val : lut_len, tb->first, tb->limit, tb->count, tb->off, tb->sorted,
                        tb->sorted + kNsymCode, which == 0 ? (uint32_t)kLut2Size : 0u, tb->lut2_base, tb->lut2_shift,
                        (int)tb->maxlen, tb->fullmask};
      ok = ihs_decode_warp(which == 0 ? p16 : p16 + vu, which == 0 ? vu : lavail, nr, bk,
                           (which == 0 ? a.runv : a.runl) + (uint64_t)b * kSlots, (int)which, &used, ring);
      ok = ok && (which == 0 ? used == vu : ((8ull + 2ull * (vu + used) + 3) & ~3ull) == bytes);
    }
    if (!ok && lane0) flag(a.st, ERR_CORRUPT);
  }
}

template <int ND, typename E>
__global__ __launch_bounds__(32 * kStreamWarps, 2) void stream_decode_kernel(DecodeArgs a) {
  chained_begin();
  stream_decode_body<ND, E>(a, 0, 0);
}

// =================================================================================
// blocks that no decoding warp reconstructs: run blocks, blocks cut by the field's edge,
// and all blocks of a batch of mixed dimensionality
//
// Bound by latency and barriers, not by bytes: one CTA a block, and what it needs arrives
// step after step.  So a thread keeps 16 consecutive slots (one row, or a piece of one) in
// registers from the codes, or straight from the runs, to the sums along x; shared memory
// only turns rows into columns for the other axes.  Runs become codes by a bit per run
// start and population counts.  (A word per slot for the starts and a scan of maxima over
// them took a dozen barriers, and the codes went through memory once more, in a launch of
// their own for single fields: 40 mixed fields, 51 M elements: 175 -> 82 us;
// 2-D 1800x3600: 12 us in two launches -> 6 us in one.)
// =================================================================================
constexpr int kRecThreads = 256;

struct RebuildSmem {
  int32_t k[kSlots];          // sums along x, swizzled; before that, codes of a cut run block
  uint16_t v[kSlots];         // run values
  uint32_t bits[kSlots / 32]; // run starts
  uint32_t tot[2][kRecThreads / 32];
  int go;
};

// The runs of run block b (m elements) as codes: thread t gets slots 16t .. 16t + 15, two a
// word (slots beyond m hold no code).  Returns false, the same in every thread, when the
// block is corrupt (flagged).  Contains barriers.
__device__ __forceinline__ bool expand_runs(const DecodeArgs& a, uint32_t b, int codec, uint32_t m, RebuildSmem& S,
                                            uint32_t (&c)[8]) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const uint64_t bytes = a.blk_off[b + 1] - a.blk_off[b];
  const uint8_t* pay = a.ar + a.off_pay + a.blk_off[b];
  const uint32_t lim = 2 * a.radius;
  uint32_t nr;
  const uint16_t *v, *l;
  if (codec == CODEC_RLE) {
    nr = (uint32_t)(bytes / 4);
    v = reinterpret_cast<const uint16_t*>(pay);
    l = v + nr;
  } else {
    nr = reinterpret_cast<const uint32_t*>(pay)[0];
    v = a.runv + (uint64_t)b * kSlots;
    l = a.runl + (uint64_t)b * kSlots;
  }
  if (nr > m) {
    if (tid == 0) flag(a.st, ERR_CORRUPT);
    return false;
  }
  if (tid < kSlots / 32) S.bits[tid] = 0;
  bool bad = false;
  uint32_t total = 0;
  for (uint32_t i0 = 0, k = 0; i0 < nr; i0 += kRecThreads, k ^= 1) {
    const uint32_t i = i0 + tid;
    uint32_t len = 0;
    if (i < nr) {
      const uint16_t val = v[i];
      len = l[i];
      S.v[i] = val;
      bad |= val >= lim || len == 0;
    }
    const uint32_t incl = warp_incl_scan(len);
    if (lane == 31) S.tot[k][wid] = incl;
    __syncthreads();  // (the other half of tot is free: every thread has read it before this barrier)
    uint32_t start = total + incl - len;
#pragma unroll
    for (uint32_t w = 0; w < kRecThreads / 32; w++) {
      const uint32_t t = S.tot[k][w];
      if (w < wid) start += t;
      total += t;
    }
    if (len && start < (uint32_t)kSlots) atomicOr(&S.bits[start >> 5], 1u << (start & 31));
  }
  if (__syncthreads_or(bad) || total != m) {
    if (tid == 0) flag(a.st, ERR_CORRUPT);
    return false;
  }
  // runs that start before slot 16t: the words of earlier warps, then the warp's own
  const uint32_t hb = (S.bits[tid >> 1] >> (16 * (tid & 1))) & 0xffffu;
  const uint4 w4 = reinterpret_cast<const uint4*>(S.bits)[lane];
  const uint32_t n4 = __popc(w4.x) + __popc(w4.y) + __popc(w4.z) + __popc(w4.w), n = __popc(hb);
  uint32_t run = __reduce_add_sync(~0u, lane < 4 * wid ? n4 : 0u) + warp_incl_scan(n) - n;
  uint32_t cur = run ? S.v[run - 1] : 0u;
#pragma unroll
  for (int i = 0; i < 16; i++) {
    if ((hb >> i) & 1u) cur = S.v[run++];
    c[i >> 1] = i & 1 ? c[i >> 1] | cur << 16 : cur;
  }
  return true;
}

// Global prediction: the codes of a listed run block into the code stream (the list the
// set-up wrote holds exactly the header's count unless the archive is corrupt, which the
// set-up has flagged).
__global__ __launch_bounds__(kRecThreads) void rle_expand_kernel(DecodeArgs a) {
  chained_begin();
  __shared__ __align__(16) RebuildSmem S;
  if (a.dead) return;
  const uint32_t b = a.runblk[blockIdx.x];
  if (b >= a.g.nblk) return;
  const int codec = a.ar[a.off_codec + b];
  if (codec != CODEC_RLE && codec != CODEC_RLE_HUFF) return;
  // the status is read once, by thread 0, and acted on after the barrier, so that a
  // corruption flagged by another CTA meanwhile cannot split this CTA's threads
  if (threadIdx.x == 0) S.go = !undecodable(a.st->status);
  __syncthreads();
  if (!S.go) return;
  uint32_t org[3], w[3], c[8];
  block_box(a.g, b, org, w);
  if (!expand_runs(a, b, codec, w[0] * w[1] * w[2], S, c)) return;
  uint4* o = reinterpret_cast<uint4*>(a.codes + (uint64_t)b * kSlots + 16 * threadIdx.x);
  o[0] = make_uint4(c[0], c[1], c[2], c[3]);
  o[1] = make_uint4(c[4], c[5], c[6], c[7]);
}

// The row piece of thread t of a block: 3-D row (z, y) = (t / 16, t % 16), up to 16
// elements; 2-D piece t % 4 (16 elements) of row t / 4; 1-D elements 16t on.
struct RowPiece {
  uint32_t j0, n;  // first slot and number of slots
  uint32_t z, y;   // in the block
  bool valid;
};
template <int ND>
__device__ __forceinline__ RowPiece row_piece(const uint32_t* w) {
  const uint32_t t = threadIdx.x;
  RowPiece p;
  const uint32_t x0 = ND == 3 ? 0u : (ND == 2 ? 16u * (t & 3u) : 16u * t);
  p.z = ND == 3 ? t >> 4 : 0u;
  p.y = ND == 3 ? t & 15u : (ND == 2 ? t >> 2 : 0u);
  p.valid = p.z < w[0] && p.y < w[1] && x0 < w[2];
  p.n = p.valid ? min(16u, w[2] - x0) : 0u;
  p.j0 = p.valid ? (p.z * w[1] + p.y) * w[2] + x0 : 0u;
  return p;
}

// q = code - r of n <= 16 slots (zeros behind them)
__device__ __forceinline__ void load_codes16(const uint16_t* codes, uint32_t j0, uint32_t n, int32_t r,
                                             int32_t (&q)[16]) {
  codes += j0;
  if (n == 16 && (j0 & 7) == 0) {
    const uint4 v[2] = {reinterpret_cast<const uint4*>(codes)[0], reinterpret_cast<const uint4*>(codes)[1]};
    const uint32_t u[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
#pragma unroll
    for (int i = 0; i < 8; i++) {
      q[2 * i] = (int32_t)(u[i] & 0xffffu) - r;
      q[2 * i + 1] = (int32_t)(u[i] >> 16) - r;
    }
  } else {
#pragma unroll
    for (uint32_t i = 0; i < 16; i++) q[i] = i < n ? (int32_t)codes[i] - r : 0;
  }
}

// The outliers' deltas among block b's slots j0 .. j0 + n - 1: the records (sorted by key)
// from the first one there, found by a search.
__device__ __forceinline__ void overlay_outliers(const DecodeArgs& a, uint32_t b, uint32_t j0, uint32_t n,
                                                 int32_t (&q)[16]) {
  uint32_t lo = a.rec_start[b];
  const uint32_t re = a.rec_start[b + 1];
  if (lo == re || n == 0) return;
  const uint2* rec = reinterpret_cast<const uint2*>(a.ar + a.off_rec);
  const uint32_t k0 = (b * (uint32_t)kSlots + j0) * 2u, k1 = k0 + 2u * n;
  uint32_t hi = re;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (rec[mid].x < k0) lo = mid + 1;
    else hi = mid;
  }
  for (; lo < re; lo++) {
    const uint2 kv = rec[lo];
    if (kv.x >= k1) break;
    const uint32_t at = (kv.x - k0) >> 1;
#pragma unroll
    for (uint32_t i = 0; i < 16; i++)
      if (i == at && !(kv.x & 1u)) q[i] = (int32_t)kv.y;
  }
}

// The 16 k of thread t's row piece to the block's rows in shared memory: 16-byte chunk c of
// piece R sits at c ^ ((R >> 1) & 3), so that eight threads writing their pieces touch all
// banks; element e of the block (16 R + its place in the piece) is at swz_k(e).
__device__ __forceinline__ uint32_t swz_k(uint32_t e) { return e ^ ((e >> 3) & 12u); }
__device__ __forceinline__ void st_piece(int32_t* s_k, const int32_t (&k)[16], int32_t add) {
  const uint32_t tid = threadIdx.x, key = (tid >> 1) & 3;
#pragma unroll
  for (uint32_t c = 0; c < 4; c++)
    reinterpret_cast<int4*>(s_k + 16 * tid)[c ^ key] =
        make_int4(k[4 * c] + add, k[4 * c + 1] + add, k[4 * c + 2] + add, k[4 * c + 3] + add);
}

// Block b from its codes (or runs) to the output: outliers, partial sums within the Lorenzo
// chunks (Sec. IV-B2), scaled; then the verbatim patches.  (The caller has checked the
// field's status, the same way in every thread.)
template <int ND, typename E>
__device__ void reconstruct_body(const DecodeArgs& a, uint32_t b, RebuildSmem& S) {
  const uint32_t tid = threadIdx.x;
  uint32_t org[3], w[3];
  block_box(a.g, b, org, w);
  const uint32_t m = w[0] * w[1] * w[2];
  const int32_t r = (int32_t)a.radius;
  const Out<E> out(a);
  const RowPiece p = row_piece<ND>(w);
  const int codec = a.ar[a.off_codec + b];
  int32_t q[16];
  if (codec == CODEC_RLE || codec == CODEC_RLE_HUFF) {
    uint32_t c[8];
    if (!expand_runs(a, b, codec, m, S, c)) return;
    if (ND == 1 || m == (uint32_t)kSlots) {
#pragma unroll
      for (int i = 0; i < 8; i++) {
        q[2 * i] = (int32_t)(c[i] & 0xffffu) - r;
        q[2 * i + 1] = (int32_t)(c[i] >> 16) - r;
      }
    } else {  // slots to row pieces
      uint16_t* s_c = reinterpret_cast<uint16_t*>(S.k);
      reinterpret_cast<uint4*>(s_c)[2 * tid] = make_uint4(c[0], c[1], c[2], c[3]);
      reinterpret_cast<uint4*>(s_c)[2 * tid + 1] = make_uint4(c[4], c[5], c[6], c[7]);
      __syncthreads();
#pragma unroll
      for (uint32_t i = 0; i < 16; i++) q[i] = i < p.n ? (int32_t)s_c[p.j0 + i] - r : 0;
      __syncthreads();
    }
  } else {
    load_codes16(a.codes + (uint64_t)b * kSlots, p.j0, p.n, r, q);
  }
  overlay_outliers(a, b, p.j0, p.n, q);
  // sums along x: chunks of 256 (16 threads), 16 or 8
#pragma unroll
  for (int i = 1; i < 16; i++)
    if (ND != 3 || (i & 7)) q[i] += q[i - 1];
  int32_t before = 0;
  if (ND == 1) {
    int32_t t = q[15];
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
      const int32_t u = __shfl_up_sync(~0u, t, o, 16);
      if ((tid & 15) >= (uint32_t)o) t += u;
    }
    before = t - q[15];
  }
  st_piece(S.k, q, before);
  __syncthreads();
  const uint64_t ny = a.g.n[1], nx = a.g.n[2];
  if (ND == 1) {
    if (m == (uint32_t)kSlots && out.vec4(org[2])) {
#pragma unroll
      for (uint32_t i = 0; i < 4; i++) {
        const uint32_t e = 4 * (tid + kRecThreads * i);
        out.put4((uint64_t)org[2] + e, *reinterpret_cast<const int4*>(S.k + swz_k(e)));
      }
    } else {
#pragma unroll 4
      for (uint32_t i = 0; i < 16; i++) {
        const uint32_t e = tid + kRecThreads * i;
        if (e < m) out.put((uint64_t)org[2] + e, S.k[swz_k(e)]);
      }
    }
  } else if (ND == 2) {
    // column x of the 16-row chunk band
    const uint32_t x = tid & 63, y0 = 16 * (tid >> 6);
    if (x < w[2]) {
      const uint64_t base = (uint64_t)(org[1] + y0) * nx + org[2] + x;
      int32_t acc = 0;
#pragma unroll
      for (uint32_t i = 0; i < 16; i++) {
        acc += S.k[swz_k((y0 + i) * 64 + x)];
        if (y0 + i < w[1]) out.put(base + i * nx, acc);
      }
    }
  } else {
    // columns along z in place, then along y
    const uint32_t x = tid & 15, h = tid >> 4;
    {
      int32_t acc = 0;
#pragma unroll
      for (uint32_t z = 0; z < 16; z++) {
        int32_t& k = S.k[swz_k((z * 16 + h) * 16 + x)];
        acc = (z & 7) ? acc + k : k;
        k = acc;
      }
    }
    __syncthreads();
    if (x < w[2] && h < w[0]) {
      const uint64_t base = ((uint64_t)(org[0] + h) * ny + org[1]) * nx + org[2] + x;
      int32_t acc = 0;
#pragma unroll
      for (uint32_t y = 0; y < 16; y++) {
        const int32_t k = S.k[swz_k((h * 16 + y) * 16 + x)];
        acc = (y & 7) ? acc + k : k;
        if (y < w[1]) out.put(base + y * nx, acc);
      }
    }
  }
  // verbatim patches overwrite their elements (ordered after the block's stores)
  const uint32_t rs = a.rec_start[b], re = a.rec_start[b + 1];
  if (rs == re) return;
  __syncthreads();
  const uint2* rec = reinterpret_cast<const uint2*>(a.ar + a.off_rec);
  for (uint32_t i = rs + tid; i < re; i += kRecThreads) {
    const uint2 kv = rec[i];
    if (kv.x & 1u) {
      const uint32_t j = (kv.x >> 1) % kSlots;
      const uint32_t pl = w[1] * w[2];
      const uint32_t zz = j / pl, rem = j - zz * pl, yy = rem / w[2], xx = rem - yy * w[2];
      out.patch(((uint64_t)(org[0] + zz) * ny + (org[1] + yy)) * nx + org[2] + xx, kv.y);
    }
  }
}

// One CTA per listed block (the set-up's list: run blocks and cut blocks).
template <int ND, typename E>
__global__ __launch_bounds__(kRecThreads, 6) void reconstruct_kernel(DecodeArgs a) {
  chained_begin();
  __shared__ __align__(16) RebuildSmem S;
  if (a.dead) return;
  // the status is read once, by thread 0 (run expansions in other CTAs may flag
  // corruption meanwhile), so every thread takes the same path
  if (threadIdx.x == 0) S.go = !undecodable(a.st->status) && blockIdx.x < a.st->n_slow;
  __syncthreads();
  if (!S.go) return;
  reconstruct_body<ND, E>(a, a.slowblk[blockIdx.x], S);
}

// =================================================================================
// global (unchunked) Lorenzo reconstruction: the N-D partial sum of q' over the whole
// field (Sec. IV-B "Partial-Sum Lorenzo Reconstruction" holds without chunks).
//
// Bound by memory: the codes are read and the field written, and every full-size pass in
// between costs as much again.  A pass per axis (q' written out, then a scan along x, y
// and z, each reading and writing the field) took 296 us at 3-D 100x500x500, 143 of them
// in the x scan's serial 4-byte loads.  Now only sums cross blocks: each block's row sums
// (1/16 of the field) are scanned along x, each block forms the partial sums along x and
// y of its own rows, with the row's sum before it, in shared memory and writes them once,
// the strips' last rows (1/16 of the field) are scanned along y, and the last pass adds
// those on its way along z: 95 us.  1-D fields take one pass with a look-back.
// =================================================================================

// q' (q - r, or the outlier's delta) of a row piece of block b.
__device__ __forceinline__ void load_fused16(const DecodeArgs& a, uint32_t b, uint32_t j0, uint32_t n,
                                             int32_t (&q)[16]) {
  load_codes16(a.codes + (uint64_t)b * kSlots, j0, n, (int32_t)a.radius, q);
  overlay_outliers(a, b, j0, n, q);
}

// The word of block bx (along x) and row (of the field's rows) in gtotals.
__device__ __forceinline__ uint64_t total_at(const DecodeArgs& a, uint32_t bx, uint64_t row, uint64_t nrows) {
  return a.gpitch ? row * a.gpitch + bx : bx * nrows + row;
}

// Sums of the block's rows.
template <int ND>
__global__ __launch_bounds__(kRecThreads) void grow_totals_kernel(DecodeArgs a) {
  chained_begin();
  if (a.dead || undecodable(a.st->status)) return;
  const uint32_t b = blockIdx.x;
  uint32_t org[3], w[3];
  block_box(a.g, b, org, w);
  const RowPiece p = row_piece<ND>(w);
  int32_t q[16], sum = 0;
  load_fused16(a, b, p.j0, p.n, q);
#pragma unroll
  for (int i = 0; i < 16; i++) sum += q[i];
  if (ND == 2) {
    sum += __shfl_xor_sync(~0u, sum, 1);
    sum += __shfl_xor_sync(~0u, sum, 2);
  }
  const uint64_t nrows = (uint64_t)a.g.n[0] * a.g.n[1];
  if (p.valid && (ND == 3 || (threadIdx.x & 3) == 0))
    a.gtotals[total_at(a, b % a.g.g[2], (uint64_t)(org[0] + p.z) * a.g.n[1] + org[1] + p.y, nrows)] = sum;
}

// Row sums to the sums before each block, in place (a thread per row).
__global__ __launch_bounds__(256) void gx_carry_kernel(DecodeArgs a) {
  chained_begin();
  if (a.dead || undecodable(a.st->status)) return;
  const uint64_t nrows = (uint64_t)a.g.n[0] * a.g.n[1];
  const uint64_t row = blockIdx.x * 256ull + threadIdx.x;
  if (row >= nrows) return;
  const uint32_t nb = a.g.g[2];
  int32_t* t = a.gtotals + row;
  int32_t acc = 0;
  for (uint32_t i = 0; i < nb; i += 8) {
    int32_t v[8];
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) v[k] = i + k < nb ? t[(i + k) * nrows] : 0;
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) {
      if (i + k < nb) t[(i + k) * nrows] = acc;
      acc += v[k];
    }
  }
}

// The same, a CTA per row and eight blocks a thread, the row's words side by side: for fields
// much wider than they have rows, where a thread per row walks along x alone (4 x 4 x 1 M
// elements: 2239 -> 17 us of a decompression that takes 2708 -> 368 us; 16 x 1.5 M: 842 us).
__global__ __launch_bounds__(1024) void gx_carry_wide_kernel(DecodeArgs a) {
  chained_begin();
  __shared__ int32_t s_scan[33];
  if (a.dead || undecodable(a.st->status)) return;
  const uint32_t nb = a.g.g[2];
  int4* t = reinterpret_cast<int4*>(a.gtotals + blockIdx.x * a.gpitch);
  int32_t carry = 0;
  for (uint32_t i0 = 0; i0 < nb; i0 += 8 * blockDim.x) {
    // (what lies between the row's end and its pitch comes behind every sum that is used)
    const uint32_t i = i0 + 8 * threadIdx.x;
    int4 v = make_int4(0, 0, 0, 0), w = v;
    if (i < nb) v = t[i / 4];
    if (i + 4 < nb) w = t[i / 4 + 1];
    int32_t all;
    const int32_t s0 = carry + block_excl_scan<int32_t>(v.x + v.y + v.z + v.w + w.x + w.y + w.z + w.w, s_scan, &all);
    const int32_t s1 = s0 + v.x + v.y + v.z + v.w;
    if (i < nb) t[i / 4] = make_int4(s0, s0 + v.x, s0 + v.x + v.y, s0 + v.x + v.y + v.z);
    if (i + 4 < nb) t[i / 4 + 1] = make_int4(s1, s1 + w.x, s1 + w.x + w.y, s1 + w.x + w.y + w.z);
    carry += all;
  }
}

// Partial sums along x, over the whole row, and along y, within the block, of one block.
template <int ND>
__global__ __launch_bounds__(kRecThreads) void gblock_kernel(DecodeArgs a) {
  chained_begin();
  __shared__ __align__(16) int32_t s_k[kSlots];
  __shared__ int32_t s_band[4][64];
  if (a.dead || undecodable(a.st->status)) return;
  const uint32_t b = blockIdx.x, tid = threadIdx.x;
  uint32_t org[3], w[3];
  block_box(a.g, b, org, w);
  const uint64_t ny = a.g.n[1], nx = a.g.n[2], nrows = (uint64_t)a.g.n[0] * ny;
  const RowPiece p = row_piece<ND>(w);
  int32_t k[16];
  load_fused16(a, b, p.j0, p.n, k);
  int32_t carry =
      p.valid ? a.gtotals[total_at(a, b % a.g.g[2], (uint64_t)(org[0] + p.z) * ny + org[1] + p.y, nrows)] : 0;
#pragma unroll
  for (int i = 1; i < 16; i++) k[i] += k[i - 1];
  if (ND == 2) {
    // the row's earlier pieces
    const int32_t u1 = __shfl_up_sync(~0u, k[15], 1, 4), u2 = __shfl_up_sync(~0u, k[15], 2, 4),
                  u3 = __shfl_up_sync(~0u, k[15], 3, 4);
    const uint32_t at = tid & 3;
    carry += (at >= 1 ? u1 : 0) + (at >= 2 ? u2 : 0) + (at >= 3 ? u3 : 0);
  }
  st_piece(s_k, k, carry);
  __syncthreads();
  auto at = [&](uint32_t e) -> int32_t { return s_k[swz_k(e)]; };
  int32_t* q = reinterpret_cast<int32_t*>(a.out);
  if (ND == 3) {
    const uint32_t x = tid & 15, z = tid >> 4;
    if (x < w[2] && z < w[0]) {
      int32_t* o = q + ((uint64_t)(org[0] + z) * ny + org[1]) * nx + org[2] + x;
      int32_t acc = 0;
#pragma unroll
      for (uint32_t y = 0; y < 16; y++) {
        acc += at((z * 16 + y) * 16 + x);
        if (y < w[1]) o[y * nx] = acc;
      }
    }
  } else {
    // column x, rows 16 band .. 16 band + 15; bands chain through their sums
    const uint32_t x = tid & 63, band = tid >> 6;
    int32_t v[16], sum = 0;
#pragma unroll
    for (uint32_t i = 0; i < 16; i++) {
      const uint32_t y = 16 * band + i;
      sum += y < w[1] ? at(y * 64 + x) : 0;
      v[i] = sum;
    }
    s_band[band][x] = sum;
    __syncthreads();
    int32_t before = 0;
    for (uint32_t i = 0; i < band; i++) before += s_band[i][x];
    if (x < w[2]) {
      int32_t* o = q + (uint64_t)(org[1] + 16 * band) * nx + org[2] + x;
#pragma unroll
      for (uint32_t i = 0; i < 16; i++)
        if (16 * band + i < w[1]) o[i * nx] = v[i] + before;
    }
  }
}

// Strips of block height along y: the sums before each strip, from the last row of the
// strips before it (a thread per plane and column): gstrips[(z gy + by) nx + x].
__global__ __launch_bounds__(256) void gy_carry_kernel(DecodeArgs a) {
  chained_begin();
  if (a.dead || undecodable(a.st->status)) return;
  const uint64_t nz = a.g.n[0], ny = a.g.n[1], nx = a.g.n[2];
  const uint64_t c = blockIdx.x * 256ull + threadIdx.x;
  if (c >= nz * nx) return;
  const uint64_t z = c / nx, x = c - z * nx;
  const uint32_t gy = a.g.g[1], h = a.g.blk[1];
  const int32_t* q = reinterpret_cast<const int32_t*>(a.out) + (z * ny + h - 1) * nx + x;
  int32_t* o = a.gstrips + z * gy * nx + x;
  int32_t acc = 0;
  o[0] = 0;
  for (uint32_t i = 0; i + 1 < gy; i += 8) {
    int32_t v[8];
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) v[k] = i + k + 1 < gy ? q[(uint64_t)(i + k) * h * nx] : 0;
#pragma unroll
    for (uint32_t k = 0; k < 8; k++) {
      acc += v[k];
      if (i + k + 1 < gy) o[(uint64_t)(i + k + 1) * nx] = acc;
    }
  }
}

// The last pass, in place: the strips' sums added, partial sums along z (a thread per
// column; 2-D fields have one plane), scaled.
__global__ __launch_bounds__(256) void gfinal_kernel(DecodeArgs a) {
  chained_begin();
  if (a.dead || undecodable(a.st->status)) return;
  const uint64_t nz = a.g.n[0], ny = a.g.n[1], nx = a.g.n[2];
  const uint64_t c = blockIdx.x * 256ull + threadIdx.x;
  if (c >= ny * nx) return;
  const uint64_t y = c / nx, x = c - y * nx;
  const uint32_t gy = a.g.g[1];
  float* out = a.out + c;
  const int32_t* q = reinterpret_cast<const int32_t*>(out);
  const int32_t* st = a.gstrips + (y / a.g.blk[1]) * nx + x;
  const uint64_t plane = ny * nx, splane = (uint64_t)gy * nx;
  const float ebx2 = a.ebx2_f;
  int32_t acc = 0;
  uint64_t z = 0;
  for (; z + 8 <= nz; z += 8) {
    int32_t v[8];
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = q[(z + i) * plane] + st[(z + i) * splane];
#pragma unroll
    for (int i = 0; i < 8; i++) {
      acc += v[i];
      __stcs(&out[(z + i) * plane], scale(acc, ebx2));
    }
  }
  for (; z < nz; z++) {
    acc += q[z * plane] + st[z * splane];
    __stcs(&out[z * plane], scale(acc, ebx2));
  }
}

// Exclusive prefix of the tiles before `tile`: the aggregates back to the nearest tile
// that published an inclusive value, summed modulo 2^62 and read back as a signed value.
// One full warp calls; the wait is bounded (ERR_TIMEOUT and 0 on expiry).
__device__ int64_t signed_lookback_warp(const uint64_t* state, uint32_t tile, uint32_t* status, uint32_t spin_limit) {
  const int lane = threadIdx.x & 31;
  if (tile == 0) return 0;
  uint64_t excl = 0;
  int64_t base = (int64_t)tile - 1;
  uint32_t spins = 0;
  while (true) {
    const int64_t idx = base - lane;
    const uint64_t v = idx >= 0 ? ld_relaxed(&state[idx]) : LB_INC;
    const uint32_t inc = __ballot_sync(~0u, (v & LB_INC) != 0);
    const uint32_t bad = __ballot_sync(~0u, (v & (LB_INC | LB_AGG)) == 0);
    const int first = inc ? __ffs(inc) : 32;
    const uint32_t upto = first >= 32 ? ~0u : ((1u << first) - 1u);
    if (bad & upto) {
      if (++spins > spin_limit) {
        if (lane == 0) atomicOr(status, ERR_TIMEOUT);
        return 0;
      }
      __nanosleep(64);
      continue;
    }
    const uint64_t add = warp_sum(((1u << lane) & upto) ? (v & LB_VAL) : 0ull);
    excl = (excl + add) & LB_VAL;
    if (inc) break;
    base -= 32;
  }
  return (int64_t)(excl << 2) >> 2;
}

// 1-D fields: the inclusive scan of the whole field in one pass, one codec block (4096
// consecutive elements) per CTA in ticket order; blocks chain by decoupled look-back.
__global__ __launch_bounds__(256) void g1d_kernel(DecodeArgs a, uint64_t* state) {
  chained_begin();
  __shared__ uint32_t s_tile;
  __shared__ int s_go;
  __shared__ int32_t s_ws[8];
  __shared__ int32_t s_carry;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) {
    s_go = !undecodable(a.st->status);
    s_tile = atomicAdd(&a.st->ticket_construct, 1u);
  }
  __syncthreads();
  if (!s_go) return;  // every CTA leaves: no tile waits on another
  const uint32_t tile = s_tile;
  const uint64_t first = (uint64_t)tile * kSlots + 16u * tid;
  const uint32_t n = first < a.g.nelem ? (uint32_t)min((unsigned long long)16, (unsigned long long)(a.g.nelem - first)) : 0u;
  int32_t k[16];
  load_fused16(a, tile, 16u * tid, n, k);
#pragma unroll
  for (int i = 1; i < 16; i++) k[i] += k[i - 1];
  const int32_t incl = warp_incl_scan(k[15]);
  if (lane == 31) s_ws[wid] = incl;
  __syncthreads();
  int32_t pre = incl - k[15];
  for (int v = 0; v < wid; v++) pre += s_ws[v];
  if (wid == 0) {
    const int64_t total = (int64_t)warp_sum(lane < 8 ? s_ws[lane] : 0);
    if (lane == 0) st_relaxed(&state[tile], (tile == 0 ? LB_INC : LB_AGG) | ((uint64_t)total & LB_VAL));
    const int64_t c = signed_lookback_warp(state, tile, &a.st->status, kSpinLimit);
    if (lane == 0) {
      if (tile) st_relaxed(&state[tile], LB_INC | ((uint64_t)(c + total) & LB_VAL));
      s_carry = (int32_t)c;
    }
  }
  __syncthreads();
  pre += s_carry;
  float* out = a.out + first;
  if (n == 16 && ((uintptr_t)out & 15) == 0) {
#pragma unroll
    for (int i = 0; i < 4; i++)
      __stcs(reinterpret_cast<float4*>(out) + i,
             make_float4(scale(k[4 * i] + pre, a.ebx2_f), scale(k[4 * i + 1] + pre, a.ebx2_f),
                         scale(k[4 * i + 2] + pre, a.ebx2_f), scale(k[4 * i + 3] + pre, a.ebx2_f)));
  } else {
#pragma unroll
    for (uint32_t i = 0; i < 16; i++)
      if (i < n) out[i] = scale(k[i] + pre, a.ebx2_f);
  }
}

// The last pass of 2-D fields: a thread per column and eight rows (which lie in one strip).
__global__ __launch_bounds__(256) void gfinal_rows_kernel(DecodeArgs a) {
  chained_begin();
  if (a.dead || undecodable(a.st->status)) return;
  const uint32_t ny = a.g.n[1], nx = a.g.n[2], nxb = (nx + 255) / 256;
  const uint32_t y0 = 8 * (blockIdx.x / nxb), x = 256 * (blockIdx.x % nxb) + threadIdx.x;
  if (x >= nx) return;
  float* out = a.out + (uint64_t)y0 * nx + x;
  const int32_t* q = reinterpret_cast<const int32_t*>(out);
  const int32_t before = a.gstrips[(uint64_t)(y0 / a.g.blk[1]) * nx + x];
  int32_t v[8];
#pragma unroll
  for (uint32_t i = 0; i < 8; i++) v[i] = y0 + i < ny ? q[(uint64_t)i * nx] : 0;
#pragma unroll
  for (uint32_t i = 0; i < 8; i++)
    if (y0 + i < ny) __stcs(&out[(uint64_t)i * nx], scale(v[i] + before, a.ebx2_f));
}

// Verbatim patches (after the last pass).
__global__ void gpatch_kernel(DecodeArgs a) {
  chained_begin();
  if (a.dead || undecodable(a.st->status)) return;
  const uint2* rec = reinterpret_cast<const uint2*>(a.ar + a.off_rec);
  const uint64_t ny = a.g.n[1], nx = a.g.n[2];
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < a.n_rec; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint2 kv = rec[i];
    if ((kv.x & 1u) == 0) continue;
    const uint32_t slot = kv.x >> 1, b = slot / kSlots, j = slot % kSlots;
    uint32_t org[3], w[3];
    block_box(a.g, b, org, w);
    const uint32_t pl = w[1] * w[2], zz = j / pl, rr = j - zz * pl, yy = rr / w[2], xx = rr - yy * w[2];
    a.out[((uint64_t)(org[0] + zz) * ny + (org[1] + yy)) * nx + org[2] + xx] = __uint_as_float(kv.y);
  }
}

// The global reconstruction's launches (after set-up, decoding and run expansion).
cudaError_t launch_global_reconstruct(DecodeArgs a, cudaStream_t s) {
  trace_begin(K_RECONSTRUCT, s);
  const int nd = a.g.ndim;
  const uint64_t nz = a.g.n[0], ny = a.g.n[1], nx = a.g.n[2];
  auto ctas = [](uint64_t threads) { return (unsigned)((threads + 255) / 256); };
  if (nd == 1) {
    launch_chained(g1d_kernel, a.g.nblk, 256, 0, s, a, a.scan_state);
  } else {
    // a block's CTA needs no more threads than the field's rows and columns have work for
    // (2-D: 64 columns by 16 rows a band, 3-D: 16 rows a plane)
    const unsigned threads = nd == 2 ? 64u * (unsigned)((imin(64, ny) + 15) / 16) : (16u * imin(16, nz) + 31u) & ~31u;
    // Row sums: a thread per row walks along its blocks alone, a CTA per row takes thousands at
    // a time but the SMs hold few of them (eight of 256 threads an SM, or two of 1024 for as few
    // rows).  A call with a thread and with a CTA per row: 16 rows of 40, 84 and 800 blocks 44 and
    // 45, 46 and 46, 70 and 46 us; 3000 rows of 40, 84 and 400 blocks 87 and 89, 127 and 124, 445
    // and 427 us; 8000 rows of 84 and 160 blocks 272 and 277, 530 and 531 us.  Hence the line.
    const uint64_t nrows = nz * ny;
    const bool wide = a.g.g[2] > 64 + nrows / 80;
    a.gpitch = wide ? (a.g.g[2] + 3ull) & ~3ull : 0;
    if (nd == 2) launch_chained(grow_totals_kernel<2>, a.g.nblk, threads, 0, s, a);
    else launch_chained(grow_totals_kernel<3>, a.g.nblk, threads, 0, s, a);
    if (wide)
      launch_chained(gx_carry_wide_kernel, (unsigned)nrows, nrows <= 2ull * sm_count() ? 1024 : 256, 0, s, a);
    else
      launch_chained(gx_carry_kernel, ctas(nrows), 256, 0, s, a);
    if (nd == 2) launch_chained(gblock_kernel<2>, a.g.nblk, threads, 0, s, a);
    else launch_chained(gblock_kernel<3>, a.g.nblk, threads, 0, s, a);
    launch_chained(gy_carry_kernel, ctas(nz * nx), 256, 0, s, a);
    if (nd == 2 && nx >= 256)
      launch_chained(gfinal_rows_kernel, (unsigned)((nx + 255) / 256 * ((ny + 7) / 8)), 256, 0, s, a);
    else
      launch_chained(gfinal_kernel, ctas(ny * nx), 256, 0, s, a);
  }
  trace_further(K_GLOBAL_PASSES, (nd == 1 ? 0 : 4) + (a.n_rec ? 1 : 0));
  if (a.n_rec) launch_chained(gpatch_kernel, (unsigned)((a.n_rec + 255) / 256 < 1024 ? (a.n_rec + 255) / 256 : 1024), 256, 0, s, a);
  trace_end(K_RECONSTRUCT, s);
  return cudaGetLastError();
}

// =================================================================================
// batches: device-side header checks and table-driven launches
// =================================================================================
__device__ __forceinline__ uint64_t dev_a8(uint64_t v) { return (v + 7) & ~7ull; }

// Reads field f's archive header on the device, checks it against the shape the
// batch was planned for (the same checks the single-field entry makes on the host)
// and completes the field's decode arguments; a failing header marks the field
// dead (every later stage skips it) and corrupt.
__global__ void dec_header_batch_kernel(DecodeArgs* tasks, int nfields) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= nfields) return;
  DecodeArgs& a = tasks[f];
  const Geom& g = a.g;
  bool ok = a.bytes >= (uint64_t)kHdr;
  uint64_t n_rec = 0, n_out = 0, n_patch = 0, payload = 0, total = 0, nblk = 0, dims[3] = {0, 0, 0};
  uint32_t magic = 0, radius = 0, lanes = 0, flags = 0;
  uint16_t version = 0;
  uint8_t ndim = 0, mode = 0;
  float eb_f = 0.0f;
  if (ok) {
    const uint8_t* h = a.ar;
    memcpy(&magic, h, 4);
    memcpy(&version, h + 4, 2);
    ndim = h[6];
    mode = h[7];
    memcpy(dims, h + 8, 24);
    memcpy(&eb_f, h + 48, 4);
    memcpy(&radius, h + 52, 4);
    memcpy(&lanes, h + 56, 4);
    memcpy(&flags, h + 60, 4);
    memcpy(&nblk, h + 64, 8);
    memcpy(&n_rec, h + 72, 8);
    memcpy(&n_out, h + 80, 8);
    memcpy(&n_patch, h + 88, 8);
    memcpy(&payload, h + 96, 8);
    memcpy(&total, h + 104, 8);
    memcpy(a.n_codec, h + 116, 12);
    ok = magic == kMagic && version == kVersion && ndim == g.ndim && mode <= 1;
    for (int d = 0; d < 3 && ok; d++) {
      const uint64_t want = d < g.ndim ? (uint64_t)g.n[3 - g.ndim + d] : 0ull;
      ok = dims[d] == want;
    }
    ok = ok && radius >= 1 && radius <= 512 && lanes == (uint32_t)kLanes && flags <= 3;
    ok = ok && nblk == g.nblk && n_rec == n_out + n_patch && eb_f > 0.0f && isfinite(2.0f * eb_f);
    ok = ok && n_rec <= 2 * g.nelem && payload <= a.bytes && (payload & 3) == 0;
    const uint64_t off_bb = kHdr + dev_a8(g.nblk);
    const uint64_t off_rec = off_bb + dev_a8(4ull * g.nblk);
    const uint64_t off_books = off_rec + 8 * n_rec + dev_a8(payload);
    const uint64_t want_total = off_books + ((flags & 1) ? kNsymCode : 0) + ((flags & 2) ? kNsymCode + kNsymLen : 0);
    ok = ok && total == want_total && total <= a.bytes;
    if (ok) {
      a.off_codec = kHdr;
      a.off_bb = off_bb;
      a.off_rec = off_rec;
      a.off_pay = off_rec + 8 * n_rec;
      a.off_books = off_books;
      a.n_rec = n_rec;
      a.payload = payload;
      a.flags = flags;
      a.radius = radius;
      a.ebx2_f = 2.0f * eb_f;
    }
  }
  a.dead = ok ? 0 : 1;
  if (!ok) atomicOr(&a.st->status, ERR_CORRUPT);
}

__device__ __forceinline__ int field_of(const uint32_t* prefix, int nfields, uint32_t c) {
  int lo = 0, hi = nfields - 1;  // last field with prefix[f] <= c
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= c) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// set-up: per field its prep chunks (one CTA per 1024 blocks, chained by look-back),
// 3 table CTAs, then its record CTAs (setup0 prefix)
__global__ __launch_bounds__(1024) void dec_setup_batch_kernel(const DecodeArgs* __restrict__ tasks,
                                                               const uint32_t* __restrict__ setup0, int nfields) {
  const int f = field_of(setup0, nfields, blockIdx.x);
  const DecodeArgs& a = tasks[f];
  const uint32_t role = blockIdx.x - setup0[f], nroles = setup0[f + 1] - setup0[f];
  const uint32_t nprep = (a.g.nblk + 1023) / 1024;
  if (role < nprep) dec_prep_chunk_body(a, nprep);
  else if (role < nprep + 3) dec_tables_body(a, (int)(role - nprep));
  else dec_records_body(a, role - nprep - 3, nroles - nprep - 3);
}

// entropy decoding: per field ceil(nblk / (rounds W / 2)) CTAs of W warps (W = blockDim.x /
// 32, chosen by the batch's tuner: 8, 16 or 32), whose warps draw the streams of the CTA's
// blocks one at a time; ND != 0 (the batch's common dimensionality): full Huffman blocks
// reconstructed in the decoding warps, as for single fields
template <int ND>
__global__ __launch_bounds__(1024) void stream_decode_batch_kernel(const DecodeArgs* __restrict__ tasks,
                                                                   const uint32_t* __restrict__ chunk0, int nfields,
                                                                   uint32_t rounds) {
  const int f = field_of(chunk0, nfields, blockIdx.x);
  const DecodeArgs& a = tasks[f];
  const uint32_t per = rounds * (blockDim.x / 64);  // blocks per CTA: two streams each
  const uint32_t b0 = (blockIdx.x - chunk0[f]) * per;
  const uint32_t b1 = min(a.g.nblk, b0 + per);
  stream_decode_body<ND, float>(a, b0, b1);
}

// Reconstruction of a batch, one CTA per codec block of every field.
__global__ __launch_bounds__(kRecThreads, 6) void reconstruct_batch_kernel(const DecodeArgs* __restrict__ tasks,
                                                                        const uint32_t* __restrict__ tile0, int nfields) {
  __shared__ __align__(16) RebuildSmem S;
  const int f = field_of(tile0, nfields, blockIdx.x);
  const DecodeArgs& a = tasks[f];
  const uint32_t b = blockIdx.x - tile0[f];
  if (a.dead) return;
  // full Huffman blocks were reconstructed by the decoding warps (fused batches)
  if (a.fuse && a.ar[a.off_codec + b] == CODEC_HUFF && block_is_full(a.g, b)) return;
  // the status is read once, by thread 0 (run expansions in other CTAs may flag
  // corruption meanwhile), so every thread takes the same path
  if (threadIdx.x == 0) S.go = !undecodable(a.st->status);
  __syncthreads();
  if (!S.go) return;
  if (a.g.ndim == 1) reconstruct_body<1, float>(a, b, S);
  else if (a.g.ndim == 2) reconstruct_body<2, float>(a, b, S);
  else reconstruct_body<3, float>(a, b, S);
}

cudaError_t launch_decode_batch(const DecodeBatchLaunch& L, cudaStream_t s) {
  cudaError_t e;
  trace_begin(K_DEC_HEADER, s);
  dec_header_batch_kernel<<<(L.nfields + 127) / 128, 128, 0, s>>>(L.tasks, L.nfields);
  trace_end(K_DEC_HEADER, s);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  trace_begin(K_DEC_SETUP, s);
  dec_setup_batch_kernel<<<L.nsetup, 1024, 0, s>>>(L.tasks, L.setup0, L.nfields);
  trace_end(K_DEC_SETUP, s);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int warps = L.warps ? L.warps : kStreamWarps;
  const size_t smem = stream_smem_bytes(3, warps);
  auto k = L.nd == 1 ? stream_decode_batch_kernel<1>
                     : (L.nd == 2 ? stream_decode_batch_kernel<2>
                                  : (L.nd == 3 ? stream_decode_batch_kernel<3> : stream_decode_batch_kernel<0>));
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  trace_begin(K_STREAM_DECODE, s);
  k<<<L.nchunks, 32 * warps, smem, s>>>(L.tasks, L.chunk0, L.nfields, L.rounds);
  trace_end(K_STREAM_DECODE, s);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // (run blocks are expanded inside the reconstruction)
  trace_begin(K_RECONSTRUCT, s);
  reconstruct_batch_kernel<<<L.ntiles, kRecThreads, 0, s>>>(L.tasks, L.tile0, L.nfields);
  trace_end(K_RECONSTRUCT, s);
  return cudaGetLastError();
}

// One bounded wait that nothing satisfies (a test aid for the failure path): which 0,
// the look-back of tile 1 behind a tile 0 that never publishes; which 1, an
// mbarrier phase no copy or arrival completes.  Either gives up after `spin_limit`
// tries and leaves ERR_TIMEOUT in the status, and the kernel returns normally.
__global__ void wait_selftest_kernel(int which, uint32_t spin_limit, uint64_t* lb, DevState* st) {
  __shared__ unsigned long long s_bar;
  if (which == 0) {
    if (threadIdx.x < 32) lookback_warp(lb, 1, 5, &st->status, spin_limit);
  } else if (which == 2) {
    // a field hand-over of the batched persistent kernel that no producer releases
    if (threadIdx.x == 0 && !wait_ge_acquire(&st->tiles_flushed, 1u, spin_limit)) atomicOr(&st->status, ERR_TIMEOUT);
  } else if (threadIdx.x == 0) {
    mbar_init(&s_bar);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!mbar_wait(&s_bar, 0, spin_limit)) atomicOr(&st->status, ERR_TIMEOUT);
  }
}

cudaError_t launch_wait_selftest(int which, uint32_t spin_limit, uint64_t* lb, DevState* st, cudaStream_t s) {
  wait_selftest_kernel<<<1, 32, 0, s>>>(which, spin_limit, lb, st);
  return cudaGetLastError();
}

__global__ void dec_status_kernel(const DevState* st, uint32_t* d_status) {
  chained_begin();
  *d_status = (uint32_t)fold(st->status);
}

cudaError_t launch_dec_status(const DevState* st, uint32_t* d_status, cudaStream_t s) {
  trace_begin(K_DEC_STATUS, s);
  launch_chained(dec_status_kernel, 1, 1, 0, s, st, d_status);
  trace_end(K_DEC_STATUS, s);
  return cudaGetLastError();
}

// The entropy decoding and reconstruction launches of one field, for element type E.
template <typename E>
cudaError_t launch_decode_stages(const DecodeArgs& a, cudaStream_t s) {
  const int nd = a.g.ndim;
  const int nluts = ((a.flags & 1u) ? 1 : 0) + ((a.flags & 2u) ? 2 : 0);
  if (nluts) {
    // warps per CTA: a stream is a chain of dependent steps, so a field with fewer streams
    // than the chip's SMs take at full occupancy spreads them over more, smaller CTAs
    // (each stages its own tables)
    auto k = nd == 1 ? stream_decode_kernel<1, E> : (nd == 2 ? stream_decode_kernel<2, E> : stream_decode_kernel<3, E>);
    const int sms = sm_count();
    const uint64_t streams = 2ull * a.g.nblk;
    const int wi = streams >= 32ull * sms ? 2 : (streams >= 8ull * sms ? 1 : 0);
    const int warps = 4 << wi;
    static_assert(kStreamWarps == 16, "4, 8 or 16 warps");
    const size_t smem = stream_smem_bytes(nluts, warps);
    static PerDevice occ[4][4][3];
    const int per_sm = occ[nd][nluts][wi].get(
        [&] { return allow_and_count(k, 32 * warps, smem, stream_smem_bytes(3, kStreamWarps)); });
    const uint64_t want = (streams + warps - 1) / warps;
    const uint64_t cap = (uint64_t)sms * per_sm;
    const unsigned grid = (unsigned)(want < cap ? want : cap);
    trace_begin(K_STREAM_DECODE, s);
    launch_chained(k, grid, 32 * warps, smem, s, a);
    trace_end(K_STREAM_DECODE, s);
  }
  const uint32_t nrun = a.n_codec[CODEC_RLE] + a.n_codec[CODEC_RLE_HUFF];
  if (a.global) {
    if (nrun) {
      trace_begin(K_RLE_EXPAND, s);
      launch_chained(rle_expand_kernel, nrun, kRecThreads, 0, s, a);
      trace_end(K_RLE_EXPAND, s);
    }
    return launch_global_reconstruct(a, s);
  }
  // blocks left to the reconstruction kernel: at most the cut blocks and the run blocks
  // (the header's counts, which the set-up checks); none, and the launch is skipped
  uint64_t full = 1;
  for (int d = 0; d < 3; d++) full *= a.g.n[d] / a.g.blk[d];
  uint64_t work = (a.g.nblk - full) + nrun;
  if (work > a.g.nblk) work = a.g.nblk;
  if (work) {
    auto k = nd == 1 ? reconstruct_kernel<1, E> : (nd == 2 ? reconstruct_kernel<2, E> : reconstruct_kernel<3, E>);
    trace_begin(K_RECONSTRUCT, s);
    launch_chained(k, (unsigned)work, kRecThreads, 0, s, a);
    trace_end(K_RECONSTRUCT, s);
  }
  return cudaGetLastError();
}

cudaError_t launch_decode(const DecodeArgs& a, cudaStream_t s) {
  const uint64_t n = (a.n_rec > (uint64_t)a.g.nblk + 1 ? a.n_rec : (uint64_t)a.g.nblk + 1);
  uint64_t rec_ctas = (n + 1023) / 1024;
  if (rec_ctas > 1024) rec_ctas = 1024;
  const uint32_t nchunks = (a.g.nblk + 1023) / 1024;
  trace_begin(K_DEC_SETUP, s);
  dec_setup_kernel<<<(unsigned)(nchunks + 3 + rec_ctas), 1024, 0, s>>>(a, nchunks);
  trace_end(K_DEC_SETUP, s);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return a.f64 ? launch_decode_stages<double>(a, s) : launch_decode_stages<float>(a, s);
}

}  // namespace cszp
