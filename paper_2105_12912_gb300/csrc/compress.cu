// Compression kernels of cszp (sm_103a).
//
// Pipeline (one stream, no host round trip until the end):
//   range_kernel / abs_params_kernel  value range (REL) and the FP32 error bound
//   construct_kernel (construct.cu,   prequant + chunk-local Lorenzo + postquant,
//     device code construct_body.cuh) record counts, bit words, residuals, histograms
//   codebook_kernel                   three canonical Huffman books; a fourth CTA
//                                     scans the blocks' record counts
//   plan_kernel                       per block: its records, exact sizes or heuristic /
//                                     MLP pick
//   payload_kernel                    per block: its place among the payloads, payload;
//                                     block 0: header, padding, books
//                                     (plan_rle_kernel, payload_rle_kernel: RLE forced)
// Batches run the same bodies either as one launch per stage (the *_batch kernels)
// or as the phases of one persistent kernel (batch_persistent_kernel).
#include "common.cuh"
#include "construct_body.cuh"
#include "kernels.h"

namespace cszp {

// =================================================================================
// value range and error bound
// =================================================================================

__device__ __forceinline__ uint32_t order_key(float f) {
  uint32_t b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float key_to_float(uint32_t k) {
  uint32_t b = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
  return __uint_as_float(b);
}

// ABS: eb_d = eb; REL: eb_d = eb * (max - min) in double.  eb_f = largest float <= eb_d,
// ebx2_f = 2 eb_f, ebx2_r = fl32(1 / (double)ebx2_f).  Degenerate bounds -> ERR_ARG.
__device__ void derive_eb(DevState* st, int mode, double eb, float vmin, float vmax) {
  double d = mode == 0 ? eb : eb * ((double)vmax - (double)vmin);
  float f = __double2float_rd(d);
  float x2 = 2.0f * f;
  float r = __double2float_rn(1.0 / (double)x2);
  st->eb_d = d;
  st->eb_f = f;
  st->ebx2_f = x2;
  st->ebx2_r = r;
  st->vmin = vmin;
  st->vmax = vmax;
  if (!(f > 0.0f) || !isfinite(x2) || !(r > 0.0f) || !isfinite(r)) atomicOr(&st->status, ERR_ARG);
}

__global__ void abs_params_kernel(DevState* st, double eb) {
  chained_begin();
  if (threadIdx.x == 0 && blockIdx.x == 0) derive_eb(st, 0, eb, 0.0f, 0.0f);
}

// Double-precision fields: eb_d as above (from the double range), the quantization
// step fl64(2 eb_d (1 - 2^-24)) and its inverse; eb_f is the largest float <= eb_d
// (informational, in the header).  Degenerate bounds -> ERR_ARG.
__device__ void derive_eb_d(DevState* st, int mode, double eb, double vmin, double vmax) {
  const double d = mode == 0 ? eb : __dmul_rn(eb, __dsub_rn(vmax, vmin));
  const double stp = __dmul_rn(__dmul_rn(2.0, d), kStepShrink);
  const double r = __ddiv_rn(1.0, stp);
  st->eb_d = d;
  st->eb_f = __double2float_rd(d);
  st->step_d = stp;
  st->rstep_d = r;
  if (!(d > 0.0) || !isfinite(d) || !(stp > 0.0) || !isfinite(stp) || !(r > 0.0) || !isfinite(r))
    atomicOr(&st->status, ERR_ARG);
}

__global__ void abs_params_d_kernel(DevState* st, double eb) {
  chained_begin();
  if (threadIdx.x == 0 && blockIdx.x == 0) derive_eb_d(st, 0, eb, 0.0, 0.0);
}

__device__ __forceinline__ unsigned long long order_key_d(double f) {
  const uint32_t hi = (uint32_t)__double2hiint(f), lo = (uint32_t)__double2loint(f);
  const uint32_t neg = (uint32_t)((int32_t)hi >> 31);  // all ones: every bit flips, else the sign
  return (unsigned long long)(hi ^ (neg | 0x80000000u)) << 32 | (lo ^ neg);
}
__device__ __forceinline__ double key_to_double(unsigned long long k) {
  return __longlong_as_double((long long)((k >> 63) ? (k & ~(1ull << 63)) : ~k));
}

// Min / max of a double field (grid-stride, 16-byte loads); the last CTA derives the
// bound and the step.
__global__ __launch_bounds__(256) void range_d_kernel(const double* __restrict__ x, uint64_t n, DevState* st,
                                                      int mode, double eb) {
  chained_begin();
  __shared__ unsigned long long s_red[2][33];
  __shared__ bool s_last;
  unsigned long long lo_inv = 0, hi = 0;
  uint32_t bad = 0;
  const uint64_t tid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  const uint64_t nth = (uint64_t)gridDim.x * blockDim.x;
  const bool vec = (((uintptr_t)x) & 15) == 0;
  const uint64_t nvec = vec ? n / 2 : 0;
  const double2* x2 = reinterpret_cast<const double2*>(x);
  // (integers only: one FP64 compare an element, at 2 a cycle and SM, took as long as the
  // field's bytes; and no branch: a non-finite value only has to be seen, the range of such a
  // field is not used.  3-D 256^3: 71 -> 39 -> 33 us)
  auto take = [&](double a) {
    const unsigned long long key = order_key_d(a);
    bad |= ((uint32_t)__double2hiint(a) & 0x7ff00000u) == 0x7ff00000u;
    lo_inv = max(lo_inv, ~key);
    hi = max(hi, key);
  };
  // four independent 16-byte loads in flight per thread per iteration
  uint64_t i = tid;
  for (; i + 3 * nth < nvec; i += 4 * nth) {
    const double2 v0 = __ldcs(&x2[i]), v1 = __ldcs(&x2[i + nth]), v2 = __ldcs(&x2[i + 2 * nth]),
                  v3 = __ldcs(&x2[i + 3 * nth]);
    take(v0.x);
    take(v0.y);
    take(v1.x);
    take(v1.y);
    take(v2.x);
    take(v2.y);
    take(v3.x);
    take(v3.y);
  }
  for (; i < nvec; i += nth) {
    const double2 v = __ldcs(&x2[i]);
    take(v.x);
    take(v.y);
  }
  for (uint64_t i = nvec * 2 + tid; i < n; i += nth) take(x[i]);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    lo_inv = max(lo_inv, __shfl_xor_sync(~0u, lo_inv, o));
    hi = max(hi, __shfl_xor_sync(~0u, hi, o));
  }
  bad = __any_sync(~0u, bad);
  if (lane == 0) {
    s_red[0][wid] = lo_inv;
    s_red[1][wid] = hi;
  }
  if (bad && lane == 0) atomicOr(&st->status, ERR_NONFINITE);
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long a = 0, b = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
      a = max(a, s_red[0][w]);
      b = max(b, s_red[1][w]);
    }
    atomicMax(&st->range64_lo_inv, a);
    atomicMax(&st->range64_hi, b);
    __threadfence();
    s_last = atomicAdd(&st->range_done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (s_last && threadIdx.x == 0) {
    __threadfence();
    const unsigned long long a = atomicAdd(&st->range64_lo_inv, 0ull);
    const unsigned long long b = atomicAdd(&st->range64_hi, 0ull);
    if (b == 0) {  // nothing finite was seen
      atomicOr(&st->status, ERR_NONFINITE);
      return;
    }
    derive_eb_d(st, mode, eb, key_to_double(~a), key_to_double(b));
  }
}

// Grid-stride min/max with float4 loads; non-finite values are flagged.  The last CTA
// to finish derives the error bound.
// ready (batched persistent kernel only, else nullptr): released as 1 by the last CTA
// once the bound is derived or found impossible.
__device__ __forceinline__ void range_body(const float* __restrict__ x, uint64_t n, DevState* st, int mode, double eb,
                           uint32_t cta, uint32_t nctas, uint32_t* ready = nullptr) {
  __shared__ uint32_t s_red[2][33];
  __shared__ bool s_last;
  uint32_t lo_inv = 0, hi = 0, bad = 0;
  const uint64_t tid = cta * (uint64_t)blockDim.x + threadIdx.x;
  const uint64_t nth = (uint64_t)nctas * blockDim.x;
  const bool vec = (((uintptr_t)x) & 15) == 0;
  uint64_t nvec = vec ? n / 4 : 0;
  const float4* x4 = reinterpret_cast<const float4*>(x);
  auto take = [&](float4 v) {
    const float a[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < 4; k++) {
      if (!isfinite(a[k])) {
        bad = 1;
      } else {
        const uint32_t key = order_key(a[k]);
        lo_inv = max(lo_inv, ~key);
        hi = max(hi, key);
      }
    }
  };
  // four independent 16-byte loads in flight per thread per iteration
  uint64_t i = tid;
  for (; i + 3 * nth < nvec; i += 4 * nth) {
    const float4 v0 = __ldcs(&x4[i]), v1 = __ldcs(&x4[i + nth]), v2 = __ldcs(&x4[i + 2 * nth]),
                 v3 = __ldcs(&x4[i + 3 * nth]);
    take(v0);
    take(v1);
    take(v2);
    take(v3);
  }
  for (; i < nvec; i += nth) take(__ldcs(&x4[i]));
  for (uint64_t i = nvec * 4 + tid; i < n; i += nth) {
    float a = x[i];
    if (!isfinite(a)) {
      bad = 1;
    } else {
      uint32_t key = order_key(a);
      lo_inv = max(lo_inv, ~key);
      hi = max(hi, key);
    }
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    lo_inv = max(lo_inv, __shfl_xor_sync(~0u, lo_inv, o));
    hi = max(hi, __shfl_xor_sync(~0u, hi, o));
  }
  bad = __any_sync(~0u, bad);
  if (lane == 0) {
    s_red[0][wid] = lo_inv;
    s_red[1][wid] = hi;
  }
  if (bad && lane == 0) atomicOr(&st->status, ERR_NONFINITE);
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t a = 0, b = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
      a = max(a, s_red[0][w]);
      b = max(b, s_red[1][w]);
    }
    atomicMax(&st->range_lo_inv, a);
    atomicMax(&st->range_hi, b);
    __threadfence();
    s_last = atomicAdd(&st->range_done, 1u) == nctas - 1;
  }
  __syncthreads();
  if (s_last && threadIdx.x == 0) {
    __threadfence();
    uint32_t a = atomicAdd(&st->range_lo_inv, 0u);
    uint32_t b = atomicAdd(&st->range_hi, 0u);
    if (b == 0) {  // nothing finite was seen
      atomicOr(&st->status, ERR_NONFINITE);
    } else {
      derive_eb(st, mode, eb, key_to_float(~a), key_to_float(b));
    }
    if (ready) release_flag(ready);
  }
}

__global__ __launch_bounds__(256) void range_kernel(const float* __restrict__ x, uint64_t n, DevState* st, int mode,
                                                    double eb) {
  chained_begin();
  range_body(x, n, st, mode, eb, blockIdx.x, gridDim.x);
}

// Batch: cta0[f] .. cta0[f+1]-1 are field f's CTAs; an ABS field has one CTA, which
// only derives the bound.
__global__ __launch_bounds__(256) void range_batch_kernel(const RangeTask* __restrict__ tasks,
                                                          const uint32_t* __restrict__ cta0, int nfields) {
  const uint32_t c = blockIdx.x;
  int lo = 0, hi = nfields - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (cta0[mid] <= c) lo = mid;
    else hi = mid - 1;
  }
  const RangeTask& t = tasks[lo];
  if (t.mode == 0) {
    if (threadIdx.x == 0) derive_eb(t.st, 0, t.eb, 0.0f, 0.0f);
    return;
  }
  range_body(t.x, t.n, t.st, t.mode, t.eb, c - cta0[lo], cta0[lo + 1] - cta0[lo]);
}


// =================================================================================
// canonical Huffman books (two-queue construction, Sec. II-A Step-6 via cuSZ)
// =================================================================================

constexpr int kBookThreads = 1024;

// Ascending sort of L distinct keys.  Warps first sort runs of 32 in registers (bitonic,
// by shuffles; no barrier), then runs merge: an element's place in the merged run is its
// index in its own run plus the number of smaller keys in the partner run (binary
// search).  a holds the keys on entry and on exit; b is scratch.  Both have room for L
// rounded up to 32.
__device__ void rank_merge_sort_u64(uint64_t* a, uint64_t* b, int L) {
  uint64_t* src = a;
  uint64_t* dst = b;
  const int lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < ((L + 31) & ~31); i += blockDim.x) {
    uint64_t k = i < L ? a[i] : ~0ull;
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
      for (int o = size >> 1; o; o >>= 1) {
        const uint64_t z = __shfl_xor_sync(~0u, k, o);
        const bool low = ((lane & o) == 0) == ((lane & size) == 0 || size == 32);
        k = (z < k) == low ? z : k;
      }
    }
    a[i] = k;
  }
  __syncthreads();
  for (int run = 32; run < L; run <<= 1) {
    for (int i = threadIdx.x; i < L; i += blockDim.x) {
      const uint64_t k = src[i];
      const int r = i / run;
      const int r0 = r * run;
      const bool left = (r & 1) == 0;
      const int p0 = left ? r0 + run : r0 - run;
      const int pn = left ? max(0, min(run, L - p0)) : run;
      int lo = 0, hi = pn;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (src[p0 + mid] < k) lo = mid + 1;
        else hi = mid;
      }
      dst[(left ? r0 : p0) + (i - r0) + lo] = k;
    }
    __syncthreads();
    uint64_t* t = src;
    src = dst;
    dst = t;
  }
  if (src != a) {
    for (int i = threadIdx.x; i < L; i += blockDim.x) a[i] = src[i];
    __syncthreads();
  }
}

// =================================================================================
// record offsets: exclusive prefix of the blocks' record counts (one CTA)
// =================================================================================
__device__ void record_offsets_body(const BookArgs& a) {
  __shared__ uint64_t s_scan[33];
  constexpr int kPerThread = 8;
  const int tid = threadIdx.x;
  const uint32_t nblk = a.nblk;
  uint64_t carry = 0;
  for (uint32_t base = 0; base < nblk; base += blockDim.x * kPerThread) {
    const uint32_t b0 = base + tid * kPerThread;
    uint32_t c[kPerThread];
    uint64_t mine = 0;
#pragma unroll
    for (int i = 0; i < kPerThread; i++) {
      const uint32_t v = b0 + i < nblk ? a.rec.counts[b0 + i] : 0u;
      c[i] = (v >> 16) + (v & 0xffffu);
      mine += c[i];
    }
    uint64_t agg;
    uint64_t off = carry + block_excl_scan<uint64_t>(mine, s_scan, &agg);
#pragma unroll
    for (int i = 0; i < kPerThread; i++) {
      if (b0 + i < nblk) a.rec.rec_off[b0 + i] = off;
      off += c[i];
    }
    carry += agg;
  }
}

// One CTA per book: 0 quant codes [1024], 1 run values [1024], 2 run lengths [4096].
// Working memory of one over nsym symbols: len nsym B | sym 2 nsym | parent by node
// 4 nsym | region A 8 nsym (sort keys, live node list, canonical scratch) | region B
// 8 nsym (sort scratch, new nodes, depth pass): 92 KB for the run lengths, two such CTAs
// an SM.
__host__ __device__ constexpr uint32_t book_mem_bytes(int nsym) { return 23u * (uint32_t)nsym; }

// Keys of live nodes: (weight, internal, node id), the order in which the sequential
// two-queue method picks them (weight, leaves before internal nodes, creation order).
constexpr uint64_t kNodeClass = 1ull << 13, kNodeId = kNodeClass - 1;

// Merging rounds of one warp (no barrier) over the sorted live list A[0..n) and the
// queue B[0..) of the nodes made here, which come in nondecreasing order: each round the
// warp takes the 32 lightest live nodes in order (the elementwise minimum of one list
// and the other reversed holds them as a bitonic sequence), and with t the sum of the
// two lightest merges every consecutive pair whose second member weighs <= t: those
// precede the node of weight t in the order above, so the sequential method would merge
// them too before it comes up again.  Node ids next, next + 1, ...  Returns the number
// of nodes made; *p_out, *q_out: the first live elements of A and B.  Stops when one
// node is left, or after kDenseRounds full rounds in a row.
//
// Bound by latency: about 400 cycles a round for up to 16 merges, where the two-queue
// method took one thread 190-220 cycles a merge (code histograms are sparse at their
// rare end, so few pairs qualify at a time and rounds of the whole CTA, 2500 cycles
// each, do not pay).  The launch with the 2-D 1800x3600 field's 1024-symbol book: 90 us
// before, 33 us so (a run of 324 symbols: 39 and 19 us).
constexpr int kDenseRounds = 12;
__device__ __forceinline__ int merge_warp(const uint64_t* A, int n, uint64_t* B, uint16_t* par, uint32_t next,
                                          int* p_out, int* q_out) {
  const int lane = threadIdx.x & 31;
  int p = 0, q = 0, e = 0, dense = 0;
  while (n - p + e - q > 1 && dense < kDenseRounds) {
    uint64_t x = p + lane < n ? A[p + lane] : ~0ull;
    const int j = q + 31 - lane;
    const uint64_t y = j < e ? B[j] : ~0ull;
    x = y < x ? y : x;
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const uint64_t z = __shfl_xor_sync(~0u, x, o);
      x = (z < x) == ((lane & o) == 0) ? z : x;
    }
    const uint64_t mate = __shfl_xor_sync(~0u, x, 1);
    const uint64_t sum = (x >> 14) + (mate >> 14);
    const uint64_t t = __shfl_sync(~0u, sum, 0);
    // (the pairs' heavier weights ascend: those within t are the first k)
    const int k = __popc(__ballot_sync(~0u, !(lane & 1) && mate != ~0ull && (mate >> 14) <= t));
    const bool in = lane < 2 * k;
    const uint32_t id = next + (uint32_t)(e + (lane >> 1));
    if (in) par[x & kNodeId] = (uint16_t)id;
    if (in && !(lane & 1)) B[e + (lane >> 1)] = (sum << 14) | kNodeClass | id;
    const int from_b = __popc(__ballot_sync(~0u, in && (uint32_t)(x & kNodeId) >= next));
    q += from_b;
    p += 2 * k - from_b;
    e += k;
    dense = k == 16 ? dense + 1 : 0;
    __syncwarp();
  }
  *p_out = p;
  *q_out = q;
  return e;
}

// One canonical book (role 0 code, 1 run value, 2 run length) or, role 3, the
// record offsets of a field, by a CTA of NT threads.  mem: book_mem_bytes(nsym) of
// working memory, shared (the book kernels) or global (the batched persistent
// kernel's run-length books).
template <int NT>
__device__ void codebook_core(const BookArgs& a, int role, unsigned char* mem) {
  if (role == 3) {
    record_offsets_body(a);
    return;
  }
  const int book = role;
  const int nsym = book == 2 ? kNsymLen : kNsymCode;
  const uint32_t* hist = book == 0 ? a.hist_code : (book == 1 ? a.hist_val : a.hist_len);
  uint8_t* len_out = a.lens + (book == 0 ? 0 : (book == 1 ? kNsymCode : 2 * kNsymCode));
  uint64_t* code_out = a.codes + (book == 0 ? 0 : (book == 1 ? kNsymCode : 2 * kNsymCode));
  uint32_t* packed_out = packed_books(a.codes) + (code_out - a.codes);

  uint8_t* s_len = mem;
  uint16_t* s_sym = reinterpret_cast<uint16_t*>(mem + nsym);
  uint16_t* s_par = reinterpret_cast<uint16_t*>(mem + 3 * nsym);
  uint64_t* A = reinterpret_cast<uint64_t*>(mem + 7 * nsym);
  uint64_t* B = reinterpret_cast<uint64_t*>(mem + 15 * nsym);
  __shared__ uint32_t s_L;
  __shared__ int s_n, s_k, s_next, s_p, s_q, s_e;
  __shared__ CanonSmem cs;
  const int tid = threadIdx.x;

  if (tid == 0) s_L = 0;
  for (int s = tid; s < nsym; s += blockDim.x) s_len[s] = 0;
  __syncthreads();
  // the symbols that occur, in any order (one counter update a warp)
#pragma unroll 4
  for (int s = tid; s < nsym; s += blockDim.x) {
    const uint32_t f = hist[s];
    const uint32_t has = __ballot_sync(~0u, f != 0);
    uint32_t at = 0;
    if ((tid & 31) == 0 && has) at = atomicAdd(&s_L, (uint32_t)__popc(has));
    at = __shfl_sync(~0u, at, 0) + __popc(has & ((1u << (tid & 31)) - 1u));
    if (f) A[at] = ((uint64_t)f << 12) | (uint64_t)s;
  }
  __syncthreads();
  const int L = (int)s_L;
  if (L == 1) {
    if (tid == 0) s_len[A[0] & 0xfff] = 1;
  } else if (L > 1) {
    // leaves in (frequency, symbol) order
    rank_merge_sort_u64(A, B, L);
    for (int i = tid; i < L; i += blockDim.x) {
      const uint64_t key = A[i];
      s_sym[i] = (uint16_t)(key & 0xfff);
      A[i] = ((key >> 12) << 14) | (uint64_t)i;
    }
    if (tid == 0) {
      s_n = L;
      s_next = L;
    }
    __syncthreads();
    const int nn = 2 * L - 1;
    // ---- merging rounds ----------------------------------------------------------
    // A round of the whole CTA merges every qualifying pair of the live list (the rule of
    // merge_warp) and rank-merges the new nodes back; it costs as much as six rounds of
    // one warp, so warp 0 goes alone unless kBlockPairs pairs qualify, and the CTA
    // rank-merges what it leaves in the same way.
    constexpr int kBlockPairs = 96;
    while (true) {
      const int n = s_n;
      if (n <= 1) break;
      const int next = s_next;
      if (tid < 32) {
        // qualifying pairs i, weight(A[2i+1]) <= t, up to kBlockPairs or, if that many, all
        const uint64_t t = (A[0] >> 14) + (A[1] >> 14);
        int k = 0;
        if (n >= 2 * kBlockPairs && (A[2 * kBlockPairs - 1] >> 14) <= t) {
          int lo = kBlockPairs, hi = n / 2;
          while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((A[2 * mid + 1] >> 14) <= t) lo = mid + 1;
            else hi = mid;
          }
          k = lo;
        } else {
          int p, q;
          const int e = merge_warp(A, n, B, s_par, (uint32_t)next, &p, &q);
          if (tid == 0) {
            s_p = p;
            s_q = q;
            s_e = e;
          }
        }
        if (tid == 0) s_k = k;
      }
      __syncthreads();
      const int k = s_k;
      // left over after the round: A[p..n) and the new nodes B[q..e)
      int p = 2 * k, q = 0, e = k;
      if (k) {
        for (int i = tid; i < k; i += blockDim.x) {
          const uint64_t x = A[2 * i], y = A[2 * i + 1];
          const uint64_t wn = (x >> 14) + (y >> 14);
          const uint32_t id = (uint32_t)next + i;
          s_par[x & kNodeId] = (uint16_t)id;
          s_par[y & kNodeId] = (uint16_t)id;
          B[i] = (wn << 14) | kNodeClass | id;
        }
        __syncthreads();
      } else {
        p = s_p;
        q = s_q;
        e = s_e;
      }
      const int na = n - p, live = na + e - q;
      if (live == 1) break;  // the root
      uint64_t mine[(kNsymLen + NT - 1) / NT];
      int dst[(kNsymLen + NT - 1) / NT], cnt = 0;
      for (int i = tid; i < live; i += blockDim.x) {
        const bool from_a = i < na;
        const uint64_t x = from_a ? A[p + i] : B[q + i - na];
        const uint64_t* other = from_a ? B + q : A + p;
        int lo = 0, hi = from_a ? e - q : na;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (other[mid] < x) lo = mid + 1;
          else hi = mid;
        }
        mine[cnt] = x;
        dst[cnt] = (from_a ? i : i - na) + lo;
        cnt++;
      }
      __syncthreads();
      for (int c = 0; c < cnt; c++) A[dst[c]] = mine[c];
      if (tid == 0) {
        s_n = live;
        s_next = next + e;
      }
      __syncthreads();
    }
    if (tid == 0) s_par[nn - 1] = (uint16_t)(nn - 1);
    __syncthreads();
    // depths by pointer jumping (region B): word i holds node i's ancestor and how far up
    // it is.  The words are updated in place: one that has already moved on this round
    // still names an ancestor and its distance.  Done once every ancestor is the root.
    volatile uint32_t* s_up = reinterpret_cast<uint32_t*>(B);
    for (int i = tid; i < nn; i += blockDim.x) s_up[i] = ((uint32_t)s_par[i] << 16) | (i == nn - 1 ? 0u : 1u);
    __syncthreads();
    bool open = true;
    while (__syncthreads_or(open)) {
      open = false;
      for (int i = tid; i < nn; i += blockDim.x) {
        const uint32_t w = s_up[i], u = s_up[w >> 16];
        const uint32_t v = (u & 0xffff0000u) | ((w & 0xffffu) + (u & 0xffffu));
        s_up[i] = v;
        open |= (v >> 16) != (uint32_t)(nn - 1);
      }
    }
    for (int i = tid; i < L; i += blockDim.x) {
      const uint32_t d = s_up[i] & 0xffffu;
      if (d > (uint32_t)kMaxLen) atomicOr(&a.st->status, ERR_RANGE);
      s_len[s_sym[i]] = (uint8_t)d;
    }
  }
  __syncthreads();
  for (int s = tid; s < nsym; s += blockDim.x) len_out[s] = s_len[s];
  canonical_build(s_len, nsym, &cs, reinterpret_cast<uint16_t*>(A), code_out, packed_out, nullptr);
}

__global__ __launch_bounds__(kBookThreads) void codebook_kernel(BookArgs a) {
  chained_begin();
  extern __shared__ __align__(16) unsigned char smem[];
  codebook_core<kBookThreads>(a, blockIdx.x, smem);
}

// Batch: four CTAs per field (three books and the record offsets).
__global__ __launch_bounds__(kBookThreads) void codebook_batch_kernel(const BookArgs* __restrict__ tasks) {
  extern __shared__ __align__(16) unsigned char smem[];
  codebook_core<kBookThreads>(tasks[blockIdx.x >> 2], blockIdx.x & 3, smem);
}

static size_t codebook_smem_bytes() { return book_mem_bytes(kNsymLen); }

// =================================================================================
// header, section padding and books
// =================================================================================
__device__ void finalize_body(const FinalizeArgs& a) {
  __shared__ uint32_t s_hdr[kHdr / 4];
  __shared__ uint64_t s_total, s_off_books, s_pay_end;
  __shared__ uint32_t s_flags;
  DevState* st = a.st;
  const int tid = threadIdx.x;
  if (tid == 0) {
    const uint64_t n_rec = st->n_rec, payload = st->payload;
    const uint32_t flags = (st->ncodec[CODEC_HUFF] ? 1u : 0u) | (st->ncodec[CODEC_RLE_HUFF] ? 2u : 0u) |
                           (a.f64 ? kFlagF64 : 0u) | (a.global ? kFlagGlobal : 0u);
    const uint64_t off_pay = a.off_rec + 8 * n_rec;
    const uint64_t off_books = off_pay + ((payload + 7) & ~7ull);
    const uint64_t total = off_books + ((flags & 1) ? kNsymCode : 0) + ((flags & 2) ? kNsymCode + kNsymLen : 0);
    s_total = total;
    s_off_books = off_books;
    s_pay_end = off_pay + payload;
    s_flags = flags;
    st->total = total;
    if (total > a.cap) atomicOr(&st->status, ERR_CAPACITY);
    for (int i = 0; i < kHdr / 4; i++) s_hdr[i] = 0;
    unsigned char* h = reinterpret_cast<unsigned char*>(s_hdr);
    auto put32 = [&](int off, uint32_t v) { memcpy(h + off, &v, 4); };
    auto put64 = [&](int off, uint64_t v) { memcpy(h + off, &v, 8); };
    put32(0, kMagic);
    h[4] = (unsigned char)(kVersion & 0xff);
    h[5] = (unsigned char)(kVersion >> 8);
    h[6] = (unsigned char)a.ndim;
    h[7] = (unsigned char)a.eb_mode;
    for (int i = 0; i < 3; i++) put64(8 + 8 * i, i < a.ndim ? a.dims[i] : 0ull);
    double eu = a.eb_user, ed = st->eb_d;
    memcpy(h + 32, &eu, 8);
    memcpy(h + 40, &ed, 8);
    float ef = st->eb_f;
    memcpy(h + 48, &ef, 4);
    put32(52, a.radius);
    put32(56, (uint32_t)kLanes);
    put32(60, flags);
    put64(64, a.nblk);
    put64(72, n_rec);
    put64(80, n_rec - st->n_patch);
    put64(88, st->n_patch);
    put64(96, payload);
    put64(104, total);
    put32(112, (uint32_t)a.select);
    for (int i = 0; i < 3; i++) put32(116 + 4 * i, st->ncodec[i]);
  }
  __syncthreads();
  if (s_total > a.cap) return;
  uint8_t* ar = a.ar;
  for (int i = tid; i < kHdr / 4; i += blockDim.x) {
    reinterpret_cast<uint32_t*>(ar)[i] = s_hdr[i];
    if (a.hdr_copy) a.hdr_copy[i] = s_hdr[i];
  }
  // zero padding: codec section, blk_bytes section, payload tail
  for (uint64_t i = kHdr + a.nblk + tid; i < a.off_bb; i += blockDim.x) ar[i] = 0;
  for (uint64_t i = a.off_bb + 4ull * a.nblk + tid; i < a.off_rec; i += blockDim.x) ar[i] = 0;
  for (uint64_t i = s_pay_end + tid; i < s_off_books; i += blockDim.x) ar[i] = 0;
  uint64_t o = s_off_books;
  if (s_flags & 1) {
    for (int i = tid; i < kNsymCode; i += blockDim.x) ar[o + i] = a.lens[i];
    o += kNsymCode;
  }
  if (s_flags & 2) {
    for (int i = tid; i < kNsymCode + kNsymLen; i += blockDim.x) ar[o + i] = a.lens[kNsymCode + i];
  }
}

// =================================================================================
// per-block selection and encoding
// =================================================================================
constexpr int kEncThreads = 256;
constexpr int kBufBytes = 16384;  // payload assembly buffer

// Learned pick from the network's three predictions (identical in every lane): the
// smallest (first index on ties), and whether the runner-up lies within the margin,
// in which case the caller decides by exact sizes.  Plain FP32 compares only.
__device__ __forceinline__ int learned_pick(const float* y, bool& fallback) {
  int c = 0;
  if (y[1] < y[c]) c = 1;
  if (y[2] < y[c]) c = 2;
  int r = -1;
#pragma unroll
  for (int k = 0; k < 3; k++)
    if (k != c && (r < 0 || y[k] < y[r])) r = k;
  const float gap = y[r] - y[c];
  fallback = gap < kMlpMargin;
  return c;
}

// The network's parameters staged in shared memory for one forward pass per block:
// the weight matrices transposed (the 32 lanes' weights for one input are consecutive
// words) and padded to 33 words per row, so each multiply-add step of the warp reads
// one conflict-free row instead of 32 scattered cache lines of the packed layout.
constexpr int kSwW1 = 0;                     // [8][33]  W1 transposed
constexpr int kSwB1 = kSwW1 + kMlpIn * 33;   // [32]
constexpr int kSwW2 = kSwB1 + kMlpHid;       // [32][33] W2 transposed
constexpr int kSwB2 = kSwW2 + kMlpHid * 33;  // [32]
constexpr int kSwW3 = kSwB2 + kMlpHid;       // [3][33]  W3 rows
constexpr int kSwB3 = kSwW3 + kMlpOut * 33;  // [3]
constexpr int kSwWords = kSwB3 + kMlpOut;

__device__ __forceinline__ void stage_mlp(const float* __restrict__ w, float* sw) {
  for (int i = threadIdx.x; i < kMlpParams; i += kEncThreads) {
    const float v = __ldg(&w[i]);
    int d;
    if (i < kMlpB1) {
      d = kSwW1 + (i % kMlpIn) * 33 + i / kMlpIn;
    } else if (i < kMlpW2) {
      d = kSwB1 + (i - kMlpB1);
    } else if (i < kMlpB2) {
      const int k = i - kMlpW2;
      d = kSwW2 + (k % kMlpHid) * 33 + k / kMlpHid;
    } else if (i < kMlpW3) {
      d = kSwB2 + (i - kMlpB2);
    } else if (i < kMlpB3) {
      const int k = i - kMlpW3;
      d = kSwW3 + (k / kMlpHid) * 33 + k % kMlpHid;
    } else {
      d = kSwB3 + (i - kMlpB3);
    }
    sw[d] = v;
  }
}

// mlp_forward_warp on the staged parameters: the same operands in the same order, so
// the same FP32 results.  f: the 8 features (same in every lane).
__device__ __forceinline__ void mlp_forward_staged(const float* sw, const float (&f)[kMlpIn], float* y) {
  const int lane = threadIdx.x & 31;
  float acc = sw[kSwB1 + lane];
#pragma unroll
  for (int j = 0; j < kMlpIn; j++) acc = fmaf(sw[kSwW1 + 33 * j + lane], f[j], acc);
  const float h1 = acc > 0.0f ? acc : 0.0f;
  acc = sw[kSwB2 + lane];
#pragma unroll
  for (int j = 0; j < kMlpHid; j++) acc = fmaf(sw[kSwW2 + 33 * j + lane], __shfl_sync(~0u, h1, j), acc);
  const float h2 = acc > 0.0f ? acc : 0.0f;
  const int o = lane < kMlpOut ? lane : 0;
  acc = sw[kSwB3 + o];
#pragma unroll
  for (int j = 0; j < kMlpHid; j++) acc = fmaf(sw[kSwW3 + 33 * o + j], __shfl_sync(~0u, h2, j), acc);
#pragma unroll
  for (int c = 0; c < kMlpOut; c++) y[c] = __shfl_sync(~0u, acc, c);
}

// smallest exact size; ties prefer HUFF, then RLE_HUFF, then RLE
__device__ __forceinline__ int exhaustive_pick(uint32_t sh, uint32_t sr, uint32_t srh) {
  int c = CODEC_HUFF;
  uint32_t best = sh;
  if (srh < best) {
    c = CODEC_RLE_HUFF;
    best = srh;
  }
  if (sr < best) c = CODEC_RLE;
  return c;
}

static_assert(kEncThreads % kMadoN == 0, "madogram distances by thread");

// Block b's outlier and patch records, in slot order, at its record offset (all threads;
// not inlined: few blocks have any, and the registers are the payload's).
__device__ __noinline__ void place_records(const EncodeArgs& a, uint32_t b, const uint32_t* org, const uint32_t* w,
                                           uint64_t* s_scan64) {
  const uint32_t tid = threadIdx.x;
  const RecordArgs& R = a.rec;
  const uint32_t lo = tid * 16;
  const uint32_t* mw = R.masks + (uint64_t)b * kMaskWords;
  const uint32_t pb = (mw[lo >> 5] >> (lo & 31)) & 0xffffu;
  const uint32_t ob = (mw[128 + (lo >> 5)] >> (lo & 31)) & 0xffffu;
  uint64_t pos = R.rec_off[b] + block_excl_scan<uint64_t>((uint64_t)(__popc(ob) + __popc(pb)), s_scan64, nullptr);
  if (ob | pb) {
    const int32_t* dl = R.deltas + (uint64_t)b * kSlots;
    const uint64_t ny = a.g.n[1], nx = a.g.n[2];
    uint32_t err = 0;
    for (int i = 0; i < 16; i++) {
      const uint32_t j = lo + i;
      const uint32_t slot2 = (b * (uint32_t)kSlots + j) * 2u;
      if ((ob >> i) & 1u) {
        if (pos < R.rec_cap) reinterpret_cast<uint2*>(R.rec)[pos] = make_uint2(slot2, (uint32_t)dl[j]);
        else err |= ERR_CAPACITY;
        pos++;
      }
      if ((pb >> i) & 1u) {
        uint32_t zz = 0, yy = 0, xx = j;
        if (a.g.ndim == 2) {
          yy = j / w[2];
          xx = j - yy * w[2];
        } else if (a.g.ndim == 3) {
          const uint32_t pl = w[1] * w[2];
          zz = j / pl;
          const uint32_t rr = j - zz * pl;
          yy = rr / w[2];
          xx = rr - yy * w[2];
        }
        const uint64_t e = ((uint64_t)(org[0] + zz) * ny + (org[1] + yy)) * nx + (org[2] + xx);
        if (pos < R.rec_cap) reinterpret_cast<uint2*>(R.rec)[pos] = make_uint2(slot2 + 1u, __float_as_uint(R.x[e]));
        else err |= ERR_CAPACITY;
        pos++;
      }
    }
    if (err) atomicOr(&a.st->status, err);
  }
}

// The runs of a block: their values and starts, in order, from its codes and the run starts
// that construction left as bits.  A thread takes 16 consecutive codes; runs before them are
// counted in the bit words, which every warp reads for itself.  All threads; a barrier
// follows at the caller.
__device__ __forceinline__ void scatter_runs(const uint16_t* codes, const uint32_t* heads, uint16_t* s_at,
                                             uint16_t* s_rv) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const uint4* src = reinterpret_cast<const uint4*>(codes + 16 * tid);
  const uint4 c0 = __ldcg(&src[0]), c1 = __ldcg(&src[1]), w4 = __ldcg(&reinterpret_cast<const uint4*>(heads)[lane]);
  const uint32_t hb = (__ldcg(&heads[tid >> 1]) >> (16 * (tid & 1))) & 0xffffu;
  const uint32_t c[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
  const uint32_t n4 = __popc(w4.x) + __popc(w4.y) + __popc(w4.z) + __popc(w4.w), n = __popc(hb);
  uint32_t run = __reduce_add_sync(~0u, lane < 4 * wid ? n4 : 0u) + warp_incl_scan(n) - n;
#pragma unroll
  for (uint32_t i = 0; i < 16; i++) {
    if ((hb >> i) & 1u) {
      s_rv[run] = (uint16_t)(c[i >> 1] >> (16 * (i & 1)));
      s_at[run] = (uint16_t)(16 * tid + i);
      run++;
    }
  }
}

// Length of run i of nr in a block of m codes, the starts being at.
__device__ __forceinline__ uint32_t run_length(const uint16_t* at, uint32_t i, uint32_t nr, uint32_t m) {
  return (i + 1 < nr ? at[i + 1] : m) - at[i];
}

// The nr runs of a block: their values and lengths, with one barrier before the lengths and one
// after them.  s_at: scratch, the run starts.  (Finding the starts again from codes in shared
// memory took three more barriers, with one warp's index of the words between them: 40 mixed
// fields, most of their blocks in runs, compression 553 -> 511 us.)  All threads.
__device__ __noinline__ void extract_runs(const uint16_t* codes, const uint32_t* heads, uint32_t m, uint32_t nr,
                                          uint16_t* s_at, uint16_t* s_rv, uint16_t* s_rl) {
  const uint32_t tid = threadIdx.x;
  scatter_runs(codes, heads, s_at, s_rv);
  __syncthreads();
  for (uint32_t i = tid; i < nr; i += kEncThreads) s_rl[i] = (uint16_t)run_length(s_at, i, nr, m);
  __syncthreads();
}

// Encoding takes two launches (or phases): the plan of every block -- records, runs,
// statistics, exact sizes, the pick -- then, when every size is known, the payloads.  One
// launch with a decoupled look-back for the payload offsets held a CTA's place on its SM
// until the slowest of the hundreds of blocks before it had its size, half of the time it
// was resident (100x500x500 learned: 176 us with the look-back, 96 us with made-up
// offsets).  Now the plan adds each block's size to its group's total and a payload CTA
// sums what precedes it, with nothing to wait for; the codes are read twice for it.
// 3-D 512^3: 525 -> 390 us for both.
//
// Groups of kGroup blocks: one 64-bit total each, payload bytes below bit 40, the numbers
// of RLE and of RLE+Huffman blocks from bits 40 and 52.
constexpr uint32_t kGroup = 256;
static_assert(kGroup == kEncThreads, "a thread per block of the group");
constexpr uint64_t kGroupBytes = (1ull << 40) - 1;

// The Huffman streams' symbols of this thread (pair_plan); kNsymCode behind the last.
struct HuffPart {
  const uint16_t* src;
  uint32_t n, steps, j0;
  bool full;
  __device__ __forceinline__ HuffPart(const uint16_t* codes, uint32_t m) {
    const uint32_t w = threadIdx.x >> 5, h = huff_split(m);
    n = w >> 2 ? m - h : h;
    steps = quarter_steps(n);
    j0 = 32 * (w & 3) * steps + (threadIdx.x & 31);
    src = codes + (w >> 2 ? h : 0u) + j0;
    full = m == (uint32_t)kSlots;
  }
  __device__ __forceinline__ void load(uint32_t (&sym)[16]) const {
    if (full) {
#pragma unroll
      for (uint32_t i = 0; i < 16; i++) sym[i] = __ldcg(&src[32 * i]);
    } else {
#pragma unroll
      for (uint32_t i = 0; i < 16; i++)
        sym[i] = i < steps && j0 + 32 * i < n ? (uint32_t)__ldcg(&src[32 * i]) : (uint32_t)kNsymCode;
    }
  }
};

// The code book's packed codes in shared memory, and an empty one for "no symbol" (a
// barrier follows at the caller)
__device__ __forceinline__ void stage_book(const EncodeArgs& a, uint32_t* s_tab) {
  reinterpret_cast<uint4*>(s_tab)[threadIdx.x] = __ldcg(&reinterpret_cast<const uint4*>(packed_books(a.bcodes))[threadIdx.x]);
  if (threadIdx.x == 0) s_tab[kNsymCode] = 0;
}

// P of the Huffman block whose symbols the thread holds.  Contains one barrier.
__device__ __forceinline__ void plan_huff(PairPlan& P, const EncodeArgs& a, const HuffPart& part, uint32_t (&sym)[16],
                                          const uint32_t* s_tab, uint32_t* s_part) {
  uint32_t cum = 0, odd = 0, longest = 0;
#pragma unroll
  for (int i = 0; i < 16; i++) {
    P.e[i] = s_tab[sym[i]];
    cum += P.e[i] & 31u;
    longest = max(longest, P.e[i] & 31u);
  }
  if (longest == kPackedLong) {
    part.load(sym);  // (again: not held for this rare case)
    odd = 1u << 31;
#pragma unroll
    for (int i = 0; i < 16; i++)
      if ((P.e[i] & 31u) == kPackedLong) cum += a.lens[sym[i]] - kPackedLong;
  }
  pair_plan(P, cum | odd, s_part);
}

// The runs of this thread (values or lengths) in an RLE+Huffman block of nr runs.
struct RunPart {
  const uint16_t* sy;
  const uint32_t* book;
  const uint8_t* lens;
  uint32_t which, steps, j0, nr;
  __device__ __forceinline__ RunPart(const EncodeArgs& a, const uint16_t* rv, const uint16_t* rl, uint32_t n) {
    which = threadIdx.x >> 7;
    nr = n;
    steps = quarter_steps(n);
    j0 = 32 * ((threadIdx.x >> 5) & 3) * steps + (threadIdx.x & 31);
    sy = which ? rl : rv;
    const uint32_t at = which ? 2 * kNsymCode : kNsymCode;
    book = packed_books(a.bcodes) + at;
    lens = a.lens + at;
  }
  // Packed codes of the steps from `first` on; returns their bits (odd: bit 31 set where a
  // code is not packed).
  __device__ __forceinline__ uint32_t load(uint32_t first, uint32_t (&e)[16], uint32_t& odd) const {
    uint32_t cum = 0;
#pragma unroll
    for (uint32_t i = 0; i < 16; i++) {
      const uint32_t j = j0 + 32 * (first + i);
      e[i] = 0;
      if (first + i < steps && j < nr) {
        const uint32_t sym = (uint32_t)sy[j] - which;  // (run lengths are coded less one)
        e[i] = book[sym];
        uint32_t L = e[i] & 31u;
        if (L == kPackedLong) {
          odd = 1u << 31;
          L = lens[sym];
        }
        cum += L;
      }
    }
    return cum;
  }
};

// P of an RLE+Huffman block's runs, with the codes of their first 16 steps.  Contains one
// barrier.
__device__ __forceinline__ void plan_runs(PairPlan& P, const RunPart& part, uint32_t* s_part) {
  uint32_t cum = 0, odd = 0;
#pragma unroll 1
  for (uint32_t first = part.steps > 16 ? 16u : 0u;; first -= 16) {  // (the later steps first)
    cum += part.load(first, P.e, odd);
    if (first == 0) break;
  }
  pair_plan(P, cum | odd, s_part);
}

// Payload bytes of a Huffman block (u16 unit count, both streams) and of an RLE+Huffman
// block (two words, both streams), from its plan
__device__ __forceinline__ uint32_t huff_bytes(const PairPlan& P) { return (2 * (1 + P.units_a + P.units_b) + 3) & ~3u; }
__device__ __forceinline__ uint32_t rlehuff_bytes(const PairPlan& P) { return (8 + 2 * (P.units_a + P.units_b) + 3) & ~3u; }

// Where the plan leaves the runs of a block that is coded by them: values, then lengths, in
// the block's outlier residuals, which its records no longer need.
__device__ __forceinline__ uint16_t* block_run_store(const EncodeArgs& a, uint32_t b) {
  return reinterpret_cast<uint16_t*>(const_cast<int32_t*>(a.rec.deltas) + (uint64_t)b * kSlots);
}

// The field's status as far as encoding goes by it.  An expired wait (ERR_TIMEOUT) may have
// left blocks that construction never wrote: their codes, run counts, sizes and picks are
// whatever the memory held, good for no index, so such a field's blocks are passed over (the
// call reports the status).  Every other error leaves valid codes.  Read through L2, by every
// thread beside loads it waits for anyway; the launches before have set all there is to set.
__device__ __forceinline__ uint32_t encode_status(const EncodeArgs& a) { return __ldcg(&a.st->status); }

// The plan of codec block b of one field (all threads of the CTA).  box: its origin and
// extent (block_box).  status: the field's, the same in every thread.  smem:
// plan_smem_bytes() of dynamic shared memory.
__device__ void plan_body(const EncodeArgs& a, uint32_t b, const uint32_t* box, uint32_t status, unsigned char* smem) {
  uint16_t* s_c = reinterpret_cast<uint16_t*>(smem);              // 4096 codes; before them the run starts
  uint16_t* s_rv = s_c + kSlots;                                  // run values
  uint16_t* s_rl = s_rv + kSlots;                                 // run lengths
  uint32_t* s_hist = reinterpret_cast<uint32_t*>(s_rl + kSlots);  // 1024: the statistics' code histogram
  uint32_t* s_sw = s_hist + kNsymCode;                            // the learned selector's parameters
  uint32_t* s_tab = s_sw + (kSwWords + 3) / 4 * 4;                // the code book, packed (+4)
  uint32_t* s_part = s_tab + kNsymCode + 4;                       // 2 x 256
  uint64_t* s_scan64 = reinterpret_cast<uint64_t*>(s_part + 2 * kEncThreads);  // 33
  __shared__ int s_codec;
  __shared__ float s_feat[8];

  const int tid = threadIdx.x, wid = tid >> 5;
  const uint32_t m = box[3] * box[4] * box[5];
  const int sel = a.select;
  const uint32_t r = a.radius;
  // the symbols are on their way while the block's run count and records are looked at; read
  // again where that takes more (L2 has them), rather than held
  const uint16_t* codes = a.codes + (uint64_t)b * kSlots;
  const uint32_t* heads = a.masks + (uint64_t)b * kMaskWords + 2 * (kSlots / 32);
  const HuffPart part(codes, m);
  uint32_t sym[16];
  part.load(sym);
  bool fresh = true;  // sym holds the symbols
  // the run count comes from construction; forced Huffman does without
  const bool analyze = a.analyze != 0;
  const uint32_t nr = sel != SEL_HUFF || analyze ? a.block_runs[b] : 0u;
  const uint32_t records = a.place_records ? a.rec.counts[b] : 0u;
  if (status & ERR_TIMEOUT) return;  // (every load above is on its way by now)
  const bool eligible = a.all_runs || 4 * nr <= m;
  // Runs are extracted (values, lengths) when a run codec or the statistics may need them.
  bool runs = analyze || (sel != SEL_HUFF && eligible);
  const bool statistics = analyze || ((sel == SEL_HEURISTIC || sel == SEL_LEARNED) && eligible);
  // the histogram starts at zero; it and the parameters are ready at the barriers of the
  // run extraction
  static_assert(kNsymCode == 4 * kEncThreads, "a 16-byte store a thread");
  if (statistics) {
    reinterpret_cast<uint4*>(s_hist)[tid] = make_uint4(0u, 0u, 0u, 0u);
    if (sel == SEL_LEARNED) stage_mlp(a.mlp_w, reinterpret_cast<float*>(s_sw));
  }
  if (records != 0) {
    place_records(a, b, box, box + 3, s_scan64);
    fresh = false;
  }
  if (runs) {
    extract_runs(codes, heads, m, nr, s_c, s_rv, s_rl);
    fresh = false;
  }

  // selection by the block's statistics; -1: by exact sizes
  int codec = sel == SEL_HUFF || (!eligible && (sel == SEL_HEURISTIC || sel == SEL_LEARNED)) ? CODEC_HUFF
              : sel == SEL_RLE || sel == SEL_RLE_HUFF                                       ? sel
                                                                                            : -1;
  if (analyze) codec = -1;
  if (statistics) {
    const bool heuristic = sel == SEL_HEURISTIC && !analyze;
    for (uint32_t i = tid; i < nr; i += kEncThreads) atomicAdd(&s_hist[s_rv[i]], (uint32_t)s_rl[i]);
    const bool want_mado = !heuristic;
    if (want_mado) {  // the codes, in the place of the run starts
      const uint4* src = reinterpret_cast<const uint4*>(codes);
      for (int i = tid; i < kSlots / 8; i += kEncThreads) reinterpret_cast<uint4*>(s_c)[i] = __ldcg(&src[i]);
    }
    __syncthreads();
    // block statistics in one pass and one reduction: entropy sum, |delta| sum, top
    // count and largest in-range |delta|, and (selector) the madogram's code changes
    // on the pairs (j, j + 1 + 25 (j mod 8))
    uint64_t S_ = 0, absd = 0;
    uint32_t f1 = 0, maxd = 0, mism = 0;
    for (int c = tid; c < kNsymCode; c += kEncThreads) {
      const uint32_t h = s_hist[c];
      if (h) {
        S_ += (uint64_t)h * log2_q16_small(h);
        f1 = max(f1, h);
        if (c != 0) {
          const uint32_t d = (uint32_t)abs((int)c - (int)r);
          absd += (uint64_t)h * d;
          maxd = max(maxd, d);
        }
      }
    }
    if (want_mado) {
      // kEncThreads is a multiple of kMadoN, so a thread's distance is fixed
      const uint32_t d = kMadoD0 + kMadoStep * (tid % kMadoN);
      for (uint32_t j = tid; j + d < m; j += kEncThreads) mism += s_c[j] != s_c[j + d];
    }
    S_ = warp_sum(S_);
    absd = warp_sum(absd);
    mism = warp_sum(mism);
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      f1 = max(f1, __shfl_xor_sync(~0u, f1, o));
      maxd = max(maxd, __shfl_xor_sync(~0u, maxd, o));
    }
    if ((tid & 31) == 0) {
      s_scan64[4 * wid + 0] = S_;
      s_scan64[4 * wid + 1] = absd;
      s_scan64[4 * wid + 2] = ((uint64_t)f1 << 32) | maxd;
      s_scan64[4 * wid + 3] = mism;
    }
    __syncthreads();
    const int64_t Lm = log2_q16_small(m);
    if (heuristic) {
      if (tid == 0) {
        S_ = 0;
        f1 = 0;
        for (int v = 0; v < kEncThreads / 32; v++) {
          S_ += s_scan64[4 * v + 0];
          f1 = max(f1, (uint32_t)(s_scan64[4 * v + 2] >> 32));
        }
        const int64_t NH = (int64_t)m * Lm - (int64_t)S_;
        int64_t Rm = 0;
        if (10ll * f1 > 4ll * m) {
          const int64_t rest = (int64_t)m - f1;
          Rm = (int64_t)m * 65536 + (int64_t)f1 * log2_q16_small(f1) +
               (rest > 0 ? rest * (int64_t)log2_q16_small((uint32_t)rest) : 0) - (int64_t)m * Lm;
          if (Rm < 0) Rm = 0;
        }
        const int64_t est = NH + Rm;
        s_codec = (100 * est <= 109ll * (int64_t)m * 65536) ? CODEC_RLE_HUFF : CODEC_HUFF;
      }
    } else {
      if (wid == 0) {
        // warp 0: the block totals (lane v < 8 brings warp v's partials), one feature
        // per lane k < 8, then the network on the staged parameters
        const int lane = tid & 31;
        uint64_t tS = 0, tA = 0, tM = 0;
        uint32_t tF = 0, tD = 0;
        if (lane < kEncThreads / 32) {
          tS = s_scan64[4 * lane + 0];
          tA = s_scan64[4 * lane + 1];
          tF = (uint32_t)(s_scan64[4 * lane + 2] >> 32);
          tD = (uint32_t)s_scan64[4 * lane + 2];
          tM = s_scan64[4 * lane + 3];
        }
        tS = warp_sum(tS);
        tA = warp_sum(tA);
        tM = warp_sum(tM);
#pragma unroll
        for (int o = 16; o; o >>= 1) {
          tF = max(tF, __shfl_xor_sync(~0u, tF, o));
          tD = max(tD, __shfl_xor_sync(~0u, tD, o));
        }
        const float fm = (float)m;
        float fk = 0.0f;
        if (lane == 0) {
          fk = (float)s_hist[r] / fm;  // zero residuals
        } else if (lane == 1) {
          const int64_t NH = (int64_t)m * Lm - (int64_t)tS;
          fk = (float)NH / (float)((uint64_t)m * 65536ull);
        } else if (lane == 2) {
          fk = (float)tF / fm;
        } else if (lane == 3) {
          fk = (float)log2_q16_small(1u + tD) / 65536.0f;
        } else if (lane == 4) {
          fk = (float)nr / fm;
        } else if (lane == 5) {
          fk = (float)s_hist[0] / fm;  // outliers
        } else if (lane == 6) {
          fk = (float)tA / (float)((uint64_t)m * r);
        } else if (lane == 7) {
          // pairs inside the block: positions j < m - d for each residue class j mod 8
          uint32_t pairs = 0;
          for (uint32_t k = 0; k < kMadoN; k++) {
            const uint32_t d = kMadoD0 + kMadoStep * k;
            if (m > d + k) pairs += (m - d - k + kMadoN - 1) / kMadoN;
          }
          fk = pairs ? (float)(uint32_t)tM / (float)pairs : 0.0f;
        }
        if (analyze) {
          if (lane < kMlpIn) s_feat[lane] = fk;
        } else {
          float f[kMlpIn], y[kMlpOut];
#pragma unroll
          for (int j = 0; j < kMlpIn; j++) f[j] = __shfl_sync(~0u, fk, j);
          mlp_forward_staged(reinterpret_cast<const float*>(s_sw), f, y);
          bool fb;
          const int c = learned_pick(y, fb);
          if (lane == 0) s_codec = fb ? -1 : c;
        }
      }
    }
    __syncthreads();
    if (!analyze) codec = s_codec;  // (-1 where the network is unsure)
  }

  // A pick by sizes takes the runs' first, then the Huffman size, unless a run codec is
  // already smaller than any Huffman payload can be: every code takes at least one bit, so
  // a block of m codes holds at least m / 16 units plus its unit count, 2 + m / 8 bytes.
  PairPlan plan;
  uint32_t size_h = ~0u, size_rh = ~0u;
  const uint32_t size_r = 4 * nr;
  if (codec == CODEC_RLE_HUFF || (codec < 0 && eligible)) {
    plan_runs(plan, RunPart(a, s_rv, s_rl, nr), s_part);
    size_rh = rlehuff_bytes(plan);
  }
  if (codec == CODEC_HUFF || (codec < 0 && (analyze || min(size_r, size_rh) >= 2 + m / 8))) {
    stage_book(a, s_tab);
    if (!fresh) part.load(sym);
    __syncthreads();
    plan_huff(plan, a, part, sym, s_tab, s_part + kEncThreads);
    size_h = huff_bytes(plan);
  }
  if (analyze) {
    // one training row: features, log2 bits per element of each codec (Q16-exact),
    // exact sizes, and whether the learned selector decides this block
    if (tid < kMlpIn) a.feat_out[(uint64_t)b * kMlpIn + tid] = s_feat[tid];
    if (tid < kMlpOut) {
      const uint32_t sz = tid == CODEC_HUFF ? size_h : (tid == CODEC_RLE ? size_r : size_rh);
      const bool have = sz != ~0u;
      a.size_out[(uint64_t)b * kMlpOut + tid] = have ? sz : 0xffffffffu;
      a.tgt_out[(uint64_t)b * kMlpOut + tid] =
          have ? (float)((int64_t)log2_q16(8ull * sz) - (int64_t)log2_q16(m)) * (1.0f / 65536.0f) : 0.0f;
      if (tid == 0) a.valid_out[b] = eligible ? 1 : 0;
    }
    return;
  }
  if (codec < 0) codec = exhaustive_pick(size_h, size_r, size_rh);  // (the same in every thread)
  const uint32_t size = codec == CODEC_HUFF ? size_h : (codec == CODEC_RLE ? size_r : size_rh);
  if (codec != CODEC_HUFF) {
    if (!runs) extract_runs(codes, heads, m, nr, s_c, s_rv, s_rl);
    uint16_t* rv = block_run_store(a, b);
    for (uint32_t i = tid; i < nr; i += kEncThreads) {
      rv[i] = s_rv[i];
      rv[kSlots + i] = s_rl[i];
    }
  }
  if (tid == 0) {
    a.ar[a.off_codec + b] = (uint8_t)codec;
    reinterpret_cast<uint32_t*>(a.ar + a.off_bb)[b] = size;
    atomicAdd(reinterpret_cast<unsigned long long*>(a.groups) + b / kGroup,
              (unsigned long long)size | (codec == CODEC_RLE ? 1ull << 40 : (codec == CODEC_RLE_HUFF ? 1ull << 52 : 0ull)));
  }
}

// The field's totals from its groups', then the header, section padding and books (one
// CTA; not inlined, as the two below, for the registers of the common path).
__device__ __noinline__ void finish_field(const EncodeArgs& a) {
  __shared__ uint64_t s_sum[kEncThreads / 32], s_all[kEncThreads / 32];
  const uint32_t tid = threadIdx.x, wid = tid >> 5;
  const uint32_t ngroups = (a.g.nblk + kGroup - 1) / kGroup;
  uint64_t bytes = 0, counts = 0;  // (RLE blocks, RLE+Huffman blocks from bit 32)
  for (uint32_t k = tid; k < ngroups; k += kEncThreads) {
    const uint64_t v = __ldcg(&a.groups[k]);
    bytes += v & kGroupBytes;
    counts += ((v >> 40) & 0xfffu) | (v >> 52) << 32;
  }
  bytes = warp_sum(bytes);
  counts = warp_sum(counts);
  if ((tid & 31) == 0) {
    s_sum[wid] = bytes;
    s_all[wid] = counts;
  }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < kEncThreads / 32; w++) {
      bytes += s_sum[w];
      counts += s_all[w];
    }
    a.st->payload = bytes;
    a.st->ncodec[CODEC_RLE] = (uint32_t)counts;
    a.st->ncodec[CODEC_RLE_HUFF] = (uint32_t)(counts >> 32);
    a.st->ncodec[CODEC_HUFF] = a.g.nblk - (uint32_t)counts - (uint32_t)(counts >> 32);
  }
  finalize_body(a.fin);
}

// A block with codes longer than a packed one's, or one whose payload does not fit the
// buffer: both streams by the gathering encoder.  first: units before stream A.
__device__ __noinline__ void encode_long(const EncodeArgs& a, int codec, const uint16_t* codes, uint32_t m,
                                         const uint16_t* rv, uint32_t nr, uint32_t ua, uint16_t* out16,
                                         uint32_t* s_part) {
  if (codec == CODEC_HUFF) {
    const uint32_t h = huff_split(m);
    ihs_encode_block(codes, h, 0, a.lens, a.bcodes, out16 + 1, s_part);
    ihs_encode_block(codes + h, m - h, 0, a.lens, a.bcodes, out16 + 1 + ua, s_part);
  } else {
    const uint8_t* vlen = a.lens + kNsymCode;
    const uint64_t* vcode = a.bcodes + kNsymCode;
    ihs_encode_block(rv, nr, 0, vlen, vcode, out16 + 4, s_part);
    ihs_encode_block(rv + kSlots, nr, -1, vlen + kNsymCode, vcode + kNsymCode, out16 + 4 + ua, s_part);
  }
}

// The streams of an RLE+Huffman block of more than 2048 runs (forced modes): two turns of
// 16 steps, the codes read again.  (Not inlined: a loop in the payload's common path costs it
// its registers, 3-D 512^3 compression 803 -> 842 us.  The gathering encoder, which such
// blocks took before: 1426 us for 60 M elements of a walk; now 897.)
__device__ __noinline__ void emit_many_runs(const EncodeArgs& a, uint32_t pre, uint32_t base, uint32_t units_a,
                                            const uint16_t* rv, uint32_t nr, uint32_t* s_buf, uint32_t* s_heads) {
  PairPlan P;
  P.pre = pre;
  P.base = base;
  P.units_a = units_a;
  const RunPart part(a, rv, rv + kSlots, nr);
  PairEmitter em;
  em.init(P, reinterpret_cast<uint16_t*>(s_buf), 4u, s_heads);
  uint32_t odd = 0;
#pragma unroll 1
  for (uint32_t f = 0; f < part.steps; f += 16) {
    part.load(f, P.e, odd);
    em.steps(P.e);
  }
  em.finish(s_heads);
}

// The payload of codec block b (all threads of the CTA), after the plans of all the field's
// blocks; block 0 also writes the header, section padding and books.  m: the block's
// elements.  status: the field's, the same in every thread.  smem: payload_smem_bytes() of
// dynamic shared memory.
__device__ void payload_body(const EncodeArgs& a, uint32_t b, uint32_t m, uint32_t status, unsigned char* smem) {
  uint32_t* s_buf = reinterpret_cast<uint32_t*>(smem);  // 16 KB: the payload; before it, the code book
  uint32_t* s_part = s_buf + kBufBytes / 4;             // 256 (+ 8)
  uint32_t* s_heads = s_part + kEncThreads + 8;         // 256
  __shared__ uint64_t s_sum[kEncThreads / 32];
  const uint32_t tid = threadIdx.x, wid = tid >> 5;
  const uint16_t* codes = a.codes + (uint64_t)b * kSlots;
  const HuffPart part(codes, m);
  uint32_t sym[16];
  part.load(sym);
  const int codec = __ldcg(&a.ar[a.off_codec + b]);
  const uint32_t* bb = reinterpret_cast<const uint32_t*>(a.ar + a.off_bb);
  const uint32_t size = __ldcg(&bb[b]);
  const uint64_t n_rec = __ldcg(&a.st->n_rec);
  // what precedes the block: the groups before its own, the blocks before it in its own
  const uint32_t group = b / kGroup, in_group = b % kGroup;
  uint64_t before = tid < in_group ? (uint64_t)__ldcg(&bb[group * kGroup + tid]) : 0ull;
  for (uint32_t k = tid; k < group; k += kEncThreads) before += __ldcg(&a.groups[k]) & kGroupBytes;
  const uint32_t nr = a.block_runs[b];
  const uint16_t* rv = block_run_store(a, b);
  if (status & ERR_TIMEOUT) return;  // (every load above is on its way by now)
  before = warp_sum(before);
  if ((tid & 31) == 0) s_sum[wid] = before;
  PairPlan plan;
  const bool in_smem = size <= (uint32_t)kBufBytes;
  if (codec == CODEC_HUFF) {
    stage_book(a, s_buf);
    __syncthreads();
    plan_huff(plan, a, part, sym, s_buf, s_part);
  } else if (codec == CODEC_RLE_HUFF) {
    plan_runs(plan, RunPart(a, rv, rv + kSlots, nr), s_part);
  } else {
    __syncthreads();
  }
  uint64_t dst_off = a.off_rec + 8ull * n_rec;
#pragma unroll
  for (int w = 0; w < kEncThreads / 32; w++) dst_off += s_sum[w];
  if (dst_off + size > a.cap) {
    if (tid == 0) atomicOr(&a.st->status, ERR_CAPACITY);
  } else {
    uint32_t* dst = reinterpret_cast<uint32_t*>(a.ar + dst_off);
    if (codec == CODEC_RLE) {
      uint16_t* d16 = reinterpret_cast<uint16_t*>(dst);
      for (uint32_t i = tid; i < nr; i += kEncThreads) {
        d16[i] = rv[i];
        d16[nr + i] = rv[kSlots + i];
      }
    } else {
      // assembled in shared memory (every chosen size fits 16 KB unless a forced mode meets
      // very long codes; those go direct)
      uint16_t* out16 = in_smem ? reinterpret_cast<uint16_t*>(s_buf) : reinterpret_cast<uint16_t*>(dst);
      const uint32_t ua = plan.units_a, ub = plan.units_b;
      const uint32_t first = codec == CODEC_HUFF ? 1u : 4u, units = first + ua + ub;  // before stream A; in all
      if (plan.packed && in_smem) {
        if (codec == CODEC_RLE_HUFF && quarter_steps(nr) > 16) {
          emit_many_runs(a, plan.pre, plan.base, plan.units_a, rv, nr, s_buf, s_heads);
        } else {
          PairEmitter em;
          em.init(plan, reinterpret_cast<uint16_t*>(s_buf), first, s_heads);
          em.steps(plan.e);
          em.finish(s_heads);
        }
      } else {
        encode_long(a, codec, codes, m, rv, nr, ua, out16, s_part);
      }
      if (tid == 0) {
        if (codec == CODEC_HUFF) {
          out16[0] = (uint16_t)ua;
        } else {
          reinterpret_cast<uint32_t*>(out16)[0] = nr;
          reinterpret_cast<uint32_t*>(out16)[1] = ua;
        }
        if (units & 1u) out16[units] = 0;
      }
      if (in_smem) {
        __syncthreads();
        for (uint32_t i = tid; i < size / 4; i += kEncThreads) dst[i] = s_buf[i];
      }
    }
  }
  if (b == 0) finish_field(a);
}

// Forced RLE: a block's size is its run count's, so its plan needs no runs, and its payload
// takes them from the codes.  (A store and a reload of every run between the two, as for blocks
// picked by size, took more than the rest where runs are short: 100x500x500 walk, rel 1e-4,
// compression 427 us; now 271.)  Kernels of their own, for the registers of the others.
__device__ void plan_rle_body(const EncodeArgs& a, uint32_t b, const uint32_t* box, unsigned char* smem) {
  const uint32_t nr = a.block_runs[b], records = a.rec.counts[b];
  if (encode_status(a) & ERR_TIMEOUT) return;
  if (records != 0) place_records(a, b, box, box + 3, reinterpret_cast<uint64_t*>(smem));
  if (threadIdx.x == 0) {
    a.ar[a.off_codec + b] = (uint8_t)CODEC_RLE;
    reinterpret_cast<uint32_t*>(a.ar + a.off_bb)[b] = 4 * nr;
    atomicAdd(reinterpret_cast<unsigned long long*>(a.groups) + b / kGroup, (unsigned long long)(4 * nr) | 1ull << 40);
  }
}

__device__ void payload_rle_body(const EncodeArgs& a, uint32_t b, uint32_t m, unsigned char* smem) {
  uint16_t* s_rv = reinterpret_cast<uint16_t*>(smem);  // 4096 run values, 4096 run starts
  uint16_t* s_at = s_rv + kSlots;
  __shared__ uint64_t s_sum[kEncThreads / 32];
  const uint32_t tid = threadIdx.x;
  const uint32_t* bb = reinterpret_cast<const uint32_t*>(a.ar + a.off_bb);
  const uint32_t nr = a.block_runs[b], group = b / kGroup;
  uint64_t before = tid < b % kGroup ? (uint64_t)__ldcg(&bb[group * kGroup + tid]) : 0ull;
  for (uint32_t k = tid; k < group; k += kEncThreads) before += __ldcg(&a.groups[k]) & kGroupBytes;
  uint64_t dst_off = a.off_rec + 8ull * __ldcg(&a.st->n_rec);
  if (encode_status(a) & ERR_TIMEOUT) return;
  scatter_runs(a.codes + (uint64_t)b * kSlots, a.masks + (uint64_t)b * kMaskWords + 2 * (kSlots / 32), s_at, s_rv);
  before = warp_sum(before);
  if ((tid & 31) == 0) s_sum[tid >> 5] = before;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kEncThreads / 32; w++) dst_off += s_sum[w];
  if (dst_off + 4 * nr > a.cap) {
    if (tid == 0) atomicOr(&a.st->status, ERR_CAPACITY);
  } else {
    // nr values, then nr lengths, two a word
    uint32_t* dst = reinterpret_cast<uint32_t*>(a.ar + dst_off);
    auto unit = [&](uint32_t i) -> uint32_t { return i < nr ? s_rv[i] : run_length(s_at, i - nr, nr, m); };
    for (uint32_t i = tid; i < nr; i += kEncThreads) dst[i] = unit(2 * i) | unit(2 * i + 1) << 16;
  }
  if (b == 0) finish_field(a);
}

// (four CTAs an SM: with the registers of five the plan spills, 3-D 512^3 compression 818
// against 805 us, 40 mixed fields 486 against 474; the payload's place is better at five)
__global__ __launch_bounds__(kEncThreads, 4) void plan_kernel(EncodeArgs a) {
  chained_begin();
  __shared__ uint32_t s_box[6];
  extern __shared__ __align__(16) unsigned char smem[];
  if (threadIdx.x == 0) block_box(a.g, blockIdx.x, s_box, s_box + 3);
  __syncthreads();
  plan_body(a, blockIdx.x, s_box, encode_status(a), smem);
}

__global__ __launch_bounds__(kEncThreads, 5) void payload_kernel(EncodeArgs a) {
  chained_begin();
  __shared__ uint32_t s_m;
  extern __shared__ __align__(16) unsigned char smem[];
  if (threadIdx.x == 0) s_m = block_elems(a.g, blockIdx.x);
  __syncthreads();
  payload_body(a, blockIdx.x, s_m, encode_status(a), smem);
}

__global__ __launch_bounds__(kEncThreads) void plan_rle_kernel(EncodeArgs a) {
  chained_begin();
  __shared__ uint32_t s_box[6];
  extern __shared__ __align__(16) unsigned char smem[];
  if (threadIdx.x == 0) block_box(a.g, blockIdx.x, s_box, s_box + 3);
  __syncthreads();
  plan_rle_body(a, blockIdx.x, s_box, smem);
}

__global__ __launch_bounds__(kEncThreads) void payload_rle_kernel(EncodeArgs a) {
  chained_begin();
  __shared__ uint32_t s_m;
  extern __shared__ __align__(16) unsigned char smem[];
  if (threadIdx.x == 0) s_m = block_elems(a.g, blockIdx.x);
  __syncthreads();
  payload_rle_body(a, blockIdx.x, s_m, smem);
}

__device__ __forceinline__ int field_of_prefix(const uint32_t* prefix, int nfields, uint32_t c) {
  int lo = 0, hi = nfields - 1;  // last field with prefix[f] <= c
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= c) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Batch: one CTA per codec block of every field (tile0[f] = first block of field f).
__global__ __launch_bounds__(kEncThreads, 4) void plan_batch_kernel(const EncodeArgs* __restrict__ tasks,
                                                                 const uint32_t* __restrict__ tile0, int nfields) {
  chained_begin();
  __shared__ uint32_t s_box[6];
  __shared__ int s_field;
  extern __shared__ __align__(16) unsigned char smem[];
  if (threadIdx.x == 0) {
    const int f = field_of_prefix(tile0, nfields, blockIdx.x);
    s_field = f;
    block_box(tasks[f].g, blockIdx.x - tile0[f], s_box, s_box + 3);
  }
  __syncthreads();
  const EncodeArgs& a = tasks[s_field];
  plan_body(a, blockIdx.x - tile0[s_field], s_box, encode_status(a), smem);
}

__global__ __launch_bounds__(kEncThreads, 5) void payload_batch_kernel(const EncodeArgs* __restrict__ tasks,
                                                                    const uint32_t* __restrict__ tile0, int nfields) {
  chained_begin();
  __shared__ uint32_t s_m;
  __shared__ int s_field;
  extern __shared__ __align__(16) unsigned char smem[];
  if (threadIdx.x == 0) {
    const int f = field_of_prefix(tile0, nfields, blockIdx.x);
    s_field = f;
    s_m = block_elems(tasks[f].g, blockIdx.x - tile0[f]);
  }
  __syncthreads();
  const EncodeArgs& a = tasks[s_field];
  payload_body(a, blockIdx.x - tile0[s_field], s_m, encode_status(a), smem);
}

static size_t plan_smem_bytes() {
  return kSlots * 2 * 3 + 4 * (kNsymCode + (kSwWords + 3) / 4 * 4 + kNsymCode + 4 + 2 * kEncThreads) +
         33 * 8 + 16;
}
static size_t payload_smem_bytes() { return kBufBytes + 4 * (2 * kEncThreads + 8); }

// =================================================================================
// batched compression in one persistent launch
// =================================================================================
// Every CTA runs the phases of the staged batch in order, so the work items of
// each phase are taken (by ticket) only after those of the phases before it were all
// taken: a waiting CTA waits on items that running CTAs hold (only a running CTA takes
// an item), and those wait only on earlier phases, so the launch cannot deadlock even
// when not all of its CTAs are resident at once.  The
// hand-overs are per field (DevState ready_range, tiles_flushed, books_done, encode_done: a
// release by the producer, an acquire by thread 0 of the consumer, then a CTA
// barrier), so one field's books and encoding start while other fields are still
// being constructed.  Every wait is bounded (ERR_TIMEOUT in the field's status).
// The output is the staged path's, byte for byte: the same bodies run on the same
// items.
constexpr int kPersistThreads = 256;
static_assert(kPersistThreads == kEncThreads, "one CTA shape for every phase");

// thread 0 draws the next item of a phase; every thread gets it (two barriers, so the
// word is free for the next draw)
__device__ __forceinline__ uint32_t draw_item(uint32_t* ticket, uint32_t* s_word) {
  if (threadIdx.x == 0) *s_word = atomicAdd(ticket, 1u);
  __syncthreads();
  const uint32_t v = *s_word;
  __syncthreads();
  return v;
}

// thread 0 waits for a field's hand-over counter, then the CTA proceeds together
__device__ __forceinline__ void await_field(const uint32_t* counter, uint32_t target, DevState* st, uint32_t limit) {
  if (threadIdx.x == 0 && !wait_ge_acquire(counter, target, limit)) atomicOr(&st->status, ERR_TIMEOUT);
  __syncthreads();
}

template <int ND>
__global__ __launch_bounds__(kPersistThreads, 4) void batch_persistent_kernel(const __grid_constant__ PersistArgs p) {
  // the construction phase's swizzled TMA tiles want 1024-byte aligned buffers; the
  // alignment is taken here (1 KB of slack in the dynamic size) rather than declared,
  // which would pad the static shared memory of every kernel in this file
  extern __shared__ __align__(16) unsigned char smem_dyn[];
  unsigned char* smem_raw = smem_dyn + ((1024u - (smem_u32(smem_dyn) & 1023u)) & 1023u);
  __shared__ uint32_t s_word, s_box[6], s_status;
  const int tid = threadIdx.x;
  // ---- phase 1: value ranges and bounds ---------------------------------------------
  while (true) {
    const uint32_t c = draw_item(&p.tickets[2], &s_word);
    if (c >= p.nrange) break;
    const int f = field_of_prefix(p.cta0, p.nfields, c);
    const RangeTask& t = p.rtasks[f];
    if (t.mode == 0) {
      if (tid == 0) {
        derive_eb(t.st, 0, t.eb, 0.0f, 0.0f);
        release_flag(&t.st->ready_range);
      }
    } else {
      range_body(t.x, t.n, t.st, t.mode, t.eb, c - p.cta0[f], p.cta0[f + 1] - p.cta0[f], &t.st->ready_range);
    }
    __syncthreads();
  }
  // ---- phase 2: construction (waits for each field's bound) ---------------------------
  cons::construct_loop<ND, float, false, true>(p.ctasks[0], p.ctasks, p.tile0, p.nfields, p.ntiles, &p.tickets[0],
                                               p.spin_limit, smem_raw);
  // ---- phase 3: books and record offsets (wait for each field's tiles) ---------------
  while (true) {
    const uint32_t j = draw_item(&p.tickets[3], &s_word);
    if (j >= 4u * (uint32_t)p.nfields) break;
    const int f = (int)(j >> 2), role = (int)(j & 3);
    const BookArgs& ba = p.btasks[f];
    await_field(&ba.st->tiles_flushed, p.tile0[f + 1] - p.tile0[f], ba.st, p.spin_limit);
    unsigned char* mem = role == 2 ? p.len_books + (size_t)f * book_mem_bytes(kNsymLen) : smem_raw;
    codebook_core<kPersistThreads>(ba, role, mem);
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      atomicAdd(&ba.st->books_done, 1u);
    }
  }
  // ---- phase 4: block plans (wait for each field's books) ------------------------------
  int ready_field = -1;
  while (true) {
    const uint32_t t = draw_item(&p.tickets[1], &s_word);
    if (t >= p.ntiles) break;
    const int f = field_of_prefix(p.tile0, p.nfields, t);
    const EncodeArgs& ea = p.etasks[f];
    if (f != ready_field) {
      await_field(&ea.st->books_done, 4u, ea.st, p.spin_limit);
      ready_field = f;
    }
    // (the status once, by thread 0: other CTAs' waits may expire meanwhile)
    if (tid == 0) {
      block_box(ea.g, t - p.tile0[f], s_box, s_box + 3);
      s_status = encode_status(ea);
    }
    __syncthreads();
    plan_body(ea, t - p.tile0[f], s_box, s_status, smem_raw);
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      atomicAdd(&ea.st->encode_done, 1u);
    }
  }
  // ---- phase 5: payloads (wait for each field's plans) ---------------------------------
  ready_field = -1;
  while (true) {
    const uint32_t t = draw_item(&p.tickets[4], &s_word);
    if (t >= p.ntiles) break;
    const int f = field_of_prefix(p.tile0, p.nfields, t);
    const EncodeArgs& ea = p.etasks[f];
    if (f != ready_field) {
      await_field(&ea.st->encode_done, ea.g.nblk, ea.st, p.spin_limit);
      ready_field = f;
    }
    if (tid == 0) {
      s_box[0] = block_elems(ea.g, t - p.tile0[f]);
      s_status = encode_status(ea);
    }
    __syncthreads();
    payload_body(ea, t - p.tile0[f], s_box[0], s_status, smem_raw);
    __syncthreads();
  }
}

static size_t persist_smem_bytes() {
  size_t b = construct_smem_bytes();
  if (plan_smem_bytes() > b) b = plan_smem_bytes();
  if (payload_smem_bytes() > b) b = payload_smem_bytes();
  if (book_mem_bytes(kNsymCode) > b) b = book_mem_bytes(kNsymCode);
  return b + 1024;  // alignment slack
}

size_t persist_len_book_bytes() { return book_mem_bytes(kNsymLen); }

template <int ND>
static int persist_occupancy() {
  static PerDevice occ_and_one;
  return occ_and_one.get([] {
    int occ = 0;
    const int sm = (int)persist_smem_bytes();
    if (cudaFuncSetAttribute(batch_persistent_kernel<ND>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, batch_persistent_kernel<ND>, kPersistThreads, sm) !=
            cudaSuccess)
      occ = 0;
    return occ + 1;
  }) - 1;
}

int persist_grid_max() {
  int occ = persist_occupancy<0>();
  for (int o : {persist_occupancy<1>(), persist_occupancy<2>(), persist_occupancy<3>()})
    if (o < occ) occ = o;
  return occ * sm_count();
}

cudaError_t launch_batch_persistent(const PersistArgs& p, int grid, int nd, cudaStream_t s) {
  auto k = nd == 1 ? batch_persistent_kernel<1>
                   : (nd == 2 ? batch_persistent_kernel<2> : (nd == 3 ? batch_persistent_kernel<3> : batch_persistent_kernel<0>));
  if (grid <= 0 || grid > persist_grid_max()) return cudaErrorInvalidConfiguration;
  trace_begin(K_BATCH, s);
  k<<<grid, kPersistThreads, persist_smem_bytes(), s>>>(p);
  trace_end(K_BATCH, s);
  return cudaGetLastError();
}

// =================================================================================
// launchers
// =================================================================================
cudaError_t launch_abs_params(DevState* st, double eb, cudaStream_t s) {
  trace_begin(K_PARAMS, s);
  abs_params_kernel<<<1, 32, 0, s>>>(st, eb);
  trace_end(K_PARAMS, s);
  return cudaGetLastError();
}

cudaError_t launch_range(const float* x, uint64_t n, DevState* st, int mode, double eb, cudaStream_t s) {
  const uint32_t grid = range_ctas(n);
  trace_begin(K_RANGE, s);
  range_kernel<<<grid, 256, 0, s>>>(x, n, st, mode, eb);
  trace_end(K_RANGE, s);
  return cudaGetLastError();
}

cudaError_t launch_range_d(const double* x, uint64_t n, DevState* st, int mode, double eb, cudaStream_t s) {
  trace_begin(K_RANGE, s);
  if (mode == 0) abs_params_d_kernel<<<1, 32, 0, s>>>(st, eb);
  else range_d_kernel<<<range_ctas(2 * n), 256, 0, s>>>(x, n, st, mode, eb);
  trace_end(K_RANGE, s);
  return cudaGetLastError();
}

cudaError_t launch_codebook(const BookArgs& a, cudaStream_t s) {
  const size_t sm = codebook_smem_bytes();
  cudaError_t e = cudaFuncSetAttribute(codebook_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  const int grid = a.place_records ? 4 : 3;
  trace_begin(K_CODEBOOK, s);
  launch_chained(codebook_kernel, grid, kBookThreads, sm, s, a);
  trace_end(K_CODEBOOK, s);
  return cudaGetLastError();
}

cudaError_t launch_encode(const EncodeArgs& a, cudaStream_t s) {
  trace_begin(K_ENCODE, s);
  if (a.select == SEL_RLE && !a.analyze) {
    launch_chained(plan_rle_kernel, a.g.nblk, kEncThreads, 33 * 8, s, a);
    launch_chained(payload_rle_kernel, a.g.nblk, kEncThreads, 4 * kSlots, s, a);
    trace_further(K_ENCODE_PAYLOAD, 1);
    trace_end(K_ENCODE, s);
    return cudaGetLastError();
  }
  launch_chained(plan_kernel, a.g.nblk, kEncThreads, plan_smem_bytes(), s, a);
  if (!a.analyze) {
    launch_chained(payload_kernel, a.g.nblk, kEncThreads, payload_smem_bytes(), s, a);
    trace_further(K_ENCODE_PAYLOAD, 1);
  }
  trace_end(K_ENCODE, s);
  return cudaGetLastError();
}

uint32_t range_ctas(uint64_t n) {
  const uint64_t want = (n / 4 + 255) / 256, most = 8ull * sm_count();
  const uint64_t grid = want < most ? want : most;
  return grid ? (uint32_t)grid : 1u;
}

// A single field's CTAs take as little as one 16-byte load a thread, for its latency; a
// batch's fields fill the SMs together, so a CTA takes at least 64 KB there: its reduction,
// two atomics and a fence, about 2 us, would otherwise outweigh its loads (40 mixed fields,
// 51 M elements: 57 -> 39 us).
uint32_t range_ctas_batch(uint64_t n) {
  const uint64_t want = (n + 16383) / 16384;
  const uint32_t most = range_ctas(n);
  return want < most ? (uint32_t)want : most;
}

cudaError_t launch_range_batch(const RangeTask* d_tasks, const uint32_t* d_cta0, int nfields, uint32_t nctas,
                               cudaStream_t s) {
  trace_begin(K_RANGE, s);
  range_batch_kernel<<<nctas, 256, 0, s>>>(d_tasks, d_cta0, nfields);
  trace_end(K_RANGE, s);
  return cudaGetLastError();
}

cudaError_t launch_codebook_batch(const BookArgs* d_tasks, int nfields, cudaStream_t s) {
  const size_t sm = codebook_smem_bytes();
  cudaError_t e =
      cudaFuncSetAttribute(codebook_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  trace_begin(K_CODEBOOK, s);
  codebook_batch_kernel<<<4 * nfields, kBookThreads, sm, s>>>(d_tasks);
  trace_end(K_CODEBOOK, s);
  return cudaGetLastError();
}

cudaError_t launch_encode_batch(const EncodeArgs* d_tasks, const uint32_t* d_tile0, int nfields, uint32_t ntiles,
                                cudaStream_t s) {
  trace_begin(K_ENCODE, s);
  plan_batch_kernel<<<ntiles, kEncThreads, plan_smem_bytes(), s>>>(d_tasks, d_tile0, nfields);
  // (chained to the plans: two launches cost a small batch about as much as the one they
  // replaced; 4 x 64 K elements, forced RLE, staged: 54 -> 53 us, 52 in one launch)
  launch_chained(payload_batch_kernel, ntiles, kEncThreads, payload_smem_bytes(), s, d_tasks, d_tile0, nfields);
  trace_further(K_ENCODE_PAYLOAD, 1);
  trace_end(K_ENCODE, s);
  return cudaGetLastError();
}


}  // namespace cszp
