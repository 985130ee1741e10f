// Test aid (built by test_gpu_expired_wait.py against libcszp.so): the launches that follow a
// bounded wait, on a workspace whose state says that one expired.
#include "host.h"
#include "kernels.h"

using namespace cszp;

// The encoding launches (csz_compress's) for a workspace that csz_compress has filled for
// this field.  spoil: first overwrites what construction left with 0xff, as memory that was
// never written may hold anything.
extern "C" int probe_encode(const float* x, int ndim, const uint64_t* dims, int select, void* ws, uint8_t* ar,
                            uint64_t cap, int spoil) {
  Geom g;
  if (!make_geom(ndim, dims, g)) return 1;
  const Layout L = layout(g);
  DevState* st = at<DevState>(ws, L.st);
  const uint32_t bit = ERR_TIMEOUT;
  if (cudaMemcpy(&st->status, &bit, sizeof(bit), cudaMemcpyHostToDevice) != cudaSuccess) return 2;
  if (cudaMemset(at<void>(ws, L.lb_e), 0, L.zero_end - L.lb_e) != cudaSuccess) return 2;
  if (spoil && (cudaMemset(at<void>(ws, L.codes), 0xff, 2ull * kSlots * g.nblk) != cudaSuccess ||
                cudaMemset(at<void>(ws, L.counts), 0xff, 4ull * g.nblk) != cudaSuccess ||
                cudaMemset(at<void>(ws, L.masks), 0xff, 4ull * kMaskWords * g.nblk) != cudaSuccess ||
                cudaMemset(at<void>(ws, L.runs), 0xff, 2ull * g.nblk) != cudaSuccess))
    return 2;
  const uint64_t off_bb = kHdr + a8(g.nblk), off_rec = off_bb + a8(4ull * g.nblk);
  EncodeArgs a;
  memset(&a, 0, sizeof(a));
  a.g = g;
  a.st = st;
  a.radius = 512;
  a.select = select;
  a.all_runs = select == SEL_RLE || select == SEL_RLE_HUFF;
  a.codes = at<uint16_t>(ws, L.codes);
  a.block_runs = at<uint16_t>(ws, L.runs);
  a.masks = at<uint32_t>(ws, L.masks);
  a.lens = at<uint8_t>(ws, L.lens);
  a.bcodes = at<uint64_t>(ws, L.bcodes);
  a.ar = ar;
  a.cap = cap;
  a.off_codec = kHdr;
  a.off_bb = off_bb;
  a.off_rec = off_rec;
  a.groups = at<uint64_t>(ws, L.lb_e);
  a.place_records = 1;
  a.rec.x = x;
  a.rec.counts = at<uint32_t>(ws, L.counts);
  a.rec.masks = a.masks;
  a.rec.deltas = at<int32_t>(ws, L.deltas);
  a.rec.rec_off = at<uint64_t>(ws, L.rec_off);
  a.rec.rec = reinterpret_cast<uint32_t*>(ar + off_rec);
  a.rec.rec_cap = (cap - off_rec) / 8;
  a.fin.st = st;
  a.fin.ar = ar;
  a.fin.cap = cap;
  a.fin.ndim = ndim;
  a.fin.radius = 512;
  a.fin.select = select;
  a.fin.nblk = g.nblk;
  a.fin.off_bb = off_bb;
  a.fin.off_rec = off_rec;
  a.fin.lens = a.lens;
  if (launch_encode(a, nullptr) != cudaSuccess) return 3;
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 4;
}

// The decoding launches (csz_decompress's) of an FP32 archive whose header is hdr, with the
// status set before them.
extern "C" int probe_decode(const uint8_t* ar, uint64_t bytes, const uint8_t* hdr, int ndim, const uint64_t* dims,
                            void* ws, float* out) {
  Geom g;
  if (!make_geom(ndim, dims, g)) return 1;
  const Layout L = layout(g);
  DevState* st = at<DevState>(ws, L.st);
  const uint32_t bit = ERR_TIMEOUT;
  if (cudaMemset(st, 0, L.hist_code - L.st) != cudaSuccess) return 2;
  if (cudaMemset(at<void>(ws, L.lb_e), 0, 8ull * g.nblk) != cudaSuccess) return 2;
  if (cudaMemcpy(&st->status, &bit, sizeof(bit), cudaMemcpyHostToDevice) != cudaSuccess) return 2;
  float eb = 0.0f;
  DecodeArgs a;
  memset(&a, 0, sizeof(a));
  memcpy(&eb, hdr + 48, 4);
  memcpy(&a.radius, hdr + 52, 4);
  memcpy(&a.flags, hdr + 60, 4);
  memcpy(&a.n_rec, hdr + 72, 8);
  memcpy(&a.payload, hdr + 96, 8);
  memcpy(a.n_codec, hdr + 116, 12);
  a.g = g;
  a.st = st;
  a.ar = ar;
  a.bytes = bytes;
  a.off_codec = kHdr;
  a.off_bb = kHdr + a8(g.nblk);
  a.off_rec = a.off_bb + a8(4ull * g.nblk);
  a.off_pay = a.off_rec + 8 * a.n_rec;
  a.off_books = a.off_pay + a8(a.payload);
  a.ebx2_f = 2.0f * eb;
  a.blk_off = at<uint64_t>(ws, L.blk_off);
  a.rec_start = at<uint32_t>(ws, L.rec_start);
  a.tabs = at<DecTab>(ws, L.tabs);
  a.codes = at<uint16_t>(ws, L.codes);
  a.runv = a.codes;
  a.runl = at<uint16_t>(ws, L.runl);
  a.runblk = at<uint32_t>(ws, L.runblk);
  a.slowblk = at<uint32_t>(ws, L.slowblk);
  a.prep_lb = at<uint64_t>(ws, L.prep_lb);
  a.global = (a.flags & kFlagGlobal) != 0;
  a.fuse = !a.global;
  a.scan_state = at<uint64_t>(ws, L.lb_e);
  a.gtotals = reinterpret_cast<int32_t*>(a.runl);
  a.gstrips = a.gtotals + 512ull * g.nblk;
  a.out = out;
  if (launch_decode(a, nullptr) != cudaSuccess) return 3;
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 4;
}
