// Storage-type dispatch and launch configuration of the fused step.
#include <algorithm>
#include <functional>
#include <vector>

#include "lbm_internal.h"

namespace lbm {

cudaError_t launch_fused(int storage, const void* src, void* dst,
                         const StepArgs& a, const FusedConfig& cfg,
                         cudaStream_t s) {
  switch (storage) {
    case 0: return launch_fused_storage<float>(src, dst, a, cfg, s);
    case 1: return launch_fused_storage<__half>(src, dst, a, cfg, s);
    case 2: return launch_fused_storage<__nv_bfloat16>(src, dst, a, cfg, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_fused_box(int storage, const void* src, void* dst, const StepArgs& a, int box,
                             cudaStream_t s) {
  switch (storage) {
    case 0: return launch_fused_box_storage<float>(src, dst, a, box, s);
    case 1: return launch_fused_box_storage<__half>(src, dst, a, box, s);
    case 2: return launch_fused_box_storage<__nv_bfloat16>(src, dst, a, box, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_fused_batch(int storage, const void* src, void* dst,
                               const BatchCase* cases, int ncases,
                               int total_items, bool walls, bool bgk,
                               const FusedConfig& cfg, int sms, cudaStream_t s) {
  switch (storage) {
    case 0: return launch_fused_batch_storage<float>(src, dst, cases, ncases, total_items, walls, bgk, cfg, sms, s);
    case 1: return launch_fused_batch_storage<__half>(src, dst, cases, ncases, total_items, walls, bgk, cfg, sms, s);
    case 2: return launch_fused_batch_storage<__nv_bfloat16>(src, dst, cases, ncases, total_items, walls, bgk, cfg, sms, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_fused_tma(int storage, const void* src, void* dst, const StepArgs& a,
                             const CUtensorMap* maps, int kind, int ns, int zchunk, int* err,
                             cudaStream_t s) {
  switch (storage) {
    case 0: return launch_fused_tma_storage<float>(src, dst, a, maps, kind, ns, zchunk, err, s);
    case 1: return launch_fused_tma_storage<__half>(src, dst, a, maps, kind, ns, zchunk, err, s);
    case 2:
      return launch_fused_tma_storage<__nv_bfloat16>(src, dst, a, maps, kind, ns, zchunk, err,
                                                     s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_fused_tma_batch(int storage, const void* src, void* dst,
                                   const BatchCase* cases, int ncases, int total_items,
                                   bool walls, const CUtensorMap* maps, int kind, int ns, int zc,
                                   int* err, int sms, cudaStream_t s) {
  if (kind != 0 && kind != 2) return cudaErrorInvalidValue;
  switch (storage) {
    case 0:
      return launch_fused_tma_batch_storage<float>(src, dst, cases, ncases, total_items, walls,
                                                   maps, kind, ns, zc, err, sms, s);
    case 1:
      return launch_fused_tma_batch_storage<__half>(src, dst, cases, ncases, total_items, walls,
                                                    maps, kind, ns, zc, err, sms, s);
    case 2:
      return launch_fused_tma_batch_storage<__nv_bfloat16>(src, dst, cases, ncases, total_items,
                                                           walls, maps, kind, ns, zc, err, sms,
                                                           s);
  }
  return cudaErrorInvalidValue;
}

int tma_kind(int tile_y) { return tile_y == 8 ? 0 : (tile_y == 16 ? 1 : (tile_y == 15 ? 2 : -1)); }

static const int kTmaTW[3] = {32, 16, 34}, kTmaBY[3] = {8, 16, 15};

bool tma_config_fits(int storage, int kind, int ns) {
  if (kind < 0 || kind > 2 || ns < 1 || ns > 2) return false;
  switch (storage) {
    case 0: return tma_config_fits_storage<float>(kind, ns);
    case 1: return tma_config_fits_storage<__half>(kind, ns);
    case 2: return tma_config_fits_storage<__nv_bfloat16>(kind, ns);
  }
  return false;
}

// Pair bytes of a storage type (red and blue value of one direction and cell).
static int pair_bytes(int storage) { return storage == 0 ? 8 : 4; }

// The TMA forms are built for the MRT operator only (a BGK context runs the
// shared-memory-hold form).
bool tma_eligible(const StepArgs& a, int storage) {
  return ((long long)a.nx * pair_bytes(storage)) % 16 == 0 && a.nz >= 3 && !a.bgk;
}

// Default TMA configuration.  Tile: the one with more interior cells per
// launched thread for this nx x ny (the 34 x 15 tile wins where nx is a
// multiple of 32, the 32 x 8 tile where it is a multiple of 30).  Stages:
// two for FP32, one for 16-bit storage.  z chunk: each CTA refills two halo
// planes (about half a plane of work), and CTAs run in rounds of (SMs x
// CTAs per SM), so the chunk minimises rounds x (zchunk + 1/2).  On GB300 at
// 128^3 this picks the 34 x 15 tile with 12-plane chunks: 14.4 GLUPS (FP32)
// and 15.7 GLUPS (FP16) against 13.1 and 14.6 for the shared-memory hold.
// 16-bit storage on a lattice where the 32 x 8 tile fits better keeps the
// plain shared-memory hold, which is ahead of its TMA form there.
bool tma_default_config(const StepArgs& a, int storage, int sms, const bool kind_ok[3],
                        FusedConfig* out) {
  if (!tma_eligible(a, storage)) return false;
  double best_eff = -1.0;
  int kind = -1;
  for (int k : {0, 2}) {
    if (!kind_ok[k]) continue;
    const int tw = kTmaTW[k], by = kTmaBY[k];
    const double tiles = (double)((a.nx + tw - 3) / (tw - 2)) * ((a.ny + by - 3) / (by - 2));
    const double eff = (double)a.nx * a.ny / (tiles * tw * by);
    if (eff > best_eff * 1.02) {
      best_eff = eff;
      kind = k;
    }
  }
  if (kind < 0) return false;
  const int ns = storage == 0 ? 2 : 1;
  if (storage != 0 && kind == 0) return false;
  if (!tma_config_fits(storage, kind, ns)) return false;
  const int tw = kTmaTW[kind], by = kTmaBY[kind];
  const long long cols = (long long)((a.nx + tw - 3) / (tw - 2)) * ((a.ny + by - 3) / (by - 2));
  const long long slots = (long long)(sms > 0 ? sms : 152) * (kind == 2 ? 1 : 2);
  int best_zc = 12;
  double best_cost = 1e300;
  for (int zc = 6; zc <= 24; ++zc) {
    const long long ctas = cols * ((a.nz + zc - 1) / zc);
    const double cost = (double)((ctas + slots - 1) / slots) * (zc + 1.5);
    if (cost <= best_cost + 1e-9) {
      best_cost = cost;
      best_zc = zc;
    }
  }
  out->tile_y = by;
  out->hold = ns == 2 ? 7 : 8;
  out->zchunk = best_zc < a.nz ? best_zc : a.nz;
  return true;
}

// Two tensor maps over a population buffer seen as a 4-D array of pairs
// [direction][z][y][x] (x fastest; direction stride = the padded plane),
// for a tile of tw x by threads: FP32 map 0 has tw-pair boxes, map 1
// (tw + 2)-pair boxes; 16-bit storage uses tw + 4 pairs rounded up to a
// multiple of 4 (map 1 = map 0).  Boxes are by rows by one plane by one direction, no swizzle; cells
// beyond the array read as zero.
// One tensor map over a population buffer seen as [direction][z][y][x]
// pairs, with a box of w x h pairs (one plane, one direction).
cudaError_t tensor_map_encoder(EncodeTiledFn* out) {
  static EncodeTiledFn encode = nullptr;
  if (!encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                     cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn)
      return e != cudaSuccess ? e : cudaErrorNotSupported;
    encode = (EncodeTiledFn)fn;
  }
  *out = encode;
  return cudaSuccess;
}

static cudaError_t encode_box(int storage, const void* base, const StepArgs& a, unsigned w,
                              unsigned h, CUtensorMap* map) {
  EncodeTiledFn encode = nullptr;
  const cudaError_t e = tensor_map_encoder(&encode);
  if (e != cudaSuccess) return e;
  const cuuint64_t E = (cuuint64_t)pair_bytes(storage);
  const cuuint64_t dims[4] = {(cuuint64_t)a.nx, (cuuint64_t)a.ny, (cuuint64_t)a.nz, 19};
  const cuuint64_t strides[3] = {E * a.nx, E * a.nx * a.ny, E * (cuuint64_t)a.plane};
  const cuuint32_t es[4] = {1, 1, 1, 1};
  const CUtensorMapDataType dt =
      storage == 0 ? CU_TENSOR_MAP_DATA_TYPE_UINT64 : CU_TENSOR_MAP_DATA_TYPE_UINT32;
  const cuuint32_t box[4] = {(cuuint32_t)w, (cuuint32_t)h, 1, 1};
  const CUresult r = encode(map, dt, 4, const_cast<void*>(base), dims, strides, box, es,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t tma_build_maps(int storage, const void* base, const StepArgs& a, int kind,
                           CUtensorMap maps[2]) {
  if (kind < 0 || kind > 2) return cudaErrorInvalidValue;
  if (!tma_eligible(a, storage)) return cudaErrorInvalidValue;
  const int tw = kTmaTW[kind], by = kTmaBY[kind];
  for (int m = 0; m < 2; ++m) {
    const unsigned w = (unsigned)(storage == 0 ? (m == 0 ? tw : tw + 2) : (tw + 4 + 3) / 4 * 4);
    cudaError_t e = encode_box(storage, base, a, w, (unsigned)by, &maps[m]);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// z chunk in [lo, hi] whose list schedule of cols x ceil(nz / chunk) CTAs over
// `slots` places ends first, a CTA of p planes costing p + overhead (ties: the
// longer chunk); at most nz.
static int schedule_zchunk(long long cols, int nz, int slots, int lo, int hi, double overhead);

int seam12_zchunk(const StepArgs& a, int sms) { return list_schedule_zchunk(a, sms, 10); }

int list_schedule_zchunk(const StepArgs& a, int sms, int rows) {
  // One CTA per SM; the hardware hands the CTAs out in launch order (tile
  // columns fastest, then z chunks) to whichever SM falls free, so a step
  // lasts as long as that list schedule.  A CTA of p planes costs p + 3
  // plane-times (two halo planes and a pipeline start).  The full chunks all
  // last the same and fill the SMs round by round; the shorter last chunk's
  // CTAs are placed one by one.  Over 6..32 planes at 128^3..256^3 this
  // picks the measured fastest chunk, where counting whole rounds of
  // equal CTAs picked 16 planes at 128^3 (4.5 % slower than 24).  Chunks
  // up to 48 planes: measured against the 32-plane limit it had before,
  // its picks run 3.4 % faster on the 256 x 256 x 1024 lattice, 0.9-2.2 %
  // faster at 128^3 (16-bit) and 192^3 / 256^3, within 0.1 % at 192^3
  // FP32 and 1.6-3.2 % slower at 160^3; beyond 48 planes the CTAs marching
  // neighbouring columns drift apart and the model, which does not see
  // that, goes wrong (128 planes on the 1024-plane lattice: 12 % slower).
  const long long cols = (long long)((a.nx + 31) / 32) * ((a.ny + rows - 1) / rows);
  return schedule_zchunk(cols, a.nz, sms > 0 ? sms : 152, 6, 48, 3.0);
}

static int schedule_zchunk(long long cols, int nz, int slots, int lo, int hi, double overhead) {
  std::vector<double> heap((size_t)slots);
  int best_zc = 12;
  double best_span = 1e300;
  for (int zc = lo; zc <= hi; ++zc) {
    const long long full = (long long)(nz / zc) * cols;
    const int tail = nz % zc;
    const double d = zc + overhead;
    const long long rounds = full / slots, extra = full % slots;
    for (int j = 0; j < slots; ++j) heap[(size_t)j] = (double)(rounds + (j < extra)) * d;
    double span = (double)(rounds + (extra > 0)) * d;
    if (tail > 0) {
      auto later = std::greater<double>();
      std::make_heap(heap.begin(), heap.end(), later);
      for (long long c = 0; c < cols; ++c) {
        std::pop_heap(heap.begin(), heap.end(), later);
        heap.back() += tail + overhead;
        span = std::max(span, heap.back());
        std::push_heap(heap.begin(), heap.end(), later);
      }
    }
    if (span <= best_span + 1e-9) {
      best_span = span;
      best_zc = zc;
    }
  }
  return best_zc < nz ? best_zc : nz;
}

bool seam_eligible(const StepArgs& a, int storage) {
  return storage == 0 && tma_eligible(a, storage) && !a.wx && !a.wy && a.nx >= kTmaTW[2] &&
         a.ny >= kTmaBY[2];
}

cudaError_t tma_build_seam_maps(const void* base, const StepArgs& a, int tile_y,
                                CUtensorMap maps[6]) {
  // the strips need periodic x and y; the batched form also builds them for
  // cases narrower than a tile (its lanes fall back to global pulls there)
  if (!tma_eligible(a, 0) || a.wx || a.wy || (tile_y != 15 && tile_y != 12))
    return cudaErrorInvalidValue;
  const unsigned tw = (unsigned)kTmaTW[2], by = (unsigned)tile_y;
  const unsigned shape[6][2] = {{tw, by}, {tw + 2, by}, {2, by}, {tw, 2}, {tw + 2, 2}, {2, 2}};
  for (int m = 0; m < 6; ++m) {
    cudaError_t e = encode_box(0, base, a, shape[m][0], shape[m][1], &maps[m]);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

bool seam16_eligible(const StepArgs& a, int storage) {
  return storage != 0 && tma_eligible(a, storage) && !a.wx && !a.wy && a.nx >= kTmaTW[2] &&
         a.ny >= kTmaBY[2];
}

cudaError_t tma_build_seam16_maps(int storage, const void* base, const StepArgs& a, int tile_y,
                                  CUtensorMap maps[4]) {
  if (!seam16_eligible(a, storage) || (tile_y != 15 && tile_y != 12))
    return cudaErrorInvalidValue;
  const unsigned w = (unsigned)(kTmaTW[2] + 4 + 3) / 4 * 4, by = (unsigned)tile_y;
  const unsigned shape[4][2] = {{w, by}, {4, by}, {w, 2}, {4, 2}};
  for (int m = 0; m < 4; ++m) {
    cudaError_t e = encode_box(storage, base, a, shape[m][0], shape[m][1], &maps[m]);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_fused_tma_seam16(int storage, const void* src, void* dst, const StepArgs& a,
                                    int tile_y, const CUtensorMap* maps4, int zchunk, int* err,
                                    cudaStream_t s, MonAcc* mon) {
  if (storage == 1)
    return launch_fused_tma_seam16_storage<__half>(src, dst, a, tile_y, maps4, zchunk, err, s,
                                                   mon);
  if (storage == 2)
    return launch_fused_tma_seam16_storage<__nv_bfloat16>(src, dst, a, tile_y, maps4, zchunk,
                                                          err, s, mon);
  return cudaErrorInvalidValue;
}

// Batched kernel variants: (tile_y, hold) = (8, 2), (8, 0), (16, 1), and
// the TMA forms (8 or 15, 7 or 8) where the context built tensor maps.
bool valid_batch_config(const FusedConfig& c) {
  const bool shape = (c.tile_y == 8 && (c.hold == 2 || c.hold == 0)) ||
                     (c.tile_y == 16 && c.hold == 1) ||
                     ((c.tile_y == 8 || c.tile_y == 15) && (c.hold == 7 || c.hold == 8)) ||
                     (c.tile_y == 12 && c.hold == 7);
  return shape && c.zchunk > 0;
}

// A batch's CTAs in one form of the step: places (SMs x CTAs per SM), and when
// the last CTA ends, in plane-times.  The CTAs are handed out in launch order
// to the place that falls free first; past 8192 of them the schedule is taken
// as their work over the places and half a CTA's for the ragged end.
namespace {
class BatchSpan {
 public:
  explicit BatchSpan(int places) : free_((size_t)places, 0.0) {}
  void add(const StepArgs& a, int iw, int ih, int zc, double overhead) {
    const long long tiles = (long long)((a.nx + iw - 1) / iw) * ((a.ny + ih - 1) / ih);
    for (int z = 0; z < a.nz; z += zc) {
      const double d = std::min(zc, a.nz - z) + overhead;
      longest_ = std::max(longest_, d);
      work_ += (double)tiles * d;
      if ((items_ += tiles) > 8192) continue;
      auto later = std::greater<double>();
      for (long long t = 0; t < tiles; ++t) {
        std::pop_heap(free_.begin(), free_.end(), later);
        free_.back() += d;
        end_ = std::max(end_, free_.back());
        std::push_heap(free_.begin(), free_.end(), later);
      }
    }
  }
  long long items() const { return items_; }
  double end() const {
    return items_ > 8192 ? work_ / (double)free_.size() + 0.5 * longest_ : end_;
  }

 private:
  std::vector<double> free_;
  long long items_ = 0;
  double work_ = 0.0, longest_ = 0.0, end_ = 0.0;
};
}  // namespace

// Which form a batch runs: the one whose schedule ends first, a plane-time
// taking 3.75 us on the 34 x 15 tile (its seam lanes pull from global memory),
// 2.75 us on the 34 x 12 seam form and 2.85 us on the 32 x 8 tile with two CTAs
// per SM.  GB300, us per step in these three, FP32: 128 boxes of 64 x 64 x 32
// with a floor 1226 / 1140 / 1657; 60 of 64 x 64 x 24 426 / 456 / 557; 60 of 40 x
// 40 x 24 367 / 304 / 242; 60 of 48 x 51 x 37 562 / 647 / 493; 60 of 96 x 40 x 32
// 624 / 502 / 649; 60 of 96 x 64 x 24 602 / 657 / 752; 48 droplet boxes of 32 to
// 96 cells 1268 / 1535 / 1481; 16 bits, 34 x 15 / 32 x 8: 60 of 40 x 40 x 24 326 /
// 241, 60 of 64 x 72 x 32 670 / 812.  The seam form only where no box is narrower
// than its tile (the droplet boxes' 32-cell ones are what slows it there).  A
// batch of fewer than 32 CTAs keeps the tensor-copy form, the slower one there
// (three boxes of 40 x 40 x 24 100 us against 31 on the 32 x 8 tile, two of 32^3
// and two of 64 x 64 x 32 133 and 131 against 31 and 42): its bounded waits and
// their report are what is specified of the smallest batches; lbm_set_fused_config
// gives a program the faster form.
void batch_default_config(const StepArgs* const* args, int ncases, int storage, int sms,
                          bool seam_ok, FusedConfig* c) {
  BatchSpan t15(sms), t12(sms), t8(2 * sms);
  bool seam = storage == 0 && seam_ok;
  for (int k = 0; k < ncases; ++k) {
    const StepArgs& a = *args[k];
    t15.add(a, 32, 13, 32, 3.0);
    t12.add(a, 32, 10, 32, 3.0);
    t8.add(a, 30, 6, 12, 2.5);
    seam = seam && a.nx >= kTmaTW[2] && a.ny >= kTmaBY[2];
  }
  if (t15.items() < 32) return;
  const double c15 = 3.75 * t15.end(), c12 = 2.75 * t12.end(), c8 = 2.85 * t8.end();
  if (seam && c12 < c15 && c12 <= c8) {
    c->tile_y = 12;
    c->zchunk = 32;
    c->hold = 7;
  } else if (c8 < c15) {
    c->tile_y = 8;
    c->zchunk = 12;
    c->hold = 2;
  }
}

bool batch_seam_eligible(const StepArgs& a, int storage) {
  return storage == 0 && tma_eligible(a, storage) && !a.wx && !a.wy && !a.bgk;
}

bool valid_fused_config(const FusedConfig& c, int storage) {
  if (c.tile_y == 15) return (c.hold == 7 || c.hold == 8) && c.zchunk > 0;
  if (c.tile_y != 8 && c.tile_y != 16) return false;
  if (c.hold < 0 || c.hold > 8) return false;
  if ((c.hold == 2 || c.hold == 3 || c.hold == 5 || c.hold == 6) && c.tile_y != 8) return false;
  if (c.hold == 4 && c.tile_y != 16) return false;
  (void)storage;
  return c.zchunk > 0;
}

// Default: 30 x 6 interior tiles, reduced state held in shared memory, two
// CTAs per SM.  The z chunk is the one whose list schedule over the 2 x 152
// slots ends first, as for the seam forms (list_schedule_zchunk); halo planes
// and start cost 2.5 planes here.  GB300, us per step, against 12 planes halved
// while the grid left slots empty: 101 x 99 x 67 with walls 16 planes 61.7, 12
// planes 81.5 (408 CTAs for 304 slots: a second round a third full); 129 x 65
// x 150 28 planes 108, 12 planes 122; 200 x 100 x 100 BGK 41 planes 149, 12
// planes 161; within 4 % of the fastest of 15 chunks on seven odd, walled and
// 16-bit lattices.
FusedConfig default_fused_config(const StepArgs& a, int storage) {
  (void)storage;
  FusedConfig c;
  c.tile_y = 8;
  c.hold = 2;
  const long long cols = (long long)((a.nx + 29) / 30) * ((a.ny + 5) / 6);
  c.zchunk = schedule_zchunk(cols, a.nz, 2 * 152, 3, 48, 2.5);
  return c;
}

// The box form's range, GB300, us per step (box / the fastest marching chunk).
// Without a seam form it wins up to about 180,000 cells: walls all round 45^3
// 11.4 / 14.4, 53^3 17.0 / 18.4, 57^3 21.2 / 18.4, 59^3 21.4 / 18.4; FP16 10.5 /
// 14.3, 15.9 / 17.4, 19.3 / 17.4, 19.5 / 17.4.
// On the lattices of the seam forms the line at 81,920 cells is not where the two
// are equal: 64 x 40 x 32 9.2 / 24.6, 64 x 40 x 36 (beyond it) 9.5 / 25.6, 48^3 10.6
// / 24.6, 56^3 16.2 / 24.7, 64^3 23.9 / 28.5, 72^3 36.2 / 39.9; FP16 48^3 9.7 / 13.3,
// 56^3 14.9 / 16.4, 60^3 18.8 / 16.4, 64^3 21.7 / 28.7.  It keeps the tensor-copy
// kernels, whose bounded waits report through the error word, the default of the
// lattices on which that is specified (from 92,160 cells on); lbm_set_box gives a
// program the faster form there.
// BGK lattices keep the shared-memory-hold kernel: its multiply-adds and the box
// form's are contracted differently, and under that operator a changed last bit
// grows near tau_v = 1/2 (a closed box of drops 4e-5 apart after 60 steps, a
// Rayleigh-Taylor column overflowing in other cells).
int default_box(const StepArgs& a, int storage) {
  if (a.bgk) return 0;
  const long long N = (long long)a.nx * a.ny * a.nz;
  const bool seam = seam_eligible(a, storage) || seam16_eligible(a, storage);
  if (N > (seam ? 81920 : 180000)) return 0;
  return N <= 16384 ? 1 : 2;
}

}  // namespace lbm
