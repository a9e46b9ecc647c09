// Fused step of small lattices (included once per storage type): one CTA per
// box of BX x BY x BZ cells, one thread per cell of the box and its one-cell
// ring.  Every thread pulls its cell and writes (rho^N, Qbar) into a
// shared-memory window; after one barrier the box's own threads -- whose
// populations stayed in registers -- take the Eq. 49 gradients, collide and
// store.
//
// Why a form of its own: on a few ten thousand cells the step is bound by the
// length of a CTA's serial chain, not by memory.  The z-marching kernels walk
// at least six planes plus two halo planes one after the other (pull latency,
// barrier, collision each time) in 10 to 20 CTAs; here a step is one pull, one
// barrier and one collision, spread over every SM.  The ring's pulls are
// redundant (a 4 x 4 x 4 box pulls 208 cells for 64, an 8 x 4 x 4 box 352 for
// 128) but hit L2, which holds both buffers at these sizes.  GB300, us per
// step in a run of 200, marching kernel -> box: 4 x 128 x 4 with walls 19.6
// -> 2.6, 16^3 16.4 -> 2.7, 24^3 17.6 -> 3.5, 32^3 26.4 -> 4.4, 40^3 24.6 ->
// 7.2, FP16 13.3 -> 6.7.  Which box: 4 x 4 x 4 while its CTAs leave SMs idle
// (20^3: 125 CTAs 2.7, 8 x 4 x 4 3.1), the larger box with less ring on more
// cells (32^3: 512 CTAs 6.8, 256 CTAs 4.4).  The two are level at about 10,000
// cells (22^3 3.4 / 3.2, 25^3 4.2 / 4.4, 32 x 32 x 16 4.7 / 3.2); the line in
// default_box, 16,384, is that of an earlier overlap of the launches, under
// which 24^3 took 3.6 / 3.9.  8 x 8 x 4 and 16 x 4 x 4 boxes were no faster
// anywhere (then: 32^3 4.5 and 4.3, 48^3 12.0 and 11.5 against 10.8).
#pragma once

#include "lbm_fused.cuh"

namespace lbm {

// Thread -> site of the box with its ring, in window coordinates (0 .. B + 1
// on each axis): the box's cells first, so that the collision's warps are
// full, then the z faces, then the perimeter of every inner plane.
template <int BX, int BY, int BZ>
struct BoxShape {
  static constexpr int SX = BX + 2, SY = BY + 2, SZ = BZ + 2;
  static constexpr int kCells = BX * BY * BZ;
  static constexpr int kSites = SX * SY * SZ;
  static constexpr int kThreads = (kSites + 31) / 32 * 32;
  // CTAs per SM the registers must allow (96 and 80 a thread)
  static constexpr int kCtasPerSm = kThreads <= 224 ? 3 : 2;
  __device__ __forceinline__ static void site(int t, int& sx, int& sy, int& sz) {
    if (t < kCells) {
      sx = 1 + t % BX;
      sy = 1 + t / BX % BY;
      sz = 1 + t / (BX * BY);
      return;
    }
    int r = t - kCells;
    if (r < 2 * SX * SY) {
      sz = r < SX * SY ? 0 : SZ - 1;
      r = r < SX * SY ? r : r - SX * SY;
      sx = r % SX;
      sy = r / SX;
      return;
    }
    r -= 2 * SX * SY;
    constexpr int P = 2 * SX + 2 * BY;  // perimeter of an inner plane
    sz = 1 + r / P;
    r %= P;
    if (r < 2 * SX) {
      sx = r % SX;
      sy = r < SX ? 0 : SY - 1;
    } else {
      r -= 2 * SX;
      sx = r < BY ? 0 : SX - 1;
      sy = 1 + (r < BY ? r : r - BY);
    }
  }
};

template <typename T, int BX, int BY, int BZ, bool WALLS>
__global__ void __launch_bounds__((BoxShape<BX, BY, BZ>::kThreads),
                                  (BoxShape<BX, BY, BZ>::kCtasPerSm))
    k_fused_box(const T* src, T* dst, const __grid_constant__ StepArgs a) {
  using S = BoxShape<BX, BY, BZ>;
  using Pair = typename Store<T>::Pair;
  __shared__ float4 win[S::SZ][S::SY][S::SX];
  const int t = threadIdx.x;
  int sx, sy, sz;
  S::site(t, sx, sy, sz);
  // launched with programmatic stream serialisation: the next step's CTAs may
  // start (and wait here) while this one runs, which hides their launch
  after_previous_kernel();
  const int cx = blockIdx.x * BX + sx - 1, cy = blockIdx.y * BY + sy - 1,
            cz = blockIdx.z * BZ + sz - 1;  // unwrapped
  // sites that some cell of the box reads: inside the lattice or one cell
  // beyond a periodic face; the stencil reads no corner of the ring
  const bool corner = (sx == 0 || sx == S::SX - 1) && (sy == 0 || sy == S::SY - 1) &&
                      (sz == 0 || sz == S::SZ - 1);
  bool used = t < S::kSites && !corner && cx <= a.nx && cy <= a.ny && cz <= a.nz;
  if (WALLS)
    used = used && !(a.wx && (cx < 0 || cx >= a.nx)) && !(a.wy && (cy < 0 || cy >= a.ny)) &&
           !(a.wz && (cz < 0 || cz >= a.nz));
  float f[19], rR = 0.f, rB = 0.f;
  Macro m;
  unsigned cell = 0;
  if (used) {
    const int x = cx < 0 ? a.nx - 1 : (cx == a.nx ? 0 : cx);
    const int y = cy < 0 ? a.ny - 1 : (cy == a.ny ? 0 : cy);
    const int z = cz < 0 ? a.nz - 1 : (cz == a.nz ? 0 : cz);
    const ColOff co = col_off(a, x, y);
    const PlaneOff po = plane_off(a, z);
    cell = po.zo[1] + co.yo[1] + co.xo[1];
    pull_reduce<T, WALLS, true>(reinterpret_cast<const Pair*>(src), (unsigned)a.plane, a, co, po,
                                f, rR, rB);
    m = macro_total(a, f, rR, rB);
    win[sz][sy][sx] = stencil_entry(a, m);
  }
  __syncthreads();
  if (t >= S::kCells || cx >= a.nx || cy >= a.ny || cz >= a.nz) return;
  const bool xlo = WALLS && a.wx && cx == 0, xhi = WALLS && a.wx && cx == a.nx - 1;
  const bool ylo = WALLS && a.wy && cy == 0, yhi = WALLS && a.wy && cy == a.ny - 1;
  const bool zlo = WALLS && a.wz && cz == 0, zhi = WALLS && a.wz && cz == a.nz - 1;
  const float4 ctr = win[sz][sy][sx];
  float Gx, Gy, Gz, Qx, Qy, Qz;
  stencil_gradients(
      [&](int dx, int dy, int dz) -> const float4& { return win[sz + dz][sy + dy][sx + dx]; },
      ctr, xlo, xhi, ylo, yhi, zlo, zhi, Gx, Gy, Gz, Qx, Qy, Qz);
  if (WALLS && a.wetting) wetting_rule(a, xlo, xhi, ylo, yhi, zlo, zhi, Gx, Gy, Gz);
  const Recolour rc = collide_total<false>(a, f, m, ctr.x, Gx, Gy, Gz, Qx, Qy, Qz);
  store_recoloured<T>(dst, (unsigned)a.plane, a, cell, rc, f);
}

template <typename T, int BX, int BY, int BZ, bool WALLS>
static cudaError_t launch_box_v(const void* src, void* dst, const StepArgs& a, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((a.nx + BX - 1) / BX, (a.ny + BY - 1) / BY, (a.nz + BZ - 1) / BZ);
  cfg.blockDim = dim3(BoxShape<BX, BY, BZ>::kThreads);
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_fused_box<T, BX, BY, BZ, WALLS>, (const T*)src, (T*)dst, a);
}

template <typename T, int BX, int BY, int BZ>
static cudaError_t launch_box_b(const void* src, void* dst, const StepArgs& a, cudaStream_t s) {
  return a.wx || a.wy || a.wz ? launch_box_v<T, BX, BY, BZ, true>(src, dst, a, s)
                              : launch_box_v<T, BX, BY, BZ, false>(src, dst, a, s);
}

template <typename T>
cudaError_t launch_fused_box_storage(const void* src, void* dst, const StepArgs& a, int box,
                                     cudaStream_t s) {
  switch (box) {
    case 1: return launch_box_b<T, 4, 4, 4>(src, dst, a, s);
    case 2: return launch_box_b<T, 8, 4, 4>(src, dst, a, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace lbm
