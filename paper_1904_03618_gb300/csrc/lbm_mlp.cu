// Surrogate network on the 5th-generation tensor cores (sm_103a).
//
// The network maps impact parameters to a spreading-factor series: dense
// layers x -> tanh(x W + b) -> ... -> (. W_out + b_out), trained with mean
// squared error and Adam.  Every matrix product of the forward and backward
// passes runs on the tensor cores: inference and training steps of up to 4096
// rows in the whole-network kernels of lbm_net.cuh; the products of larger
// training batches (and lbm_gemm_bf16) in k_gemm_ws when K is at most 256
// (a persistent warp-specialised kernel, described above it) or split over
// it, and otherwise in k_gemm_tc:
//   - a CTA owns a 128-row tile of C (all of C's columns, N <= 256);
//   - the A (128 x 64) and B (N x 64) K-slices are converted to BF16 and
//     written into shared memory in the canonical K-major layout without
//     swizzle (8-row x 16-byte core matrices; K-adjacent core matrices 128 B
//     apart, 8-row groups 1024 B apart);
//   - one elected thread issues tcgen05.mma (kind::f16, BF16 x BF16 -> FP32,
//     M = 128, K = 16 per instruction) into a TMEM accumulator, then
//     tcgen05.commit signals an mbarrier; every thread waits on it with a
//     bounded spin before the slices are overwritten;
//   - the epilogue reads the accumulator with tcgen05.ld (one TMEM lane per
//     row) and applies bias + tanh, or the tanh derivative of the backward
//     pass, before storing FP32.
// FP32 master weights and activations live in global memory; operands are
// rounded to BF16 when staged (FP32 accumulation).
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <cstddef>
#include <cstdint>
#include <new>
#include <type_traits>

#include "lbm_internal.h"

namespace lbm {
namespace mlp {

constexpr int kM = 128;     // rows per CTA (UMMA M)
constexpr int kKT = 64;     // K per shared-memory slice
constexpr int kNMax = 256;  // UMMA N limit for M = 128
constexpr int kThreads = 128;
// Bounded mbarrier wait: g_mma_wait_ns, kWaitNs unless a test has shortened
// it to exercise the give-up path; the second chance before TMEM is released
// always waits up to kWaitNs.
constexpr unsigned long long kWaitNs = 200ull * 1000 * 1000;
static __device__ unsigned long long g_mma_wait_ns = kWaitNs;

struct GemmArgs {
  const float* A;
  long long sa_m, sa_k;  // A(m, k) = A[m * sa_m + k * sa_k]
  const float* B;
  long long sb_k, sb_n;  // B(k, n) = B[k * sb_k + n * sb_n]
  int M, N, K;
  const float* bias;     // epilogue: C = act(acc + bias) (bias nullable)
  int act;               // 0 identity, 1 tanh
  const float* H;        // if non-null: C = acc * (1 - H^2) (tanh backward)
  long long sh_m;
  float* C;
  long long sc_m;
  int* err;              // set to 1 if a bounded wait gives up
  int splits;            // K split over gridDim.y CTAs; > 1: C zeroed, partials added
  int ws_bn;             // k_gemm_ws: columns per CTA
};

struct GemmSmem {
  __nv_bfloat16 a[kM * kKT];      // 16 KB
  __nv_bfloat16 b[kNMax * kKT];   // 32 KB
  unsigned long long mbar;
  unsigned tmem_base;
};

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}

// Byte offset of element (row, k) of a K-major slice in the canonical
// no-swizzle layout.
__device__ __forceinline__ unsigned core_offset(int row, int k) {
  return (unsigned)(((row >> 3) * (kKT / 8) + (k >> 3)) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

// Shared-memory matrix descriptor (SM100 form): start address, leading-
// dimension byte offset (between K-adjacent core matrices), stride byte
// offset (between 8-row groups), version 1, no swizzle.
__device__ __forceinline__ unsigned long long smem_desc(unsigned addr, unsigned lbo,
                                                        unsigned sbo) {
  unsigned long long d = 0;
  d |= (unsigned long long)((addr >> 4) & 0x3FFFu);
  d |= (unsigned long long)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (unsigned long long)((sbo >> 4) & 0x3FFFu) << 32;
  d |= 1ull << 46;
  return d;
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, M = 128, N.
__device__ __forceinline__ unsigned instr_desc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(n >> 3) << 17) |
         ((unsigned)(kM >> 4) << 24);
}

__device__ __forceinline__ bool mbar_poll(unsigned addr, unsigned phase) {
  unsigned done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(done)
      : "r"(addr), "r"(phase)
      : "memory");
  return done != 0;
}
__device__ __forceinline__ bool mbar_test(unsigned addr, unsigned phase) {
  unsigned done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(done)
      : "r"(addr), "r"(phase)
      : "memory");
  return done != 0;
}
// The give-up limit of this launch, read once per CTA (a volatile read:
// only the host writes it, so its initial value is no constant).
__device__ __forceinline__ unsigned long long mma_wait_limit() {
  return *(const volatile unsigned long long*)&g_mma_wait_ns;
}
// Bounded wait: `limit` ns of wall time on the global timer.  A limit below
// 1000 ns (shorter than a tick of that timer, and than the time a blocking
// try_wait may suspend the thread) is a test of the give-up path: one
// non-blocking poll decides.
__device__ __forceinline__ bool mbar_wait(unsigned addr, unsigned phase,
                                          unsigned long long limit = kWaitNs) {
  if (limit < 1000) return mbar_test(addr, phase);
  if (mbar_poll(addr, phase)) return true;
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  while (!mbar_poll(addr, phase)) {
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t - t0 > limit) return false;
  }
  return true;
}

// Stages the ROWS x 64 slice X(r, k), r in [r0, r0 + ROWS), k in [k0, k0 + 64),
// of X(r, k) = X[r * s_r + k * s_k] into the K-major core layout as BF16, zero
// outside [0, R) x [0, K).  Where one stride is 1 and 16-byte groups are
// aligned, each thread issues a batch of 16-byte loads before converting
// and storing any of them (memory-level parallelism); the ragged edge and
// other strides take scalar loads.
template <int ROWS>
__device__ __forceinline__ void stage_slice(unsigned char* dst, const float* __restrict__ X,
                                            long long s_r, long long s_k, int r0, int R,
                                            int k0, int K, int tid) {
  constexpr int kBatch = 8;
  const bool aligned = (reinterpret_cast<unsigned long long>(X) & 15u) == 0;
  if (s_k == 1 && aligned && (s_r & 3) == 0) {
    // groups of 4 consecutive k: ROWS x 16 groups
    constexpr int G = ROWS * (kKT / 4);
    for (int base = 0; base < G; base += kThreads * kBatch) {
      float4 v[kBatch];
#pragma unroll
      for (int b = 0; b < kBatch; ++b) {
        const int t = base + b * kThreads + tid;
        const int r = t / (kKT / 4), kq = (t % (kKT / 4)) * 4;
        const int m = r0 + r, kk = k0 + kq;
        v[b] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (t < G && m < R) {
          const float* p = X + m * s_r + kk;
          if (kk + 3 < K) {
            v[b] = __ldg(reinterpret_cast<const float4*>(p));
          } else {
            if (kk < K) v[b].x = __ldg(p);
            if (kk + 1 < K) v[b].y = __ldg(p + 1);
            if (kk + 2 < K) v[b].z = __ldg(p + 2);
          }
        }
      }
#pragma unroll
      for (int b = 0; b < kBatch; ++b) {
        const int t = base + b * kThreads + tid;
        if (t >= G) continue;
        const int r = t / (kKT / 4), kq = (t % (kKT / 4)) * 4;
        __nv_bfloat162 lo = __floats2bfloat162_rn(v[b].x, v[b].y);
        __nv_bfloat162 hi = __floats2bfloat162_rn(v[b].z, v[b].w);
        uint2 w;
        w.x = *reinterpret_cast<unsigned*>(&lo);
        w.y = *reinterpret_cast<unsigned*>(&hi);
        *reinterpret_cast<uint2*>(dst + core_offset(r, kq)) = w;
      }
    }
  } else if (s_r == 1 && aligned && (s_k & 3) == 0) {
    // groups of 4 consecutive rows: (ROWS / 4) x 64 groups
    constexpr int G = (ROWS / 4) * kKT;
    for (int base = 0; base < G; base += kThreads * kBatch) {
      float4 v[kBatch];
#pragma unroll
      for (int b = 0; b < kBatch; ++b) {
        const int t = base + b * kThreads + tid;
        const int k = t / (ROWS / 4), rq = (t % (ROWS / 4)) * 4;
        const int m = r0 + rq, kk = k0 + k;
        v[b] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (t < G && kk < K) {
          const float* p = X + m + kk * s_k;
          if (m + 3 < R) {
            v[b] = __ldg(reinterpret_cast<const float4*>(p));
          } else {
            if (m < R) v[b].x = __ldg(p);
            if (m + 1 < R) v[b].y = __ldg(p + 1);
            if (m + 2 < R) v[b].z = __ldg(p + 2);
          }
        }
      }
#pragma unroll
      for (int b = 0; b < kBatch; ++b) {
        const int t = base + b * kThreads + tid;
        if (t >= G) continue;
        const int k = t / (ROWS / 4), rq = (t % (ROWS / 4)) * 4;
        const float e[4] = {v[b].x, v[b].y, v[b].z, v[b].w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          *reinterpret_cast<__nv_bfloat16*>(dst + core_offset(rq + j, k)) =
              __float2bfloat16_rn(e[j]);
      }
    }
  } else {
    for (int e = tid; e < ROWS * kKT; e += kThreads) {
      const int r = e / kKT, k = e % kKT;
      const int m = r0 + r, kk = k0 + k;
      const float v = (m < R && kk < K) ? X[m * s_r + kk * s_k] : 0.f;
      *reinterpret_cast<__nv_bfloat16*>(dst + core_offset(r, k)) = __float2bfloat16_rn(v);
    }
  }
}

__global__ void __launch_bounds__(kThreads, 1) k_gemm_tc(GemmArgs g) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  GemmSmem& sm = *reinterpret_cast<GemmSmem*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * kM;
  const int n_mma = (g.N + 15) / 16 * 16;  // UMMA N: multiple of 16
  unsigned ncols = 32;
  while ((int)ncols < n_mma) ncols <<= 1;  // TMEM allocation: power of 2 >= 32
  const unsigned mbar = smem_u32(&sm.mbar);

  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(mbar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(&sm.tmem_base)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const unsigned tmem = sm.tmem_base;
  const unsigned long long wait_ns = mma_wait_limit();

  const unsigned a_base = smem_u32(sm.a), b_base = smem_u32(sm.b);
  const unsigned idesc = instr_desc(n_mma);
  bool ok = true;
  unsigned phase = 0;
  const int nk = (g.K + kKT - 1) / kKT;
  // this CTA's share of the K slices (split K over gridDim.y)
  const int per = (nk + (int)gridDim.y - 1) / (int)gridDim.y;
  const int kt0 = (int)blockIdx.y * per, kt1 = min(nk, kt0 + per);
  for (int kt = kt0; kt < kt1 && ok; ++kt) {
    const int k0 = kt * kKT;
    // stage A (128 x 64) and B (n_mma x 64; B as rows n) as BF16, zero
    // outside the matrix
    stage_slice<kM>(reinterpret_cast<unsigned char*>(sm.a), g.A, g.sa_m, g.sa_k, m0, g.M, k0,
                    g.K, tid);
    if (n_mma <= 128)
      stage_slice<128>(reinterpret_cast<unsigned char*>(sm.b), g.B, g.sb_n, g.sb_k, 0, g.N,
                       k0, g.K, tid);
    else
      stage_slice<kNMax>(reinterpret_cast<unsigned char*>(sm.b), g.B, g.sb_n, g.sb_k, 0, g.N,
                         k0, g.K, tid);
    // make the generic-proxy writes visible to the tensor core (async proxy)
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
      for (int s = 0; s < kKT / 16; ++s) {
        // K slice s = core matrices 2s, 2s + 1 along K
        const unsigned long long da = smem_desc(a_base + s * 256, 128, 1024);
        const unsigned long long db = smem_desc(b_base + s * 256, 128, 1024);
        const unsigned accum = (kt > kt0 || s > 0) ? 1u : 0u;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
            "l"(da), "l"(db), "r"(idesc), "r"(accum)
            : "memory");
      }
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
              mbar)
          : "memory");
    }
    // wait for the MMAs of this slice before the slices are rewritten; the
    // verdict is made uniform over the CTA so every thread leaves together
    ok = __syncthreads_and(mbar_wait(mbar, phase, wait_ns) ? 1 : 0) != 0;
    phase ^= 1u;
  }
  if (!ok) {
    if (tid == 0) atomicExch(g.err, 1);
    // give in-flight MMAs a second bounded chance (at the full limit)
    // before TMEM is released
    mbar_wait(mbar, phase ^ 1u, kWaitNs);
  } else if (kt0 < kt1) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    // epilogue: warp w reads TMEM lanes 32w .. 32w + 31 = rows of the tile
    const int row = warp * 32 + lane;
    const int m = m0 + row;
    const bool vec = g.splits == 1 && (g.sc_m & 3) == 0 &&
                     (reinterpret_cast<unsigned long long>(g.C) & 15u) == 0;
    for (int c0 = 0; c0 < n_mma; c0 += 8) {
      unsigned r[8];
      const unsigned taddr = tmem + ((unsigned)(warp * 32) << 16) + (unsigned)c0;
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
            "=r"(r[6]), "=r"(r[7])
          : "r"(taddr)
          : "memory");
      asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
      if (m >= g.M) continue;
      float v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int n = c0 + j;
        v[j] = __uint_as_float(r[j]);
        if (n >= g.N) continue;
        if (g.H) {
          const float h = g.H[m * g.sh_m + n];
          v[j] *= (1.f - h * h);
        } else {
          if (g.bias) v[j] += g.bias[n];
          // tanh on the special-function unit: its error (about 2^-11
          // relative) is below the BF16 rounding of the operands
          if (g.act == 1) asm("tanh.approx.f32 %0, %0;" : "+f"(v[j]));
        }
      }
      float* crow = g.C + m * g.sc_m + c0;
      if (vec && c0 + 7 < g.N) {
        reinterpret_cast<float4*>(crow)[0] = make_float4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<float4*>(crow)[1] = make_float4(v[4], v[5], v[6], v[7]);
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (c0 + j >= g.N) continue;
          if (g.splits > 1) atomicAdd(crow + j, v[j]);
          else crow[j] = v[j];
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"(ncols)
                 : "memory");
}

// ---------------------------------------------------------------------------
// Warp-specialised persistent GEMM for products whose whole B fits in shared
// memory (K <= 256): every forward layer and every dZ W^T of the network;
// and, with one grid z-slice per 256 of K whose partial tiles are added into
// a zeroed C, the plain products with K > 256 (weight gradients).
//   - B (bn columns x K, BF16) is staged once per CTA and stays resident;
//   - a CTA walks the 128-row tiles blockIdx.x, blockIdx.x + gridDim.x, ...
//     of its column block blockIdx.y;
//   - the FP32 A slices (128 x 64) reach a BF16 ring (full / empty
//     mbarriers) one of two ways.  Where A's rows are K-contiguous with a
//     16-byte multiple stride (the TMA form, column blocks <= 128), one
//     thread issues tensor copies of each slice into a three-stage FP32
//     ring and 8 converter warps round it into a two-stage BF16 ring;
//     elsewhere (the register form) 8 producer warps load, round and store
//     the slices themselves into a four-stage ring, starting while the
//     epilogue and MMA warps stage B;
//   - one thread issues the tcgen05.mma of each slice into one of two TMEM
//     accumulators and commits them to the slice's empty barrier, and the
//     finished tile to its accumulator's full barrier;
//   - 8 epilogue warps (two per TMEM lane quadrant, alternate 32-column
//     chunks) drain the other accumulator (tcgen05.ld, bias + tanh or the
//     tanh derivative, FP32 stores) while the next tile accumulates.
// Every wait is bounded; a role that gives up raises a CTA-wide flag that
// ends the other roles' waits, and the MMA thread waits (at the full limit)
// for its last commit before the accumulators are released.
// ---------------------------------------------------------------------------
namespace ws {
constexpr int kEpiWarps = 8;                 // warps 0-7: TMEM lane quadrant warp % 4
constexpr int kProdWarps = 8;                // warps 8-15
constexpr int kProd = 32 * kProdWarps;
constexpr int kMmaWarp = kEpiWarps + kProdWarps;  // warp 16
constexpr int kThreads = 32 * (kMmaWarp + 1);     // 544
constexpr int kStages = 4;
constexpr int kKMax = 256;
constexpr int kStagesT = 2;  // the TMA form: BF16 ring stages
constexpr int kFStages = 3;  // the TMA form: FP32 ring stages (96 KB in flight)
}  // namespace ws

struct WsSmem {
  __nv_bfloat16 b[kNMax * ws::kKMax];       // B: K / 64 slices of bn x 64, 128 KB
  __nv_bfloat16 a[ws::kStages][kM * kKT];   // A ring, 4 x 16 KB
  float bias[kNMax];
  float ctile[ws::kEpiWarps][32 * 32];  // per-warp 32 x 32 transpose of C (swizzled)
  unsigned long long full[ws::kStages], empty[ws::kStages], acc_full[2], acc_empty[2];
  unsigned tmem_base;
  int give_up;
};
// The TMA form (k_gemm_ws<true>): column blocks of at most 128, and the FP32
// A slices arrive by tensor copies -- two 32-k boxes of 128 rows each, with
// the 128-byte swizzle (16-byte chunk c of row r at chunk c ^ (r & 7)) --
// into a three-stage FP32 ring that the converter warps turn into a
// two-stage BF16 ring (the MMA of a slice takes a fraction of a copy's
// latency, so the bytes go to copies in flight).  The FP32 ring starts on a
// 1024-byte boundary (the swizzle's period).
constexpr int kTmaBn = 128;
struct WsSmemT {
  __nv_bfloat16 b[kTmaBn * ws::kKMax];       // 64 KB
  __nv_bfloat16 a[ws::kStagesT][kM * kKT];   // 32 KB
  float af[ws::kFStages][2][kM * 32];        // 96 KB: stage, 32-k box, 128 rows x 32
  float bias[kNMax];
  float ctile[ws::kEpiWarps][32 * 32];
  unsigned long long full[ws::kStagesT], empty[ws::kStagesT], acc_full[2], acc_empty[2];
  unsigned long long ffull[ws::kFStages], fempty[ws::kFStages];  // copies landed / consumed
  unsigned tmem_base;
  int give_up;
};
static_assert(offsetof(WsSmemT, af) % 1024 == 0, "the swizzled boxes need 1024-byte alignment");

__device__ __forceinline__ void tma_load_2d(unsigned dst, const CUtensorMap* map, int x, int y,
                                            unsigned mbar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];\n" ::"r"(dst),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(mbar)
      : "memory");
}

__device__ __forceinline__ void mbar_arrive(unsigned addr) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(addr) : "memory");
}

// Bounded wait that also ends when another role of the CTA has given up.
__device__ __forceinline__ bool ws_wait(unsigned addr, unsigned parity,
                                        unsigned long long limit, const volatile int* give_up) {
  if (limit < 1000) return mbar_test(addr, parity);
  if (mbar_poll(addr, parity)) return true;
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  while (!mbar_poll(addr, parity)) {
    if (*give_up) return false;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t - t0 > limit) return false;
  }
  return true;
}

__device__ __forceinline__ unsigned pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<unsigned*>(&v);
}

// Stages the `rows` x 64 slice X(r, k), r in [r0, r0 + rows), k in [k0, k0 +
// 64), into the K-major core layout as BF16, zero outside [0, R) x [0, K);
// rows is a multiple of 8, t in [0, NT).
//   k contiguous: a task is 8 consecutive k of one row (two 16-byte loads,
//     one 16-byte store: a full row of one core matrix); the 8 tasks of a
//     quarter-warp take 8 different rows of one core-matrix group, so the
//     stores hit 8 different bank groups;
//   rows contiguous: a task is 4 rows x 8 k (eight 16-byte loads along the
//     rows, transposed in registers into four 16-byte stores); the lanes of
//     a warp take consecutive row quads, so each load instruction reads 512
//     contiguous bytes;
//   other strides: one element per task.
template <int NT>
__device__ __forceinline__ void ws_stage(unsigned char* dst, const float* __restrict__ X,
                                         long long s_r, long long s_k, int r0, int R, int rows,
                                         int k0, int K, int t) {
  const bool aligned = (reinterpret_cast<unsigned long long>(X) & 15u) == 0;
  if (s_k == 1 && aligned && (s_r & 3) == 0) {
    const int G = rows * 8;
    constexpr int kB = 4;
    for (int base = 0; base < G; base += NT * kB) {
      float4 v[kB][2];
#pragma unroll
      for (int b = 0; b < kB; ++b) {
        const int g = base + b * NT + t;
        const int r = (g >> 6) * 8 + (g & 7), kq = ((g >> 3) & 7) * 8;
        const int m = r0 + r, kk = k0 + kq;
        v[b][0] = v[b][1] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (g < G && m < R) {
          const float* p = X + (long long)m * s_r + kk;
          if (kk + 7 < K) {
            v[b][0] = __ldg(reinterpret_cast<const float4*>(p));
            v[b][1] = __ldg(reinterpret_cast<const float4*>(p) + 1);
          } else {
            float e[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) e[j] = kk + j < K ? __ldg(p + j) : 0.f;
            v[b][0] = make_float4(e[0], e[1], e[2], e[3]);
            v[b][1] = make_float4(e[4], e[5], e[6], e[7]);
          }
        }
      }
#pragma unroll
      for (int b = 0; b < kB; ++b) {
        const int g = base + b * NT + t;
        if (g >= G) continue;
        const int r = (g >> 6) * 8 + (g & 7), kq = ((g >> 3) & 7) * 8;
        uint4 w;
        w.x = pack_bf16x2(v[b][0].x, v[b][0].y);
        w.y = pack_bf16x2(v[b][0].z, v[b][0].w);
        w.z = pack_bf16x2(v[b][1].x, v[b][1].y);
        w.w = pack_bf16x2(v[b][1].z, v[b][1].w);
        *reinterpret_cast<uint4*>(dst + core_offset(r, kq)) = w;
      }
    }
  } else if (s_r == 1 && aligned && (s_k & 3) == 0) {
    const int quads = rows / 4, G = quads * 8;
    for (int g = t; g < G; g += NT) {
      const int r4 = (g % quads) * 4, kq = (g / quads) * 8;
      const int m = r0 + r4;
      float4 v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int kk = k0 + kq + j;
        v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (kk < K && m < R) {
          const float* p = X + m + (long long)kk * s_k;
          if (m + 3 < R) {
            v[j] = __ldg(reinterpret_cast<const float4*>(p));
          } else {
            v[j].x = __ldg(p);
            if (m + 1 < R) v[j].y = __ldg(p + 1);
            if (m + 2 < R) v[j].z = __ldg(p + 2);
          }
        }
      }
      uint4 w;
      w.x = pack_bf16x2(v[0].x, v[1].x);
      w.y = pack_bf16x2(v[2].x, v[3].x);
      w.z = pack_bf16x2(v[4].x, v[5].x);
      w.w = pack_bf16x2(v[6].x, v[7].x);
      *reinterpret_cast<uint4*>(dst + core_offset(r4, kq)) = w;
      w.x = pack_bf16x2(v[0].y, v[1].y);
      w.y = pack_bf16x2(v[2].y, v[3].y);
      w.z = pack_bf16x2(v[4].y, v[5].y);
      w.w = pack_bf16x2(v[6].y, v[7].y);
      *reinterpret_cast<uint4*>(dst + core_offset(r4 + 1, kq)) = w;
      w.x = pack_bf16x2(v[0].z, v[1].z);
      w.y = pack_bf16x2(v[2].z, v[3].z);
      w.z = pack_bf16x2(v[4].z, v[5].z);
      w.w = pack_bf16x2(v[6].z, v[7].z);
      *reinterpret_cast<uint4*>(dst + core_offset(r4 + 2, kq)) = w;
      w.x = pack_bf16x2(v[0].w, v[1].w);
      w.y = pack_bf16x2(v[2].w, v[3].w);
      w.z = pack_bf16x2(v[4].w, v[5].w);
      w.w = pack_bf16x2(v[6].w, v[7].w);
      *reinterpret_cast<uint4*>(dst + core_offset(r4 + 3, kq)) = w;
    }
  } else {
    for (int e = t; e < rows * kKT; e += NT) {
      const int r = e / kKT, k = e % kKT;
      const int m = r0 + r, kk = k0 + k;
      const float v = (m < R && kk < K) ? X[(long long)m * s_r + (long long)kk * s_k] : 0.f;
      *reinterpret_cast<__nv_bfloat16*>(dst + core_offset(r, k)) = __float2bfloat16_rn(v);
    }
  }
}

// B (rows n in [r0, r0 + rows), all nk slices of 64 k) staged once per CTA by
// all its threads: the same tasks as ws_stage, numbered across the slices
// so that each thread keeps several tasks' loads in flight (4 tasks of two
// 16-byte loads, or 2 tasks of eight).
template <int NT>
__device__ __forceinline__ void ws_stage_b(unsigned char* dst, const float* __restrict__ X,
                                           long long s_r, long long s_k, int r0, int R,
                                           int rows, int nk, int K, int t) {
  const bool aligned = (reinterpret_cast<unsigned long long>(X) & 15u) == 0;
  const size_t slice_bytes = (size_t)rows * 128;
  if (s_k == 1 && aligned && (s_r & 3) == 0) {
    const int Gs = rows * 8, G = nk * Gs;
    constexpr int kB = 4;
    for (int base = 0; base < G; base += NT * kB) {
      float4 v[kB][2];
#pragma unroll
      for (int b = 0; b < kB; ++b) {
        const int gt = base + b * NT + t;
        const int sl = gt / Gs, g = gt % Gs;
        const int r = (g >> 6) * 8 + (g & 7), kq = ((g >> 3) & 7) * 8;
        const int m = r0 + r, kk = sl * kKT + kq;
        v[b][0] = v[b][1] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (gt < G && m < R) {
          const float* p = X + (long long)m * s_r + kk;
          if (kk + 7 < K) {
            v[b][0] = __ldg(reinterpret_cast<const float4*>(p));
            v[b][1] = __ldg(reinterpret_cast<const float4*>(p) + 1);
          } else {
            float e[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) e[j] = kk + j < K ? __ldg(p + j) : 0.f;
            v[b][0] = make_float4(e[0], e[1], e[2], e[3]);
            v[b][1] = make_float4(e[4], e[5], e[6], e[7]);
          }
        }
      }
#pragma unroll
      for (int b = 0; b < kB; ++b) {
        const int gt = base + b * NT + t;
        if (gt >= G) continue;
        const int sl = gt / Gs, g = gt % Gs;
        const int r = (g >> 6) * 8 + (g & 7), kq = ((g >> 3) & 7) * 8;
        uint4 w;
        w.x = pack_bf16x2(v[b][0].x, v[b][0].y);
        w.y = pack_bf16x2(v[b][0].z, v[b][0].w);
        w.z = pack_bf16x2(v[b][1].x, v[b][1].y);
        w.w = pack_bf16x2(v[b][1].z, v[b][1].w);
        *reinterpret_cast<uint4*>(dst + sl * slice_bytes + core_offset(r, kq)) = w;
      }
    }
  } else if (s_r == 1 && aligned && (s_k & 3) == 0) {
    const int quads = rows / 4, Gs = quads * 8, G = nk * Gs;
    constexpr int kB = 2;
    for (int base = 0; base < G; base += NT * kB) {
      float4 v[kB][8];
#pragma unroll
      for (int b = 0; b < kB; ++b) {
        const int gt = base + b * NT + t;
        const int sl = gt / Gs, g = gt % Gs;
        const int r4 = (g % quads) * 4, kq = (g / quads) * 8;
        const int m = r0 + r4;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int kk = sl * kKT + kq + j;
          v[b][j] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (gt < G && kk < K && m < R) {
            const float* p = X + m + (long long)kk * s_k;
            if (m + 3 < R) {
              v[b][j] = __ldg(reinterpret_cast<const float4*>(p));
            } else {
              v[b][j].x = __ldg(p);
              if (m + 1 < R) v[b][j].y = __ldg(p + 1);
              if (m + 2 < R) v[b][j].z = __ldg(p + 2);
            }
          }
        }
      }
#pragma unroll
      for (int b = 0; b < kB; ++b) {
        const int gt = base + b * NT + t;
        if (gt >= G) continue;
        const int sl = gt / Gs, g = gt % Gs;
        const int r4 = (g % quads) * 4, kq = (g / quads) * 8;
        unsigned char* d = dst + sl * slice_bytes;
        const float4* u = v[b];
        *reinterpret_cast<uint4*>(d + core_offset(r4, kq)) =
            make_uint4(pack_bf16x2(u[0].x, u[1].x), pack_bf16x2(u[2].x, u[3].x),
                       pack_bf16x2(u[4].x, u[5].x), pack_bf16x2(u[6].x, u[7].x));
        *reinterpret_cast<uint4*>(d + core_offset(r4 + 1, kq)) =
            make_uint4(pack_bf16x2(u[0].y, u[1].y), pack_bf16x2(u[2].y, u[3].y),
                       pack_bf16x2(u[4].y, u[5].y), pack_bf16x2(u[6].y, u[7].y));
        *reinterpret_cast<uint4*>(d + core_offset(r4 + 2, kq)) =
            make_uint4(pack_bf16x2(u[0].z, u[1].z), pack_bf16x2(u[2].z, u[3].z),
                       pack_bf16x2(u[4].z, u[5].z), pack_bf16x2(u[6].z, u[7].z));
        *reinterpret_cast<uint4*>(d + core_offset(r4 + 3, kq)) =
            make_uint4(pack_bf16x2(u[0].w, u[1].w), pack_bf16x2(u[2].w, u[3].w),
                       pack_bf16x2(u[4].w, u[5].w), pack_bf16x2(u[6].w, u[7].w));
      }
    }
  } else {
    for (int sl = 0; sl < nk; ++sl)
      ws_stage<NT>(dst + sl * slice_bytes, X, s_r, s_k, r0, R, rows, sl * kKT, K, t);
  }
}

// The K-contiguous A slice (128 x 64) of the producers split into a load and
// a store phase, so that a producer thread keeps the loads of two slices in
// flight: task b of thread t is group g = 256 b + t of ws_stage's mapping.
struct ASlice {
  float4 v[4][2];
};
__device__ __forceinline__ void ws_load_a(ASlice& x, const float* __restrict__ X, long long s_r,
                                          int r0, int R, int k0, int K, int t) {
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int g = b * ws::kProd + t;
    const int r = (g >> 6) * 8 + (g & 7), kq = ((g >> 3) & 7) * 8;
    const int m = r0 + r, kk = k0 + kq;
    x.v[b][0] = x.v[b][1] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (m < R) {
      const float* p = X + (long long)m * s_r + kk;
      if (kk + 7 < K) {
        x.v[b][0] = __ldg(reinterpret_cast<const float4*>(p));
        x.v[b][1] = __ldg(reinterpret_cast<const float4*>(p) + 1);
      } else {
        float e[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) e[j] = kk + j < K ? __ldg(p + j) : 0.f;
        x.v[b][0] = make_float4(e[0], e[1], e[2], e[3]);
        x.v[b][1] = make_float4(e[4], e[5], e[6], e[7]);
      }
    }
  }
}
__device__ __forceinline__ void ws_store_a(unsigned char* dst, const ASlice& x, int t) {
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int g = b * ws::kProd + t;
    const int r = (g >> 6) * 8 + (g & 7), kq = ((g >> 3) & 7) * 8;
    uint4 w;
    w.x = pack_bf16x2(x.v[b][0].x, x.v[b][0].y);
    w.y = pack_bf16x2(x.v[b][0].z, x.v[b][0].w);
    w.z = pack_bf16x2(x.v[b][1].x, x.v[b][1].y);
    w.w = pack_bf16x2(x.v[b][1].z, x.v[b][1].w);
    *reinterpret_cast<uint4*>(dst + core_offset(r, kq)) = w;
  }
}

// g.ws_bn: columns per CTA (a multiple of 16, <= 256; <= kTmaBn for TA);
// K <= 256.  TA: the A slices arrive by tensor copies of amap (warp 17 lane
// 0 issues them; the producer warps convert), else the producer warps load
// them.
template <bool TA>
__global__ void __launch_bounds__(TA ? ws::kThreads + 32 : ws::kThreads, 1)
    k_gemm_ws(GemmArgs g, const __grid_constant__ CUtensorMap amap) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  using S = std::conditional_t<TA, WsSmemT, WsSmem>;
  constexpr int NTH = TA ? ws::kThreads + 32 : ws::kThreads;
  constexpr int NS = TA ? ws::kStagesT : ws::kStages;  // BF16 ring stages
  constexpr int kTmaWarp = ws::kMmaWarp + 1;
  // the TMA form's swizzled boxes need a 1024-byte aligned base (the
  // launch allocates 1 KB more)
  unsigned char* base = smem_raw;
  if constexpr (TA) base += (1024u - (smem_u32(smem_raw) & 1023u)) & 1023u;
  S& sm = *reinterpret_cast<S*>(base);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // split K (gridDim.z > 1, the register form only): this CTA's products
  // cover K range [z kKMax, (z + 1) kKMax) and add into the zeroed C
  const bool split = gridDim.z > 1;
  if (split) {
    const int kb = (int)blockIdx.z * ws::kKMax;
    g.A += (long long)kb * g.sa_k;
    g.B += (long long)kb * g.sb_k;
    g.K = min(ws::kKMax, g.K - kb);
  }
  const int bn = g.ws_bn;
  const int n0 = (int)blockIdx.y * bn;
  const int nk = (g.K + kKT - 1) / kKT;
  const int mt = (g.M + kM - 1) / kM;
  unsigned acc_cols = 32;
  while ((int)acc_cols < bn) acc_cols <<= 1;
  volatile int* give_up = &sm.give_up;

  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(&sm.full[s])),
                   "r"(ws::kProd)
                   : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&sm.empty[s]))
                   : "memory");
    }
    for (int b = 0; b < 2; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&sm.acc_full[b]))
                   : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(
                       smem_u32(&sm.acc_empty[b])),
                   "r"(32 * ws::kEpiWarps)
                   : "memory");
    }
    sm.give_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == ws::kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(&sm.tmem_base)),
                 "r"(2 * acc_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  const int my_tiles = (mt - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  const int total = my_tiles * nk;  // A slices this CTA consumes
  // the TMA form: the copy thread owns the FP32 ring's barriers and has its
  // first kFStages copies in flight while the others stage B
  [[maybe_unused]] auto issue_a = [&](auto& smr, int q) {
    const int st2 = q % ws::kFStages;
    const int mi = (int)blockIdx.x + (q / nk) * (int)gridDim.x, k0 = (q % nk) * kKT;
    const unsigned mb = smem_u32(&smr.ffull[st2]);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mb),
                 "r"((unsigned)(2 * kM * 32 * sizeof(float)))
                 : "memory");
    tma_load_2d(smem_u32(smr.af[st2][0]), &amap, k0, mi * kM, mb);
    tma_load_2d(smem_u32(smr.af[st2][1]), &amap, k0 + 32, mi * kM, mb);
  };
  int pre = 0;
  if constexpr (TA) {
    if (warp == kTmaWarp && lane == 0) {
      for (int b = 0; b < ws::kFStages; ++b) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&sm.ffull[b]))
                     : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(&sm.fempty[b])),
                     "r"(ws::kProd)
                     : "memory");
      }
      asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      pre = total < ws::kFStages ? total : ws::kFStages;
      for (int q = 0; q < pre; ++q) issue_a(sm, q);
    }
  }
  // B (bn x K) of this column block, staged once: in the TMA form by every
  // thread but the copy warp's, before the barrier; in the register form
  // after it by the epilogue and MMA warps only (kBStagers threads, their
  // own named barrier), while the producer warps already load A
  constexpr int kBStagers = 32 * (ws::kEpiWarps + 1);
  if (TA)
    if (tid < ws::kThreads)
      ws_stage_b<ws::kThreads>(reinterpret_cast<unsigned char*>(sm.b), g.B, g.sb_n, g.sb_k, n0,
                               g.N, bn, nk, g.K, tid);
  for (int n = tid; n < bn; n += NTH)
    sm.bias[n] = (g.bias && n0 + n < g.N) ? g.bias[n0 + n] : 0.f;
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const unsigned tmem = sm.tmem_base;
  const unsigned long long wait_ns = mma_wait_limit();
  if (!TA && (warp < ws::kEpiWarps || warp == ws::kMmaWarp)) {
    ws_stage_b<kBStagers>(reinterpret_cast<unsigned char*>(sm.b), g.B, g.sb_n, g.sb_k, n0, g.N,
                          bn, nk, g.K, warp < ws::kEpiWarps ? tid : tid - 32 * ws::kProdWarps);
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("bar.sync 1, %0;\n" ::"n"(kBStagers) : "memory");
  }

  if (TA && warp >= ws::kEpiWarps && warp < ws::kMmaWarp) {
    // converters: each FP32 slice (two swizzled 32-k boxes) into the BF16
    // ring; task g = (row r, 8-k group kg) as in ws_stage, whose eight lanes
    // of a quarter-warp read eight rows of one chunk column -- eight
    // different swizzled chunks, no bank conflict -- and write eight rows of
    // one core-matrix column
    if constexpr (TA) {
      const int pt = tid - 32 * ws::kEpiWarps;
      bool ok = true;
      for (int q = 0; q < total && ok; ++q) {
        const int st = q % NS, use = q / NS;
        const int st2 = q % ws::kFStages, use2 = q / ws::kFStages;
        ok = ws_wait(smem_u32(&sm.empty[st]), (use & 1) ^ 1, wait_ns, give_up) &&
             ws_wait(smem_u32(&sm.ffull[st2]), use2 & 1, wait_ns, give_up);
        if (!ok) break;
        unsigned char* dst = reinterpret_cast<unsigned char*>(sm.a[st]);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int g = b * ws::kProd + pt;
          const int r = (g >> 6) * 8 + (g & 7), kg = (g >> 3) & 7;
          const float* row = sm.af[st2][kg >> 2] + r * 32;
          const int c0 = (kg & 3) * 2, sw = r & 7;
          const float4 v0 = *reinterpret_cast<const float4*>(row + 4 * (c0 ^ sw));
          const float4 v1 = *reinterpret_cast<const float4*>(row + 4 * ((c0 + 1) ^ sw));
          uint4 w;
          w.x = pack_bf16x2(v0.x, v0.y);
          w.y = pack_bf16x2(v0.z, v0.w);
          w.z = pack_bf16x2(v1.x, v1.y);
          w.w = pack_bf16x2(v1.z, v1.w);
          *reinterpret_cast<uint4*>(dst + core_offset(r, kg * 8)) = w;
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        mbar_arrive(smem_u32(&sm.full[st]));
        mbar_arrive(smem_u32(&sm.fempty[st2]));
      }
      if (!ok) {
        *give_up = 1;
        atomicExch(g.err, 1);
      }
    }
  } else if (TA && warp == kTmaWarp) {
    // the tensor copies of the FP32 slices, kFStages ahead of the
    // converters; before leaving, the last copies issued are waited for
    // (at the full limit), so that none lands after the CTA has gone
    if constexpr (TA) {
      if (lane == 0) {
        int issued = pre;
        bool ok = true;
        for (int q = pre; q < total; ++q) {
          const int use2 = q / ws::kFStages;
          if (!ws_wait(smem_u32(&sm.fempty[q % ws::kFStages]), (use2 & 1) ^ 1, wait_ns,
                       give_up)) {
            ok = false;
            break;
          }
          issue_a(sm, q);
          ++issued;
        }
        if (!ok) {
          *give_up = 1;
          atomicExch(g.err, 1);
        }
        for (int q = issued - ws::kFStages < 0 ? 0 : issued - ws::kFStages; q < issued; ++q)
          mbar_wait(smem_u32(&sm.ffull[q % ws::kFStages]),
                    (unsigned)((q / ws::kFStages) & 1), kWaitNs);
      }
    }
  } else if (!TA && warp >= ws::kEpiWarps && warp < ws::kMmaWarp) {
    // producers: A slices into the ring, two at a time where A is
    // K-contiguous (both slices' loads in flight before either is stored)
    const int pt = tid - 32 * ws::kEpiWarps;
    const bool pair = g.sa_k == 1 && (g.sa_m & 3) == 0 &&
                      (reinterpret_cast<unsigned long long>(g.A) & 15u) == 0;
    bool ok = true;
    for (int q = 0; q < total; q += pair ? 2 : 1) {
      const int nq = pair && q + 1 < total ? 2 : 1;
      for (int i = 0; i < nq && ok; ++i) {
        const int use = (q + i) / ws::kStages;
        ok = ws_wait(smem_u32(&sm.empty[(q + i) % ws::kStages]), (use & 1) ^ 1, wait_ns,
                     give_up);
      }
      if (!ok) break;
      const int mi0 = (int)blockIdx.x + (q / nk) * (int)gridDim.x, s0 = q % nk;
      if (pair) {
        ASlice x0, x1;
        ws_load_a(x0, g.A, g.sa_m, mi0 * kM, g.M, s0 * kKT, g.K, pt);
        if (nq == 2) {
          const int mi1 = (int)blockIdx.x + ((q + 1) / nk) * (int)gridDim.x, s1 = (q + 1) % nk;
          ws_load_a(x1, g.A, g.sa_m, mi1 * kM, g.M, s1 * kKT, g.K, pt);
        }
        ws_store_a(reinterpret_cast<unsigned char*>(sm.a[q % ws::kStages]), x0, pt);
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        mbar_arrive(smem_u32(&sm.full[q % ws::kStages]));
        if (nq == 2) {
          ws_store_a(reinterpret_cast<unsigned char*>(sm.a[(q + 1) % ws::kStages]), x1, pt);
          asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
          mbar_arrive(smem_u32(&sm.full[(q + 1) % ws::kStages]));
        }
      } else {
        ws_stage<ws::kProd>(reinterpret_cast<unsigned char*>(sm.a[q % ws::kStages]), g.A,
                            g.sa_m, g.sa_k, mi0 * kM, g.M, kM, s0 * kKT, g.K, pt);
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        mbar_arrive(smem_u32(&sm.full[q % ws::kStages]));
      }
    }
    if (!ok) {
      *give_up = 1;
      atomicExch(g.err, 1);
    }
  } else if (warp == ws::kMmaWarp) {
    if (lane == 0) {
      const unsigned idesc = instr_desc(bn);
      const unsigned b_base = smem_u32(sm.b);
      unsigned last_bar = 0, last_par = 0;
      int q = 0, j = 0;
      bool ok = true;
      for (int mi = blockIdx.x; mi < mt && ok; mi += gridDim.x, ++j) {
        const int acc = j & 1, use_acc = j >> 1;
        if (!ws_wait(smem_u32(&sm.acc_empty[acc]), (use_acc & 1) ^ 1, wait_ns, give_up)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const unsigned d_tmem = tmem + (unsigned)acc * acc_cols;
        for (int s = 0; s < nk; ++s, ++q) {
          const int st = q % NS, use = q / NS;
          if (!ws_wait(smem_u32(&sm.full[st]), use & 1, wait_ns, give_up)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
          const unsigned a_base = smem_u32(sm.a[st]);
#pragma unroll
          for (int kk = 0; kk < kKT / 16; ++kk) {
            const unsigned long long da = smem_desc(a_base + kk * 256, 128, 1024);
            const unsigned long long db =
                smem_desc(b_base + (unsigned)(s * bn * 128 + kk * 256), 128, 1024);
            const unsigned accum = (s > 0 || kk > 0) ? 1u : 0u;
            asm volatile(
                "{\n\t.reg .pred p;\n\t"
                "setp.ne.b32 p, %4, 0;\n\t"
                "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
                "l"(da), "l"(db), "r"(idesc), "r"(accum)
                : "memory");
          }
          last_bar = smem_u32(&sm.empty[st]);
          last_par = (unsigned)(use & 1);
          asm volatile(
              "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                  last_bar)
              : "memory");
        }
        if (!ok) break;
        last_bar = smem_u32(&sm.acc_full[acc]);
        last_par = (unsigned)(use_acc & 1);
        asm volatile(
            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                last_bar)
            : "memory");
      }
      if (!ok) {
        *give_up = 1;
        atomicExch(g.err, 1);
      }
      // the accumulators are released only after the last MMA has completed
      if (last_bar != 0) mbar_wait(last_bar, last_par, kWaitNs);
    }
  } else {
    // epilogue: warp w drains TMEM lanes 32 (w % 4) .. 32 (w % 4) + 31 (rows
    // of the tile), the 32-column chunks w / 4, w / 4 + 2, ...  Lane l
    // reads row l; the 32 x 32 block goes through the warp's shared-memory
    // buffer with its 16-byte chunks swizzled (chunk i of row r at slot
    // i ^ (r & 7)), so the writes (8 lanes: 8 rows, one chunk) and the reads
    // (8 lanes: one row, 8 chunks) both touch 8 different bank groups; each
    // lane then owns 4 consecutive columns of rows r = 4 i + l / 8, so a
    // store instruction writes 4 rows x 128 bytes.
    const bool vec = (g.sc_m & 3) == 0 && (reinterpret_cast<unsigned long long>(g.C) & 15u) == 0;
    const bool hvec =
        g.H && (g.sh_m & 3) == 0 && (reinterpret_cast<unsigned long long>(g.H) & 15u) == 0;
    float* buf = sm.ctile[warp];
    const int cq = (lane & 7) * 4;  // this lane's 4 columns in phase 2
    int j = 0;
    bool ok = true;
    for (int mi = blockIdx.x; mi < mt && ok; mi += gridDim.x, ++j) {
      const int acc = j & 1, use_acc = j >> 1;
      ok = __all_sync(0xffffffffu,
                      ws_wait(smem_u32(&sm.acc_full[acc]), use_acc & 1, wait_ns, give_up));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      const int quad = warp & 3;
      const int row0 = mi * kM + quad * 32;
      for (int c0 = (warp >> 2) * 32; c0 < bn; c0 += 64) {
        unsigned r[32];
        const unsigned taddr =
            tmem + ((unsigned)(quad * 32) << 16) + (unsigned)acc * acc_cols + (unsigned)c0;
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, "
            "%10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, "
            "%26, %27, %28, %29, %30, %31}, [%32];\n"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
              "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
              "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]),
              "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
              "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]),
              "=r"(r[30]), "=r"(r[31])
            : "r"(taddr)
            : "memory");
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
        for (int i = 0; i < 8; ++i)
          *reinterpret_cast<uint4*>(buf + lane * 32 + 4 * (i ^ (lane & 7))) =
              make_uint4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
        __syncwarp();
        const int c = c0 + cq;      // column within the block
        const int n = n0 + c;       // column of C
        float4 bq = make_float4(0.f, 0.f, 0.f, 0.f);
        if (!g.H && c < bn) bq = *reinterpret_cast<const float4*>(sm.bias + c);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int rr = 4 * i + (lane >> 3);
          const int m = row0 + rr;
          float4 v = *reinterpret_cast<const float4*>(buf + rr * 32 + 4 * ((lane & 7) ^ (rr & 7)));
          if (m >= g.M || c >= bn || n >= g.N) continue;
          const bool full4 = c + 3 < bn && n + 3 < g.N;
          if (g.H) {
            float4 h;
            const float* hp = g.H + (long long)m * g.sh_m + n;
            if (hvec && full4) {
              h = __ldg(reinterpret_cast<const float4*>(hp));
            } else {
              h.x = hp[0];
              h.y = n + 1 < g.N ? hp[1] : 0.f;
              h.z = n + 2 < g.N ? hp[2] : 0.f;
              h.w = n + 3 < g.N ? hp[3] : 0.f;
            }
            v.x *= 1.f - h.x * h.x;
            v.y *= 1.f - h.y * h.y;
            v.z *= 1.f - h.z * h.z;
            v.w *= 1.f - h.w * h.w;
          } else {
            v.x += bq.x;
            v.y += bq.y;
            v.z += bq.z;
            v.w += bq.w;
            // tanh on the special-function unit: its error (about 2^-11
            // relative) is below the BF16 rounding of the operands
            if (g.act == 1) {
              asm("tanh.approx.f32 %0, %0;" : "+f"(v.x));
              asm("tanh.approx.f32 %0, %0;" : "+f"(v.y));
              asm("tanh.approx.f32 %0, %0;" : "+f"(v.z));
              asm("tanh.approx.f32 %0, %0;" : "+f"(v.w));
            }
          }
          float* cp = g.C + (long long)m * g.sc_m + n;
          if (split) {
            if (vec && full4) {
              atomicAdd(reinterpret_cast<float4*>(cp), v);
            } else {
              atomicAdd(cp, v.x);
              if (c + 1 < bn && n + 1 < g.N) atomicAdd(cp + 1, v.y);
              if (c + 2 < bn && n + 2 < g.N) atomicAdd(cp + 2, v.z);
              if (c + 3 < bn && n + 3 < g.N) atomicAdd(cp + 3, v.w);
            }
          } else if (vec && full4) {
            *reinterpret_cast<float4*>(cp) = v;
          } else {
            cp[0] = v.x;
            if (c + 1 < bn && n + 1 < g.N) cp[1] = v.y;
            if (c + 2 < bn && n + 2 < g.N) cp[2] = v.z;
            if (c + 3 < bn && n + 3 < g.N) cp[3] = v.w;
          }
        }
        __syncwarp();
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      mbar_arrive(smem_u32(&sm.acc_empty[acc]));
    }
    if (!ok) {
      *give_up = 1;
      if (lane == 0) atomicExch(g.err, 1);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  if (warp == ws::kMmaWarp)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"(2 * acc_cols)
                 : "memory");
}

// K split for products with few row tiles and many K slices (linear
// epilogues only: no bias, no activation); C is zeroed and the CTAs add.
static int sm_count();
static int choose_splits(const GemmArgs& g) {
  const int sms = sm_count();
  if (g.bias || g.act || g.sc_m != g.N) return 1;  // contiguous C: one memset zeroes it
  const int mt = (g.M + kM - 1) / kM, nk = (g.K + kKT - 1) / kKT;
  int want = (2 * sms) / mt;  // about two CTAs per SM in all
  if (want > nk) want = nk;
  if (want <= 1) return 1;
  const int per = (nk + want - 1) / want;
  return (nk + per - 1) / per;  // no split left without slices
}

static int sm_count() {
  static int sms_dev[kMaxDevices] = {};
  int& sms = sms_dev[device_slot()];
  if (sms == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      sms = 148;
  }
  return sms;
}

// k_gemm_ws launch plan (host only).  The TMA form wherever A's layout
// allows one: K-contiguous rows whose stride is a 16-byte multiple, a
// 16-byte aligned base, at least one full row tile and one 32-k box.  The
// column block is halved (down to 16 columns) while the row tiles alone
// leave SMs idle, and in the TMA form until it is at most kTmaBn; the
// grid's x extent is at most the SMs per column block (persistent CTAs over
// the row tiles).
struct WsPlan {
  bool ta;
  int bn, nt, gx;  // columns per CTA, column blocks, CTAs per column block
};
static WsPlan ws_plan(int M, int N, int K, long long sa_m, long long sa_k, bool a_aligned16,
                      int sms) {
  WsPlan p;
  p.ta = sa_k == 1 && (sa_m & 3) == 0 && a_aligned16 && M >= kM && K >= 32;
  const int n_mma = (N + 15) / 16 * 16;
  const int mt = (M + kM - 1) / kM;
  int nt = 1;
  while ((long long)mt * nt * 2 <= sms && n_mma / (nt * 2) >= 16) nt *= 2;
  if (p.ta)
    while ((n_mma + nt - 1) / nt > kTmaBn) nt *= 2;
  p.bn = ((n_mma + nt - 1) / nt + 15) / 16 * 16;
  p.nt = (N + p.bn - 1) / p.bn;
  p.gx = sms / p.nt;
  if (p.gx < 1) p.gx = 1;
  if (p.gx > mt) p.gx = mt;
  return p;
}

// The A map of the TMA form: FP32 A seen as K x M (K innermost), boxes of
// 32 x 128 with the 128-byte swizzle; rows and columns beyond A read as
// zero.
static bool encode_a_map(const GemmArgs& g, CUtensorMap* map) {
  EncodeTiledFn encode = nullptr;
  if (tensor_map_encoder(&encode) != cudaSuccess) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)g.K, (cuuint64_t)g.M};
  const cuuint64_t strides[1] = {(cuuint64_t)g.sa_m * sizeof(float)};
  const cuuint32_t box[2] = {32, (cuuint32_t)kM};
  const cuuint32_t es[2] = {1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(g.A), dims, strides,
                box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <bool TA>
static cudaError_t launch_ws_form(const GemmArgs& g, const CUtensorMap& amap, int gx, int nt,
                                  cudaStream_t s, int splits = 1) {
  static bool attr_dev[kMaxDevices] = {};
  bool& attr = attr_dev[device_slot()];
  const int bytes = TA ? (int)sizeof(WsSmemT) + 1024 : (int)sizeof(WsSmem);
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(k_gemm_ws<TA>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  k_gemm_ws<TA><<<dim3((unsigned)gx, (unsigned)nt, (unsigned)splits),
                  TA ? ws::kThreads + 32 : ws::kThreads, bytes, s>>>(g, amap);
  return cudaGetLastError();
}

static cudaError_t launch_gemm_ws(GemmArgs g, cudaStream_t s) {
  const int sms = sm_count();
  const bool aligned = (reinterpret_cast<uintptr_t>(g.A) & 15u) == 0;
  WsPlan p = ws_plan(g.M, g.N, g.K, g.sa_m, g.sa_k, aligned, sms);
  CUtensorMap amap;
  memset(&amap, 0, sizeof(amap));
  if (p.ta && !encode_a_map(g, &amap))  // no tensor map: the register form
    p = ws_plan(g.M, g.N, g.K, g.sa_m, g.sa_k, false, sms);
  g.ws_bn = p.bn;
  g.splits = 1;
  return p.ta ? launch_ws_form<true>(g, amap, p.gx, p.nt, s)
              : launch_ws_form<false>(g, amap, p.gx, p.nt, s);
}

// Split-K plan (host only) for K > kKMax: the register form with one grid
// z-slice per kKMax of K, the column block the whole (16-padded) N, and per
// slice the CTAs the SMs leave for it, at most the row tiles.  Ineligible
// (splits = 0): more than 65,535 slices.
static WsPlan ws_split_plan(int M, int N, int K, int sms, int* splits) {
  WsPlan p;
  p.ta = false;
  const long long sl = ((long long)K + ws::kKMax - 1) / ws::kKMax;
  *splits = sl > 65535 ? 0 : (int)sl;
  p.bn = (N + 15) / 16 * 16;
  p.nt = 1;
  const int mt = (M + kM - 1) / kM;
  p.gx = *splits > 0 ? sms / *splits : 1;
  if (p.gx < 1) p.gx = 1;
  if (p.gx > mt) p.gx = mt;
  return p;
}

// K > kKMax without an epilogue (no bias, activation or tanh derivative)
// into a contiguous C: split K over the persistent kernel, partial
// products added into C after one memset.
static cudaError_t launch_gemm_ws_split(GemmArgs g, int splits, const WsPlan& p,
                                        cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(g.C, 0, sizeof(float) * (size_t)g.M * g.N, s);
  if (e != cudaSuccess) return e;
  CUtensorMap amap;
  memset(&amap, 0, sizeof(amap));
  g.ws_bn = p.bn;
  g.splits = 1;
  return launch_ws_form<false>(g, amap, p.gx, p.nt, s, splits);
}

cudaError_t launch_gemm(const GemmArgs& g_in, cudaStream_t s) {
  if (g_in.N < 1 || g_in.N > kNMax || g_in.M < 1 || g_in.K < 1) return cudaErrorInvalidValue;
  if (g_in.K <= ws::kKMax) return launch_gemm_ws(g_in, s);
  if (!g_in.bias && !g_in.act && !g_in.H && g_in.sc_m == g_in.N) {
    int splits = 0;
    const WsPlan p = ws_split_plan(g_in.M, g_in.N, g_in.K, sm_count(), &splits);
    if (splits > 0) return launch_gemm_ws_split(g_in, splits, p, s);
  }
  GemmArgs g = g_in;
  g.splits = choose_splits(g);
  static bool attr_dev[kMaxDevices] = {};
  bool& attr = attr_dev[device_slot()];
  // 100 KB of shared memory per CTA keeps at most two CTAs on an SM, so
  // their TMEM allocations (<= 256 columns each) never exceed the SM's 512.
  const int bytes = (int)sizeof(GemmSmem) + 1024 > 100 * 1024 ? (int)sizeof(GemmSmem) + 1024
                                                              : 100 * 1024;
  if (!attr) {
    cudaError_t e =
        cudaFuncSetAttribute(k_gemm_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  if (g.splits > 1) {
    cudaError_t e = cudaMemsetAsync(g.C, 0, sizeof(float) * (size_t)g.M * g.N, s);
    if (e != cudaSuccess) return e;
  }
  const dim3 grid((unsigned)((g.M + kM - 1) / kM), (unsigned)g.splits);
  k_gemm_tc<<<grid, kThreads, bytes, s>>>(g);
  return cudaGetLastError();
}

// dY = 2 (Y - T) / (B n_out) and the loss sum((Y - T)^2) / (B n_out) (one
// block, fixed-order reduction).
__global__ void k_mse(const float* __restrict__ y, const float* __restrict__ t, int n,
                      float scale, float* __restrict__ dy, float* __restrict__ loss) {
  __shared__ float sh[1024];
  float acc = 0.f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const float d = y[i] - t[i];
    dy[i] = 2.f * d * scale;
    acc += d * d;
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) sh[threadIdx.x] += sh[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = sh[0] * scale;
}

// db[n] = sum_b dZ[b, n] (one thread per column, fixed order).
__global__ void k_colsum(const float* __restrict__ dz, int rows, int cols,
                         float* __restrict__ db) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= cols) return;
  float s = 0.f;
  for (int b = 0; b < rows; ++b) s += dz[(size_t)b * cols + n];
  db[n] = s;
}

}  // namespace mlp
}  // namespace lbm

#include "lbm_net.cuh"

namespace lbm {
cudaError_t mlp_set_wait_ns(unsigned long long ns) {
  const unsigned long long v = ns ? ns : mlp::kWaitNs;
  return cudaMemcpyToSymbol(mlp::g_mma_wait_ns, &v, sizeof v);
}
}  // namespace lbm

// ---------------------------------------------------------------------------
// C ABI of the surrogate network.
// ---------------------------------------------------------------------------
using namespace lbm::mlp;

struct lbm_mlp {
  int n_in, width, depth, n_out, max_batch, nlayers;
  int dims[66];
  long long woff[65], boff[65];  // offsets of W_l, b_l in the flat vector
  long long nparams;
  float *theta, *grad, *adam_m, *adam_v;
  NetShape shape;
  __nv_bfloat16 *fwd, *bwd;  // BF16 copies of the weights, behind theta (its allocation)
  int net_rows;              // rows the training kernels of lbm_net.cuh take
  float* acts;         // activations: layer l input at acts + aoff[l]
  long long aoff[66];
  float* dz[2];        // ping-pong backward buffers (max_batch x max width); dz[0] also
                       // holds dZ of every layer for net_rows rows
  float* dy;           // loss gradient (max_batch x n_out)
  float* loss;         // device scalar, then a partial sum per CTA of k_net_cluster
  int* err;            // error word of the kernels (pinned host memory)
  long long step;
  cudaStream_t stream;
  char msg[512];
};

static thread_local char g_mlp_create_err[512];

static lbm_status mlp_fail(lbm_mlp* m, lbm_status s, const char* fmt, ...) {
  char* dst = m ? m->msg : g_mlp_create_err;
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(dst, 512, fmt, ap);
  va_end(ap);
  return s;
}

#define MLP_CUDA(m, call, what)                                                     \
  do {                                                                              \
    cudaError_t e_ = (call);                                                        \
    if (e_ != cudaSuccess) return mlp_fail(m, LBM_ERR_CUDA, "%s: %s", what,         \
                                           cudaGetErrorString(e_));                 \
  } while (0)

static void mlp_release(lbm_mlp* m) {
  lbm::dev_free(m->theta);
  lbm::dev_free(m->grad);
  lbm::dev_free(m->adam_m);
  lbm::dev_free(m->adam_v);
  lbm::dev_free(m->acts);
  lbm::dev_free(m->dz[0]);
  lbm::dev_free(m->dz[1]);
  lbm::dev_free(m->dy);
  lbm::dev_free(m->loss);
  lbm::host_free(m->err);
}

extern "C" lbm_status lbm_mlp_create(int n_in, int width, int depth, int n_out,
                                     int max_batch, void* cuda_stream, lbm_mlp** out) {
  g_mlp_create_err[0] = 0;
  if (!out) return mlp_fail(nullptr, LBM_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (n_in < 1 || n_in > kNMax || width < 1 || width > kNMax || depth < 0 || depth > 64 ||
      n_out < 1 || n_out > kNMax || max_batch < 1 || max_batch > (1 << 20))
    return mlp_fail(nullptr, LBM_ERR_ARG,
                    "need 1 <= n_in, width, n_out <= 256, 0 <= depth <= 64, "
                    "1 <= max_batch <= 2^20");
  lbm_mlp* m = new (std::nothrow) lbm_mlp;
  if (!m) return mlp_fail(nullptr, LBM_ERR_OOM, "host allocation failed");
  memset(m, 0, sizeof(*m));
  m->n_in = n_in;
  m->width = width;
  m->depth = depth;
  m->n_out = n_out;
  m->max_batch = max_batch;
  m->stream = (cudaStream_t)cuda_stream;
  m->nlayers = depth + 1;
  m->dims[0] = n_in;
  for (int l = 1; l <= depth; ++l) m->dims[l] = width;
  m->dims[depth + 1] = n_out;
  long long o = 0, ao = 0;
  for (int l = 0; l < m->nlayers; ++l) {
    m->woff[l] = o;
    o += (long long)m->dims[l] * m->dims[l + 1];
    m->boff[l] = o;
    o += m->dims[l + 1];
  }
  for (int l = 0; l <= m->nlayers; ++l) {
    m->aoff[l] = ao;
    ao += (long long)max_batch * m->dims[l];
  }
  m->nparams = o;
  const size_t pb = sizeof(float) * (size_t)o;
  m->shape = NetShape{n_in, width, depth, n_out};
  m->net_rows = max_batch < kNetTrainRows ? max_batch : kNetTrainRows;
  const size_t pack_at = (pb + 255) / 256 * 256;
  const size_t pack_bytes = sizeof(__nv_bfloat16) * (size_t)m->shape.packed();
  const size_t theta_bytes = pack_at + 2 * pack_bytes;
  const size_t dz_all = (size_t)m->net_rows * ((size_t)depth * width + n_out);
  const size_t wmax = (size_t)max_batch * (size_t)(width > n_out ? (width > n_in ? width : n_in)
                                                                  : (n_out > n_in ? n_out : n_in));
  using lbm::dev_alloc;
  bool okay = dev_alloc((void**)&m->theta, theta_bytes) == cudaSuccess &&
              dev_alloc((void**)&m->grad, pb) == cudaSuccess &&
              dev_alloc((void**)&m->adam_m, pb) == cudaSuccess &&
              dev_alloc((void**)&m->adam_v, pb) == cudaSuccess &&
              dev_alloc((void**)&m->acts, sizeof(float) * (size_t)ao) == cudaSuccess &&
              dev_alloc((void**)&m->dz[0], sizeof(float) * (wmax > dz_all ? wmax : dz_all)) ==
                  cudaSuccess &&
              dev_alloc((void**)&m->dz[1], sizeof(float) * wmax) == cudaSuccess &&
              dev_alloc((void**)&m->dy, sizeof(float) * (size_t)max_batch * n_out) == cudaSuccess &&
              dev_alloc((void**)&m->loss, sizeof(float) * (1 + 8 * kNetTrainRows / kM)) ==
                  cudaSuccess &&
              lbm::host_alloc((void**)&m->err, sizeof(int)) == cudaSuccess;
  if (!okay) {
    cudaGetLastError();
    mlp_release(m);
    delete m;
    return mlp_fail(nullptr, LBM_ERR_OOM, "cudaMalloc failed");
  }
  m->fwd = reinterpret_cast<__nv_bfloat16*>(reinterpret_cast<char*>(m->theta) + pack_at);
  m->bwd = m->fwd + m->shape.packed();
  cudaMemsetAsync(m->theta, 0, theta_bytes, m->stream);  // the copies' padding stays zero
  cudaMemsetAsync(m->adam_m, 0, pb, m->stream);
  cudaMemsetAsync(m->adam_v, 0, pb, m->stream);
  *m->err = 0;
  *out = m;
  return LBM_OK;
}

extern "C" void lbm_mlp_destroy(lbm_mlp* m) {
  if (!m) return;
  if (m->stream) cudaStreamSynchronize(m->stream);
  else cudaDeviceSynchronize();
  mlp_release(m);
  delete m;
}

extern "C" const char* lbm_mlp_last_error(const lbm_mlp* m) {
  return m ? m->msg : g_mlp_create_err;
}

extern "C" size_t lbm_mlp_num_params(const lbm_mlp* m) { return m ? (size_t)m->nparams : 0; }

extern "C" lbm_status lbm_mlp_set_params(lbm_mlp* m, const float* theta) {
  if (!m || !theta) return m ? mlp_fail(m, LBM_ERR_ARG, "theta is NULL") : LBM_ERR_ARG;
  MLP_CUDA(m, cudaMemcpyAsync(m->theta, theta, sizeof(float) * (size_t)m->nparams,
                              cudaMemcpyDefault, m->stream),
           "cudaMemcpyAsync");
  MLP_CUDA(m, cudaMemsetAsync(m->adam_m, 0, sizeof(float) * (size_t)m->nparams, m->stream),
           "cudaMemsetAsync");
  MLP_CUDA(m, cudaMemsetAsync(m->adam_v, 0, sizeof(float) * (size_t)m->nparams, m->stream),
           "cudaMemsetAsync");
  k_net_pack<<<(unsigned)((m->nparams + 255) / 256), 256, 0, m->stream>>>(
      m->shape, m->theta, m->nparams, m->fwd, m->bwd);
  MLP_CUDA(m, cudaGetLastError(), "weight packing kernel");
  MLP_CUDA(m, cudaStreamSynchronize(m->stream), "stream sync");
  // new parameters start a new history: a give-up reported before is cleared
  *m->err = 0;
  m->step = 0;
  return LBM_OK;
}

extern "C" lbm_status lbm_mlp_get_params(lbm_mlp* m, float* theta) {
  if (!m || !theta) return m ? mlp_fail(m, LBM_ERR_ARG, "theta is NULL") : LBM_ERR_ARG;
  MLP_CUDA(m, cudaMemcpyAsync(theta, m->theta, sizeof(float) * (size_t)m->nparams,
                              cudaMemcpyDefault, m->stream),
           "cudaMemcpyAsync");
  MLP_CUDA(m, cudaStreamSynchronize(m->stream), "stream sync");
  return LBM_OK;
}

static lbm_status gemm(lbm_mlp* m, const GemmArgs& g) {
  MLP_CUDA(m, launch_gemm(g, m->stream), "tensor-core GEMM launch");
  return LBM_OK;
}

// Forward pass for `batch` rows of x (device, batch x n_in); activations
// stay in m->acts; returns the output pointer.
static lbm_status mlp_forward_dev(lbm_mlp* m, const float* x, int batch, float** y_out) {
  MLP_CUDA(m, cudaMemcpyAsync(m->acts + m->aoff[0], x, sizeof(float) * (size_t)batch * m->n_in,
                              cudaMemcpyDeviceToDevice, m->stream),
           "cudaMemcpyAsync");
  for (int l = 0; l < m->nlayers; ++l) {
    GemmArgs g;
    memset(&g, 0, sizeof(g));
    const int din = m->dims[l], dout = m->dims[l + 1];
    g.A = m->acts + m->aoff[l];
    g.sa_m = din;
    g.sa_k = 1;
    g.B = m->theta + m->woff[l];
    g.sb_k = dout;
    g.sb_n = 1;
    g.M = batch;
    g.N = dout;
    g.K = din;
    g.bias = m->theta + m->boff[l];
    g.act = (l < m->nlayers - 1) ? 1 : 0;
    g.C = m->acts + m->aoff[l + 1];
    g.sc_m = dout;
    g.err = m->err;
    lbm_status st = gemm(m, g);
    if (st != LBM_OK) return st;
  }
  *y_out = m->acts + m->aoff[m->nlayers];
  return LBM_OK;
}

static lbm_status check_batch(lbm_mlp* m, int batch) {
  if (batch < 1 || batch > m->max_batch)
    return mlp_fail(m, LBM_ERR_ARG, "batch must lie in [1, %d]", m->max_batch);
  return LBM_OK;
}

// Waits for the stream; the error word lies in pinned host memory, which the
// kernels write only when a wait gives up, so reading it needs no copy.
static lbm_status check_err(lbm_mlp* m) {
  MLP_CUDA(m, cudaStreamSynchronize(m->stream), "stream sync");
  if (*(volatile int*)m->err)
    return mlp_fail(m, LBM_ERR_TIMEOUT, "a tensor-core GEMM wait gave up");
  return LBM_OK;
}

// Whether the kernels may use the caller's array in place: device memory of
// the current GPU, aligned to its floats.  Anything else goes through a copy.
static bool in_place(const void* ptr) {
  cudaPointerAttributes at;
  int dev = -1;
  if (((uintptr_t)ptr & 3u) != 0 || cudaGetDevice(&dev) != cudaSuccess ||
      cudaPointerGetAttributes(&at, ptr) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice && at.device == dev;
}

// The input rows where the kernels read them: x itself, or a copy in acts.
static lbm_status net_input(lbm_mlp* m, const float* x, int batch, const float** out) {
  *out = x;
  if (in_place(x)) return LBM_OK;
  MLP_CUDA(m, cudaMemcpyAsync(m->acts + m->aoff[0], x, sizeof(float) * (size_t)batch * m->n_in,
                              cudaMemcpyDeviceToDevice, m->stream),
           "cudaMemcpyAsync");
  *out = m->acts + m->aoff[0];
  return LBM_OK;
}

static NetArgs net_args(lbm_mlp* m, const float* x, int batch) {
  NetArgs a;
  memset(&a, 0, sizeof(a));
  a.s = m->shape;
  a.batch = batch;
  a.x = x;
  a.theta = m->theta;
  a.fwd = m->fwd;
  a.bwd = m->bwd;
  a.err = m->err;
  return a;
}

extern "C" lbm_status lbm_mlp_forward(lbm_mlp* m, const float* x, int batch, float* y) {
  lbm::NvtxRange nvtx_range_("lbm_mlp_forward");
  if (!m || !x || !y) return m ? mlp_fail(m, LBM_ERR_ARG, "NULL pointer") : LBM_ERR_ARG;
  lbm_status st = check_batch(m, batch);
  if (st != LBM_OK) return st;
  const float* xd = nullptr;
  if ((st = net_input(m, x, batch, &xd)) != LBM_OK) return st;
  const size_t xb = sizeof(float) * (size_t)batch * m->n_in;
  const size_t yb = sizeof(float) * (size_t)batch * m->n_out;
  // y may overlap x (its rows are then still inputs of other rows' CTAs)
  const bool apart = (const char*)y + yb <= (const char*)xd || (const char*)xd + xb <= (const char*)y;
  const bool direct = apart && in_place(y);
  NetArgs a = net_args(m, xd, batch);
  a.y = direct ? y : m->acts + m->aoff[m->nlayers];
  MLP_CUDA(m, launch_net(a, m->stream), "network kernel launch");
  if (!direct)
    MLP_CUDA(m, cudaMemcpyAsync(y, a.y, yb, cudaMemcpyDefault, m->stream), "cudaMemcpyAsync");
  return check_err(m);  // synchronises: a wait that gave up is reported
}

// Loss and gradient of up to net_rows rows: the forward pass, the loss and
// the dZ chain of every 128 rows in one kernel, then every layer's weight and
// bias gradient in another.
static lbm_status net_backward(lbm_mlp* m, const float* x, const float* t, int batch) {
  const float* xd = nullptr;
  lbm_status st = net_input(m, x, batch, &xd);
  if (st != LBM_OK) return st;
  NetArgs a = net_args(m, xd, batch);
  a.t = t;
  a.scale = 1.f / (float)(batch * m->n_out);
  a.h = m->acts + m->aoff[1];
  a.h_stride = (long long)m->max_batch * m->width;
  a.dz = m->dz[0];
  a.dz_stride = (long long)m->net_rows * m->width;
  a.loss_part = m->loss + 1;
  MLP_CUDA(m, launch_net_cluster(a, m->stream), "network kernel launch");
  DwArgs d;
  memset(&d, 0, sizeof(d));
  d.s = m->shape;
  d.batch = batch;
  d.x = xd;
  d.h = a.h;
  d.h_stride = a.h_stride;
  d.dz = a.dz;
  d.dz_stride = a.dz_stride;
  d.grad = m->grad;
  d.loss_part = a.loss_part;
  const int c = net_cluster(m->shape), rows = net_rows_per_tile(batch, c);
  d.loss_parts = (batch + rows - 1) / rows * c;
  d.scale = a.scale;
  d.loss = m->loss;
  d.err = m->err;
  MLP_CUDA(m, launch_net_dw(d, m->nparams, m->stream), "weight-gradient kernel launch");
  return LBM_OK;
}

// Loss and gradient into m->grad (device).
static lbm_status mlp_backward(lbm_mlp* m, const float* x, const float* t, int batch) {
  if (batch <= m->net_rows) return net_backward(m, x, t, batch);
  float* y = nullptr;
  lbm_status st = mlp_forward_dev(m, x, batch, &y);
  if (st != LBM_OK) return st;
  const int nout = m->n_out;
  k_mse<<<1, 1024, 0, m->stream>>>(y, t, batch * nout, 1.f / (float)(batch * nout), m->dy,
                                   m->loss);
  MLP_CUDA(m, cudaGetLastError(), "loss kernel");
  const float* dz = m->dy;  // the output layer is linear: dZ = dY
  int buf = 0;
  for (int l = m->nlayers - 1; l >= 0; --l) {
    const int din = m->dims[l], dout = m->dims[l + 1];
    const float* h_in = m->acts + m->aoff[l];
    // dW_l = H_{l-1}^T dZ_l  (M = din, N = dout, K = batch)
    GemmArgs g;
    memset(&g, 0, sizeof(g));
    g.A = h_in;
    g.sa_m = 1;
    g.sa_k = din;
    g.B = dz;
    g.sb_k = dout;
    g.sb_n = 1;
    g.M = din;
    g.N = dout;
    g.K = batch;
    g.C = m->grad + m->woff[l];
    g.sc_m = dout;
    g.err = m->err;
    if ((st = gemm(m, g)) != LBM_OK) return st;
    k_colsum<<<(dout + 127) / 128, 128, 0, m->stream>>>(dz, batch, dout, m->grad + m->boff[l]);
    MLP_CUDA(m, cudaGetLastError(), "bias-gradient kernel");
    if (l > 0) {
      // dZ_{l-1} = (dZ_l W_l^T) * (1 - H_{l-1}^2)  (M = batch, N = din, K = dout)
      GemmArgs h;
      memset(&h, 0, sizeof(h));
      h.A = dz;
      h.sa_m = dout;
      h.sa_k = 1;
      h.B = m->theta + m->woff[l];
      h.sb_k = 1;
      h.sb_n = dout;
      h.M = batch;
      h.N = din;
      h.K = dout;
      h.H = h_in;
      h.sh_m = din;
      h.C = m->dz[buf];
      h.sc_m = din;
      h.err = m->err;
      if ((st = gemm(m, h)) != LBM_OK) return st;
      dz = m->dz[buf];
      buf ^= 1;
    }
  }
  return LBM_OK;
}

extern "C" lbm_status lbm_mlp_loss_grad(lbm_mlp* m, const float* x, const float* t, int batch,
                                        float* loss, float* grad) {
  lbm::NvtxRange nvtx_range_("lbm_mlp_loss_grad");
  if (!m || !x || !t) return m ? mlp_fail(m, LBM_ERR_ARG, "NULL pointer") : LBM_ERR_ARG;
  lbm_status st = check_batch(m, batch);
  if (st != LBM_OK) return st;
  if ((st = mlp_backward(m, x, t, batch)) != LBM_OK) return st;
  if (grad)
    MLP_CUDA(m, cudaMemcpyAsync(grad, m->grad, sizeof(float) * (size_t)m->nparams,
                                cudaMemcpyDefault, m->stream),
             "cudaMemcpyAsync");
  if (loss)
    MLP_CUDA(m, cudaMemcpyAsync(loss, m->loss, sizeof(float), cudaMemcpyDefault, m->stream),
             "cudaMemcpyAsync");
  return check_err(m);
}

extern "C" lbm_status lbm_mlp_train_step(lbm_mlp* m, const float* x, const float* t, int batch,
                                         float lr, float* loss) {
  lbm::NvtxRange nvtx_range_("lbm_mlp_train_step");
  if (!m || !x || !t) return m ? mlp_fail(m, LBM_ERR_ARG, "NULL pointer") : LBM_ERR_ARG;
  lbm_status st = check_batch(m, batch);
  if (st != LBM_OK) return st;
  if ((st = mlp_backward(m, x, t, batch)) != LBM_OK) return st;
  m->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = (float)(1.0 - pow(0.9, (double)m->step));
  const float c2 = (float)(1.0 - pow(0.999, (double)m->step));
  MLP_CUDA(m, launch_serial(k_net_adam, (unsigned)((m->nparams + 255) / 256), 1, 256, 0, 0,
                            m->stream, m->shape, m->theta, m->grad, m->adam_m, m->adam_v,
                            m->nparams, lr, b1, b2, 1e-8f, c1, c2, m->fwd, m->bwd),
           "Adam kernel");
  if (loss) {
    MLP_CUDA(m, cudaMemcpyAsync(loss, m->loss, sizeof(float), cudaMemcpyDefault, m->stream),
             "cudaMemcpyAsync");
    return check_err(m);
  }
  return LBM_OK;
}

extern "C" lbm_status lbm_test_gemm_plan(int M, int N, int K, long long sa_m, long long sa_k,
                                         int a_aligned16, int sms, int out[4]) {
  if (!out || M < 1 || N < 1 || N > kNMax || K < 1 || sms < 1) return LBM_ERR_ARG;
  if (K > ws::kKMax) {
    int splits = 0;
    const WsPlan p = ws_split_plan(M, N, K, sms, &splits);
    if (splits == 0) {
      out[0] = 3;  // the one-tile-per-CTA kernel
      out[1] = out[2] = out[3] = 0;
      return LBM_OK;
    }
    out[0] = 2;
    out[1] = p.bn;
    out[2] = splits;
    out[3] = p.gx;
    return LBM_OK;
  }
  const WsPlan p = ws_plan(M, N, K, sa_m, sa_k, a_aligned16 != 0, sms);
  out[0] = p.ta ? 1 : 0;
  out[1] = p.bn;
  out[2] = p.nt;
  out[3] = p.gx;
  return LBM_OK;
}

extern "C" lbm_status lbm_gemm_bf16(const float* A, long long sa_m, long long sa_k,
                                    const float* B, long long sb_k, long long sb_n, float* C,
                                    long long sc_m, int M, int N, int K, int* err,
                                    void* cuda_stream) {
  lbm::NvtxRange nvtx_range_("lbm_gemm_bf16");
  if (!A || !B || !C || !err || M < 1 || N < 1 || N > kNMax || K < 1)
    return LBM_ERR_ARG;
  GemmArgs g;
  memset(&g, 0, sizeof(g));
  g.A = A;
  g.sa_m = sa_m;
  g.sa_k = sa_k;
  g.B = B;
  g.sb_k = sb_k;
  g.sb_n = sb_n;
  g.M = M;
  g.N = N;
  g.K = K;
  g.C = C;
  g.sc_m = sc_m;
  g.err = err;
  return launch_gemm(g, (cudaStream_t)cuda_stream) == cudaSuccess ? LBM_OK : LBM_ERR_CUDA;
}
