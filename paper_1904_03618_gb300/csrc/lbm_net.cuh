// Whole-network kernels of the surrogate (included by lbm_mlp.cu, whose
// descriptors, barriers and bounded waits they use): one launch for a forward
// pass, three for a training step.  A tile is up to 128 rows of the batch; it
// goes through every layer without leaving the chip: its activations are the
// BF16 A operand of the next layer (64 KB of shared memory), the FP32
// accumulator lies in tensor memory, and the weights come from a BF16 copy laid
// out as the tensor cores read it (pack_index).  Products, roundings and their
// order are those of the layer-by-layer kernels, in which every product's FP32
// activations went through HBM, in a launch each.
//
// k_net (inference): a CTA per SM walks pairs of tiles, one's MMAs under the
// other's epilogue.  Bound: tanh on the special-function unit (16 a clock and
// SM: 2,048 clocks for a 128 x 256 layer) next to 2,150 clocks of MMA; what it
// runs at is the chain MMA -> epilogue of a tile (2,150 + 3,300 clocks a
// layer), half hidden by the pair.  The single thread that issues the MMAs must
// not compute between them: with the descriptors and the ring's slot (a
// division) formed per 16 k the loop took 370 clocks a step instead of the
// MMA's 134, 63 instead of 43 us.  65,536 rows of the 4 x 256 network: 43 us on
// the device against 175 us in five launches.
// k_net_cluster (training, to the loss and the dZ chain of the tile's rows,
// which need no other row): a cluster of up to 8 CTAs per tile, each computing
// 32 columns of every layer and writing them into every peer's A operand
// through distributed shared memory.  On a minibatch the chain of layers is
// latency: a CTA's share of a layer's weights is 16 KB, loaded up to four
// layers ahead, its MMA and epilogue an eighth of the layer's, and a cluster
// barrier closes the layer.  256 rows: 28 us for 9 products; one CTA per 128
// rows took 109 us.
// k_net_dw: every layer's weight and bias gradient in one launch (9 us, in 19
// before: 90 us of it the bias sums, a thread a column from global memory): a
// CTA per (layer, 128 rows of W, 32 columns, 256 of the batch); with more than
// one slice of the batch the partial sums are added into a zeroed gradient; and
// one per 32 biases of a layer.
// k_net_adam: Adam over all parameters, writing the BF16 copies on the way.
// A training step of 256 rows: 37 us against 226 us.
#pragma once

#include "lbm_chained.cuh"

namespace lbm {
namespace mlp {

constexpr int kNetEpi = 256;                   // epilogue threads of a tile (8 warps)
constexpr int kNetThreads = 2 * kNetEpi + 64;  // two tiles, the MMA and the copy warp
constexpr int kNetStages = 5;                  // weight slices of 32 k (16 KB) in the ring
constexpr int kNetBlock = 32;                  // columns per CTA of a cluster
constexpr int kNetBufs = 4;                    // ... and its weight buffers, a layer each
constexpr int kClThreads = kNetEpi + 32;       // + the MMA and copy thread's warp
// Batches the training kernels take (dZ of every layer is kept: 17 MB at 4 x
// 256); larger ones go layer by layer through the persistent GEMMs.
constexpr int kNetTrainRows = 4096;
constexpr int kNetActSbo = kNMax / 8 * 128;  // bytes between 8-row groups of the A operand

__host__ __device__ constexpr int pad32(int n) { return (n + 31) & ~31; }

// The network's shape and where its layers lie.
struct NetShape {
  int n_in, width, depth, n_out;
  __host__ __device__ int layers() const { return depth + 1; }
  __host__ __device__ int din(int l) const { return l == 0 ? n_in : width; }
  __host__ __device__ int dout(int l) const { return l == depth ? n_out : width; }
  // W_l in the flat parameter vector (b_l follows it)
  __host__ __device__ long long woff(int l) const {
    return l == 0 ? 0
                  : ((long long)n_in * width + width) +
                        (long long)(l - 1) * ((long long)width * width + width);
  }
  // elements of layer l in either packed copy, both extents padded to 32
  __host__ __device__ long long poff(int l) const {
    return l == 0 ? 0
                  : (long long)pad32(n_in) * pad32(width) +
                        (long long)(l - 1) * pad32(width) * pad32(width);
  }
  __host__ __device__ long long packed() const {
    return poff(depth) + (long long)pad32(din(depth)) * pad32(n_out);
  }
};

// Element (n, k) of an operand of np rows in a packed copy: slices of 16 k,
// each the K-major core layout (8 rows x 16 bytes; K-adjacent core matrices
// 128 bytes apart, 8-row groups 256).
__host__ __device__ __forceinline__ long long pack_index(int n, int k, int np) {
  return (long long)(k >> 4) * np * 16 + ((n >> 3) * 2 + ((k >> 3) & 1)) * 64 + (n & 7) * 8 +
         (k & 7);
}
// Stores parameter W_l(i, j) into the forward copy (rows j, k = i) and the
// backward copy (rows i, k = j).
__device__ __forceinline__ void pack_weight(const NetShape& s, int l, int i, int j, float w,
                                            __nv_bfloat16* fwd, __nv_bfloat16* bwd) {
  const __nv_bfloat16 v = __float2bfloat16_rn(w);
  const long long p = s.poff(l);
  fwd[p + pack_index(j, i, pad32(s.dout(l)))] = v;
  bwd[p + pack_index(i, j, pad32(s.din(l)))] = v;
}
// Layer of parameter q of the flat vector, and its index within the layer.
__device__ __forceinline__ int param_layer(const NetShape& s, long long q, int* at) {
  int l = 0;
  if (s.depth > 0 && q >= s.woff(1)) {
    const long long per = (long long)s.width * s.width + s.width;
    const long long r = (q - s.woff(1)) / per;
    l = 1 + (int)(r < s.depth - 1 ? r : s.depth - 1);
  }
  *at = (int)(q - s.woff(l));
  return l;
}

struct NetArgs {
  NetShape s;
  int batch;
  int rows;  // k_net_cluster: rows of a tile in use (32, 64 or 128)
  const float* x;
  const float* theta;
  const __nv_bfloat16 *fwd, *bwd;  // packed weights
  float* y;                        // inference: batch x n_out
  // training (t non-null)
  const float* t;
  float scale;         // 1 / (batch n_out)
  float* h;            // hidden layer l (1..depth) at h + (l - 1) h_stride
  long long h_stride;
  float* dz;           // dZ of layer l at dz + l dz_stride
  long long dz_stride;
  float* loss_part;    // one partial sum of squares per CTA
  int* err;
};

struct NetSmem {
  __nv_bfloat16 act[2][kM * kNMax];            // A operands of the two tiles
  __nv_bfloat16 ring[kNetStages][kNMax * 32];  // weight slices
  float bias[2 * kNetEpi / 32][4][32];         // per warp: its chunks' columns
  unsigned long long full[kNetStages], empty[kNetStages], acc_full[2], act_ready[2];
  unsigned tmem_base;
  int give_up;
};

struct ClSmem {
  __nv_bfloat16 act[2][kM * kNMax];             // A operands of this layer and the next
  __nv_bfloat16 w[kNetBufs][kNetBlock * kNMax];  // weights of this CTA's columns
  unsigned long long full[kNetBufs], acc_full;
  float red[8];
  unsigned tmem_base;
  int give_up;
};

// Walks the ring's slots; par: the parity of the phase the slot is in.
constexpr unsigned kRingBytes = kNMax * 64;
struct Ring {
  unsigned slot = 0, par = 0;
  __device__ __forceinline__ void step() {
    if (++slot == kNetStages) {
      slot = 0;
      par ^= 1u;
    }
  }
};

__device__ __forceinline__ void bulk_load(unsigned dst, const void* src, unsigned bytes,
                                          unsigned mbar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
      ::"r"(dst), "l"(src), "r"(bytes), "r"(mbar)
      : "memory");
}

__device__ __forceinline__ void tmem_load32(unsigned taddr, unsigned* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, "
      "%10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, "
      "%26, %27, %28, %29, %30, %31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

__device__ __forceinline__ void mma_f16(unsigned d_tmem, unsigned long long da,
                                        unsigned long long db, unsigned idesc, unsigned accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(da), "l"(db), "r"(idesc), "r"(accum)
      : "memory");
}
__device__ __forceinline__ void mma_commit(unsigned mbar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(mbar)
      : "memory");
}
__device__ __forceinline__ void mbar_init(unsigned addr, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(addr), "r"(count) : "memory");
}

// Byte offset of element (row, k) of a 256-k operand of the core layout (k a
// multiple of 8: one 16-byte row of a core matrix).
__device__ __forceinline__ unsigned act_offset(int row, int k) {
  return (unsigned)((row >> 3) * kNetActSbo + (k >> 3) * 128 + (row & 7) * 16);
}
__device__ __forceinline__ uint4 pack8(const float* v) {
  return make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]),
                    pack_bf16x2(v[6], v[7]));
}
// Four consecutive values of a row of n (columns c ..), 16 bytes at once
// where vec allows it.
__device__ __forceinline__ void store4(float* row, int c, int n, bool vec, const float* v) {
  if (vec && c + 3 < n) {
    *reinterpret_cast<float4*>(row + c) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (c + j < n) row[c + j] = v[j];
  }
}

// Stage st of a tile: forward layer st, then (training) the dZ products from
// the last layer down to layer 1.
struct NetStage {
  int layer, N, K;  // true extents; operands are padded to 32
  bool back;
  __device__ __forceinline__ NetStage(const NetShape& s, int st) {
    back = st >= s.layers();
    layer = back ? 2 * s.layers() - 1 - st : st;
    N = back ? s.din(layer) : s.dout(layer);
    K = back ? s.dout(layer) : s.din(layer);
  }
};

// A tile's inputs as the first A operand (k >= n_in and rows beyond the batch
// zero) in the first `rows` rows, a power of two, by kNetEpi threads.
__device__ __forceinline__ void net_input_tile(const NetArgs& g, unsigned char* act, int m0,
                                               int rows, int t) {
  const int n_in = g.s.n_in;
  for (int e = t; e < rows * (pad32(n_in) / 8); e += kNetEpi) {
    const int r = e & (rows - 1), k = e / rows * 8, m = m0 + r;
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      v[j] = m < g.batch && k + j < n_in ? ld_chained(g.x + (size_t)m * n_in + k + j) : 0.f;
    *reinterpret_cast<uint4*>(act + act_offset(r, k)) = pack8(v);
  }
}

// tanh on the special-function unit: its error (about 2^-11 relative) is
// below the BF16 rounding of the operands
__device__ __forceinline__ float net_tanh(float v) {
  asm("tanh.approx.f32 %0, %0;" : "+f"(v));
  return v;
}

__global__ void __launch_bounds__(kNetThreads, 1)
    k_net(const __grid_constant__ NetArgs g, int tiles) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  NetSmem& sm = *reinterpret_cast<NetSmem*>(smem_raw);
  constexpr int kMmaWarp = 2 * kNetEpi / 32, kCopyWarp = kMmaWarp + 1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const NetShape& s = g.s;
  const int L = s.layers();
  volatile int* give_up = &sm.give_up;
  if (tid == 0) {
    for (int q = 0; q < kNetStages; ++q) {
      mbar_init(smem_u32(&sm.full[q]), 1);
      mbar_init(smem_u32(&sm.empty[q]), 1);
    }
    for (int w = 0; w < 2; ++w) {
      mbar_init(smem_u32(&sm.acc_full[w]), 1);
      mbar_init(smem_u32(&sm.act_ready[w]), kNetEpi);
    }
    sm.give_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(&sm.tmem_base)),
                 "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const unsigned tmem = sm.tmem_base;
  const unsigned long long wait_ns = mma_wait_limit();
  // this CTA's tiles: blockIdx.x + j gridDim.x, j even in slot 0, odd in slot 1
  const int mine = (tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;

  if (warp == kCopyWarp) {
    // weight slices in the MMAs' order: tile pair, layer, tile of the pair
    if (lane == 0) {
      Ring r;
      bool ok = true;
      for (int j = 0; j < mine && ok; j += 2)
        for (int l = 0; l < L && ok; ++l)
          for (int w = 0; w < 2 && j + w < mine && ok; ++w) {
            const unsigned bytes = (unsigned)pad32(s.dout(l)) * 64u;
            const char* src = reinterpret_cast<const char*>(g.fwd + s.poff(l));
            for (int k = pad32(s.din(l)) / 32; k > 0; --k, src += bytes, r.step()) {
              if (!ws_wait(smem_u32(sm.empty) + 8u * r.slot, r.par ^ 1u, wait_ns, give_up)) {
                ok = false;
                break;
              }
              const unsigned mb = smem_u32(sm.full) + 8u * r.slot;
              asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mb),
                           "r"(bytes)
                           : "memory");
              bulk_load(smem_u32(sm.ring) + r.slot * kRingBytes, src, bytes, mb);
            }
          }
      if (!ok) {
        *give_up = 1;
        atomicExch(g.err, 1);
      }
      // no copy lands after the CTA has gone: the last fill of every slot (one
      // never filled passes: the parity before its first phase)
      for (int p = 0; p < kNetStages; ++p, r.step())
        mbar_wait(smem_u32(sm.full) + 8u * r.slot, r.par ^ 1u, kWaitNs);
    }
  } else if (warp == kMmaWarp) {
    if (lane == 0) {
      unsigned last_bar = 0, last_par = 0;
      Ring r;
      bool ok = true;
      for (int j = 0; j < mine && ok; j += 2)
        for (int l = 0; l < L && ok; ++l)
          for (int w = 0; w < 2 && j + w < mine && ok; ++w) {
            const int n = (j >> 1) * L + l, np = pad32(s.dout(l));  // n: phase of the slot
            const unsigned idesc = instr_desc(np), d = tmem + 256u * (unsigned)w;
            // descriptors count 16 bytes: 256 a K step of A; a step of B and a
            // slot of the ring are added to its first
            unsigned long long da = smem_desc(smem_u32(sm.act[w]), 128, kNetActSbo);
            const unsigned long long db0 = smem_desc(smem_u32(sm.ring), 128, 256);
            if (!ws_wait(smem_u32(&sm.act_ready[w]), n & 1, wait_ns, give_up)) {
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            unsigned accum = 0;
            for (int k = pad32(s.din(l)) / 32; k > 0; --k, da += 32, r.step()) {
              if (!ws_wait(smem_u32(sm.full) + 8u * r.slot, r.par, wait_ns, give_up)) {
                ok = false;
                break;
              }
              const unsigned long long db = db0 + (unsigned long long)(r.slot * (kRingBytes / 16));
              mma_f16(d, da, db, idesc, accum);
              mma_f16(d, da + 16, db + (unsigned long long)(np * 2), idesc, 1u);
              accum = 1;
              last_bar = smem_u32(sm.empty) + 8u * r.slot;
              last_par = r.par;
              mma_commit(last_bar);
            }
            if (!ok) break;
            last_bar = smem_u32(&sm.acc_full[w]);
            last_par = (unsigned)(n & 1);
            mma_commit(last_bar);
          }
      if (!ok) {
        *give_up = 1;
        atomicExch(g.err, 1);
      }
      // the accumulators are released only after the last MMA has completed
      if (last_bar != 0) mbar_wait(last_bar, last_par, kWaitNs);
    }
  } else {
    // 8 warps per slot; TMEM lane = row: warp w reads rows 32 (w % 4) .. + 31,
    // the 32-column chunks h, h + 2, ... of its half h
    const int w = warp >> 3, h = (warp >> 2) & 1, t = tid & (kNetEpi - 1);
    const int row = (warp & 3) * 32 + lane;
    const unsigned trow = tmem + 256u * (unsigned)w + ((unsigned)((warp & 3) * 32) << 16);
    unsigned char* act = reinterpret_cast<unsigned char*>(sm.act[w]);
    int n = 0;  // phase of the slot
    bool ok = true;
    for (int j = w; j < mine && ok; j += 2) {
      const int m0 = ((int)blockIdx.x + j * (int)gridDim.x) * kM, m = m0 + row;
      net_input_tile(g, act, m0, kM, t);
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      mbar_arrive(smem_u32(&sm.act_ready[w]));
      for (int l = 0; l < L && ok; ++l, ++n) {
        const int N = s.dout(l), np = pad32(N);
        const float* b = g.theta + s.woff(l) + (long long)s.din(l) * N;
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // the warp's own copy: no barrier between the warps
          const int c = h * 32 + 64 * i + lane;
          sm.bias[warp][i][lane] = c < N ? __ldg(b + c) : 0.f;
        }
        __syncwarp();
        ok = __all_sync(0xffffffffu,
                        ws_wait(smem_u32(&sm.acc_full[w]), n & 1, wait_ns, give_up));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const bool out = l == s.depth;
        for (int c0 = h * 32; c0 < np; c0 += 64) {
          unsigned r[32];
          tmem_load32(trow + (unsigned)c0, r);
          const float* bias = sm.bias[warp][c0 >> 6];
#pragma unroll
          for (int c8 = 0; c8 < 32; c8 += 8) {
            const int c = c0 + c8;
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[c8 + i]) + bias[c8 + i];
            if (out) {
              if (m < g.batch) {
                float* yp = g.y + (size_t)m * N;
                const bool vec = (N & 3) == 0 && ((size_t)yp & 15u) == 0;
                store4(yp, c, N, vec, v);
                store4(yp, c + 4, N, vec, v + 4);
              }
            } else {
#pragma unroll
              for (int i = 0; i < 8; ++i) v[i] = net_tanh(v[i]);
              // columns from N to its padding are k of the next product: zero, also
              // where an infinite input has made a NaN of their zero weights
              if (c + 8 > N) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                  if (c + i >= N) v[i] = 0.f;
              }
              *reinterpret_cast<uint4*>(act + act_offset(row, c)) = pack8(v);
            }
          }
        }
        __syncwarp();  // every lane has read the biases
        if (!out) {
          asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
          asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
          mbar_arrive(smem_u32(&sm.act_ready[w]));
        }
      }
    }
    if (!ok) {
      *give_up = 1;
      if (lane == 0) atomicExch(g.err, 1);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  if (warp == kMmaWarp)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512u)
                 : "memory");
}

// The kernels of a training step are launched with programmatic stream
// serialisation; what one writes, the next reads with ld_chained.

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(r));
  return r;
}
// Closes a stage: this CTA's writes into the peers' operands are visible to
// their MMAs after it.  Every thread of every CTA passes every one, also after
// a wait gave up, so that none waits for a peer that has gone.
__device__ __forceinline__ void cluster_close() {
  asm volatile("fence.proxy.async;\n" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  asm volatile("fence.proxy.async;\n" ::: "memory");
}
__device__ __forceinline__ void store_peer(unsigned addr, unsigned peer, uint4 v) {
  unsigned a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(peer));
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(a), "r"(v.x),
               "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}

__global__ void __launch_bounds__(kClThreads, 1) k_net_cluster(const __grid_constant__ NetArgs g) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  ClSmem& sm = *reinterpret_cast<ClSmem*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int kMmaWarp = kNetEpi / 32;
  const NetShape& s = g.s;
  const int L = s.layers(), stages = 2 * L - 1;
  const unsigned C = cluster_size(), rank = cluster_rank();
  const int n0 = (int)rank * kNetBlock;  // this CTA's columns of every layer
  const int m0 = (int)(blockIdx.x / C) * g.rows;
  volatile int* give_up = &sm.give_up;
  if (tid == 0) {
    for (int q = 0; q < kNetBufs; ++q) mbar_init(smem_u32(&sm.full[q]), 1);
    mbar_init(smem_u32(&sm.acc_full), 1);
    sm.give_up = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(&sm.tmem_base)),
                 "r"((unsigned)kNetBlock)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  after_previous_kernel();
  if (warp != kMmaWarp) {
    net_input_tile(g, reinterpret_cast<unsigned char*>(sm.act[0]), m0, g.rows, tid);
  }
  __syncthreads();
  // also: every peer has started, its shared memory may be written
  cluster_close();
  const unsigned tmem = sm.tmem_base;
  const unsigned long long wait_ns = mma_wait_limit();
  // stages whose product has columns in this block: the q-th of them uses
  // weight buffer q % kNetBufs and phase q of the accumulator
  auto works = [&](int st) { return n0 < pad32(NetStage(s, st).N); };
  int loaded = 0, next = 0;  // the copy thread: buffers filled, next stage to look at
  auto load_next = [&]() {
    while (next < stages && !works(next)) ++next;
    if (next >= stages) return;
    const NetStage sg(s, next);
    const int np = pad32(sg.N), ks = pad32(sg.K) / 16, buf = loaded % kNetBufs;
    const __nv_bfloat16* src = (sg.back ? g.bwd : g.fwd) + s.poff(sg.layer) + n0 * 16;
    const unsigned mb = smem_u32(&sm.full[buf]);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mb),
                 "r"((unsigned)ks * kNetBlock * 32u)
                 : "memory");
    for (int k = 0; k < ks; ++k)
      bulk_load(smem_u32(sm.w[buf] + k * kNetBlock * 16), src + (size_t)k * np * 16,
                kNetBlock * 32, mb);
    ++loaded;
    ++next;
  };
  const bool mma_thread = warp == kMmaWarp && lane == 0;
  if (mma_thread)
    for (int b = 0; b < kNetBufs; ++b) load_next();

  const int h = (warp >> 2) & 1, row = (warp & 3) * 32 + lane, m = m0 + row;
  const bool live = m < g.batch;
  const bool epi = warp < kMmaWarp && (warp & 3) * 32 < g.rows;  // warps with rows in use
  const int c = n0 + 16 * h;  // first of this thread's 16 columns
  const unsigned tsrc = tmem + ((unsigned)((warp & 3) * 32) << 16) + 16u * (unsigned)h;
  float loss = 0.f;
  bool ok = true;
  int q = 0;
  for (int st = 0; st < stages; ++st) {
    const NetStage sg(s, st);
    const bool last = st == stages - 1;
    if (works(st)) {
      if (mma_thread && ok) {
        const int buf = q % kNetBufs, ks = pad32(sg.K) / 16;
        ok = ws_wait(smem_u32(&sm.full[buf]), (q / kNetBufs) & 1, wait_ns, give_up);
        if (ok) {
          unsigned long long da = smem_desc(smem_u32(sm.act[st & 1]), 128, kNetActSbo);
          unsigned long long db = smem_desc(smem_u32(sm.w[buf]), 128, 256);
          for (int k = 0; k < ks; k += 2, da += 32, db += 4 * kNetBlock) {
            mma_f16(tmem, da, db, instr_desc(kNetBlock), k > 0 ? 1u : 0u);
            mma_f16(tmem, da + 16, db + 2 * kNetBlock, instr_desc(kNetBlock), 1u);
          }
          mma_commit(smem_u32(&sm.acc_full));
          // its weight buffer is free once the MMAs are done; nothing else of
          // the CTA is released before that either
          ok = mbar_wait(smem_u32(&sm.acc_full), q & 1, wait_ns);
          if (!ok) mbar_wait(smem_u32(&sm.acc_full), q & 1, kWaitNs);
          else load_next();
        }
        if (!ok) {
          *give_up = 1;
          atomicExch(g.err, 1);
        }
      }
      if (epi && ok) {
        const int l = sg.layer, N = sg.N;
        // what the epilogue needs from global memory, under the MMAs
        float bias = 0.f, hv[16];
        const float* hp = nullptr;
        if (sg.back) {
          hp = g.h + (long long)(l - 1) * g.h_stride + (size_t)m * N;
          const bool vec = (N & 3) == 0 && ((size_t)hp & 15u) == 0;
#pragma unroll
          for (int i = 0; i < 16; i += 4) {
            if (live && vec && c + i + 3 < N) {
              const float4 a = *reinterpret_cast<const float4*>(hp + c + i);
              hv[i] = a.x, hv[i + 1] = a.y, hv[i + 2] = a.z, hv[i + 3] = a.w;
            } else {
#pragma unroll
              for (int k = i; k < i + 4; ++k) hv[k] = live && c + k < N ? hp[c + k] : 0.f;
            }
          }
        } else {
          const int n = c + (lane & 15);
          if (n < N) bias = ld_chained(g.theta + s.woff(l) + (long long)s.din(l) * N + n);
        }
        ok = __all_sync(0xffffffffu, ws_wait(smem_u32(&sm.acc_full), q & 1, wait_ns, give_up));
        if (ok) {
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
          float v[16];
          {
            unsigned r[16];
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, "
                "%9, %10, %11, %12, %13, %14, %15}, [%16];\n"
                : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                  "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
                  "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                : "r"(tsrc)
                : "memory");
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
          }
          const bool out = !sg.back && l == s.depth;
          float* dst;  // the row's values in global memory
          if (sg.back) {
            dst = g.dz + (long long)(l - 1) * g.dz_stride + (size_t)m * N;
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] *= 1.f - hv[i] * hv[i];
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] += __shfl_sync(0xffffffffu, bias, i);
            if (!out) {
#pragma unroll
              for (int i = 0; i < 16; ++i) v[i] = net_tanh(v[i]);
              dst = g.h + (long long)l * g.h_stride + (size_t)m * N;
            } else {
              // dZ = dY of the linear output layer, and the squared error
              dst = g.dz + (long long)l * g.dz_stride + (size_t)m * N;
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const float d =
                    live && c + i < N ? v[i] - ld_chained(g.t + (size_t)m * N + c + i) : 0.f;
                v[i] = 2.f * d * g.scale;
                loss += d * d;
              }
            }
          }
          if (live) {
            const bool vec = (N & 3) == 0 && ((size_t)dst & 15u) == 0;
#pragma unroll
            for (int i = 0; i < 16; i += 4) store4(dst, c + i, N, vec, v + i);
          }
          if (!last) {
            // columns from N to its padding are k of the next product: zero
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (c + i >= N) v[i] = 0.f;
            const uint4 lo = pack8(v), hi = pack8(v + 8);
            const unsigned a = smem_u32(sm.act[(st + 1) & 1]) + act_offset(row, c);
            for (unsigned p = 0; p < C; ++p) {
              store_peer(a, p, lo);
              store_peer(a + 128, p, hi);
            }
          }
        } else {
          *give_up = 1;
          if (lane == 0) atomicExch(g.err, 1);
        }
      }
      ++q;
    }
    if (!last) {
      __syncwarp();
      cluster_close();
    }
  }
  if (mma_thread)  // no copy lands after the CTA has gone
    for (int p = loaded < kNetBufs ? 0 : loaded - kNetBufs; p < loaded; ++p)
      mbar_wait(smem_u32(&sm.full[p % kNetBufs]), (unsigned)((p / kNetBufs) & 1), kWaitNs);
  if (warp < kMmaWarp) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, off);
    if (lane == 0) sm.red[warp] = loss;
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  if (tid == 0) {
    float v = 0.f;
    for (int w = 0; w < 8; ++w) v += sm.red[w];
    g.loss_part[blockIdx.x] = v;
  }
  if (warp == kMmaWarp)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"((unsigned)kNetBlock)
                 : "memory");
}

// ---------------------------------------------------------------------------
// dW_l = H_{l-1}^T dZ_l and db_l = column sums of dZ_l, all layers.
// ---------------------------------------------------------------------------
constexpr int kDwThreads = 512;
constexpr int kDwN = 32;    // columns of W per CTA
constexpr int kDwK = 256;   // batch rows per CTA

struct DwArgs {
  NetShape s;
  int batch;
  int tiles;  // CTAs of the weight gradients; those of the biases follow
  const float* x;  // layer 0's input (batch x n_in)
  const float* h;
  long long h_stride;
  const float* dz;
  long long dz_stride;
  float* grad;
  const float* loss_part;
  int loss_parts;
  float scale;
  float* loss;
  int* err;
};

struct DwSmem {
  __nv_bfloat16 a[kM * kDwK];    // 64 KB
  __nv_bfloat16 b[kDwN * kDwK];  // 16 KB
  unsigned long long mbar;
  unsigned tmem_base;
};
// Bias gradients: db_l(n) = sum over the batch of dZ_l, one CTA per 32
// columns (past the weight tiles in the grid).  The rows are added in their
// order, one lane a column, whatever the batch: 512 threads bring 256 rows at
// a time into one of two buffers while warp 0 adds up the other (a chain of
// 4 clocks a row).
__device__ __forceinline__ void dw_bias(float (*buf)[kDwK][kDwN], const float* Z, int dout, int n0,
                                        int batch, float* db, int t) {
  constexpr int P = kDwThreads / kDwN, R = kDwK / P;
  const int c = t % kDwN, p = t / kDwN;
  float v[R], sum = 0.f;
  auto load = [&](int k0) {
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int k = k0 + p + i * P;
      v[i] = k < batch && n0 + c < dout ? ld_chained(Z + (size_t)k * dout + n0 + c) : 0.f;
    }
  };
  load(0);
  for (int k0 = 0, q = 0; k0 < batch; k0 += kDwK, q ^= 1) {
#pragma unroll
    for (int i = 0; i < R; ++i) buf[q][p + i * P][c] = v[i];
    __syncthreads();
    if (k0 + kDwK < batch) load(k0 + kDwK);
    if (t < kDwN) {
#pragma unroll 32
      for (int k = 0; k < kDwK; ++k) sum += buf[q][k][t];
    }
  }
  if (t < kDwN && n0 + t < dout) db[t + n0] = sum;
}

// X(r, k) = src[k * ld + r], r in [r0, r0 + ROWS), k in [0, kDwK): BF16 into
// the core layout, zero outside R x K.  A task is 4 rows x 8 k: eight 16-byte
// loads along the rows, transposed in registers into four 16-byte stores.
template <int ROWS>
__device__ __forceinline__ void dw_stage(unsigned char* dst, const float* src, int ld,
                                         int r0, int R, int K, int t) {
  constexpr int quads = ROWS / 4, G = quads * (kDwK / 8);
  const bool vec = (ld & 3) == 0 && ((size_t)src & 15u) == 0;
#pragma unroll 2
  for (int e = t; e < G; e += kDwThreads) {
    const int r = e % quads * 4, k = e / quads * 8, m = r0 + r;
    float4 v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k + j >= K || m >= R) continue;
      const float* p = src + (size_t)(k + j) * ld + m;
      if (vec && m + 3 < R) {
        v[j] = ld_chained(reinterpret_cast<const float4*>(p));
      } else {
        v[j].x = ld_chained(p);
        if (m + 1 < R) v[j].y = ld_chained(p + 1);
        if (m + 2 < R) v[j].z = ld_chained(p + 2);
        if (m + 3 < R) v[j].w = ld_chained(p + 3);
      }
    }
    const float* f = reinterpret_cast<const float*>(v);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float c[8] = {f[i],      f[4 + i],  f[8 + i],  f[12 + i],
                          f[16 + i], f[20 + i], f[24 + i], f[28 + i]};
      *reinterpret_cast<uint4*>(dst + act_offset(r + i, k)) = pack8(c);
    }
  }
}

__global__ void __launch_bounds__(kDwThreads, 1) k_net_dw(const __grid_constant__ DwArgs g) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  DwSmem& sm = *reinterpret_cast<DwSmem*>(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const NetShape& s = g.s;
  static_assert(sizeof(float) * 2 * kDwK * kDwN <= sizeof(sm.a), "dw_bias's buffers");
  after_previous_kernel();
  // this CTA's layer and tile
  int l = 0, b = (int)blockIdx.x, mt, nt;
  const bool bias = b >= g.tiles;
  if (bias) {
    if (blockIdx.y > 0) return;
    b -= g.tiles;
  }
  for (;; ++l) {
    mt = bias ? 1 : (s.din(l) + kM - 1) / kM;
    nt = (s.dout(l) + kDwN - 1) / kDwN;
    if (b < mt * nt || l == s.depth) break;
    b -= mt * nt;
  }
  if (bias) {
    dw_bias(reinterpret_cast<float(*)[kDwK][kDwN]>(sm.a), g.dz + (long long)l * g.dz_stride,
            s.dout(l), b * kDwN, g.batch, g.grad + s.woff(l) + (long long)s.din(l) * s.dout(l),
            tid);
    return;
  }
  const int din = s.din(l), dout = s.dout(l), m0 = b % mt * kM, n0 = b / mt * kDwN;
  const int k0 = (int)blockIdx.y * kDwK, K = min(kDwK, g.batch - k0);
  const bool split = gridDim.y > 1;
  const float* H = (l == 0 ? g.x : g.h + (long long)(l - 1) * g.h_stride) + (size_t)k0 * din;
  const float* Z = g.dz + (long long)l * g.dz_stride + (size_t)k0 * dout;
  const unsigned mbar = smem_u32(&sm.mbar);
  if (tid == 0) {
    mbar_init(mbar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(&sm.tmem_base)),
                 "r"((unsigned)kDwN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  dw_stage<kM>(reinterpret_cast<unsigned char*>(sm.a), H, din, m0, din, K, tid);
  dw_stage<kDwN>(reinterpret_cast<unsigned char*>(sm.b), Z, dout, n0, dout, K, tid);
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const unsigned tmem = sm.tmem_base;
  const unsigned long long wait_ns = mma_wait_limit();
  if (tid == 0) {
    const unsigned a_base = smem_u32(sm.a), b_base = smem_u32(sm.b);
    const int ks = (K + 15) / 16;
    for (int k = 0; k < ks; ++k)
      mma_f16(tmem, smem_desc(a_base + (unsigned)k * 256, 128, kNetActSbo),
              smem_desc(b_base + (unsigned)k * 256, 128, kNetActSbo), instr_desc(kDwN),
              k > 0 ? 1u : 0u);
    mma_commit(mbar);
  }
  const bool ok = __syncthreads_and(mbar_wait(mbar, 0, wait_ns) ? 1 : 0) != 0;
  float* grad = g.grad + s.woff(l);
  if (!ok) {
    if (tid == 0) atomicExch(g.err, 1);
    mbar_wait(mbar, 0, kWaitNs);  // in-flight MMAs before TMEM is released
  } else {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (warp < 4) {
      unsigned r[32];
      tmem_load32(tmem + ((unsigned)(warp * 32) << 16), r);
      const int m = m0 + warp * 32 + lane;
      if (m < din) {
        float* wrow = grad + (size_t)m * dout;
        const bool vec = (dout & 3) == 0 && ((size_t)wrow & 15u) == 0;
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          const float v[4] = {__uint_as_float(r[j]), __uint_as_float(r[j + 1]),
                              __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3])};
          if (!split) {
            store4(wrow, n0 + j, dout, vec, v);
          } else if (vec && n0 + j + 3 < dout) {
            atomicAdd(reinterpret_cast<float4*>(wrow + n0 + j),
                      make_float4(v[0], v[1], v[2], v[3]));
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (n0 + j + i < dout) atomicAdd(wrow + n0 + j + i, v[i]);
          }
        }
      }
    } else if (warp == 4 && blockIdx.x == 0 && blockIdx.y == 0 && lane == 0) {
      float v = 0.f;
      for (int p = 0; p < g.loss_parts; ++p) v += g.loss_part[p];
      *g.loss = v * g.scale;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"((unsigned)kDwN)
                 : "memory");
}

// The packed copies of the whole parameter vector.
__global__ void k_net_pack(const __grid_constant__ NetShape s, const float* __restrict__ theta,
                           long long n, __nv_bfloat16* __restrict__ fwd,
                           __nv_bfloat16* __restrict__ bwd) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  int at;
  const int l = param_layer(s, q, &at), dout = s.dout(l);
  if (at < s.din(l) * dout) pack_weight(s, l, at / dout, at % dout, theta[q], fwd, bwd);
}

// One Adam step over all parameters (bias-corrected, Kingma & Ba); the
// updated weights also go into the packed copies.
__global__ void k_net_adam(const __grid_constant__ NetShape s, float* p, const float* g, float* m,
                           float* v, long long n, float lr, float b1, float b2, float eps,
                           float c1, float c2, __nv_bfloat16* fwd, __nv_bfloat16* bwd) {
  after_previous_kernel();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = ld_chained(g + i);
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  p[i] = pi;
  int at;
  const int l = param_layer(s, i, &at), dout = s.dout(l);
  if (at < s.din(l) * dout) pack_weight(s, l, at / dout, at % dout, pi, fwd, bwd);
}

template <typename... P, typename... A>
static cudaError_t launch_serial(void (*kernel)(P...), unsigned grid_x, unsigned grid_y,
                                 unsigned threads, int smem, int cluster, cudaStream_t s,
                                 A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid_x, grid_y);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)cluster;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 0 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// CTAs of a cluster: the 32-column blocks of the widest layer, a power of two.
static int net_cluster(const NetShape& s) {
  const int n = pad32(s.depth > 0 && s.width > s.n_out ? s.width : s.n_out) / kNetBlock;
  int c = 1;
  while (c < n) c *= 2;
  return c;
}

// Rows of a tile: what a cluster exchanges after every layer is proportional
// to them (64 KB in and out of each of 8 CTAs at 128 rows), and unused rows of
// the 128-row product cost nothing here, so as few as the clusters that run at
// once allow.  GB300, us per training step of the 4 x 256 network with at most
// 32 / 64 / 128 / 256 CTAs: 256 rows 39.5 / 37.0 / 37.1 / 37.1, 512 rows 55.5
// / 43.2 / 65.7 / 65.8, 1024 rows 62 / 62 / 76 / 96.
constexpr int kNetCtas = 64;
static int net_rows_per_tile(int batch, int c) {
  int rows = 32;
  while (rows < kM && (batch + rows - 1) / rows * c > kNetCtas) rows *= 2;
  return rows;
}

static cudaError_t launch_net_cluster(NetArgs g, cudaStream_t s) {
  static bool attr_dev[kMaxDevices] = {};
  bool& attr = attr_dev[device_slot()];
  constexpr int bytes = (int)sizeof(ClSmem);
  static_assert(sizeof(ClSmem) <= 227 * 1024, "k_net_cluster's shared memory");
  if (!attr) {
    const cudaError_t e = cudaFuncSetAttribute(
        k_net_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  const int c = net_cluster(g.s);
  g.rows = net_rows_per_tile(g.batch, c);
  return launch_serial(k_net_cluster, (unsigned)((g.batch + g.rows - 1) / g.rows * c), 1,
                       kClThreads, bytes, c, s, g);
}

// Forward pass of g.batch rows.
static cudaError_t launch_net(const NetArgs& g, cudaStream_t s) {
  const int sms = sm_count(), tiles = (g.batch + kM - 1) / kM;
  static bool attr_dev[kMaxDevices] = {};
  bool& attr = attr_dev[device_slot()];
  constexpr int bytes = (int)sizeof(NetSmem);
  static_assert(sizeof(NetSmem) <= 227 * 1024, "k_net's shared memory");
  if (!attr) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_net, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  k_net<<<(unsigned)(tiles < sms ? tiles : sms), kNetThreads, bytes, s>>>(g, tiles);
  return cudaGetLastError();
}

static cudaError_t launch_net_dw(DwArgs g, long long nparams, cudaStream_t s) {
  static bool attr_dev[kMaxDevices] = {};
  bool& attr = attr_dev[device_slot()];
  constexpr int bytes = (int)sizeof(DwSmem);
  if (!attr) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_net_dw, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  const unsigned splits = (unsigned)((g.batch + kDwK - 1) / kDwK);
  if (splits > 1) {
    const cudaError_t e = cudaMemsetAsync(g.grad, 0, sizeof(float) * (size_t)nparams, s);
    if (e != cudaSuccess) return e;
  }
  int blocks = 0;
  g.tiles = 0;
  for (int l = 0; l <= g.s.depth; ++l) {
    const int nt = (g.s.dout(l) + kDwN - 1) / kDwN;
    g.tiles += (g.s.din(l) + kM - 1) / kM * nt;
    blocks += nt;
  }
  return launch_serial(k_net_dw, (unsigned)(g.tiles + blocks), splits, kDwThreads, bytes, 0, s, g);
}

}  // namespace mlp
}  // namespace lbm
