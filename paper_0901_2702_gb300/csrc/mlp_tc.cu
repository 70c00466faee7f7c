// Inference of the initial-guess network (Sec. 5) on the fifth-generation
// tensor cores, fused end to end: one persistent kernel takes a tile of 128
// pixels from the observed Stokes samples through the input features, the
// four layers and the decoding into an initial model.  Every layer is a chain
// of tcgen05.mma (M = 128, K = 16 per instruction, BF16 operands in shared
// memory, FP32 accumulators in tensor memory); the bias + GELU epilogues read
// the accumulators back with tcgen05.ld, each warp owning a lane quarter and
// a part of the columns, and write the next layer's BF16 operand to shared
// memory.  Nothing but the observations and the outputs touches HBM.
//
// The GELUs bound it: 768 a pixel at about 25 instructions each are some
// 22,000 issue cycles a tile and SM.  A tile's own chain -- observations,
// products, decoding -- is as long again, so a CTA has two tiles in flight, a
// group of eight warps and half the tensor memory each: one computes GELUs
// while the other's products run.  1,048,576 pixels: 1.15 ms with one tile in
// flight and one thread that loaded and issued, 0.89 ms so.
//
// Shared-memory operands are in the no-swizzle K-major canonical layout of
// the MMA descriptors: core matrices of 8 rows x 16 bytes stored as 128
// contiguous bytes, core matrices adjacent along K 128 bytes apart (the
// leading-dimension offset) and 8-row groups `sbo` bytes apart (the
// stride-dimension offset).  Beside the two 64 KB activation tiles, over which
// the features lie, 80 KB hold weights: they stream, 280 KB a tile from L2, in
// chunks of 16 KB (two K = 16 steps of a hidden layer; half of one holds the
// output layer) through a ring of five slots, layer by layer for the first
// group's tile, then for the second's.  One warp loads, one issues products;
// beside 16 busy warps their bookkeeping is what a chunk costs (some 500
// cycles, whatever its size or the ring's: chunks of 8 KB in eleven slots
// took 1.00 ms), hence chunks no smaller.
//
// Every wait is bounded (about 1 s); on a timeout the kernel lets its copies
// and tensor-core work in flight finish (bounded again), frees its tensor
// memory, writes kDevErrNnWait to the error word and returns.
#include <cuda_bf16.h>
#include <stdint.h>

#include "common.cuh"
#include "nn.cuh"
#include "nn_device.cuh"
#include "tc_device.cuh"

namespace vfisv {
namespace nn {

namespace {

using bf16 = __nv_bfloat16;

constexpr int TM = 128;       // pixels per tile = MMA M
constexpr int K0 = 32;        // input width (24) padded to two K = 16 steps
constexpr int N3 = 16;        // output width (11) padded to the smallest N for M = 128
constexpr int NSLOT = 5;      // weight ring depth
constexpr int kCompute = 512;  // 16 warps, in one or two groups, each with a tile in flight
constexpr int kLaunch = kCompute + 64;  // and a warp that loads weights, one that issues
constexpr int kPerLayer = HID / 32;  // chunks of a hidden layer

constexpr uint32_t kChunkBytes = HID * 32 * 2;    // 16384
constexpr uint32_t kHChunkBytes = TM * 64 * 2;    // 16384: 64 columns of the activations
constexpr uint32_t kW3ChunkBytes = N3 * 64 * 2;   // 2048: 64 inputs of the output layer
constexpr uint32_t kW3Bytes = N3 * HID * 2;       // 8192
static_assert(K0 == 32, "layer 0 is one chunk");
static_assert((1 + 2 * kPerLayer) * kChunkBytes + kW3Bytes == kTcPackBytes, "packed weight size");

// Shared-memory carve, bytes from a 1024-byte aligned base.
constexpr uint32_t SM_RING = 0;
constexpr uint32_t kTileBytes = TM * HID * 2;     // 65536
constexpr uint32_t SM_H = SM_RING + NSLOT * kChunkBytes;  // two activation tiles, the
// features (read by layer 0 before its epilogue writes) at the start of each
constexpr uint32_t SM_BIAS = SM_H + 2 * kTileBytes;         // b0 | b1 | b2 | b3 (16)
constexpr uint32_t SM_STAT = SM_BIAS + (3 * HID + N3) * 4;  // in_mean 24 | in_std 24 | out_mean 16 | out_std 16
constexpr uint32_t SM_BAR = SM_STAT + 80 * 4;             // full[5] empty[5] mma[2] ready[2] drain
constexpr uint32_t SM_TMEM = SM_BAR + 8 * (2 * NSLOT + 5) + 8;
constexpr uint32_t SM_END = SM_TMEM + 16;
constexpr size_t kSmemBytes = SM_END + 1024;
static_assert(SM_BAR % 8 == 0 && SM_BIAS % 16 == 0, "alignment");
static_assert(kSmemBytes <= 232448, "shared memory per block");

constexpr int kTmemCols = 512;  // an M = 128 x N = 256 FP32 accumulator a group

constexpr uint32_t kIdescHid = idesc_bf16(TM, HID);
constexpr uint32_t kIdescOut = idesc_bf16(TM, N3);

// Packed weights (global, kTcPackBytes), in the order they stream: W0, W1 and
// W2 as N = 256 x K = 32 chunks, W3 as four N = 16 x K = 64 blocks; element
// (n, k) is the weight from input k to output n, BF16, zero-padded.
__global__ void tc_pack_kernel(const float* __restrict__ blob, uint8_t* __restrict__ wp) {
  constexpr int E0 = HID * K0, E1 = HID * HID, E3 = N3 * HID;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < E0 + 2 * E1 + E3;
       i += gridDim.x * blockDim.x) {
    float w;
    uint32_t off;
    if (i < E0) {
      const int n = i / K0, k = i % K0;
      w = k < IN ? blob[OFF_W0 + (size_t)k * HID + n] : 0.0f;
      off = cm_off(n, k, 512);
    } else if (i < E0 + 2 * E1) {
      const int j = i - E0, l = j / E1, n = (j % E1) / HID, k = j % HID;
      w = blob[(l ? OFF_W2 : OFF_W1) + (size_t)k * HID + n];
      off = (1 + l * kPerLayer + k / 32) * kChunkBytes + cm_off(n, k % 32, 512);
    } else {
      const int j = i - E0 - 2 * E1, n = j / HID, k = j % HID;
      w = n < OUT ? blob[OFF_W3 + (size_t)k * OUT + n] : 0.0f;
      off = (1 + 2 * kPerLayer) * kChunkBytes + (k / 64) * kW3ChunkBytes +
            cm_off(n, k % 64, 1024);
    }
    *reinterpret_cast<bf16*>(wp + off) = __float2bfloat16(w);
  }
}

// Weight chunks of a layer.
__device__ __forceinline__ int layer_chunks(int l) { return (l == 1 || l == 2) ? kPerLayer : 1; }

// A ring cursor: slot and phase parity of the next chunk.
struct Cursor {
  int slot = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ void next() {
    if (++slot == NSLOT) {
      slot = 0;
      phase ^= 1;
    }
  }
};

struct TcArgs {
  const float* obs;  // [n][24]
  int64_t n;
  const float* blob;
  const uint8_t* wp;  // packed weights
  float mu;
  float* init;  // [n][10]
  float* conf;  // [n] or null
  float* raw;   // [n][11] or null
  int* err;
};

// G groups: two where a CTA has several tiles; all 16 warps on the one where it
// has a single tile (up to a tile an SM: 1,000 pixels 32.9 us with one group of
// eight warps idle, 30.8 so).
template <int G>
__global__ void __launch_bounds__(kLaunch, 1) mlp_tc_kernel(TcArgs a) {
  constexpr int THREADS = kCompute / G;  // a group: 4 lane quarters x 2 or 4 parts of the columns
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t sb = smem_u32(sm);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int group = (threadIdx.x / THREADS) % G, tid = threadIdx.x % THREADS;  // of the group
  float* bias = reinterpret_cast<float*>(sm + SM_BIAS);
  float* stat = reinterpret_cast<float*>(sm + SM_STAT);
  const uint32_t bar_full = sb + SM_BAR, bar_empty = bar_full + 8 * NSLOT,
                 bar_mma = bar_empty + 8 * NSLOT, bar_ready = bar_mma + 16,
                 bar_drain = bar_ready + 16;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + SM_TMEM);

  const int64_t ntiles = (a.n + TM - 1) / TM;
  const int my_tiles = (int)((ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x);
  // tiles go to the groups in turn; the last of an odd number is group 0's alone

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2 * NSLOT + 5; ++i)  // ready: a group's warps
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar_full + 8 * i),
                   "r"(i / 2 == NSLOT + 1 ? THREADS / 32 : 1)
                   : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = threadIdx.x; i < 3 * HID; i += kLaunch) {
    const int l = i / HID;
    bias[i] = a.blob[(l == 0 ? OFF_B0 : l == 1 ? OFF_B1 : OFF_B2) + i % HID];
  }
  if (threadIdx.x < N3)
    bias[3 * HID + threadIdx.x] = threadIdx.x < OUT ? a.blob[OFF_B3 + threadIdx.x] : 0.0f;
  if (threadIdx.x < IN) {
    stat[threadIdx.x] = a.blob[OFF_INM + threadIdx.x];
    stat[IN + threadIdx.x] = a.blob[OFF_INS + threadIdx.x];
  }
  if (threadIdx.x < OUT - 1) {
    stat[48 + threadIdx.x] = a.blob[OFF_OUTM + threadIdx.x];
    stat[64 + threadIdx.x] = a.blob[OFF_OUTS + threadIdx.x];
  }
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  const uint32_t tmem = *tmem_slot;

  if (warp == kCompute / 32) {
    // weight loads: their own warp, so that neither they wait for an issue nor
    // an issue for a slot
    if (lane == 0) {
      Cursor c;
      int loaded = 0;
      bool bad = false;
      for (int t = 0; t < my_tiles && !bad; t += G) {
        const uint8_t* src = a.wp;
        for (int l = 0; l < 4 && !bad; ++l) {
          const int n = layer_chunks(l);
          const uint32_t bytes = l < 3 ? kChunkBytes : kW3Bytes;
          for (int q = 0; q < (G == 2 && t + 1 < my_tiles ? 2 : 1) && !bad; ++q)
            for (int i = 0; i < n; ++i, c.next()) {
              // (the first round finds the slots free)
              if (!mbar_wait(bar_empty + 8 * c.slot, c.phase ^ 1)) {
                bad = true;
                break;
              }
              expect_tx(bar_full + 8 * c.slot, bytes);
              bulk_load(sb + SM_RING + c.slot * kChunkBytes, src + i * kChunkBytes, bytes,
                        bar_full + 8 * c.slot);
              if (loaded < NSLOT) ++loaded;
            }
          src += n * kChunkBytes;
        }
      }
      // the copies land, and of a whole stream the tensor cores' last arrivals
      // come, before the memory is released (slots in the order of their last use)
      for (int i = 0; i < loaded; ++i) {
        const int back = loaded - i, slot = (c.slot + NSLOT - back) % NSLOT;
        const uint32_t phase = c.phase ^ (back > c.slot ? 1u : 0u);
        mbar_wait(bar_full + 8 * slot, phase);
        if (!bad) mbar_wait(bar_empty + 8 * slot, phase);
      }
      if (bad) atomicExch(a.err, kDevErrNnWait);
    }
    __syncwarp();
    __syncthreads();
    return;
  }

  if (warp == kCompute / 32 + 1) {
    // the products of both groups, in the order of the stream (every slot's
    // phases are then waited for one after the other)
    if (lane == 0) {
      Cursor c;
      bool bad = false;
      for (int t = 0; t < my_tiles && !bad; t += G)
        for (int l = 0; l < 4 && !bad; ++l)
          for (int q = 0; q < (G == 2 && t + 1 < my_tiles ? 2 : 1) && !bad; ++q) {
            // four phases a tile: layer l's has parity l & 1
            if (!mbar_wait(bar_ready + 8 * q, l & 1)) {
              bad = true;
              break;
            }
            tc_after_sync();
            const uint32_t d = tmem + (uint32_t)(q * HID), A = sb + SM_H + q * kTileBytes;
            const uint32_t sbo = l == 0 ? (K0 / 8) * 128 : 1024;
            const int n = layer_chunks(l);
            for (int i = 0; i < n; ++i, c.next()) {
              if (!mbar_wait(bar_full + 8 * c.slot, c.phase)) {
                bad = true;
                break;
              }
              const uint32_t w = sb + SM_RING + c.slot * kChunkBytes;
              if (l < 3) {
                const uint32_t Ai = A + (i >> 1) * kHChunkBytes + (i & 1) * 512;
#pragma unroll
                for (int k = 0; k < 2; ++k)
                  mma_bf16(d, sdesc(Ai + k * 256, 128, sbo), sdesc(w + k * 256, 128, 512),
                           kIdescHid, (i | k) != 0);
              } else {
#pragma unroll 4
                for (int k = 0; k < HID / 16; ++k)
                  mma_bf16(d, sdesc(A + (k >> 2) * kHChunkBytes + (k & 3) * 256, 128, 1024),
                           sdesc(w + (k >> 2) * kW3ChunkBytes + (k & 3) * 256, 128, 1024),
                           kIdescOut, k != 0);
              }
              mma_commit(bar_empty + 8 * c.slot);
            }
            if (!bad) mma_commit(bar_mma + 8 * q);
          }
      if (bad) {
        // let the tensor-core work in flight finish before the memory is released
        mma_commit(bar_drain);
        mbar_wait(bar_drain, 0);
        atomicExch(a.err, kDevErrNnWait);
      }
    }
    __syncwarp();
    __syncthreads();
    return;
  }

  const uint32_t td = tmem + (uint32_t)(group * HID);
  uint8_t* const H = sm + SM_H + group * kTileBytes;
  // the warp's part of a layer's operand is in shared memory, and what it read
  // of the accumulator read
  auto ready = [&]() {
    fence_async_smem();
    tc_before_sync();
    __syncwarp();
    if (lane == 0)
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar_ready + 8 * group)
                   : "memory");
  };
  uint32_t mph = 0;
  // the group's products of the layer are done
  auto sync_mma = [&]() -> bool {
    const bool ok = __all_sync(0xffffffffu, mbar_wait(bar_mma + 8 * group, mph));
    mph ^= 1;
    tc_after_sync();
    return ok;
  };

  // bias + GELU of the accumulator -> BF16 activations (next layer's A)
  auto epilogue_hidden = [&](const float* b) {
    constexpr int kCols = HID / (THREADS / 128);  // a warp's columns
    const int q = warp & 3, row = 32 * q + lane, cbeg = ((warp >> 2) % (THREADS / 128)) * kCols;
    uint8_t* hrow = H + (row >> 3) * 1024 + (row & 7) * 16;
#pragma unroll 1
    for (int col0 = cbeg; col0 < cbeg + kCols; col0 += 32) {
      float v[32];
      tmem_ld32(td + ((uint32_t)(32 * q) << 16) + (uint32_t)col0, v);
      uint8_t* hc = hrow + (col0 >> 6) * kHChunkBytes + ((col0 & 63) >> 3) * 128;
#pragma unroll
      for (int g8 = 0; g8 < 4; ++g8) {
        uint32_t pk[4];
#pragma unroll
        for (int e = 0; e < 4; e += 2) {
          const int j = 8 * g8 + 2 * e;
          const float4 bb = *reinterpret_cast<const float4*>(b + col0 + j);
          const f2 g0 = gelu2(f2_add(f2_pack(v[j], v[j + 1]), f2_pack(bb.x, bb.y)));
          const f2 g1 = gelu2(f2_add(f2_pack(v[j + 2], v[j + 3]), f2_pack(bb.z, bb.w)));
          pk[e] = pack_bf16x2(f2_lo(g0), f2_hi(g0));
          pk[e + 1] = pack_bf16x2(f2_lo(g1), f2_hi(g1));
        }
        *reinterpret_cast<uint4*>(hc + g8 * 128) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
      }
    }
    ready();
  };

  bool ok = true;
  for (int t = group; t < my_tiles; t += G) {
    const int64_t tile = blockIdx.x + (int64_t)t * gridDim.x;
    // features: thread (row, part) writes input columns 8 part .. 8 part + 7
    // and of part + 2
    float ic_row = 1.0f;
    {
      const int row = tid & (TM - 1);
      const int64_t m = tile * TM + row;
      const bool live = m < a.n;
      const float* o = a.obs + m * IN;
      float inv = 0.0f;
      if (live) {
        ic_row = ic_of(o);
        inv = 1.0f / ic_row;
      }
#pragma unroll
      for (int part = tid >> 7; part < K0 / 8; part += THREADS / TM) {
        uint32_t pk[4] = {0u, 0u, 0u, 0u};
        if (live && part < IN / 8) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int j = 8 * part + 2 * e;
            pk[e] = pack_bf16x2((o[j] * inv - stat[j]) / stat[IN + j],
                                (o[j + 1] * inv - stat[j + 1]) / stat[IN + j + 1]);
          }
        }
        *reinterpret_cast<uint4*>(H + cm_off(row, 8 * part, (K0 / 8) * 128)) =
            make_uint4(pk[0], pk[1], pk[2], pk[3]);
      }
      ready();
    }
    if (!(ok = sync_mma())) break;
    epilogue_hidden(bias);
    if (!(ok = sync_mma())) break;
    epilogue_hidden(bias + HID);
    if (!(ok = sync_mma())) break;
    epilogue_hidden(bias + 2 * HID);
    if (!(ok = sync_mma())) break;
    if (tid < TM) {  // lane quarter tid / 32, row = tid
      float v[16];
      tmem_ld16(td + ((uint32_t)(32 * (tid >> 5)) << 16), v);
      const int64_t m = tile * TM + tid;
      if (m < a.n) {
        float y[OUT];
#pragma unroll
        for (int o = 0; o < OUT; ++o) y[o] = v[o] + bias[3 * HID + o];
        decode_row(y, ic_row, a.mu, stat + 48, stat + 64, a.init + m * 10);
        if (a.conf) a.conf[m] = y[OUT - 1];
        if (a.raw)
#pragma unroll
          for (int o = 0; o < OUT; ++o) a.raw[m * OUT + o] = y[o];
      }
    }
    tc_before_sync();
  }

  if (!ok && lane == 0) atomicExch(a.err, kDevErrNnWait);
  tc_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc_after_sync();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kTmemCols)
                 : "memory");
  }
}

}  // namespace

cudaError_t nn_infer(void* ws, const float* blob, const float* obs, int64_t n, float mu,
                     float* init, float* conf, float* raw, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  uint8_t* wp = static_cast<uint8_t*>(ws) + kNnErrBytes;
  tc_pack_kernel<<<140, 256, 0, s>>>(blob, wp);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  int dev = 0, nsm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return e;
  nsm = sm_budget(nsm);
  const int64_t ntiles = (n + TM - 1) / TM;
  auto kern = ntiles <= nsm ? mlp_tc_kernel<1> : mlp_tc_kernel<2>;
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kSmemBytes)) != cudaSuccess)
    return e;
  TcArgs a{obs, n, blob, wp, mu, init, conf, raw, static_cast<int*>(ws)};
  kern<<<(unsigned)(ntiles < nsm ? ntiles : nsm), kLaunch, kSmemBytes, s>>>(a);
  return cudaGetLastError();
}

}  // namespace nn
}  // namespace vfisv
