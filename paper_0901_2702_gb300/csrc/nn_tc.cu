// Training products of the initial-guess network (Sec. 5) on the fifth-generation
// tensor cores, two kernels a step.
//
// train_pass_kernel takes a tile of 128 samples through the whole forward and
// backward pass: features, the four layers, the loss, and the gradients with
// respect to every layer's pre-activations, leaving only the transposed
// activations and gradients (the operands of the weight gradients) in global
// memory.  A tile belongs to a cluster of two CTAs, each owning one half of
// every hidden layer's 256 columns: its MMAs (M = 128, N = 128, BF16 operands,
// FP32 accumulators) stream that half of the weights by 1D bulk copies
// through a four-slot ring, its 16 warps run the GELU epilogues of that half,
// and it sends its half of the next operand to its peer by a bulk copy between
// the two shared memories (the operand is double-buffered; a half arrives on
// the peer's mbarrier).  All three layers' pre-activations stay in tensor
// memory (384 of 512 columns) until the backward epilogues read them.  The
// transposed copies are read back from the operand by transposing matrix
// loads, so that a warp stores 128 contiguous bytes.  One launch a layer took
// 64 SMs, wrote and read pre-activations and both operand forms through L2 and
// paid launch, staging and tensor-memory set-up eight times a step.
//
// train_dw_kernel forms the weight gradients of all layers: a CTA computes a
// 128-row tile of A B^T over a range of the batch (split-K), and an FP32
// partial per split.
//
// Operand layout in global memory, "tiled canonical" TL(R, C) for an R x C
// BF16 matrix (R a multiple of 8, C of 64): K-chunks of 64 columns one after
// the other, inside a chunk 8-row groups of 1024 bytes, inside a group eight
// 128-byte core matrices along K, each 8 rows x 16 bytes.  A chunk of an
// operand tile is then one contiguous block whose shared-memory copy is the
// no-swizzle K-major layout of the MMA descriptors (leading-dimension byte
// offset 128, stride-dimension byte offset 1024).
//
// Every wait is bounded (about 1 s); on a timeout the kernels let the copies
// and tensor-core work they issued finish (bounded again), free their tensor
// memory, write kDevErrNnWait to the error word and return.
#include <cuda_bf16.h>
#include <stdint.h>

#include "common.cuh"
#include "nn.cuh"
#include "nn_device.cuh"
#include "nn_tc.cuh"
#include "tc_device.cuh"

namespace vfisv {
namespace nn {

namespace {

constexpr int TMR = 128;      // rows of a D tile (MMA M)
constexpr int KCH = 64;       // K per chunk
constexpr int kThreads = 512;  // 16 warps: 4 accumulator lane quarters x 4 column quarters

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, int cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(slot)),
               "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t tmem, int cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols)
               : "memory");
}
__device__ __forceinline__ void bar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

// ---------------------------------------------------------------------------
// forward and backward pass

constexpr int NH = HID / 2;                       // columns of a CTA
constexpr uint32_t kHalf = NH * KCH * 2;          // 16384: its rows of a weight chunk
constexpr uint32_t kOpChunk = TMR * KCH * 2;      // 16384: a K-chunk of the operand
constexpr uint32_t kOp = 4 * kOpChunk;            // the operand, 128 x 256
constexpr uint32_t kSend = 2 * kOpChunk;          // a CTA's half of it
constexpr int NSLOT = 4;
constexpr int KX = XT;                            // features padded to two K = 16 steps
constexpr int NY = YN;                            // outputs padded
// columns an epilogue takes at once, in a rolled loop: a CTA runs each layer's
// code once or thrice, so that unrolling it costs instruction fetches (a step
// of 8192 samples, 76 us when this was measured and 68 now, took 1 us more with
// 16, 4 more with 32)
constexpr int kEpc = 8;
constexpr int kPassLaunch = kThreads + 32;  // and a warp that loads the weights
constexpr int kStreamed = 18;  // weight chunks a tile: W0 1, W1 4, W2 4, W3^T 1, W2^T 4, W1^T 4

constexpr uint32_t PM_RING = 0;
constexpr uint32_t PM_H = PM_RING + NSLOT * kHalf;            // two operands
constexpr uint32_t PM_X = PM_H + 2 * kOp;                     // features [128][32]
constexpr uint32_t PM_DY = PM_X + TMR * KX * 2;               // output gradient [128][16]
constexpr uint32_t PM_W3 = PM_DY + TMR * NY * 2;              // W3, 16 x 256
constexpr uint32_t PM_BIAS = PM_W3 + NY * HID * 2;            // b0 | b1 | b2 | b3 (16)
constexpr uint32_t PM_STAT = PM_BIAS + (3 * HID + NY) * 4;    // in mean 24, std 24; out 10, 10
constexpr uint32_t PM_BAR = PM_STAT + 80 * 4;  // full[4] empty[4] half[2] W3 mma
constexpr uint32_t PM_TMEM = PM_BAR + 8 * (2 * NSLOT + 4);
constexpr uint32_t PM_END = PM_TMEM + 16;
constexpr size_t kPassSmem = PM_END + 1024;
static_assert(PM_BAR % 8 == 0 && kPassSmem <= 232448, "shared memory of the pass");
// tensor-memory columns: the layers' accumulators at 0, 128, 256; the output
// layer's, then the last and first input gradient's at 384; the middle one's
// over layer 2's, which nothing reads any more
constexpr uint32_t kColOut = 3 * NH;

__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

// barriers of the computing warps
__device__ __forceinline__ void compute_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");
}
__device__ __forceinline__ bool compute_sync_or(bool p) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n"
      " selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)p), "n"(kThreads)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}

// Four transposed 8 x 8 matrices: lane l gives the address of row l % 8 of
// matrix l / 8 and gets elements (column l / 4, rows 2 (l % 4), + 1) of each.
__device__ __forceinline__ void ldmatrix4_trans(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

// Transposed copy of `groups` 8-column groups of a 128-row K-major block in
// shared memory (8-row groups sbo bytes apart; group g at off(g)) into
// TL(R, M) at row group g0, columns from m0: four 8 x 8 blocks a warp at once.
template <class Off>
__device__ __forceinline__ void put_transposed(Off off, uint32_t sbo, int groups, uint8_t* dst,
                                               int R, int g0, int64_t m0, int warp, int lane) {
  __syncwarp();
  for (int t = warp; t < groups * 4; t += kThreads / 32) {
    const int g = t >> 2, mg = (t & 3) * 4;  // row groups mg .. mg + 3
    uint32_t r[4];
    ldmatrix4_trans(off(g) + (uint32_t)(mg + (lane >> 3)) * sbo + (uint32_t)(lane & 7) * 16, r);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int64_t m = m0 + 8 * (mg + e);
      uint8_t* p = dst + (size_t)(m >> 6) * (size_t)R * 128 + (size_t)(g0 + g) * 1024 +
                   (size_t)((m >> 3) & 7) * 128 + lane * 4;
      *reinterpret_cast<uint32_t*>(p) = r[e];
    }
  }
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPassLaunch, 1)
    train_pass_kernel(TrainPassArgs a) {
  extern __shared__ uint8_t smem_raw[];
  // (the same offset in both CTAs: dynamic shared memory starts alike)
  uint8_t* sm = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t sb = smem_u32(sm);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint32_t rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int64_t m0 = (int64_t)(blockIdx.x >> 1) * TMR;
  float* bias = reinterpret_cast<float*>(sm + PM_BIAS);
  float* stat = reinterpret_cast<float*>(sm + PM_STAT);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + PM_TMEM);
  const uint32_t bar_full = sb + PM_BAR, bar_empty = bar_full + 8 * NSLOT,
                 bar_half = bar_empty + 8 * NSLOT, bar_w3 = bar_half + 16, bar_mma = bar_w3 + 8;
  if (warp == 0) tmem_alloc(tmem_slot, 512);
  if (tid == 0) {
    for (int i = 0; i < 2 * NSLOT + 4; ++i) bar_init(bar_full + 8 * i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < 3 * HID; i += kPassLaunch) {
    const int l = i / HID;
    bias[i] = a.blob[(l == 0 ? OFF_B0 : l == 1 ? OFF_B1 : OFF_B2) + i % HID];
  }
  if (tid < NY) bias[3 * HID + tid] = tid < OUT ? a.blob[OFF_B3 + tid] : 0.0f;
  if (tid < IN) {
    stat[tid] = a.blob[OFF_INM + tid];
    stat[IN + tid] = a.blob[OFF_INS + tid];
  }
  if (tid < OUT - 1) {
    stat[48 + tid] = a.blob[OFF_OUTM + tid];
    stat[64 + tid] = a.blob[OFF_OUTS + tid];
  }
  tc_before_sync();
  __syncthreads();
  // the peer's barriers are initialised before anything is sent to it
  cluster_sync();
  tc_after_sync();
  const uint32_t tmem = *tmem_slot;

  if (warp == kThreads / 32) {
    // weight loads: their own warp, so that neither they wait for an issue nor
    // an issue for a slot
    if (lane == 0) {
      expect_tx(bar_w3, NY * HID * 2);
      bulk_load(sb + PM_W3, a.P.Wt[3], NY * HID * 2, bar_w3);
      int g = 0;
      for (; g < kStreamed; ++g) {
        const int slot = g % NSLOT;
        const uint8_t* src;
        if (g < 1) src = a.P.Wt[0];
        else if (g < 5) src = a.P.Wt[1] + (size_t)(g - 1) * 2 * kHalf;
        else if (g < 9) src = a.P.Wt[2] + (size_t)(g - 5) * 2 * kHalf;
        else if (g < 10) src = a.P.Wn[3];
        else if (g < 14) src = a.P.Wn[2] + (size_t)(g - 10) * 2 * kHalf;
        else src = a.P.Wn[1] + (size_t)(g - 14) * 2 * kHalf;
        if (g >= NSLOT && !mbar_wait(bar_empty + 8 * slot, (g / NSLOT - 1) & 1)) break;
        expect_tx(bar_full + 8 * slot, kHalf);
        bulk_load(sb + PM_RING + slot * kHalf, src + rank * kHalf, kHalf, bar_full + 8 * slot);
      }
      // the copies land, and of a whole stream the tensor cores' last arrivals
      // come, before the memory is released
      mbar_wait(bar_w3, 0);
      for (int i = g > NSLOT ? g - NSLOT : 0; i < g; ++i) {
        mbar_wait(bar_full + 8 * (i % NSLOT), (i / NSLOT) & 1);
        if (g == kStreamed) mbar_wait(bar_empty + 8 * (i % NSLOT), (i / NSLOT) & 1);
      }
      if (g < kStreamed) atomicExch(a.err, kDevErrNnWait);
    }
    __syncwarp();
    __syncthreads();
    cluster_sync();
    return;
  }

  // issuer state (thread 0): weight chunks consumed, arrivals from the peer,
  // halves sent to it, a sticky timeout flag
  int g_cons = 0, n_half = 0, n_sent = 0;
  bool ibad = false;
  constexpr uint32_t kIdescHalf = idesc_bf16(TMR, NH), kIdescOut = idesc_bf16(TMR, NY);
  // MMAs of the next weight chunk: `steps` K = 16 steps of the operand at A
  auto issue_chunk = [&](uint32_t d, uint32_t A, uint32_t sbo, int steps, bool first) {
    const int g = g_cons++, slot = g % NSLOT;
    if (ibad) return;
    if (!mbar_wait(bar_full + 8 * slot, (g / NSLOT) & 1)) {
      ibad = true;
      return;
    }
    for (int ks = 0; ks < steps; ++ks)
      mma_bf16(d, sdesc(A + ks * 256, 128, sbo),
               sdesc(sb + PM_RING + slot * kHalf + ks * 256, 128, 1024), kIdescHalf,
               !(first && ks == 0));
    mma_commit(bar_empty + 8 * slot);
  };
  // a product over the whole operand in buffer `buf`, whose other half comes
  // from the peer: own K-chunks first would change the order of the sum, so
  // the half is waited for before the first
  auto issue_full = [&](uint32_t d, int buf) {
    if (!ibad && !mbar_wait(bar_half + 8 * buf, (n_half >> 1) & 1)) ibad = true;
    ++n_half;
    tc_after_sync();
    for (int c = 0; c < 4; ++c)
      issue_chunk(d, sb + PM_H + buf * kOp + c * kOpChunk, 1024, 4, c == 0);
    mma_commit(bar_mma);
  };
  uint32_t mph = 0;
  auto sync_mma = [&]() -> bool {
    const bool ok = mbar_wait(bar_mma, mph);
    mph ^= 1;
    if (compute_sync_or(!ok || (tid == 0 && ibad))) return false;
    tc_after_sync();
    return true;
  };

  const int lq = warp & 3, cq = warp >> 2, row = 32 * lq + lane;
  const uint32_t tlane = tmem + ((uint32_t)(32 * lq) << 16);
  const int c0 = (int)rank * NH + 32 * cq;  // this warp's first column
  // columns c .. c + 7 of a new operand (BF16) into buffer `buf`
  auto put_operand = [&](const f2 (&h)[4], int buf, int c) {
    *reinterpret_cast<uint4*>(sm + PM_H + buf * kOp + (c >> 6) * kOpChunk + (row >> 3) * 1024 +
                              (row & 7) * 16 + ((c & 63) >> 3) * 128) =
        make_uint4(pack_bf16x2(f2_lo(h[0]), f2_hi(h[0])), pack_bf16x2(f2_lo(h[1]), f2_hi(h[1])),
                   pack_bf16x2(f2_lo(h[2]), f2_hi(h[2])), pack_bf16x2(f2_lo(h[3]), f2_hi(h[3])));
  };
  // accumulator column pair + bias
  auto z_pair = [&](float lo, float hi, const float* b) {
    const float2 bb = *reinterpret_cast<const float2*>(b);
    return f2_add(f2_pack(lo, hi), f2_pack(bb.x, bb.y));
  };
  // after an epilogue: the CTA's half is in buffer `buf`; sends it to the peer
  auto publish = [&](int buf, bool send) {
    fence_async_smem();
    tc_before_sync();
    compute_sync();
    if (send && tid == 0) {
      const uint32_t off = sb + PM_H + buf * kOp + rank * kSend, bar = bar_half + 8 * buf;
      expect_tx(bar, kSend);  // what the peer sends here
      ++n_sent;
      asm volatile(
          "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, "
          "[%3];" ::"r"(peer_addr(off, rank ^ 1u)),
          "r"(off), "r"(kSend), "r"(peer_addr(bar, rank ^ 1u))
          : "memory");
    }
  };
  // the transposed copy of the CTA's half of buffer `buf`
  auto copy_out = [&](int buf, uint8_t* dst) {
    const uint32_t base = sb + PM_H + buf * kOp + rank * kSend;
    put_transposed([&](int g) { return base + (uint32_t)(g >> 3) * kOpChunk + (uint32_t)(g & 7) * 128; },
                   1024, NH / 8, dst, HID, (int)rank * (NH / 8), m0, warp, lane);
  };

  bool ok = true;
  const int64_t m_row = m0 + (tid & (TMR - 1));
  const int64_t sample = m_row < a.rows ? sample_of(m_row, a.perm) : 0;
  float ic_row = 1.0f;
  do {
    // ---- features: thread (row, part) writes input columns 8 part .. 8 part + 7 ----
    {
      const int r = tid & (TMR - 1), part = tid >> 7;
      uint32_t pk[4] = {0u, 0u, 0u, 0u};
      if (m_row < a.rows) {
        const float* o = a.obs + sample * IN;
        ic_row = ic_of(o);
        if (part < IN / 8) {
          const float inv = 1.0f / ic_row;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int j = 8 * part + 2 * e;
            pk[e] = pack_bf16x2((o[j] * inv - stat[j]) / stat[IN + j],
                                (o[j + 1] * inv - stat[j + 1]) / stat[IN + j + 1]);
          }
        }
      }
      *reinterpret_cast<uint4*>(sm + PM_X + cm_off(r, 8 * part, (KX / 8) * 128)) =
          make_uint4(pk[0], pk[1], pk[2], pk[3]);
      fence_async_smem();
      tc_before_sync();
      compute_sync();
    }
    // ---- forward: layers 0 to 2 into accumulators 0 to 2 ----
#pragma unroll 1
    for (int l = 0; l < 3; ++l) {
      const uint32_t d = tmem + (uint32_t)(l * NH);
      if (tid == 0) {
        if (l == 0) {
          tc_after_sync();
          issue_chunk(d, sb + PM_X, (KX / 8) * 128, KX / 16, true);
          mma_commit(bar_mma);
        } else {
          issue_full(d, (l - 1) & 1);
        }
      }
      if (l == 0 && rank == 0)
        put_transposed([&](int g) { return sb + PM_X + (uint32_t)g * 128; }, (KX / 8) * 128, KX / 8,
                       a.XT, KX, 0, m0, warp, lane);
      if (l > 0) copy_out((l - 1) & 1, a.HT[l - 1]);
      if (!(ok = sync_mma())) break;
#pragma unroll 1
      for (int c = 0; c < 32; c += kEpc) {
        float v[kEpc];
        tmem_ld8(tlane + (uint32_t)(l * NH + 32 * cq + c), v);
        f2 h[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          h[j] = gelu2(z_pair(v[2 * j], v[2 * j + 1], bias + l * HID + c0 + c + 2 * j));
        put_operand(h, l & 1, c0 + c);
      }
      publish(l & 1, true);
    }
    if (!ok) break;
    // ---- output layer (both CTAs), loss and its gradient ----
    if (tid == 0) {
      if (!ibad && !mbar_wait(bar_half + 0, (n_half >> 1) & 1)) ibad = true;
      ++n_half;
      if (!ibad && !mbar_wait(bar_w3, 0)) ibad = true;
      tc_after_sync();
      if (!ibad)
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int ks = 0; ks < KCH / 16; ++ks)
            mma_bf16(tmem + kColOut, sdesc(sb + PM_H + c * kOpChunk + ks * 256, 128, 1024),
                     sdesc(sb + PM_W3 + c * (NY * KCH * 2) + ks * 256, 128, 1024), kIdescOut,
                     (c | ks) != 0);
      mma_commit(bar_mma);
    }
    copy_out(0, a.HT[2]);
    if (!(ok = sync_mma())) break;
    if (warp < 4) {
      float y[16], d[16], l = 0.0f;
      tmem_ld16(tlane + kColOut, y);
#pragma unroll
      for (int o = 0; o < 16; ++o) d[o] = 0.0f;
      if (m_row < a.rows) {
#pragma unroll
        for (int o = 0; o < OUT; ++o) y[o] = y[o] + bias[3 * HID + o];
        l = loss_row(y, a.params + sample * 10, ic_row, stat + 48, stat + 64, (float)a.rows, d);
      }
      if (rank == 0) a.loss[m_row] = l;
#pragma unroll
      for (int j = 0; j < 16; j += 8)
        *reinterpret_cast<uint4*>(sm + PM_DY + cm_off(tid, j, (NY / 8) * 128)) =
            make_uint4(pack_bf16x2(d[j], d[j + 1]), pack_bf16x2(d[j + 2], d[j + 3]),
                       pack_bf16x2(d[j + 4], d[j + 5]), pack_bf16x2(d[j + 6], d[j + 7]));
    }
    fence_async_smem();
    tc_before_sync();
    compute_sync();
    // ---- backward: the pre-activation gradients of layers 2 to 0 ----
#pragma unroll 1
    for (int l = 2; l >= 0; --l) {
      const uint32_t dcol = (l == 1) ? 2 * NH : kColOut;
      // operands: dY, then buffers 1 and 0 (layer 2's gradient, layer 1's)
      if (tid == 0) {
        if (l == 2) {
          tc_after_sync();
          issue_chunk(tmem + dcol, sb + PM_DY, (NY / 8) * 128, 1, true);
          mma_commit(bar_mma);
        } else {
          issue_full(tmem + dcol, l);
        }
      }
      if (l == 2) {
        if (rank == 0)
          put_transposed([&](int g) { return sb + PM_DY + (uint32_t)g * 128; }, (NY / 8) * 128,
                         NY / 8, a.dYT, NY, 0, m0, warp, lane);
      } else {
        copy_out(l, a.dZT[l + 1]);
      }
      if (!(ok = sync_mma())) break;
      // layer 2's gradient goes to buffer 1, layer 1's to 0, layer 0's to 1
      const int buf = (l == 1) ? 0 : 1;
#pragma unroll 1
      for (int c = 0; c < 32; c += kEpc) {
        float v[kEpc], z[kEpc];
        tmem_ld8(tlane + dcol + (uint32_t)(32 * cq + c), v);
        tmem_ld8(tlane + (uint32_t)(l * NH + 32 * cq + c), z);
        f2 h[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          h[j] = f2_mul(f2_pack(v[2 * j], v[2 * j + 1]),
                        gelu_grad2(z_pair(z[2 * j], z[2 * j + 1],
                                          bias + l * HID + c0 + c + 2 * j)));
        put_operand(h, buf, c0 + c);
      }
      publish(buf, l > 0);
      if (l == 0) copy_out(buf, a.dZT[0]);
    }
  } while (false);

  if (!ok && tid == 0) {
    // let the tensor-core work and the peer's copies in flight land before the
    // shared and tensor memory are released
    mbar_wait(bar_mma, mph ^ 1);
    for (; n_half < n_sent; ++n_half) mbar_wait(bar_half + 8 * (n_half & 1), (n_half >> 1) & 1);
    atomicExch(a.err, kDevErrNnWait);
  }
  tc_before_sync();
  __syncthreads();
  // neither CTA leaves while the other may still send to it
  cluster_sync();
  if (warp == 0) {
    tc_after_sync();
    tmem_free(tmem, 512);
  }
}

// ---------------------------------------------------------------------------
// weight gradients

constexpr int NSTAGE = 2;
constexpr uint32_t kAChunk = TMR * KCH * 2;             // 16384
constexpr uint32_t kDwStage = kAChunk + HID * KCH * 2;  // the widest B
constexpr uint32_t DM_BAR = NSTAGE * kDwStage;          // full[2] empty[2] mma
constexpr uint32_t DM_TMEM = DM_BAR + 8 * (2 * NSTAGE + 1) + 8;
constexpr size_t kDwSmem = DM_TMEM + 16 + 1024;

// P[128][N] = A B^T over K-chunks kc0 .. kc0 + nk - 1 of operands TL(HID, M)
// (row tile mt) and TL(N, M).  The bias gradient, the row sums of the
// gradient operand (A of layer 0, else B, which the first row tile's CTA
// sums), is taken from the chunks in shared memory while the tensor cores
// read them: warp w sums the 8-row groups w and w + 16; a group of a chunk is
// 64 segments of 16 bytes, segment j holding row j % 8, lane l takes segments
// l and l + 32, and the four lanes of a row combine at the end in a fixed
// order.  A slot is free when its MMAs and all 16 warps have read it.
template <int N, bool SUM_A>
__device__ __forceinline__ void dw_tile(const uint8_t* A, const uint8_t* B, float* P, float* bias,
                                        int mt, int kc0, int nk, uint8_t* sm, int* err) {
  constexpr uint32_t kBChunk = N * KCH * 2;
  constexpr int kGroups = (SUM_A ? TMR : N) / 8;
  const uint32_t sb = smem_u32(sm);
  const uint32_t bar_full = sb + DM_BAR, bar_empty = bar_full + 8 * NSTAGE,
                 bar_mma = bar_empty + 8 * NSTAGE;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t tmem = *reinterpret_cast<uint32_t*>(sm + DM_TMEM);
  const bool sums = SUM_A || mt == 0;
  bool bad = false;
  int loaded = 0, consumed = 0;
  auto load = [&](int i) {
    const int slot = i % NSTAGE, kc = kc0 + i;
    const uint32_t dst = sb + slot * kDwStage, bar = bar_full + 8 * slot;
    expect_tx(bar, kAChunk + kBChunk);
    bulk_load(dst, A + (size_t)kc * HID * (KCH * 2) + (size_t)mt * kAChunk, kAChunk, bar);
    bulk_load(dst + kAChunk, B + (size_t)kc * N * (KCH * 2), kBChunk, bar);
  };
  if (tid == 0)
    for (; loaded < NSTAGE && loaded < nk; ++loaded) load(loaded);
  constexpr uint32_t idesc = idesc_bf16(TMR, N);
  float acc[2] = {0.0f, 0.0f};
#pragma unroll 1
  for (int i = 0; i < nk; ++i) {
    const int slot = i % NSTAGE;
    if (!mbar_wait(bar_full + 8 * slot, (i / NSTAGE) & 1)) bad = true;
    if (__any_sync(0xffffffffu, bad)) break;
    if (tid == 0) {
      consumed = i + 1;
      tc_after_sync();
      const uint32_t sa = sb + slot * kDwStage, sbb = sa + kAChunk;
#pragma unroll
      for (int ks = 0; ks < KCH / 16; ++ks)
        mma_bf16(tmem, sdesc(sa + ks * 256, 128, 1024), sdesc(sbb + ks * 256, 128, 1024), idesc,
                 (i | ks) != 0);
      mma_commit(bar_empty + 8 * slot);
      // refill the other slot (this warp's own arrival on it came with chunk i - 1)
      const int gn = i - 1 + NSTAGE;
      if (i > 0 && gn < nk) {
        if (mbar_wait(bar_empty + 8 * (gn % NSTAGE), ((i - 1) / NSTAGE) & 1))
          load(loaded++);
        else
          bad = true;
      }
    }
    if (sums) {
      const uint8_t* blk = sm + slot * kDwStage + (SUM_A ? 0u : kAChunk);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int grp = warp + 16 * h;
        if (grp < kGroups) {
#pragma unroll
          for (int k2 = 0; k2 < 2; ++k2) {
            const uint4 q = *reinterpret_cast<const uint4*>(blk + grp * 1024 + 16 * (lane + 32 * k2));
            const __nv_bfloat162* e = reinterpret_cast<const __nv_bfloat162*>(&q);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const float2 f = __bfloat1622float2(e[k]);
              acc[h] += f.x + f.y;
            }
          }
        }
      }
    }
    __syncwarp();
    if (lane == 0)
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar_empty + 8 * slot)
                   : "memory");
  }
  if (tid == 0) mma_commit(bar_mma);  // tracks every MMA issued above
  const bool ok_mma = mbar_wait(bar_mma, 0);
  if (tid == 0 && ok_mma && !bad) {
    // the last arrivals on the slot barriers precede the exit
    for (int i = consumed > NSTAGE ? consumed - NSTAGE : 0; i < consumed; ++i)
      mbar_wait(bar_empty + 8 * (i % NSTAGE), (i / NSTAGE) & 1);
  }
  if (__syncthreads_or(!ok_mma || bad)) {
    if (tid == 0) {
      // let the copies issued but not consumed land before the memory is released
      for (int i = consumed; i < loaded; ++i) mbar_wait(bar_full + 8 * (i % NSTAGE), (i / NSTAGE) & 1);
      atomicExch(err, kDevErrNnWait);
    }
    return;
  }
  tc_after_sync();
  if (sums) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int grp = warp + 16 * h;
      if (grp < kGroups) {
        acc[h] += __shfl_xor_sync(0xffffffffu, acc[h], 8);
        acc[h] += __shfl_xor_sync(0xffffffffu, acc[h], 16);
        if (lane < 8) bias[(SUM_A ? mt * TMR : 0) + grp * 8 + lane] = acc[h];
      }
    }
    __syncwarp();
  }
  // warp w reads accumulator lanes 32 (w % 4) .. + 31 and, of 256 columns, the
  // quarter w / 4 (narrower tiles: the first four warps take all)
  const int lq = warp & 3, cq = warp >> 2;
  const int m = mt * TMR + 32 * lq + lane;
  const uint32_t lane_addr = tmem + ((uint32_t)(32 * lq) << 16);
  if (N < 256 && cq > 0) return;
  float* pp = P + (size_t)m * N + (N == 256 ? cq * 64 : 0);
  if constexpr (N == 16) {
    float v[16];
    tmem_ld16(lane_addr, v);
#pragma unroll
    for (int j = 0; j < 16; j += 4)
      *reinterpret_cast<float4*>(pp + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
  } else {
    // through the warp's 4 KB of the stages, free by now, so that a store
    // instruction writes four rows' 128 bytes (16-byte pieces of 32 rows cost
    // eight times the wavefronts: 16 steps of 8192 samples 1.20 -> 1.08 ms)
    float4* t = reinterpret_cast<float4*>(sm + warp * 4096);
    float* prow = P + (size_t)(mt * TMR + 32 * lq) * N + (N == 256 ? cq * 64 : 0);
#pragma unroll 1
    for (int c = 0; c < (N == 256 ? 64 : N); c += 32) {
      float v[32];
      tmem_ld32(lane_addr + (uint32_t)((N == 256 ? cq * 64 : 0) + c), v);
      __syncwarp();
#pragma unroll
      for (int j = 0; j < 8; ++j)
        t[lane * 8 + (j ^ (lane & 7))] =
            make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
      __syncwarp();
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int r = 4 * j + (lane >> 3);
        *reinterpret_cast<float4*>(prow + (size_t)r * N + c + 4 * (lane & 7)) =
            t[r * 8 + ((lane & 7) ^ (r & 7))];
      }
    }
  }
}

// blockIdx: row tile, split, layer.  The CTAs of the narrow output layer also
// add the loss of each 256 rows (one warp; the pairwise order of a block's
// tree).
__global__ void __launch_bounds__(kThreads, 2) train_dw_kernel(TrainDwArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t sb = smem_u32(sm);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + DM_TMEM);
  if (warp == 0) tmem_alloc(tmem_slot, 256);
  if (tid == 0) {
    for (int i = 0; i < 2 * NSTAGE + 1; ++i)
      bar_init(sb + DM_BAR + 8 * i,
               (i >= NSTAGE && i < 2 * NSTAGE) ? 1 + kThreads / 32 : 1);  // empty: MMAs + warps
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc_before_sync();
  __syncthreads();
  tc_after_sync();
  const uint32_t tmem = *tmem_slot;
  const int mt = blockIdx.x, split = blockIdx.y, l = blockIdx.z;
  const int kc0 = split * a.per;
  const int nk = min(a.per, a.chunks - kc0);
  if (l == 0) {
    dw_tile<32, true>(a.dZT[0], a.XT, a.wpart[0] + (size_t)split * HID * 32,
                      a.bpart[0] + (size_t)split * HID, mt, kc0, nk, sm, a.err);
  } else if (l == 3) {
    dw_tile<16, false>(a.HT[2], a.dYT, a.wpart[3] + (size_t)split * HID * NY,
                       a.bpart[3] + (size_t)split * NY, mt, kc0, nk, sm, a.err);
    for (int p = (split * (int)gridDim.x + mt) * (kThreads / 32) + warp; p < a.nloss;
         p += (int)(gridDim.x * gridDim.y) * (kThreads / 32)) {
      float r[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int64_t m = (int64_t)p * 256 + 32 * j + lane;
        r[j] = m < (int64_t)a.chunks * KCH ? a.loss[m] : 0.0f;
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j < o; ++j) r[j] += r[j + o];
      for (int o = 16; o > 0; o >>= 1) r[0] += __shfl_down_sync(0xffffffffu, r[0], o);
      if (lane == 0) a.lossp[p] = r[0];
    }
  } else {
    dw_tile<256, false>(a.HT[l - 1], a.dZT[l], a.wpart[l] + (size_t)split * HID * HID,
                        a.bpart[l] + (size_t)split * HID, mt, kc0, nk, sm, a.err);
  }
  tc_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc_after_sync();
    tmem_free(tmem, 256);
  }
}

}  // namespace

cudaError_t train_pass(const TrainPassArgs& a, int64_t tiles, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(train_pass_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPassSmem);
  if (e != cudaSuccess) return e;
  train_pass_kernel<<<(unsigned)(2 * tiles), kPassLaunch, kPassSmem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t train_dw(const TrainDwArgs& a, int splits, cudaStream_t s) {
  if (a.per < 1 || splits < 1 || (int64_t)splits * a.per < a.chunks ||
      (int64_t)(splits - 1) * a.per >= a.chunks)
    return cudaErrorInvalidValue;  // every split must own at least one K-chunk
  cudaError_t e = cudaFuncSetAttribute(train_dw_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDwSmem);
  if (e != cudaSuccess) return e;
  train_dw_kernel<<<dim3(HID / TMR, (unsigned)splits, 4), kThreads, kDwSmem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace nn
}  // namespace vfisv
