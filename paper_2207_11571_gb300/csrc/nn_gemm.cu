// BF16 GEMM on the 5th-generation tensor cores (tcgen05) of sm_103a.
//
// One CTA computes a 128 x BN tile of C = A B^T.  Six warps:
//   warp 0 (one elected thread): TMA producer, 64-wide K slices of A and B into a
//          shared-memory ring (128-byte swizzle), mbarrier-tracked;
//   warp 1: allocates BN TMEM columns; one elected thread issues tcgen05.mma
//          (kind::f16, bf16 x bf16 -> f32, M = 128, N = BN, K = 16 per instruction)
//          and tcgen05.commit to free each stage and to signal the epilogue;
//   warps 2..5: epilogue, each reading its 32-lane quarter of the accumulator with
//          tcgen05.ld and applying the layer's epilogue before storing: bias and ReLU, the
//          loss and its gradient, the ReLU mask, with the bias gradient's column sums, so that
//          no element-wise launch stands between the products of a training step.
// An operand is read K-contiguous or, by the matrix descriptor's other major order, with its
// columns contiguous: the products of the backward pass need no transposed copies.
// Every mbarrier wait is bounded (about one second of SM clock); on expiry the thread
// sets the error flag, the pipeline drains with bounded waits, TMEM is released and the
// kernel returns.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <unordered_map>

#include "dg_common.h"
#include "nn_gemm.h"
#include "tc_common.cuh"

namespace dgnn {

using namespace tc;

namespace {

constexpr int kBM = 128;
constexpr int kBK = 64;               // 64 bf16 = 128 bytes = one swizzle span
constexpr int kBlk = kBK * kBK * 2;   // 8 KB: 64 K rows of 64 columns (operands with columns contiguous)
constexpr int kEpiWarps = 8;          // two per TMEM lane quarter, half of the tile's columns each
constexpr int kThreads = 64 + 32 * kEpiWarps;

template <int BN, int STAGES>
struct Smem {
  static constexpr int kABytes = kBM * kBK * 2;  // 16 KB
  static constexpr int kBBytes = BN * kBK * 2;
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kBarOffset = STAGES * kStageBytes;
  static constexpr int kBytes = kBarOffset + 256 + 1024;  // barriers, TMEM slot, alignment slack
};

// 32 consecutive FP32 accumulator columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float v[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// Sum over the warp's 32 lanes (rows) of each of 16 columns: lanes 2 c and 2 c + 1 return
// column c.  Halves of the columns are exchanged at each step (24 shuffles).  The order of
// the additions is fixed: rows r, r + 8, r + 16, r + 24, then r = 0 .. 7.
__device__ __forceinline__ float warp_column_sums(const float v[16], int lane) {
  float a[2][8], s[4], b[2][2], c[4], d[8];   // a: rows r, r + 16 (r < 16)
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const bool up = lane & 16;
    const float keep = up ? v[8 + i] : v[i], got = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[8 + i], 16);
    a[0][i] = up ? got : keep;
    a[1][i] = up ? keep : got;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool up = lane & 8;
    float lo[2], hi[2];   // rows r (+ 16), r + 8 (+ 16), r < 8
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float keep = up ? a[k][4 + i] : a[k][i];
      const float got = __shfl_xor_sync(0xffffffffu, up ? a[k][i] : a[k][4 + i], 8);
      lo[k] = up ? got : keep;
      hi[k] = up ? keep : got;
    }
    s[i] = ((lo[0] + hi[0]) + lo[1]) + hi[1];
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {   // b[k]: r % 4 + 4 k
    const bool up = lane & 4;
    const float keep = up ? s[2 + i] : s[i], got = __shfl_xor_sync(0xffffffffu, up ? s[i] : s[2 + i], 4);
    b[0][i] = up ? got : keep;
    b[1][i] = up ? keep : got;
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {   // c[2 k + h]: r % 2 + 2 h + 4 k
    const bool up = lane & 2;
    const float keep = up ? b[k][1] : b[k][0], got = __shfl_xor_sync(0xffffffffu, up ? b[k][0] : b[k][1], 2);
    c[2 * k] = up ? got : keep;
    c[2 * k + 1] = up ? keep : got;
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const bool up = lane & 1;
    const float got = __shfl_xor_sync(0xffffffffu, c[k], 1);
    d[2 * k] = up ? got : c[k];
    d[2 * k + 1] = up ? c[k] : got;
  }
  float t = d[0];
#pragma unroll
  for (int k = 1; k < 8; ++k) t += d[k];
  return t;
}

// 16 consecutive floats, as vectors where the address allows (vec); 0 past `left` of them.
__device__ __forceinline__ void load16(const float* p, bool vec, int left, float v[16]) {
  if (vec) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float4 a = reinterpret_cast<const float4*>(p)[i];
      v[4 * i] = a.x;
      v[4 * i + 1] = a.y;
      v[4 * i + 2] = a.z;
      v[4 * i + 3] = a.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = i < left ? p[i] : 0.f;
  }
}

// What the epilogue adds to, or applies to, 32 columns of a row, loaded while the products
// run: the bias, the ReLU mask (bit i: column i passes) or the scaled targets.
template <int KIND>
struct EpilogueData {
  float a[KIND == kGemmMaskBf16 ? 1 : 32];
  float t[KIND == kGemmLossBf16 ? 32 : 1];
  uint32_t mask = 0;
};

template <int KIND>
__device__ __forceinline__ void epilogue_load(const GemmEpilogue& ep, int m, int n, int N, bool live,
                                              EpilogueData<KIND>& d) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int nn = n + 16 * h;
    const bool full = nn + 16 <= N;   // library arrays are 256-byte aligned and nn a multiple of 16
    if (KIND == kGemmMaskBf16) {
      if (full && live) {   // 16 mask values in two 16-byte loads (ldm is a multiple of 8)
        const uint4* mp = reinterpret_cast<const uint4*>(ep.mask + (size_t)m * ep.ldm + nn);
        const uint4 lo = mp[0], hi = mp[1];
        const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const uint32_t b = (w[i / 2] >> (16 * (i % 2))) & 0xFFFFu;
          // bf16 > 0: sign bit clear and not +0
          if (b != 0u && (b & 0x8000u) == 0u) d.mask |= 1u << (16 * h + i);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (live && nn + i < N && __bfloat162float(ep.mask[(size_t)m * ep.ldm + nn + i]) > 0.f)
            d.mask |= 1u << (16 * h + i);
      }
    } else if (KIND == kGemmF32) {   // the caller's bias: any alignment
#pragma unroll
      for (int i = 0; i < 16; ++i) d.a[16 * h + i] = ep.bias && nn + i < N ? ep.bias[nn + i] : 0.f;
    } else {
      load16(ep.bias + nn, full, N - nn, d.a + 16 * h);
    }
    if (KIND == kGemmLossBf16) {
      float y[16], mean[16], sd[16];
      const long long src = live ? (ep.idx ? (long long)ep.idx[m] : m) : 0;
      load16(ep.Y + src * N + nn, full && N % 4 == 0 && (reinterpret_cast<size_t>(ep.Y) & 15) == 0, N - nn, y);
      load16(ep.mean + nn, full, N - nn, mean);
      load16(ep.sd + nn, full, N - nn, sd);
#pragma unroll
      for (int i = 0; i < 16; ++i) d.t[16 * h + i] = (y[i] - mean[i]) / sd[i];
    }
  }
}

// 16 columns nn.. (nn < N) of row m as bf16.
__device__ __forceinline__ void store_bf16_row(__nv_bfloat16* out, int nn, int N, const float* v) {
  if (nn + 16 <= N) {
    uint4 lo = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
    uint4 hi = make_uint4(pack_bf16(v[8], v[9]), pack_bf16(v[10], v[11]), pack_bf16(v[12], v[13]),
                          pack_bf16(v[14], v[15]));
    reinterpret_cast<uint4*>(out)[0] = lo;
    reinterpret_cast<uint4*>(out)[1] = hi;
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (nn + i < N) out[i] = __float2bfloat16_rn(v[i]);
  }
}

// Columns n .. n + 31 (n < N) of row m of the accumulator in v; live: m < M.  Every lane of
// the warp (32 consecutive rows) calls it.  Returns the row's squared errors (loss kind).
template <int KIND>
__device__ __forceinline__ float epilogue_store(const GemmEpilogue& ep, int m, int n, int N, bool live, int lane,
                                                const EpilogueData<KIND>& d, float v[32]) {
  float sq = 0.f;
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    if (KIND == kGemmMaskBf16) {
      v[i] = (d.mask >> i) & 1u ? v[i] : 0.f;
    } else if (KIND == kGemmLossBf16) {
      const float e = live && n + i < N ? (v[i] + d.a[i]) - d.t[i] : 0.f;
      v[i] = ep.grad_scale * e;
      sq += e * e;
    } else if (KIND == kGemmBiasReluBf16) {
      v[i] = fmaxf(v[i] + d.a[i], 0.f);
    } else {
      if (ep.bias) v[i] += d.a[i];
      if (ep.relu) v[i] = fmaxf(v[i], 0.f);
      if (KIND == kGemmAffineF32 && n + i < N) {
        if (ep.scale) v[i] *= ep.scale[n + i];
        if (ep.shift) v[i] += ep.shift[n + i];
      }
    }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int nn = n + 16 * h;
    if (nn >= N) break;
    if (KIND == kGemmMaskBf16 || KIND == kGemmLossBf16 || KIND == kGemmBiasReluBf16) {
      if (live) store_bf16_row(static_cast<__nv_bfloat16*>(ep.out) + (size_t)m * ep.ldo + nn, nn, N, v + 16 * h);
    }
    if (KIND == kGemmMaskBf16 || KIND == kGemmLossBf16) {
      const float s = warp_column_sums(v + 16 * h, lane);
      const int c = nn + (lane >> 1);
      if (!(lane & 1) && c < N) ep.colsum[(size_t)(m >> 5) * N + c] = s;
    }
    if ((KIND == kGemmF32 || KIND == kGemmAffineF32) && live) {
      float* out = static_cast<float*>(ep.out) + (size_t)m * ep.ldo + nn;
      if (nn + 16 <= N && ep.ldo % 4 == 0 && (reinterpret_cast<size_t>(ep.out) & 15) == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          reinterpret_cast<float4*>(out)[i] =
              make_float4(v[16 * h + 4 * i], v[16 * h + 4 * i + 1], v[16 * h + 4 * i + 2], v[16 * h + 4 * i + 3]);
      } else {
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (nn + i < N) out[i] = v[16 * h + i];
      }
    }
  }
  return sq;
}

// One 128 x BN tile at rows m0, columns n0 over the K slices [kb0, kb0 + KB).  A_MN, B_MN: the
// operand's rows run along K with its M (N) index contiguous; its tile arrives as 64-column
// blocks of 64 K rows.  These products are short (the layers of a training step at batch 1024
// take 4 to 8 K slices): launch, first loads and epilogue, not the tensor core, set their
// time, so barriers, TMEM and descriptors are set up ahead of the wait for the launch before.
// No operand is read ahead of it, weights neither: their last writer is two launches back, which
// only this launch's own wait makes visible (a step of 320-512x4-320 at batch 4096 with such
// reads 94.8 us, without 95.8, with them and the fences that would order them 100.9).
template <int BN, int STAGES, bool A_MN, bool B_MN, int KIND>
__device__ __forceinline__ void gemm_tile(const CUtensorMap* tmA, const CUtensorMap* tmB, int m0, int n0, int kb0,
                                          int KB, int M, int N, const GemmEpilogue& ep, int loss_slot,
                                          int* __restrict__ err_flag) {
  using S = Smem<BN, STAGES>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(base + S::kBarOffset);
  uint64_t* empty = full + STAGES;
  uint64_t* done = empty + STAGES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0), lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    prefetch_map(tmA);
    prefetch_map(tmB);
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, BN);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  auto load_a = [&](int kb, int s) {
    uint8_t* a = base + s * S::kStageBytes;
    const int k0 = (kb0 + kb) * kBK;
    if (A_MN) {
#pragma unroll
      for (int i = 0; i < kBM / kBK; ++i) tma_load_2d(a + i * kBlk, tmA, &full[s], m0 + i * kBK, k0);
    } else {
      tma_load_2d(a, tmA, &full[s], k0, m0);
    }
  };
  auto load_b = [&](int kb, int s) {
    uint8_t* b = base + s * S::kStageBytes + S::kABytes;
    const int k0 = (kb0 + kb) * kBK;
    if (B_MN) {
#pragma unroll
      for (int i = 0; i < BN / kBK; ++i) tma_load_2d(b + i * kBlk, tmB, &full[s], n0 + i * kBK, k0);
    } else {
      tma_load_2d(b, tmB, &full[s], k0, n0);
    }
  };

  auto enter = [] {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  };

  if (warp == 0) {
    enter();
    if (elect_one()) {
      int issued = 0, s = 0;
      uint32_t ph = 1;
      for (int kb = 0; kb < KB; ++kb) {
        if (!mbar_wait(&empty[s], ph)) {
          *(volatile int*)abort_flag = 1;
          atomicExch(err_flag, 1);
          break;
        }
        mbar_expect_tx(&full[s], S::kStageBytes);
        load_b(kb, s);
        load_a(kb, s);
        issued = kb + 1;
        if (++s == STAGES) {
          s = 0;
          ph ^= 1;
        }
      }
      // drain: every issued copy must land before the CTA exits (bounded)
      for (int kb = (issued > STAGES ? issued - STAGES : 0); kb < issued; ++kb)
        if (!mbar_wait(&full[kb % STAGES], (kb / STAGES) & 1)) atomicExch(err_flag, 2);
    }
  } else if (warp == 1) {
    enter();
    if (elect_one()) {
      constexpr uint32_t idesc = idesc_bf16(kBM, BN, A_MN, B_MN);
      // running stage and descriptors: what the issuing thread does besides adds to each slice
      constexpr uint32_t kStep = 32 >> 4, kStepMn = 2048 >> 4;   // 16 K values: 32 bytes of a row, 16 rows of 128 bytes
      const uint32_t a0 = smem_u32(base), b0 = a0 + S::kABytes;
      const uint64_t ad0 = A_MN ? sw128_desc_mn(a0, kBlk) : sw128_desc(a0);
      const uint64_t bd0 = B_MN ? sw128_desc_mn(b0, kBlk) : sw128_desc(b0);
      uint64_t ad = ad0, bd = bd0;
      int s = 0;
      uint32_t ph = 0, more = 0;
      for (int kb = 0; kb < KB; ++kb) {
        if (!mbar_wait(&full[s], ph)) {
          *(volatile int*)abort_flag = 1;
          atomicExch(err_flag, 3);
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int kk = 0; kk < kBK / 16; ++kk) {
          umma_bf16(tmem, ad + kk * (A_MN ? kStepMn : kStep), bd + kk * (B_MN ? kStepMn : kStep), idesc, more);
          more = 1;
        }
        umma_commit(&empty[s]);
        ad += S::kStageBytes >> 4;
        bd += S::kStageBytes >> 4;
        if (++s == STAGES) {
          s = 0;
          ph ^= 1;
          ad = ad0;
          bd = bd0;
        }
      }
      umma_commit(done);  // fires when every MMA issued above has completed
    }
    __syncwarp();
  } else {
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31, columns of its half of the tile
    const int quarter = warp % 4, half = (warp - 2) / 4;
    const int m = m0 + quarter * 32 + lane, c_begin = half * (BN / 2), c_end = c_begin + BN / 2;
    const bool rows = m0 + quarter * 32 < M;
    EpilogueData<KIND> data;
    enter();
    // after the wait, not ahead of it: this SM's L1 may hold lines of an earlier step
    if (rows && n0 + c_begin < N) epilogue_load<KIND>(ep, m, n0 + c_begin, N, m < M, data);
    const bool ok = mbar_wait(done, 0);
    if (!ok) {
      *(volatile int*)abort_flag = 1;
      atomicExch(err_flag, 4);
    }
    tc_fence_after();
    // tcgen05.ld is warp-collective: take the decision once per warp
    const bool run = __all_sync(0xffffffffu, ok && !*(volatile int*)abort_flag) && rows;
    float sq = 0.f;
    if (run) {
#pragma unroll 1
      for (int c0 = c_begin; c0 < c_end && n0 + c0 < N; c0 += 32) {
        float v[32];
        tmem_ld32(tmem + ((uint32_t)(quarter * 32) << 16) + c0, v);
        if (c0 > c_begin) {
          data.mask = 0;
          epilogue_load<KIND>(ep, m, n0 + c0, N, m < M, data);
        }
        sq += epilogue_store<KIND>(ep, m, n0 + c0, N, m < M, lane, data, v);
      }
    }
    if (KIND == kGemmLossBf16) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) sq += __shfl_down_sync(0xffffffffu, sq, off);
      if (lane == 0) ep.loss_part[loss_slot + warp - 2] = (double)sq;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, BN);
}

constexpr int kStages = 4;

template <int BN, int KIND>
__global__ void __launch_bounds__(kThreads, 1)
k_gemm_bf16(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int M, int N, int K,
            const __grid_constant__ GemmEpilogue ep, int* __restrict__ err_flag) {
  gemm_tile<BN, kStages, false, false, KIND>(
      &tmA, &tmB, blockIdx.x * kBM, blockIdx.y * BN, 0, (K + kBK - 1) / kBK, M, N, ep,
      (blockIdx.x * gridDim.y + blockIdx.y) * kEpiWarps, err_flag);
}

// Gradient of a layer's input: dx = dy W masked, with its column sums (dy K-major, W as it
// lies: its columns contiguous).  64-wide tiles: with 128 a training step at 4096 x 512 took
// 102.7 us instead of 99.1, at 1024 x 256 89.6 instead of 79.3.
constexpr int kBackBN = 64;
__global__ void __launch_bounds__(kThreads, 1)
k_input_gradient(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int M, int N, int K,
                 const __grid_constant__ GemmEpilogue ep, int* __restrict__ err_flag) {
  gemm_tile<kBackBN, kStages, false, true, kGemmMaskBf16>(&tmA, &tmB, blockIdx.x * kBM, blockIdx.y * kBackBN, 0,
                                                          (K + kBK - 1) / kBK, M, N, ep, 0, err_flag);
}

// Weight gradients of every layer in one launch: block -> (layer, M tile, N tile, split).  A
// launch of their own after the chain of input gradients: run beside it, layer by layer, a
// weight-gradient CTA with its long K loop outlived the chain's tiles (123.0 against 98.9 us
// per step at 4096 x 512, 86.2 against 79.4 at 1024 x 256).
constexpr int kGradBN = 128;
constexpr int kGradStages = 3;   // 96 KB: two CTAs per SM
struct GradTable {
  CUtensorMap G[kMaxGradLayers], A[kMaxGradLayers];
  int start[kMaxGradLayers + 1];   // first block of each layer
  int M[kMaxGradLayers], N[kMaxGradLayers], nt[kMaxGradLayers], tiles[kMaxGradLayers], splits[kMaxGradLayers];
  long long offset[kMaxGradLayers];
  int L, rows;
  float* out;
  long long split_stride;
};
__global__ void __launch_bounds__(kThreads, 2)
k_weight_gradients(const __grid_constant__ GradTable t, int* __restrict__ err_flag) {
  int l = 0;
  while (l + 1 < t.L && (int)blockIdx.x >= t.start[l + 1]) ++l;
  const int b = blockIdx.x - t.start[l], z = b / t.tiles[l], tile = b - z * t.tiles[l];
  const int mt = tile / t.nt[l], nt = tile - mt * t.nt[l];
  // this CTA's run of 64-row slices
  const int all = (t.rows + kBK - 1) / kBK;
  const int kb0 = (int)((long long)z * all / t.splits[l]);
  const int KB = (int)((long long)(z + 1) * all / t.splits[l]) - kb0;
  GemmEpilogue ep;
  ep.out = t.out + z * t.split_stride + t.offset[l];
  ep.ldo = t.N[l];
  gemm_tile<kGradBN, kGradStages, true, true, kGemmF32>(&t.G[l], &t.A[l], mt * kBM, nt * kGradBN, kb0, KB,
                                                        t.M[l], t.N[l], ep, 0, err_flag);
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

}  // namespace

// A tensor map only encodes an address, a shape, strides and a box, so maps are cached
// on exactly those: a repeated GEMM (every layer of every training step and RK stage)
// skips the driver encode.
struct MapKey {
  uintptr_t ptr;
  long long rows, cols, ld;
  int box_rows;
  bool operator==(const MapKey& o) const {
    return ptr == o.ptr && rows == o.rows && cols == o.cols && ld == o.ld && box_rows == o.box_rows;
  }
};
struct MapKeyHash {
  size_t operator()(const MapKey& k) const {
    size_t h = std::hash<uintptr_t>()(k.ptr);
    for (long long v : {k.rows, k.cols, k.ld, (long long)k.box_rows}) h = h * 1000003u ^ std::hash<long long>()(v);
    return h;
  }
};
std::mutex g_map_mu;
std::unordered_map<MapKey, CUtensorMap, MapKeyHash> g_map_cache;
constexpr size_t kMapCacheMax = 4096;

int encode_map(CUtensorMap* map, const __nv_bfloat16* ptr, long long rows, long long cols, long long ld,
               int box_rows);

int make_map(CUtensorMap* map, const __nv_bfloat16* ptr, long long rows, long long cols, long long ld, int box_rows) {
  const MapKey key{reinterpret_cast<uintptr_t>(ptr), rows, cols, ld, box_rows};
  {
    std::lock_guard<std::mutex> lock(g_map_mu);
    auto it = g_map_cache.find(key);
    if (it != g_map_cache.end()) {
      *map = it->second;
      return DG_OK;
    }
  }
  int rc = encode_map(map, ptr, rows, cols, ld, box_rows);
  if (rc) return rc;
  std::lock_guard<std::mutex> lock(g_map_mu);
  if (g_map_cache.size() >= kMapCacheMax) g_map_cache.clear();
  g_map_cache.emplace(key, *map);
  return DG_OK;
}

int encode_map(CUtensorMap* map, const __nv_bfloat16* ptr, long long rows, long long cols, long long ld,
               int box_rows) {
  auto fn = encode_fn();
  if (!fn) return fail(DG_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
  if ((reinterpret_cast<uintptr_t>(ptr) & 15) || (ld % 8)) return fail(DG_ERR_INVALID_ARG, "GEMM operand misaligned");
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)(ld * 2)};
  cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(ptr), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(DG_ERR_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
  return DG_OK;
}

namespace {

cudaLaunchConfig_t chain_config(dim3 grid, int smem, cudaStream_t st, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

template <int BN, int KIND>
int launch_gemm(const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, int M, int N, int K,
                const GemmEpilogue& ep, int* err, cudaStream_t st) {
  CUtensorMap ma, mb;
  int rc = make_map(&ma, A, M, K, lda, kBM);
  if (rc) return rc;
  rc = make_map(&mb, B, N, K, ldb, BN);
  if (rc) return rc;
  auto kern = k_gemm_bf16<BN, KIND>;
  const int smem = Smem<BN, kStages>::kBytes;
  static bool configured = false;
  if (!configured) {
    DG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    configured = true;
  }
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = chain_config(dim3((M + kBM - 1) / kBM, (N + BN - 1) / BN), smem, st, attr);
  DG_CUDA(cudaLaunchKernelEx(&cfg, kern, ma, mb, M, N, K, ep, err));
  return DG_OK;
}

// Tile width: enough CTAs to cover the SMs when possible, wider tiles otherwise.
int pick_bn(int M, int N) {
  const int mt = (M + kBM - 1) / kBM;
  if (N > 128 && mt * ((N + 255) / 256) >= kSMs) return 256;
  if (N > 64 && mt * ((N + 127) / 128) >= kSMs) return 128;
  return 64;
}

template <int KIND>
int launch_gemm_bn(const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, int M, int N, int K,
                   const GemmEpilogue& ep, int* err, cudaStream_t st) {
  switch (pick_bn(M, N)) {
    case 256: return launch_gemm<256, KIND>(A, lda, B, ldb, M, N, K, ep, err, st);
    case 128: return launch_gemm<128, KIND>(A, lda, B, ldb, M, N, K, ep, err, st);
    default: return launch_gemm<64, KIND>(A, lda, B, ldb, M, N, K, ep, err, st);
  }
}

}  // namespace

int gemm_loss_partials(int M, int N) {
  const int bn = pick_bn(M, N);
  return kEpiWarps * ((M + kBM - 1) / kBM) * ((N + bn - 1) / bn);
}

int gemm_bf16(const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, int M, int N, int K,
              const GemmEpilogue& ep, int* err_flag, cudaStream_t st) {
  if (M <= 0 || N <= 0 || K <= 0) return fail(DG_ERR_INVALID_ARG, "gemm: empty problem");
  if (!ep.out || ep.ldo < N) return fail(DG_ERR_INVALID_ARG, "gemm: bad output");
  if (ep.kind != kGemmF32 && !ep.bias) return fail(DG_ERR_INVALID_ARG, "gemm: bias missing");
  const bool half_out = ep.kind == kGemmBiasReluBf16 || ep.kind == kGemmLossBf16;
  if (half_out && (ep.ldo % 8)) return fail(DG_ERR_INVALID_ARG, "gemm: bf16 output ld % 8");
  if (ep.kind == kGemmLossBf16 && (!ep.Y || !ep.mean || !ep.sd || !ep.colsum || !ep.loss_part))
    return fail(DG_ERR_INVALID_ARG, "gemm: loss operands missing");
  switch (ep.kind) {
    case kGemmBiasReluBf16: return launch_gemm_bn<kGemmBiasReluBf16>(A, lda, B, ldb, M, N, K, ep, err_flag, st);
    case kGemmAffineF32: return launch_gemm_bn<kGemmAffineF32>(A, lda, B, ldb, M, N, K, ep, err_flag, st);
    case kGemmF32: return launch_gemm_bn<kGemmF32>(A, lda, B, ldb, M, N, K, ep, err_flag, st);
    case kGemmLossBf16: return launch_gemm_bn<kGemmLossBf16>(A, lda, B, ldb, M, N, K, ep, err_flag, st);
  }
  return fail(DG_ERR_INVALID_ARG, "gemm: unknown epilogue");
}


int input_gradient(const __nv_bfloat16* dy, int ldy, const __nv_bfloat16* W, int ldw, int rows, int in, int o,
                   const __nv_bfloat16* act, int lda, __nv_bfloat16* dx, float* colsum, int* err_flag,
                   cudaStream_t st) {
  if (rows < 1 || in < 1 || o < 1 || lda % 8) return fail(DG_ERR_INVALID_ARG, "input gradient: bad sizes");
  CUtensorMap ma, mb;
  int rc = make_map(&ma, dy, rows, o, ldy, kBM);
  if (!rc) rc = make_map(&mb, W, o, in, ldw, kBK);
  if (rc) return rc;
  GemmEpilogue ep;
  ep.kind = kGemmMaskBf16;
  ep.mask = act;
  ep.ldm = lda;
  ep.out = dx;
  ep.ldo = lda;
  ep.colsum = colsum;
  const int smem = Smem<kBackBN, kStages>::kBytes;
  static bool configured = false;
  if (!configured) {
    DG_CUDA(cudaFuncSetAttribute(k_input_gradient, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    configured = true;
  }
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = chain_config(dim3((rows + kBM - 1) / kBM, (in + kBackBN - 1) / kBackBN), smem, st, attr);
  DG_CUDA(cudaLaunchKernelEx(&cfg, k_input_gradient, ma, mb, rows, in, o, ep, err_flag));
  return DG_OK;
}

// Runs of rows of one layer's gradient.  A gradient is the sum of its runs' products in order,
// so the count is part of the result: the CTAs that a layer's own product would need to cover
// the SMs.  (Any other order is as accurate, but a weight whose bf16 copy then rounds the
// other way moves the next step's gradients by up to half a percent.)
int grad_splits(int M, int N, int rows) {
  const int bn = pick_bn(M, N), tiles = ((M + kBM - 1) / kBM) * ((N + bn - 1) / bn);
  return std::max(1, std::min({kMaxSplits, (rows + kBK - 1) / kBK, kSMs / tiles}));
}

int weight_gradients(const GradLayer* layers, int L, int rows, float* out, long long split_stride, int* err_flag,
                     cudaStream_t st) {
  if (L < 1 || L > kMaxGradLayers || rows < 1) return fail(DG_ERR_INVALID_ARG, "weight gradients: bad sizes");
  GradTable t;
  std::memset(&t, 0, sizeof(t));
  int blocks = 0;
  for (int l = 0; l < L; ++l) {
    const GradLayer& g = layers[l];
    int rc = make_map(&t.G[l], g.G, rows, g.M, g.ldg, kBK);
    if (!rc) rc = make_map(&t.A[l], g.A, rows, g.N, g.lda, kBK);
    if (rc) return rc;
    t.start[l] = blocks;
    t.tiles[l] = ((g.M + kBM - 1) / kBM) * ((g.N + kGradBN - 1) / kGradBN);
    t.splits[l] = grad_splits(g.M, g.N, rows);
    blocks += t.tiles[l] * t.splits[l];
    t.M[l] = g.M;
    t.N[l] = g.N;
    t.nt[l] = (g.N + kGradBN - 1) / kGradBN;
    t.offset[l] = g.offset;
  }
  t.start[L] = blocks;
  t.L = L;
  t.rows = rows;
  t.out = out;
  t.split_stride = split_stride;
  const int smem = Smem<kGradBN, kGradStages>::kBytes;
  static bool configured = false;
  if (!configured) {
    DG_CUDA(cudaFuncSetAttribute(k_weight_gradients, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    configured = true;
  }
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = chain_config(dim3(blocks), smem, st, attr);
  DG_CUDA(cudaLaunchKernelEx(&cfg, k_weight_gradients, t, err_flag));
  return DG_OK;
}

}  // namespace dgnn
