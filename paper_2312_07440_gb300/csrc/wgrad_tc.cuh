// Weight and bias gradients of the surrogate MLP's layers on the tensor cores:
//   dW_l [K][N] = sum over the batch rows r of H_{l-1}[r][k] dZ_l[r][n],
//   db_l [N]    = sum over r of dZ_l[r][n]      (BF16 operands, FP32 sums)
// for a run of layers in one launch.  The batch is the contraction, so both
// operands are taken as they lie in memory, row by row ("MN-major": 64 columns
// x 8 rows per 128-byte-swizzled atom), and no transposed copy is made.
//
// Work item: 128 rows of one dW_l (all N columns, one FP32 accumulator in
// tensor memory) over one slice of the batch; the partial sums of a slice lie
// in parts[slice][parameter] and are added in slice order afterwards, so the
// result is deterministic.  The items of all layers times the slices fill the
// SMs once: a batch of 16,384 rows of the 40 -> 4 x 256 network takes 7 items
// x 21 slices.  Bound by the operands' way from L2 (48 KB per 64 rows and
// item): 20 us, against 3 x 91 us for the hidden layers' slices on mma.sync
// with element-wise operand loads, 19 us for the input layer's and 41 us for
// the column sums.  Roles:
//   warp 0    TMA: 64 batch rows of the item's 128 H columns and N dZ columns
//             per stage, 4 stages;
//   warp 1    tensor memory and the MMAs (M = 128, N, K = 16);
//   warps 2-5 for a layer's first item the column sums of the staged dZ (two
//             columns per thread), then the accumulator to parts.
// Every wait is bounded as in gemm_tc.cuh.
#pragma once
#include "gemm_tc.cuh"

namespace tcg {
namespace wg {

constexpr int ROWS = 64;                                  // batch rows per stage
constexpr int STAGES = 4;
constexpr int MAX_RUN = 16;                               // layers of one launch
constexpr int THREADS = 64 + 128;
constexpr size_t BOX = (size_t)ROWS * 128;                // 64 rows x 64 columns (8 KB)
constexpr size_t STAGE_BYTES = (2 + MAX_N / 64) * BOX;    // 128 H columns, up to 256 dZ columns
constexpr size_t SMEM_BYTES = 1024 + STAGES * STAGE_BYTES + 256;
static_assert(SMEM_BYTES <= 232448, "more shared memory than a block may have");

struct Layer {
  CUtensorMap h, dz;  // [B][K] and [B][N], boxes of 64 columns x 64 rows
  long long w_off, b_off;
  int K;
  int item0;          // its first item
};

struct Args {
  Layer layer[MAX_RUN];
  int n_layers, n_items;
  int N, B, rows;     // rows: batch rows per slice, a multiple of ROWS
  float* parts;       // [slices][stride]
  long long stride;
  int* err;
};

// descriptor of an MN-major operand: atoms of 64 columns x 8 rows (1024
// bytes), the next 8 rows 1024 bytes on (stride offset), the next 64 columns
// one box on (leading offset), 128-byte swizzle
__device__ __forceinline__ uint64_t mn_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(BOX >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

__global__ void __launch_bounds__(THREADS, 1) k_wgrad_tc(const __grid_constant__ Args a) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + STAGES * STAGE_BYTES);
  const uint32_t b_full = smem_u32(bars), b_empty = smem_u32(bars + STAGES), b_acc = smem_u32(bars + 2 * STAGES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 1);
  __shared__ int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int item = blockIdx.x % a.n_items, slice = blockIdx.x / a.n_items;
  int li = 0;
  while (li + 1 < a.n_layers && item >= a.layer[li + 1].item0) ++li;
  const Layer& L = a.layer[li];
  const int m0 = (item - L.item0) * 128, N = a.N;
  const bool bias = m0 == 0;
  const int r0 = slice * a.rows, r1 = min(a.B, r0 + a.rows);
  const int blocks = max(0, (r1 - r0 + ROWS - 1) / ROWS);
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(b_full + 8 * s, 1);
      mbar_init(b_empty + 8 * s, bias ? 5 : 1);  // the MMAs, and the four summing warps
    }
    mbar_init(b_acc, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(MAX_N)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  volatile int* abort = &abort_flag;

  if (warp == 0) {
    if (lane == 0) {
      const int nb = N >> 6;
      int issued[STAGES] = {};
      for (int k = 0; k < blocks; ++k) {
        const int s = k % STAGES;
        if (!mbar_wait(b_empty + 8 * s, ((k / STAGES) & 1) ^ 1, a.err, 11, abort)) break;
        const uint32_t dst = smem_u32(base + s * STAGE_BYTES), bar = b_full + 8 * s;
        mbar_expect_tx(bar, (uint32_t)((2 + nb) * BOX));
        for (int c = 0; c < 2; ++c) tma_load_2d(dst + c * (uint32_t)BOX, &L.h, m0 + 64 * c, r0 + k * ROWS, bar);
        for (int c = 0; c < nb; ++c) tma_load_2d(dst + (2 + c) * (uint32_t)BOX, &L.dz, 64 * c, r0 + k * ROWS, bar);
        ++issued[s];
      }
      if (*abort) {  // loads still in flight land in shared memory: wait for them (bounded)
        const long long t0 = clock64();
        for (int s = 0; s < STAGES; ++s)
          while (issued[s] && !mbar_test(b_full + 8 * s, (uint32_t)((issued[s] - 1) & 1)) &&
                 clock64() - t0 < WAIT_CYCLES) {
          }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16(128, N) | (1u << 15) | (1u << 16);  // both operands MN-major
      for (int k = 0; k < blocks; ++k) {
        const int s = k % STAGES;
        if (!mbar_wait(b_full + 8 * s, (k / STAGES) & 1, a.err, 12, abort)) break;
        tc_fence_after();
        const uint32_t sa = smem_u32(base + s * STAGE_BYTES), sb = sa + 2 * (uint32_t)BOX;
#pragma unroll
        for (int i = 0; i < ROWS / 16; ++i)
          umma_bf16(tmem, mn_desc(sa + 2048 * i), mn_desc(sb + 2048 * i), idesc, (k | i) != 0);
        umma_commit(b_empty + 8 * s);
      }
      umma_commit(b_acc);  // every MMA issued so far has completed once this arrives
      const long long t0 = clock64();
      while (!mbar_test(b_acc, 0) && clock64() - t0 < WAIT_CYCLES) {
      }
    }
  } else {
    const int t = threadIdx.x - 64;
    float* out = a.parts + (long long)slice * a.stride;
    bool ok = true;
    if (bias) {
      float s0 = 0.0f, s1 = 0.0f;
      const int c = 2 * t;  // this thread's columns c, c + 1 of the staged dZ
      for (int k = 0; ok && k < blocks; ++k) {
        const int s = k % STAGES;
        ok = mbar_wait(b_full + 8 * s, (k / STAGES) & 1, a.err, 13, abort);
        if (ok && c < N) {
          const unsigned char* box = base + s * STAGE_BYTES + (2 + (c >> 6)) * BOX + (c & 7) * 2;
          const int ch = (c & 63) >> 3;
#pragma unroll 16
          for (int r = 0; r < ROWS; ++r) {
            const uint32_t v = *reinterpret_cast<const uint32_t*>(box + r * 128 + ((ch ^ (r & 7)) << 4));
            s0 += __uint_as_float(v << 16);
            s1 += __uint_as_float(v & 0xffff0000u);
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(b_empty + 8 * s);
      }
      if (ok && c < N) {
        out[L.b_off + c] = s0;
        out[L.b_off + c + 1] = s1;
      }
    }
    ok = mbar_wait(b_acc, 0, a.err, 14, abort) && ok;
    tc_fence_after();
    const int q = warp & 3, m = m0 + q * 32 + lane;  // warps 2..5 read lane quarters 2, 3, 0, 1
    if (ok)
      for (int c = 0; c < N; c += 16) {
        float v[16];
        tmem_ld16(tmem + (uint32_t)c + ((uint32_t)(q * 32) << 16), v);
        if (m < L.K) {
          float4* o = reinterpret_cast<float4*>(out + L.w_off + (long long)m * N + c);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            o[j] = blocks ? make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3])
                          : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
      }
    tc_fence_before();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(MAX_N) : "memory");
  }
}

}  // namespace wg
}  // namespace tcg
