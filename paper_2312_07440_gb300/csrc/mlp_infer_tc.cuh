// The surrogate MLP's whole inference in one persistent kernel on the
// 5th-generation tensor cores: features x [M][n_in] (FP32) -> input layer ->
// hidden layers -> output layer out [M][2], with every activation kept in
// shared memory (nothing but x and out touches HBM).
//
//   layer 0  z = x W_0 + b_0 with x and W_0 split into BF16 pairs
//            (x = x_h + x_l, W = W_h + W_l, each part rounded to nearest):
//            one MMA over K = 3 n_in of [x_h | x_l | x_h] against
//            [W_h ; W_h ; W_l] gives x_h W_h + x_l W_h + x_h W_l, i.e. the
//            FP32 product up to the dropped x_l W_l (~2^-16 relative) and
//            FP32 accumulation;
//   layer l  z = h W_l + b_l (BF16 h and W_l, FP32 accumulation), for
//            l = 1 .. L-1, h = bf16(SiLU(z)) of the layer before;
//   output   out = SiLU(z_{L-1}) W_out + b_out in FP32 from the last
//            accumulator (the activation of the last layer is not rounded).
//
// One CTA per SM walks pairs of 128-row tiles.  The two tiles of a pair
// alternate on the tensor core layer by layer, so the epilogue of one tile
// (tensor memory -> bias, SiLU -> BF16 into its shared-memory activation
// buffer, the next layer's A operand) runs while the MMAs of the other tile
// run.  Roles:
//   warp 0     one thread streams the packed weights through a ring of
//              WSTAGES k-blocks ([256 n][64 k] BF16, 128-byte swizzle, TMA
//              from L2: every CTA reads the same 448 KB);
//   warp 1     owns 512 tensor-memory columns (one 128 x 256 FP32
//              accumulator per tile slot); one thread issues tcgen05.mma
//              (M = 128, N = 256, K = 16) and commits each weight k-block to
//              its ring slot and each layer to the slot's "full" barrier;
//   warps 2-17 the epilogue, four per lane quarter and one 64-column quarter
//              (one k-block of the next layer's A operand) each; they also
//              compute the output layer (the column quarters' partial sums
//              meet in the slot's free activation k-blocks; the last warp to
//              arrive adds them in a fixed order);
//   warps 18-19 the split features of each new tile: loaded while the previous
//              tile is computed, written into its slot as soon as that tile's
//              last MMAs have read it, beside the output layer (written by the
//              epilogue warps after it, they doubled that layer's epilogue,
//              3.2k -> 7k cycles).
// Every wait is bounded (~2^31 cycles): on a timeout the error flag is set,
// every role stops, the MMA thread drains its MMAs, the TMA thread waits for
// its loads in flight, and the tensor memory is freed before the kernel
// returns.
#pragma once
#include "gemm_tc.cuh"

namespace tcg {
namespace inf {

constexpr int N = 256;                               // hidden width
constexpr int WSTAGES = 3;                           // weight ring depth
constexpr int MAX_LAYERS = 8;                        // input layer + hidden layers
constexpr int MAX_IN = 40;                           // 3 n_in <= 128: the split input fits two k-blocks
constexpr int FEATURE_WARP = 2 + EPI_WARPS;          // the first of two
constexpr int THREADS = 32 * (FEATURE_WARP + 2);
constexpr int KB_HIDDEN = N / BK;                    // k-blocks of a hidden layer
constexpr size_t KB_BYTES = (size_t)BM * 128;        // one k-block of a tile's activations (16 KB)
constexpr size_t ACT_BYTES = KB_HIDDEN * KB_BYTES;   // a tile's activations (64 KB)
constexpr size_t WBOX_BYTES = (size_t)N * 128;       // one weight k-block (32 KB)
constexpr size_t SMEM_BYTES = 1024 + 2 * ACT_BYTES + WSTAGES * WBOX_BYTES + 256;
static_assert(SMEM_BYTES <= 232448, "more shared memory than a block may have");

}  // namespace inf

struct InferArgs {
  const float* x;                       // [M][n_in] features (FP32)
  const float* bias[inf::MAX_LAYERS];   // [256] per layer (layer 0 the input layer)
  const float* w_out;                   // [256][2]
  const float* b_out;                   // [2]
  float* out;                           // [M][2]
  int* err;                             // set to a nonzero code when a wait gives up
  long long M;
  int n_in;                             // a multiple of 8, <= MAX_IN
  int kb0;                              // k-blocks of the split input layer: ceil(3 n_in / 64)
  int L;                                // layers before the output layer (input + hidden)
};

// byte offset of the BF16 pair at column c (even) of row r in a tile's
// activations: k-block c / 64, each row 128 bytes, its 16-byte chunks
// permuted by the 128-byte swizzle (chunk ^ row % 8) that TMA and the MMA
// descriptors use
__device__ __forceinline__ uint32_t act_off(int r, int c) {
  const int w = c & 63;
  return (uint32_t)((c >> 6) * inf::KB_BYTES + r * 128 + ((((w >> 3) ^ r) & 7) << 4) + ((w & 7) << 1));
}

// the features of one row, as quadruples
struct Features {
  float4 v[inf::MAX_IN / 4];
};

__device__ __forceinline__ void load_features(const InferArgs& a, long long row, bool aligned, Features& f) {
  const bool live = row < a.M;
  const float* xr = a.x + (live ? row : 0) * a.n_in;
#pragma unroll
  for (int i = 0; i < inf::MAX_IN / 4; ++i) {
    if (!live || 4 * i >= a.n_in)
      f.v[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    else if (aligned)
      f.v[i] = __ldg(reinterpret_cast<const float4*>(xr) + i);
    else
      f.v[i] = make_float4(__ldg(xr + 4 * i), __ldg(xr + 4 * i + 1), __ldg(xr + 4 * i + 2), __ldg(xr + 4 * i + 3));
  }
}

// columns [0, n) x_h, [n, 2n) x_l, [2n, 3n) x_h, [3n, 64 kb0) zero, in
// 16-byte chunks of 8 columns
__device__ __forceinline__ void store_features(unsigned char* act, const InferArgs& a, int r, const Features& f) {
  const int n = a.n_in;
#pragma unroll
  for (int i = 0; i < inf::MAX_IN / 8; ++i) {
    if (8 * i >= n) break;
    const float x[8] = {f.v[2 * i].x,     f.v[2 * i].y,     f.v[2 * i].z,     f.v[2 * i].w,
                        f.v[2 * i + 1].x, f.v[2 * i + 1].y, f.v[2 * i + 1].z, f.v[2 * i + 1].w};
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float h0 = __bfloat162float(__float2bfloat16_rn(x[2 * j])), h1 = __bfloat162float(__float2bfloat16_rn(x[2 * j + 1]));
      hi[j] = bf16x2(h0, h1);
      lo[j] = bf16x2(x[2 * j] - h0, x[2 * j + 1] - h1);
    }
    const uint4 h = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(act + act_off(r, 8 * i)) = h;
    *reinterpret_cast<uint4*>(act + act_off(r, n + 8 * i)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    *reinterpret_cast<uint4*>(act + act_off(r, 2 * n + 8 * i)) = h;
  }
  for (int c = 3 * n; c < 64 * a.kb0; c += 8)
    *reinterpret_cast<uint4*>(act + act_off(r, c)) = make_uint4(0u, 0u, 0u, 0u);
}

__global__ void __launch_bounds__(inf::THREADS, 1) k_mlp_infer(const __grid_constant__ CUtensorMap tmW, const InferArgs a) {
  using namespace inf;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* act = base;                      // [2 slots][4 k-blocks][128 rows][128 B]
  unsigned char* wring = base + 2 * ACT_BYTES;    // [WSTAGES][256 rows][128 B]
  uint64_t* bars = reinterpret_cast<uint64_t*>(wring + WSTAGES * WBOX_BYTES);
  // barrier slots: wfull[WSTAGES], wempty[WSTAGES], ready[2], full[2], drain, features[2],
  // free[2] (the slot's tile has been read by its last MMAs)
  const uint32_t b_wfull = smem_u32(bars), b_wempty = smem_u32(bars + WSTAGES);
  const uint32_t b_ready = smem_u32(bars + 2 * WSTAGES), b_full = smem_u32(bars + 2 * WSTAGES + 2);
  const uint32_t b_drain = smem_u32(bars + 2 * WSTAGES + 4);
  const uint32_t b_feat = smem_u32(bars + 2 * WSTAGES + 5);
  const uint32_t b_free = smem_u32(bars + 2 * WSTAGES + 7);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * WSTAGES + 9);
  __shared__ int abort_flag;
  __shared__ int head_count[8];  // [slot][lane quarter]: column quarters done

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long tiles = (a.M + BM - 1) / BM, pairs = (tiles + 1) / 2;
  const uint32_t tmem_cols = 2 * N;

  if (threadIdx.x < 8) head_count[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < WSTAGES; ++s) {
      mbar_init(b_wfull + 8 * s, 1);
      mbar_init(b_wempty + 8 * s, 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(b_ready + 8 * s, EPI_WARPS);  // one arrival per epilogue warp
      mbar_init(b_full + 8 * s, 1);
      mbar_init(b_feat + 8 * s, 2);
      mbar_init(b_free + 8 * s, 1);
    }
    mbar_init(b_drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(tmem_cols)
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
      int stage = 0;
      uint32_t phase = 0;
      int issued[WSTAGES] = {};
      for (long long P = blockIdx.x; P < pairs; P += gridDim.x) {
        const int ns = 2 * P + 1 < tiles ? 2 : 1;
        int kbg = 0;
        for (int l = 0; l < a.L; ++l) {
          const int KB = l == 0 ? a.kb0 : KB_HIDDEN;
          for (int s = 0; s < ns; ++s)
            for (int kb = 0; kb < KB; ++kb) {
              if (!mbar_wait(b_wempty + 8 * stage, phase ^ 1, a.err, 11, abort)) goto tma_done;
              mbar_expect_tx(b_wfull + 8 * stage, (uint32_t)WBOX_BYTES);
              tma_load_2d(smem_u32(wring + (size_t)stage * WBOX_BYTES), &tmW, 0, (kbg + kb) * N, b_wfull + 8 * stage);
              ++issued[stage];
              if (++stage == WSTAGES) {
                stage = 0;
                phase ^= 1;
              }
            }
          kbg += KB;
        }
      }
    tma_done:
      if (*abort) {
        // loads still in flight land in shared memory: wait for them (bounded)
        const long long t0 = clock64();
        for (int s = 0; s < WSTAGES; ++s) {
          if (issued[s] == 0) continue;
          const uint32_t par = (uint32_t)((issued[s] - 1) & 1);
          while (!mbar_test(b_wfull + 8 * s, par) && clock64() - t0 < WAIT_CYCLES) {
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16(BM, N);
      int stage = 0;
      uint32_t phase = 0, ready_ph = 0, feat_ph = 0;  // bit s: the parity slot s waits for next
      bool ok = true;
      for (long long P = blockIdx.x; ok && P < pairs; P += gridDim.x) {
        const int ns = 2 * P + 1 < tiles ? 2 : 1;
        for (int l = 0; ok && l < a.L; ++l) {
          const int KB = l == 0 ? a.kb0 : KB_HIDDEN;
          for (int s = 0; ok && s < ns; ++s) {
            if (!(ok = mbar_wait(b_ready + 8 * s, (ready_ph >> s) & 1u, a.err, 12, abort))) break;
            ready_ph ^= 1u << s;
            if (l == 0) {
              if (!(ok = mbar_wait(b_feat + 8 * s, (feat_ph >> s) & 1u, a.err, 15, abort))) break;
              feat_ph ^= 1u << s;
            }
            tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(s * N);
            const uint32_t a_base = smem_u32(act + (size_t)s * ACT_BYTES);
            for (int kb = 0; kb < KB; ++kb) {
              if (!(ok = mbar_wait(b_wfull + 8 * stage, phase, a.err, 13, abort))) break;
              tc_fence_after();
              const uint32_t a0 = a_base + (uint32_t)(kb * KB_BYTES);
              const uint32_t b0 = smem_u32(wring + (size_t)stage * WBOX_BYTES);
#pragma unroll
              for (int k = 0; k < BK / UMMA_K; ++k)
                umma_bf16(d, sw128_desc(a0 + 32 * k), sw128_desc(b0 + 32 * k), idesc, (kb | k) != 0);
              umma_commit(b_wempty + 8 * stage);  // the ring slot is free once these MMAs have read it
              if (++stage == WSTAGES) {
                stage = 0;
                phase ^= 1;
              }
            }
            if (ok) umma_commit(b_full + 8 * s);
            if (ok && l == a.L - 1) umma_commit(b_free + 8 * s);
          }
        }
      }
      // every MMA issued so far has completed once this commit arrives
      umma_commit(b_drain);
      const long long t0 = clock64();
      while (!mbar_test(b_drain, 0) && clock64() - t0 < WAIT_CYCLES) {
      }
    }
  } else if (warp >= FEATURE_WARP) {
    const int t = threadIdx.x - 32 * FEATURE_WARP;  // rows t and t + 64
    const bool aligned = (reinterpret_cast<uintptr_t>(a.x) & 15) == 0;
    uint32_t free_ph = 0;  // bit s: the parity slot s waits for next
    bool ok = true;
    Features f;
    auto put = [&](int s, long long tile, bool loaded) {
      unsigned char* as = act + (size_t)s * ACT_BYTES;
      if (!loaded) load_features(a, tile * BM + t, aligned, f);
      store_features(as, a, t, f);
      load_features(a, tile * BM + t + 64, aligned, f);
      store_features(as, a, t + 64, f);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // visible to the MMAs (async proxy)
      __syncwarp();
      if (lane == 0) mbar_arrive(b_feat + 8 * s);
    };
    if ((long long)blockIdx.x < pairs)
      for (int s = 0; s < 2 && 2 * (long long)blockIdx.x + s < tiles; ++s) put(s, 2 * (long long)blockIdx.x + s, false);
    for (long long P = blockIdx.x; ok && P < pairs; P += gridDim.x) {
      const int ns = 2 * P + 1 < tiles ? 2 : 1;
      const long long Pn = P + gridDim.x;
      for (int s = 0; s < ns; ++s) {
        if (Pn >= pairs || 2 * Pn + s >= tiles) continue;  // no next tile for this slot
        const long long row = (2 * Pn + s) * BM + t;
        load_features(a, row, aligned, f);  // in flight during the wait
        if (row + 64 < a.M) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.x + (row + 64) * a.n_in));
        if (!(ok = mbar_wait(b_free + 8 * s, (free_ph >> s) & 1u, a.err, 16, abort))) break;
        free_ph ^= 1u << s;
        put(s, 2 * Pn + s, true);
      }
    }
  } else {
    const int q = warp & 3;           // the lane quarter this warp may read
    const int cq = (warp - 2) >> 2;   // its 64-column quarter = one k-block of the next layer
    const int r = q * 32 + lane;      // row within the tile
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    uint32_t full_ph = 0;  // bit s: the parity slot s waits for next
    // both accumulators are free for the first pair
    if ((long long)blockIdx.x < pairs && lane == 0)
      for (int s = 0; s < 2 && 2 * (long long)blockIdx.x + s < tiles; ++s) mbar_arrive(b_ready + 8 * s);
    bool ok = true;
    for (long long P = blockIdx.x; ok && P < pairs; P += gridDim.x) {
      const int ns = 2 * P + 1 < tiles ? 2 : 1;
      const long long Pn = P + gridDim.x;  // this CTA's next pair
      for (int l = 0; ok && l < a.L; ++l) {
        const bool last = l == a.L - 1;
        const float* bias = a.bias[l];
        for (int s = 0; s < ns; ++s) {
          const long long row = (2 * P + s) * BM + r;
          const bool next = Pn < pairs && 2 * Pn + s < tiles;  // a next tile for this slot
          unsigned char* as = act + (size_t)s * ACT_BYTES;
          // 16 columns at a time, the next 16 in flight (tensor memory, bias)
          // while these are computed; the first bias before the wait
          uint32_t u[2][16];
          float4 b4[2][4];
          auto load_bias = [&](int ch) {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              b4[ch & 1][j] = __ldg(reinterpret_cast<const float4*>(bias + cq * 64 + ch * 16) + j);
          };
          load_bias(0);
          if (!(ok = mbar_wait(b_full + 8 * s, (full_ph >> s) & 1u, a.err, 14, abort))) break;
          full_ph ^= 1u << s;
          tc_fence_after();
          const uint32_t tacc = tmem + (uint32_t)(s * N) + lane_base;
          float h0 = 0.0f, h1 = 0.0f;
          tmem_ld16_nw(tacc + (uint32_t)(cq * 64), u[0]);
          if (!last) {
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
              const int c0 = cq * 64 + ch * 16;
              tmem_wait_ld16(u[ch & 1]);
              if (ch < 3) {
                tmem_ld16_nw(tacc + (uint32_t)(c0 + 16), u[(ch + 1) & 1]);
                load_bias(ch + 1);
              }
              // the next layer's A operand: 16 columns = two 16-byte chunks
#pragma unroll
              for (int j = 0; j < 2; ++j) {
                const float4 p = b4[ch & 1][2 * j], q = b4[ch & 1][2 * j + 1];
                const uint32_t* x = &u[ch & 1][8 * j];
                float h[8];
                silu_pair(__uint_as_float(x[0]), __uint_as_float(x[1]), p.x, p.y, h[0], h[1]);
                silu_pair(__uint_as_float(x[2]), __uint_as_float(x[3]), p.z, p.w, h[2], h[3]);
                silu_pair(__uint_as_float(x[4]), __uint_as_float(x[5]), q.x, q.y, h[4], h[5]);
                silu_pair(__uint_as_float(x[6]), __uint_as_float(x[7]), q.z, q.w, h[6], h[7]);
                *reinterpret_cast<uint4*>(as + act_off(r, c0 + 8 * j)) =
                    make_uint4(bf16x2(h[0], h[1]), bf16x2(h[2], h[3]), bf16x2(h[4], h[5]), bf16x2(h[6], h[7]));
              }
            }
          } else {
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
              // with their output weights ([c][2]: two columns per float4)
              const int c0 = cq * 64 + ch * 16;
              float4 w4[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) w4[j] = __ldg(reinterpret_cast<const float4*>(a.w_out + 2 * c0) + j);
              tmem_wait_ld16(u[ch & 1]);
              if (ch < 3) {
                tmem_ld16_nw(tacc + (uint32_t)(c0 + 16), u[(ch + 1) & 1]);
                load_bias(ch + 1);
              }
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const float4 p = b4[ch & 1][j >> 1];
                const float bl = (j & 1) ? p.z : p.x, bh = (j & 1) ? p.w : p.y;
                const uint32_t* x = &u[ch & 1][2 * j];
                float v0, v1;
                silu_pair(__uint_as_float(x[0]), __uint_as_float(x[1]), bl, bh, v0, v1);
                h0 = fmaf(v0, w4[j].x, h0);
                h1 = fmaf(v0, w4[j].y, h1);
                h0 = fmaf(v1, w4[j].z, h0);
                h1 = fmaf(v1, w4[j].w, h1);
              }
            }
          }
          if (last) {
            // the column quarters' partial sums in the slot's k-blocks 2-3
            // (the input features of the slot's next tile take k-blocks 0-1)
            float* hp = reinterpret_cast<float*>(as + 2 * KB_BYTES);
            hp[(cq * BM + r) * 2] = h0;
            hp[(cq * BM + r) * 2 + 1] = h1;
            __syncwarp();
            int prior = 0;
            if (lane == 0) {
              __threadfence_block();
              prior = atomicAdd(&head_count[s * 4 + q], 1);
            }
            prior = __shfl_sync(0xffffffffu, prior, 0);
            if (prior == 3) {
              __threadfence_block();
              if (row < a.M) {
                float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                  s0 += hp[(c * BM + r) * 2];
                  s1 += hp[(c * BM + r) * 2 + 1];
                }
                *reinterpret_cast<float2*>(a.out + 2 * row) = make_float2(s0 + a.b_out[0], s1 + a.b_out[1]);
              }
              __syncwarp();
              if (lane == 0) head_count[s * 4 + q] = 0;
            }
          }
          if (!last || next) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(b_ready + 8 * s);
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
  }
}

}  // namespace tcg
