// Inference-path loop: a linear softmax policy over the 84x84x4 stack and a
// device rollout ring (paper Section 4: inference-only throughput, with the
// emulator and the network both on the GPU and no host copies).
//
// Policy: logits[j] = sum_k stack[k] * W[k][j], stack flattened as plane *
// 7056 + row * 84 + column, W bf16 [28224][18], fp32 accumulation in a fixed
// order so every run (and the oracle) gets the same bits: 441 chunks of 64
// sequential fused multiply-adds, chunk partials reduced by the pairwise
// tree s[i] += s[i + h], h = 256 .. 1, over 512 zero-padded slots.  Softmax
// weights exp(l_j - max l) by Cody-Waite reduction (ln 2 split into 355/512
// and a remainder) and a degree-7 Taylor polynomial; the action is the
// smallest j whose running sum of weights exceeds u * total, with u the
// 24-bit fraction of the env's Philox word (env key, step, 4 << 8, episode),
// or the last action of nonzero weight when rounding leaves none.
#pragma once
#include <cstdint>

#include "device_machine.cuh"

namespace atari {

constexpr int POLICY_K = 28224, POLICY_A = 18, POLICY_CHUNKS = 441;
constexpr uint32_t PURPOSE_POLICY = 4;

__device__ __forceinline__ float exp_cw(float x) {
  if (x < -87.0f) return 0.0f;
  const float kf = rintf(__fmul_rn(x, 1.44269504088896341f));
  float r = __fmaf_rn(-kf, 0.693359375f, x);
  r = __fmaf_rn(-kf, -2.12194440e-4f, r);
  float p = 1.0f / 5040.0f;
  p = __fmaf_rn(p, r, 1.0f / 720.0f);
  p = __fmaf_rn(p, r, 1.0f / 120.0f);
  p = __fmaf_rn(p, r, 1.0f / 24.0f);
  p = __fmaf_rn(p, r, 1.0f / 6.0f);
  p = __fmaf_rn(p, r, 0.5f);
  p = __fmaf_rn(p, r, 1.0f);
  p = __fmaf_rn(p, r, 1.0f);
  const int k = (int)kf;
  if (k < -126) return 0.0f;
  return __fmul_rn(p, __int_as_float((k + 127) << 23));
}

// A block serves 128 envs with eight warps: warp p takes the chunk slots
// i = p mod 8, a subtree of the halving tree (its levels h = 256 .. 8), and
// every lane four envs, so that a weight read from shared memory (a 16-byte
// load occupies the load path for four cycles of the SM, in which it could
// issue 16 warp-wide multiply-adds) serves four envs' sums.  With one env a
// lane the loads took four times the multiply-adds' time.  Two neighbouring
// sums share one packed fp32x2 multiply-add.
//
// A subtree's 64 slots are visited in bit-reversed order, in which the two
// slots the tree adds at every level are neighbours, so the tree is the one a
// binary counter builds from left to right: the first of two leaves waits in
// registers, and the pair's sum is pushed on a stack (two levels in shared
// memory, the deeper, rarely touched ones in local memory) and added to the
// entries below it as the carry of the pair number ripples.  The eight
// subtree sums meet in the levels h = 4, 2, 1.  They are the same additions of
// the same operands as the halving tree, hence the same bits.
//
// 16384 envs: 8.3 G multiply-adds are 0.21 ms at 152 SMs x 128 lanes x 2.07 GHz.
// Measured 0.45 ms, 1.77 before (128 of the SMs hold a block, and the byte
// conversions share the FMA pipe); a block takes the same time whatever the
// number of envs it holds.
constexpr int POLICY_PARTS = 8, POLICY_E = 4, POLICY_ENVS = 32 * POLICY_E, POLICY_TPB = 32 * POLICY_PARTS;
constexpr int POLICY_V = POLICY_E * POLICY_A;             // sums a thread keeps
constexpr int POLICY_WROW = 20;                           // floats per staged row of W (16-byte rows)
constexpr int POLICY_WBUF = 64 * POLICY_WROW;             // floats per staged chunk
constexpr int POLICY_LEVELS = 6;                          // stack entries of a subtree (its 32 pairs)
constexpr size_t POLICY_SMEM = 4 * ((size_t)POLICY_PARTS * POLICY_WBUF + (size_t)2 * POLICY_V * POLICY_TPB);

__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// mu_out (may be null) receives the behaviour probability of the sampled
// action, its weight over the total (fp32 division), for a V-trace buffer.
__global__ void __launch_bounds__(POLICY_TPB, 1) k_policy(const uint8_t *obs, const uint16_t *W, const uint8_t *state,
                                                         uint8_t *actions, float *logits_out, float *mu_out, int n,
                                                         uint64_t seed) {
  extern __shared__ __align__(16) uint8_t g_smem[];
  float *wsm = reinterpret_cast<float *>(g_smem) + (threadIdx.x >> 5) * POLICY_WBUF;
  uint64_t *stk = reinterpret_cast<uint64_t *>(reinterpret_cast<float *>(g_smem) + POLICY_PARTS * POLICY_WBUF);
  constexpr int H = POLICY_V / 2;  // packed sums
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
  const int env0 = blockIdx.x * POLICY_ENVS + lane;  // and + 32, + 64, + 96
  const uint8_t *xs[POLICY_E];
#pragma unroll
  for (int e = 0; e < POLICY_E; ++e)  // idle lanes read env 0 and discard it
    xs[e] = obs + (size_t)(env0 + 32 * e < n ? env0 + 32 * e : 0) * POLICY_K;
  const bool words = (reinterpret_cast<uintptr_t>(W) & 3u) == 0;  // W in 4-byte loads
  uint64_t acc[H], first[H], deep[POLICY_LEVELS - 2][H];
  int sp = 0;
#pragma unroll 1
  for (uint32_t k = 0; k < 64; ++k) {
    const uint32_t c = (__brev(k) >> 26) * POLICY_PARTS + part;
#pragma unroll
    for (int q = 0; q < H; ++q) acc[q] = 0;
    if (c < (uint32_t)POLICY_CHUNKS) {  // the same for every lane of the warp
      const uint16_t *wc = W + (size_t)c * 64 * POLICY_A;
      __syncwarp();  // the previous chunk's readers are done
#pragma unroll
      for (int t = 0; t < POLICY_A; ++t) {
        const int q = 2 * (t * 32 + lane);  // pairs do not straddle rows: POLICY_A is even
        const uint32_t w2 = words ? *reinterpret_cast<const uint32_t *>(wc + q) : wc[q] | (uint32_t)wc[q + 1] << 16;
        *reinterpret_cast<float2 *>(wsm + q / POLICY_A * POLICY_WROW + q % POLICY_A) =
            make_float2(__uint_as_float(w2 << 16), __uint_as_float(w2 & 0xFFFF0000u));
      }
      __syncwarp();
#pragma unroll 1
      for (int q4 = 0; q4 < 4; ++q4) {
        uint4 xv[POLICY_E];
#pragma unroll
        for (int e = 0; e < POLICY_E; ++e) xv[e] = reinterpret_cast<const uint4 *>(xs[e] + (size_t)c * 64)[q4];
#pragma unroll
        for (int b = 0; b < 16; ++b) {
          const float *wr = wsm + (q4 * 16 + b) * POLICY_WROW;
          uint64_t w[POLICY_A / 2];
#pragma unroll
          for (int j = 0; j < POLICY_A / 4; ++j) {
            const ulonglong2 v = reinterpret_cast<const ulonglong2 *>(wr)[j];
            w[2 * j] = v.x;
            w[2 * j + 1] = v.y;
          }
          w[POLICY_A / 2 - 1] = reinterpret_cast<const uint64_t *>(wr)[POLICY_A / 2 - 1];
#pragma unroll
          for (int e = 0; e < POLICY_E; ++e) {
            const uint32_t xw = (b >> 2) == 0 ? xv[e].x : (b >> 2) == 1 ? xv[e].y : (b >> 2) == 2 ? xv[e].z : xv[e].w;
            // 2^23 + byte as fp32 bits, less 2^23: the byte, exactly
            const float x = __fsub_rn(__uint_as_float(__byte_perm(xw, 0x4B000000u, 0x7440u | (b & 3))), 8388608.0f);
            uint64_t x2;
            asm("mov.b64 %0, {%1, %1};" : "=l"(x2) : "f"(x));
#pragma unroll
            for (int j = 0; j < POLICY_A / 2; ++j) acc[e * (POLICY_A / 2) + j] = fma2(x2, w[j], acc[e * (POLICY_A / 2) + j]);
          }
        }
      }
    }
    if ((k & 1u) == 0) {
#pragma unroll
      for (int q = 0; q < H; ++q) first[q] = acc[q];
      continue;
    }
#pragma unroll
    for (int q = 0; q < H; ++q) acc[q] = add2(first[q], acc[q]);
#pragma unroll 1
    for (uint32_t m = __ffs(~(k >> 1)) - 1; m > 0; --m) {
      --sp;
      if (sp < 2) {
#pragma unroll
        for (int q = 0; q < H; ++q) acc[q] = add2(stk[(size_t)(sp * H + q) * POLICY_TPB + threadIdx.x], acc[q]);
      } else {
#pragma unroll
        for (int q = 0; q < H; ++q) acc[q] = add2(deep[sp - 2][q], acc[q]);
      }
    }
    if (sp < 2) {
#pragma unroll
      for (int q = 0; q < H; ++q) stk[(size_t)(sp * H + q) * POLICY_TPB + threadIdx.x] = acc[q];
    } else {
#pragma unroll
      for (int q = 0; q < H; ++q) deep[sp - 2][q] = acc[q];
    }
    ++sp;
  }
  // entry 0 of every thread's stack is its subtree's sum
  __syncthreads();
  const int t = threadIdx.x;
  const int i = blockIdx.x * POLICY_ENVS + t;
  if (t < POLICY_ENVS && i < n) {
    float l[POLICY_A];
    const int e = t >> 5;
#pragma unroll
    for (int jj = 0; jj < POLICY_A / 2; ++jj) {
      uint64_t v[POLICY_PARTS];
#pragma unroll
      for (int p = 0; p < POLICY_PARTS; ++p) v[p] = stk[(size_t)(e * (POLICY_A / 2) + jj) * POLICY_TPB + p * 32 + lane];
#pragma unroll
      for (int h = POLICY_PARTS / 2; h > 0; h >>= 1)
#pragma unroll
        for (int p = 0; p < h; ++p) v[p] = add2(v[p], v[p + h]);
      l[2 * jj] = __uint_as_float((uint32_t)v[0]);
      l[2 * jj + 1] = __uint_as_float((uint32_t)(v[0] >> 32));
    }
    float m = l[0];
#pragma unroll
    for (int j = 0; j < POLICY_A; ++j) m = l[j] > m ? l[j] : m;
    float ex[POLICY_A], tot = 0.0f;
#pragma unroll
    for (int j = 0; j < POLICY_A; ++j) {
      ex[j] = exp_cw(__fsub_rn(l[j], m));
      tot = __fadd_rn(tot, ex[j]);
    }
    const uint8_t *st = state + (size_t)i * 256;
    const uint32_t *ew = reinterpret_cast<const uint32_t *>(st + S::EPISODE);
    const uint32_t x = philox_x0(seed, ew[2], ew[1], PURPOSE_POLICY << 8, ew[0]);
    const float thr = __fmul_rn(__fmul_rn(__uint2float_rn(x >> 8), 5.9604644775390625e-08f), tot);
    float c = 0.0f;
    int act = -1, last = 0;
#pragma unroll
    for (int j = 0; j < POLICY_A; ++j) {
      c = __fadd_rn(c, ex[j]);
      if (ex[j] > 0.0f) last = j;
      if (act < 0 && c > thr) act = j;
    }
    const int a = act < 0 ? last : act;
    actions[i] = (uint8_t)a;
    if (mu_out) {
      float ea = ex[0];
#pragma unroll
      for (int j = 1; j < POLICY_A; ++j) ea = j == a ? ex[j] : ea;
      mu_out[i] = __fdiv_rn(ea, tot);
    }
    if (logits_out) {
#pragma unroll
      for (int j = 0; j < POLICY_A; ++j) logits_out[(size_t)i * POLICY_A + j] = l[j];
    }
  }
}

// Append the newest stack plane, the reward and (ring_dones not null) the
// done flag of every env to ring slot `slot`.
__global__ void k_ring_append(const uint8_t *obs, const int32_t *rewards, const uint8_t *dones, uint8_t *ring_planes,
                              float *ring_rewards, uint8_t *ring_dones, int n, int slot) {
  const int i = blockIdx.x;
  if (i >= n) return;
  const uint4 *src = reinterpret_cast<const uint4 *>(obs + (size_t)i * 4 * 7056 + 3 * 7056);
  uint4 *dst = reinterpret_cast<uint4 *>(ring_planes + ((size_t)slot * n + i) * 7056);
  for (int q = threadIdx.x; q < 7056 / 16; q += blockDim.x) dst[q] = src[q];
  if (threadIdx.x == 0) {
    ring_rewards[(size_t)slot * n + i] = (float)rewards[i];
    if (ring_dones) ring_dones[(size_t)slot * n + i] = dones[i];
  }
}

}  // namespace atari
