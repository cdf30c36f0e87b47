// Learner-side targets over a rollout kept on the device (paper Appendix,
// "A2C": the bootstrapped N-step return of the policy and value costs;
// "V-trace": the off-policy target with truncated importance weights, in
// the recursive form the paper implements, and the actor's advantage).
//
// Layout: the rollout's per-step rewards, dones and behaviour probabilities
// live in a ring of `depth` slots of n envs each (time-major, as the rollout
// loop writes them); step t of the T steps is slot (start + t) mod depth.
// Values V(s_t) ([T + 1][n], row T the bootstrap value) and target
// probabilities pi ([T][n]) come from the learner; outputs are [T][n].
//
// One thread per env walks its T steps from the last back to the first, so
// every load and store of a step is one coalesced row of the time-major
// arrays.  A walk is bound by the latency of its loads (a learner's batch is a
// few warps an SM), so the steps go in groups of TARGET_STEPS (the last one of
// what is left, so a five-step return is one group) whose loads are all issued
// before the first is used, and blocks are small to spread the
// envs over the SMs (V-trace over 60 x 32768: 67 -> 22 us a call).  fp32
// throughout, each operation rounded once (no contraction into
// fused multiply-adds), in this order per step t (g = gamma, or 0 after a
// done):
//   N-step:   R_t = r_t + g R_{t+1},  R_T = V(s_T)
//   V-trace:  ratio = pi_t / mu_t,  rho = min(rho_bar, ratio),  c = min(c_bar, ratio)
//             delta = rho ((r_t + g V_{t+1}) - V_t)
//             v_t   = (V_t + delta) + (g c)(v_{t+1} - V_{t+1}),  v_T = V(s_T)
//             A_t   = rho ((r_t + g v_{t+1}) - V_t)
#pragma once
#include <cstdint>

namespace atari {

constexpr int TARGET_STEPS = 8, TARGET_TPB = 64;

// Steps t = first .. first - N + 1 of env i's walk, those below 0 left out.
template <int N>
__device__ __forceinline__ float nstep_group(const float *rew, const uint8_t *done, int depth, int start, int first,
                                             int n, int i, float gamma, float R, float *ret) {
  float r[N];
  uint8_t d[N];
#pragma unroll
  for (int k = 0; k < N; ++k) {
    if (k > first) continue;
    int slot = start + first - k;  // start < depth and t < T <= depth
    slot -= slot >= depth ? depth : 0;
    const size_t s = (size_t)slot * n + i;
    r[k] = rew[s];
    d[k] = done[s];
  }
#pragma unroll
  for (int k = 0; k < N; ++k) {
    if (k > first) continue;
    R = __fadd_rn(r[k], __fmul_rn(d[k] ? 0.0f : gamma, R));
    ret[(size_t)(first - k) * n + i] = R;
  }
  return R;
}
__global__ void __launch_bounds__(TARGET_TPB) k_nstep_returns(const float *rew,
                                                             const uint8_t *done, int depth, int start,
                                                             const float *values, int T, int n,
                                                             float gamma, float *ret) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float R = values[(size_t)T * n + i];
  for (int t = T - 1; t >= 0; t -= TARGET_STEPS)
    R = nstep_group<TARGET_STEPS>(rew, done, depth, start, t, n, i, gamma, R, ret);
}

struct VtraceArgs {
  const float *rew;
  const uint8_t *done;
  const float *mu;
  const float *values;
  const float *pi;
  float *vs;
  float *adv;
  int depth, start, n;
  float gamma, rho_bar, c_bar;
};
template <int N>
__device__ __forceinline__ void vtrace_group(const VtraceArgs &a, int first, int i, float &v_next, float &V_next) {
  float r[N], m[N], p[N], V[N];
  uint8_t d[N];
#pragma unroll
  for (int k = 0; k < N; ++k) {
    if (k > first) continue;
    int slot = a.start + first - k;
    slot -= slot >= a.depth ? a.depth : 0;
    const size_t s = (size_t)slot * a.n + i, o = (size_t)(first - k) * a.n + i;
    r[k] = a.rew[s];
    d[k] = a.done[s];
    m[k] = a.mu[s];
    p[k] = a.pi[o];
    V[k] = a.values[o];
  }
#pragma unroll
  for (int k = 0; k < N; ++k) {
    if (k > first) continue;
    const size_t o = (size_t)(first - k) * a.n + i;
    const float g = d[k] ? 0.0f : a.gamma;
    const float ratio = __fdiv_rn(p[k], m[k]);
    // a NaN ratio (0 / 0) takes the truncation level, as min(level, NaN) does below
    const float rho = ratio < a.rho_bar ? ratio : a.rho_bar;
    const float c = ratio < a.c_bar ? ratio : a.c_bar;
    const float delta = __fmul_rn(rho, __fsub_rn(__fadd_rn(r[k], __fmul_rn(g, V_next)), V[k]));
    const float v = __fadd_rn(__fadd_rn(V[k], delta), __fmul_rn(__fmul_rn(g, c), __fsub_rn(v_next, V_next)));
    a.adv[o] = __fmul_rn(rho, __fsub_rn(__fadd_rn(r[k], __fmul_rn(g, v_next)), V[k]));
    a.vs[o] = v;
    v_next = v;
    V_next = V[k];
  }
}
__global__ void __launch_bounds__(TARGET_TPB) k_vtrace(const float *rew, const uint8_t *done, const float *mu, int depth,
                                                      int start, const float *values, const float *pi, int T, int n,
                                                      float gamma, float rho_bar, float c_bar, float *vs, float *adv) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const VtraceArgs a{rew, done, mu, values, pi, vs, adv, depth, start, n, gamma, rho_bar, c_bar};
  float v_next = values[(size_t)T * n + i];  // v_T = V(s_T)
  float V_next = v_next;
  for (int t = T - 1; t >= 0; t -= TARGET_STEPS) vtrace_group<TARGET_STEPS>(a, t, i, v_next, V_next);
}

}  // namespace atari
