// qa_soft_fit.cuh -- the fit step's kernel beyond 8 dots: one candidate at a
// time.  The table form of the other modes (k_soft_wide) sums the same terms in
// another order; Adam divides each gradient entry by its own magnitude, so the
// FP32 rounding of a small entry reaches the FP64 parameters (1e-7 relative
// where an entry's gradient is below 1e-6), and a fit's trajectory is kept to
// the bit instead.  What bounds it: issue of the divergent per-candidate sums
// and 136 register moments (two blocks per SM): 12 dots, 75 x 60, 1.5 - 2.6 ms.
#pragma once

#include "qa_soft.cuh"

namespace qa {

// D(b) = E(b) - E(b*) from the slots that differ from b*: the first-order
// terms gp / gm of each and the pair terms between them, read from the team's
// slot-ordered copy of M (Ms[s * 16 + s2] = M of the dots of slots s, s2).
__device__ __forceinline__ float delta_energy(const TeamSlots& ts, const float* Ms, unsigned b) {
  const unsigned d = b ^ ts.bstar;
  float D = 0.f;
  for (unsigned m = d; m; m &= m - 1u) {
    const int s = __ffs(m) - 1;
    const bool add = (b >> s) & 1u;
    D += add ? ts.gp[s] : ts.gm[s];
    const float* row = Ms + s * kMaxDot;
    for (unsigned q = d & ((1u << s) - 1u); q; q &= q - 1u) {
      const int s2 = __ffs(q) - 1;
      const bool add2 = (b >> s2) & 1u;
      const float v = row[s2];
      D += (add == add2) ? v : -v;
    }
  }
  return D;
}

// <n>, loss and the per-block gradient partials of a fit step.
template <bool CLOSED>
__global__ void __launch_bounds__(kSoftThreads) k_soft_fit(SoftLaunch a) {
  constexpr int KMAX = kMaxDot;               // slots
  constexpr int kTeams = kSoftThreads / 32;   // pixels: a warp each
  __shared__ ModelConsts cs;
  __shared__ TeamSlots tsm[kTeams];
  __shared__ float slotM[kTeams][KMAX * KMAX];         // slot-ordered M of a team
  __shared__ float sQa[kTeams][tri(KMAX) + KMAX + 1];  // Qa, va, sa of a team
  __shared__ float sGf[kTeams][kMaxDot];               // g of a team
  extern __shared__ float s_contrib[];  // [teams][contrib_len]
  const int n = a.n;
  stage_consts(&a.md->k, &cs);
  __syncthreads();
  const float* sM = cs.Mhi;
  const float* sMlo = cs.Mlo;
  // 32 (run_soft_fit sees to it), but read at run time: with T or the block's
  // teams known when compiled the kernel takes 255 registers instead of 196 and
  // the step a tenth longer (12 dots, 75 x 60: 2635 -> 2907 us)
  const int T = a.cfg.T;
  const int team = threadIdx.x / T, lt = threadIdx.x % T;
  const int teams = blockDim.x / T;
  const long long p = (long long)blockIdx.x * teams + team;
  const bool active = p < a.sc.P;
  TeamSlots& ts = tsm[team];
  const float kT = (float)a.kT;

  soft_setup_team<CLOSED>(a, ts, p, lt, T, active);
  float* Ms = slotM[team];
  if (active)
    for (int e = lt; e < KMAX * KMAX; e += T) {
      const int s = e / KMAX, s2 = e % KMAX;
      Ms[e] = (s < ts.k && s2 < ts.k) ? sM[ts.dot[s] * kLdM + ts.dot[s2]] : 0.f;
    }
  __syncwarp();

  // pass 1: the minimum-energy candidate b*
  float m1 = kInf, m2 = kInf;
  unsigned b1 = 0u;
  unsigned long long ev = 0;
  if (active) {
    SlotView sv{ts.dot, ts.h, ts.k, ts.w};
    search_lane<5, 4, CLOSED, false>(sM, sv, lt, T, 0.f, nullptr, nullptr, 0u, m1, b1, m2, ev);
  }
  for (int off = 1; off < T; off <<= 1) {
    const float om1 = __shfl_xor_sync(kFullS, m1, off);
    const unsigned ob1 = __shfl_xor_sync(kFullS, b1, off);
    const float om2 = __shfl_xor_sync(kFullS, m2, off);
    top2_merge(m1, b1, m2, om1, ob1, om2);
  }
  soft_anchor<kMaxDot>(a, ts, sM, sMlo, T, lt, active, b1);

  // pass 2: Boltzmann weights relative to b*
  const int k = active ? ts.k : 0;
  const unsigned total = 1u << k;
  float Z = 0.f;
  float acc[KMAX];
#pragma unroll
  for (int s = 0; s < KMAX; ++s) acc[s] = 0.f;
  const float inv_kT = 1.0f / kT;
  if (active) {
    for (unsigned b = (unsigned)lt; b < total; b += (unsigned)T) {
      if (CLOSED && __popc(b) != ts.w) continue;
      const float wgt = expf(-delta_energy(ts, Ms, b) * inv_kT);
      Z += wgt;
#pragma unroll
      for (int s = 0; s < KMAX; ++s)
        if ((b >> s) & 1u) acc[s] += wgt;
    }
  }
  for (int off = 1; off < T; off <<= 1) {
    Z += __shfl_xor_sync(kFullS, Z, off);
#pragma unroll
    for (int s = 0; s < KMAX; ++s) acc[s] += __shfl_xor_sync(kFullS, acc[s], off);
  }

  // ---- backward: a_b = -(w_b / kT) (g . n_b - g . <n>), w_b normalised ----
  const int L = contrib_len(n);
  float* my = s_contrib + team * L;
  float gs[KMAX];      // g of each slot's dot
  float gmean = 0.f;   // g . <n> - g . base
  const float invZ = 1.0f / Z;
#pragma unroll
  for (int s = 0; s < KMAX; ++s) gs[s] = 0.f;
  const float lossp = fit_loss_grad_team(
      a, ts, [&](int s) { return pick<KMAX>(acc, s); }, Z, p, sGf[team], lt, T, active);
  if (active) {
    const float* g = sGf[team];
#pragma unroll
    for (int s = 0; s < KMAX; ++s)
      if (s < k) gs[s] = g[ts.dot[s]];
    // g . <n> - g . base = sum_s g_s <b_s>, so that gn - gmean below is formed
    // without the large g . base on both sides
#pragma unroll
    for (int s = 0; s < KMAX; ++s)
      if (s < k) gmean += gs[s] * acc[s] * invZ;
  }
  float sa = 0.f;
  float va[KMAX];
  float Qa[tri(KMAX)];
#pragma unroll
  for (int s = 0; s < KMAX; ++s) va[s] = 0.f;
#pragma unroll
  for (int e = 0; e < tri(KMAX); ++e) Qa[e] = 0.f;
  if (active) {
    for (unsigned b = (unsigned)lt; b < total; b += (unsigned)T) {
      if (CLOSED && __popc(b) != ts.w) continue;
      const float wgt = expf(-delta_energy(ts, Ms, b) * inv_kT) * invZ;
      float gn = 0.f;
#pragma unroll
      for (int s = 0; s < KMAX; ++s)
        if ((b >> s) & 1u) gn += gs[s];
      const float av = -(wgt * inv_kT) * (gn - gmean);
      sa += av;
#pragma unroll
      for (int s = 0; s < KMAX; ++s) {
        if ((b >> s) & 1u) {
          va[s] += av;
#pragma unroll
          for (int s2 = s; s2 < KMAX; ++s2)
            if ((b >> s2) & 1u) Qa[s * KMAX - s * (s - 1) / 2 + (s2 - s)] += av;
        }
      }
    }
  }
  for (int off = 1; off < T; off <<= 1) {
    sa += __shfl_xor_sync(kFullS, sa, off);
#pragma unroll
    for (int s = 0; s < KMAX; ++s) va[s] += __shfl_xor_sync(kFullS, va[s], off);
#pragma unroll
    for (int e = 0; e < tri(KMAX); ++e) Qa[e] += __shfl_xor_sync(kFullS, Qa[e], off);
  }
  // pixel contribution: dM_p = 1/2 [sa r0 r0^T + r0 va^T + va r0^T + Qa],
  // rho = sa r0 + va, dc_p = -M rho (dot coordinates); the team's lanes split
  // the entries
  float* q_s = sQa[team];
  if (lt == 0) {
#pragma unroll
    for (int e = 0; e < tri(KMAX); ++e) q_s[e] = Qa[e];
#pragma unroll
    for (int s = 0; s < KMAX; ++s) q_s[tri(KMAX) + s] = va[s];
    q_s[tri(KMAX) + KMAX] = sa;
  }
  __syncwarp();
  soft_contrib<KMAX>(a, ts, q_s, my, s_contrib, sM, T, lt, teams, active, p, lossp);
}

template <bool CLOSED>
static cudaError_t run_soft_fit(const SoftLaunch& a, cudaStream_t st) {
  if (a.cfg.T != 32) return cudaErrorInvalidValue;  // the kernel's shared arrays
  constexpr int teams = kSoftThreads / 32;
  const unsigned grid = (unsigned)((a.sc.P + teams - 1) / teams);
  const size_t smem = (size_t)teams * contrib_len(a.n) * sizeof(float);
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(k_soft_fit<CLOSED>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  if (a.ev) cudaEventRecord(a.ev[0], st);
  k_soft_fit<CLOSED><<<grid, kSoftThreads, smem, st>>>(a);
  k_soft_reduce<<<contrib_len(a.n), 256, 0, st>>>(a, (int)grid);
  if (a.ev) cudaEventRecord(a.ev[1], st);
  return cudaGetLastError();
}

}  // namespace qa
