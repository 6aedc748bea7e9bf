// qa_sphere.cuh -- the candidate search of large arrays as a sphere decoder:
// an exact depth-first search over the candidate set whose partial sums bound
// every energy below them from below.
//
// With M = W^T W, W lower triangular in a fixed order of the dots (W is the
// inverse of the Cholesky factor of Cdd in that order, so no M is factored),
// x the pixel's continuous minimum, f = x - base and zeta = M (x - c) its
// gradient, a candidate base + b has the energy
//     E(b) = const + zeta . b + sum_k y_k^2,
//     y_k = (sum_{l <= k} W_kl (b_l - f_l)) / sqrt 2,
// and zeta is zero on every free dot and at least zero on the active ones
// (open: the KKT conditions; closed: up to one multiple of 1, which adds the
// same to every candidate of the right weight).  All terms are non-negative,
// so the sum over the first dots bounds every completion: the closest-vector
// search of Fincke and Pohst (Math. Comp. 44 (1985) 463; Agrell et al., IEEE
// Trans. Inf. Theory 48 (2002) 2201).  Unlike a bound by single coefficients
// it sees the pair terms, and it needs no table per pixel: W belongs to the
// model.
//
// The result is the argmin of the candidate set together with a certificate:
// `doubt` is false only when every other candidate's energy is above the
// minimum by more than twice the pixel's near-tie bound plus twice the
// rounding error of this search (sphere_margin).  The FP32 search of
// qa_search.cuh errs by at most that near-tie bound in the gap of two
// energies, so for such a pixel it finds the same argmin and a gap above the
// bound, i.e. no near tie: its outputs and flags are known without running
// it.  The other pixels (about twice the near ties: 1 % of the 16-dot
// diagrams) are settled from the candidates within the margin, which a second
// pass lists: their exact energies give the argmin, and the FP32 search's
// energies of those candidates alone its near-tie flag.
#pragma once

#include "qa_device.cuh"

namespace qa {

constexpr int kSphT = 16;                  // lanes per pixel
constexpr int kSphRow = 4 * kMaxDot + 17;  // table row: four 16-entry tables; odd, and rows of
                                           // neighbouring levels start 17 banks apart
constexpr int kSphStack = 160;             // waiting nodes per pixel
constexpr int kSphRoom = 3 * kMaxDot / 2;  // what one node's descendants add at most
constexpr int kSphSteps = 512;             // expansion steps per pixel at most
constexpr int kSphList = 16;               // candidates within the margin that are listed

// A block's copy of a model's factor: for each level k and each group g of
// four earlier levels the sums of W_kl over every subset of the group, so a
// row's sum over a bit pattern is four loads.
struct SphereModel {
  float tab[kMaxDot * kSphRow];
  float4 rowc[kMaxDot / 2];     // levels 2p, 2p + 1: their diagonals, W_{2p+1,2p}
  unsigned char ord[kMaxDot];   // dot of each level
  unsigned char pos[kMaxDot];   // level of each dot
};

// Stage a model's tables (all threads; sync after).  Thread (k, g) forms one
// group's sixteen sums by doubling.
__device__ __forceinline__ void sphere_stage(const SphereConsts& g, SphereModel& s) {
  for (int e = threadIdx.x; e < kMaxDot * 4; e += blockDim.x) {
    const int k = e >> 2, q = e & 3;
    const float4 w = *reinterpret_cast<const float4*>(&g.W[k][4 * q]);
    const float wv[4] = {w.x, w.y, w.z, w.w};
    float v[16];
    v[0] = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int b = 0; b < (1 << i); ++b) v[b + (1 << i)] = v[b] + wv[i];
    float* t = s.tab + k * kSphRow + q * 16;
#pragma unroll
    for (int b = 0; b < 16; ++b) t[b] = v[b];
  }
  if (threadIdx.x < kMaxDot) {
    s.ord[threadIdx.x] = g.ord[threadIdx.x];
    s.pos[threadIdx.x] = g.pos[threadIdx.x];
  }
  if (threadIdx.x < kMaxDot / 2) {
    const int k = 2 * threadIdx.x;
    s.rowc[threadIdx.x] = make_float4(g.wd[k], g.wd[k + 1], g.W[k + 1][k], 0.f);
  }
}

// The margin of the certificate and of the pruning: twice the near-tie bound
// (see above) plus the rounding errors of this search's sums on both sides of
// a gap.  With u = 2^-24 and Y_k = sum_l |W_kl| (|b_l - f_l| <= 1 or so),
// y_k is off by at most 28 u Y_k (the rounded W, a sixteen-term sum for the
// centre, three additions in a table and six after), so sum y_k^2 by
// 56 u sqrt(sum y^2 sum Y^2) and, with its own additions, 32 u sum y^2; ez
// bounds the error of zeta . b, the negative parts of zeta, which are left
// out, among it.
__device__ __forceinline__ float sphere_margin(const SphereConsts& g, float bound, float cost,
                                               float ez) {
  constexpr float u = 5.9604645e-8f;
  const float c = cost + 4.f * bound;  // a pruned sum is this far up
  const float d = 56.f * u * sqrtf(c * g.ysq) + 32.f * u * c + ez;
  return 2.f * bound + 2.5f * d;
}

// One node's four children: the patterns of levels 2p, 2p + 1 below the
// pattern b of the earlier levels.  c[j]: the cost with bit 0 of j at level
// 2p and bit 1 at level 2p + 1; +inf where a dot is not ambiguous or (closed)
// the rest cannot reach the weight.  lev: the pixel's centres and gradients.
template <bool CLOSED>
__device__ __forceinline__ void sphere_expand(const SphereModel& s, const float4* lev, int p,
                                              unsigned b, float C, int w, unsigned maskpos,
                                              float* c) {
  constexpr float inf = __builtin_huge_valf();
  const float4 lv = lev[p], rc = s.rowc[p];
  const float* t = s.tab + 2 * p * kSphRow;
  const unsigned i0 = b & 15u, i1 = 16u + ((b >> 4) & 15u), i2 = 32u + ((b >> 8) & 15u),
                 i3 = 48u + (b >> 12);
  const float s0 = ((t[i0] + t[i1]) + (t[i2] + t[i3])) - lv.x;
  const float* t1 = t + kSphRow;
  const float s1 = ((t1[i0] + t1[i1]) + (t1[i2] + t1[i3])) - lv.y;
  const float y1 = s0 + rc.x;
  const float c0 = fmaf(s0, s0, C), c1 = fmaf(y1, y1, C) + lv.z;
  const float a0 = s1, a1 = s1 + rc.z;
  const float d0 = a0 + rc.y, d1 = a1 + rc.y;
  c[0] = fmaf(a0, a0, c0);
  c[1] = fmaf(a1, a1, c1);
  c[2] = fmaf(d0, d0, c0) + lv.w;
  c[3] = fmaf(d1, d1, c1) + lv.w;
  if (CLOSED) {
    const int r = w - __popc(b), left = __popc(maskpos >> (2 * p + 2));
    if (r < 0 || r > left) c[0] = inf;
    if (r < 1 || r - 1 > left) c[1] = c[2] = inf;
    if (r < 2 || r - 2 > left) c[3] = inf;
  }
}

// The search of one pixel by its team of 16 lanes (lane lt owns dot lt in the
// inputs); both teams of a warp must call together.  active: the team has a
// pixel.  f: the dot's centre x - base; a1: its gradient (>= 0; ignored for
// dots that are not ambiguous); mask: the ambiguous dots; w: closed weight;
// bound: at least the near-tie bound; ez: see sphere_margin.  scr0, scr1: 16
// floats of scratch, lev: the pixel's centres and gradients, stk: kSphStack
// entries.  Returns the best pattern over the dots; close: the number of
// candidates within the margin of the minimum, 1 when it is certain, their
// patterns (over the levels) then in scr1; 0: not settled.
// What bounds it: instruction issue and shared-memory latency.  An array of
// 16 dots expands 80 to 330 nodes per pixel out of 2^16 candidates, 14 dots
// about 50, most of them in full steps of 16.
template <bool CLOSED>
__device__ __forceinline__ unsigned sphere_search(const SphereConsts& g, const SphereModel& s,
                                                  int n, int lt, bool active, float f, float a1,
                                                  unsigned mask, int w, float bound, float ez,
                                                  float* scr0, float* scr1, float4* lev,
                                                  uint2* stk, int& close,
                                                  unsigned& evaluated) {
  constexpr unsigned kAll = 0xffffffffu;
  constexpr float inf = __builtin_huge_valf();
  const unsigned hw = threadIdx.x & 16u;       // the team's first lane in the warp
  const unsigned below = (1u << lt) - 1u;
  const int np = (n + 1) >> 1;                 // level pairs (a level past n adds nothing)
  auto team = [&](bool pred) { return (__ballot_sync(kAll, pred) >> hw) & 0xffffu; };

  // centres and gradients by level; a dot that is not ambiguous keeps bit 0
  const int pos = s.pos[lt], dot = s.ord[lt];
  const bool mine = active && lt < n;
  __syncwarp();
  if (lt < n) {
    scr0[pos] = mine ? f : 0.f;
    scr1[pos] = (mine && ((mask >> lt) & 1u)) ? a1 : inf;
  } else {
    scr0[lt] = 0.f;
    scr1[lt] = inf;
  }
  __syncwarp();
  const unsigned maskpos = team(lt < n && ((mask >> dot) & 1u));
  {
    // F_k = sum_{l <= k} W_kl f_l, lane k its row (the single-bit entries of
    // the row's tables; zero from k on)
    const float* row = s.tab + lt * kSphRow;
    const float4 rc = s.rowc[lt >> 1];
    float F = ((lt & 1) ? rc.y : rc.x) * scr0[lt];
#pragma unroll
    for (int l = 0; l < kMaxDot; ++l) F = fmaf(row[(l >> 2) * 16 + (1 << (l & 3))], scr0[l], F);
    float* lf = reinterpret_cast<float*>(lev + (lt >> 1));
    lf[lt & 1] = F;
    lf[2 + (lt & 1)] = scr1[lt];
  }
  __syncwarp();

  // the first four levels: lane t their pattern t
  unsigned b = (unsigned)lt;
  float C = 0.f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float4 lv = lev[k >> 1], rc = s.rowc[k >> 1];
    const bool bit = (b >> k) & 1u;
    const float y = (s.tab[k * kSphRow + (b & ((1u << k) - 1u))] - ((k & 1) ? lv.y : lv.x)) +
                    (bit ? ((k & 1) ? rc.y : rc.x) : 0.f);
    C = fmaf(y, y, C) + (bit ? ((k & 1) ? lv.w : lv.z) : 0.f);
  }
  if (CLOSED) {
    const int r = w - __popc(b);
    if (r < 0 || r > __popc(maskpos >> 4)) C = inf;
  }
  if (!active) C = inf;
  evaluated += active ? 1u : 0u;

  // each lane completes its pattern greedily, two levels at a time; the
  // lowest of the sixteen is the first cut
  float inc = C;
  {
    unsigned rb = b;
    for (int p = 2; p < np; ++p) {
      float c[4];
      sphere_expand<CLOSED>(s, lev, p, rb, inc, w, maskpos, c);
      const bool o = c[1] < c[0], q = c[3] < c[2];
      const float e0 = o ? c[1] : c[0], e1 = q ? c[3] : c[2];
      const bool hi = e1 < e0;
      inc = hi ? e1 : e0;
      rb |= (hi ? (q ? 3u : 2u) : (o ? 1u : 0u)) << (2 * p);
    }
    evaluated += active ? (unsigned)(4 * (np - 2)) : 0u;
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) inc = fminf(inc, __shfl_xor_sync(kAll, inc, off));
  }
  bool hard = !(inc < inf);
  const float G = sphere_margin(g, bound, inc, ez);
  float cut = inc + G;

  // depth first, sixteen waiting nodes a step; a node: cost, pattern, levels.
  // A second pass, at the final cut, lists the candidates where more than one
  // lies below it.
  float m1 = inf, m2 = inf;
  unsigned b1 = 0u;
  int nl = 0;
  unsigned* lst = reinterpret_cast<unsigned*>(scr1);
#pragma unroll 1
  for (bool list = false;; list = true) {
    int sp;
    {
      const bool keep = C <= cut && C < inf && !hard;
      const unsigned m = team(keep);
      if (keep) stk[__popc(m & below)] = make_uint2(__float_as_uint(C), b | (2u << 16));
      sp = __popc(m);
    }
    __syncwarp();
#pragma unroll 1
    for (int step = 0; step < kSphSteps; ++step) {
      if (!__any_sync(kAll, sp > 0)) break;
      // as many as leave room for one node's way down (three more a level), so
      // the stack cannot overflow
      const int take = min(min(sp, kSphT), max(1, (kSphStack - kSphRoom - sp) / 3));
      bool valid = lt < take;
      uint2 nd = make_uint2(0u, 2u << 16);
      if (valid) nd = stk[sp - 1 - lt];
      sp -= take;
      const float cn = __uint_as_float(nd.x);
      valid = valid && cn <= cut;
      const int p = (int)(nd.y >> 16);
      const unsigned nb = nd.y & 0xffffu;
      float c[4];
      sphere_expand<CLOSED>(s, lev, p, nb, cn, w, maskpos, c);
      evaluated += valid ? 4u : 0u;
      const bool leaf = p + 1 == np;
      const bool vl = valid && leaf;
      if (__any_sync(kAll, vl)) {
        if (!list) {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float e = vl ? c[j] : inf;
            m2 = fminf(m2, fmaxf(m1, e));
            if (e < m1) {
              m1 = e;
              b1 = nb | ((unsigned)j << (2 * p));
            }
          }
          float t = m1;
#pragma unroll
          for (int off = 8; off > 0; off >>= 1) t = fminf(t, __shfl_xor_sync(kAll, t, off));
          cut = fminf(cut, t + G);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const bool keep = vl && c[j] <= cut;
            const unsigned m = team(keep);
            const int at = nl + __popc(m & below);
            nl += __popc(m);
            if (keep && at < kSphList) lst[at] = nb | ((unsigned)j << (2 * p));
          }
        }
      }
      __syncwarp();  // the nodes are read: their places are free
      const bool vi = valid && !leaf;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool keep = vi && c[j] <= cut;
        const unsigned m = team(keep);
        const int at = sp + __popc(m & below);
        sp += __popc(m);
        if (keep && at < kSphStack)
          stk[at] = make_uint2(__float_as_uint(c[j]),
                               (nb | ((unsigned)j << (2 * p))) | ((unsigned)(p + 1) << 16));
      }
      __syncwarp();
    }
    hard = hard || sp > 0;
    if (list) break;
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) {
      const float o1 = __shfl_xor_sync(kAll, m1, off), o2 = __shfl_xor_sync(kAll, m2, off);
      const unsigned ob = __shfl_xor_sync(kAll, b1, off);
      m2 = fminf(fminf(m2, o2), fmaxf(m1, o1));
      if (o1 < m1) {
        m1 = o1;
        b1 = ob;
      }
    }
    hard = hard || !(m1 < inf);
    cut = m1 + G;
    const bool sure = m2 > cut;
    if (!hard && sure) nl = 1;
    if (!__any_sync(kAll, !hard && !sure)) break;
    if (sure) C = inf;  // only the other team goes on
  }
  // (the same in all lanes of a team: a tie of m1 between lanes is listed)
  close = (hard || nl > kSphList || (nl < 2 && !(m2 > cut))) ? 0 : nl;
  // the pattern over the dots
  return team(lt < n && ((b1 >> pos) & 1u));
}

}  // namespace qa
