// qa_gs_tiles.cuh -- the ground-state stages as per-tile device functions,
// shared by the single-array kernels (qa_kernels_gs.cu) and the persistent
// batched kernels (qa_batch.cu).  A tile is one block's worth of pixels of one
// array; the stage functions take the array's descriptor and the tile's first
// pixel-team index, so both launch shapes run exactly the same code.
#pragma once

#include "qa_launch.h"
#include "qa_prep.cuh"
#include "qa_search.cuh"
#include "qa_sphere.cuh"

namespace qa {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kPrepThreads = 128;
constexpr int kRecheckThreads = 512;  // the tail kernel's block: resolve and recheck alike
constexpr int kResolveThreads = 512;  // the walk's 512 outer states at k = 16, one per thread
constexpr int kCheckL1 = 4, kCheckL2 = 3;  // resolve/recheck split: 2^9 outer states at k = 16
constexpr unsigned kBcap = 1024;

// One charge of the output map: int8 (saturating at 127) or int16 (at
// 32767) by the array's output width; saturation sets kFlagOverflow.
__device__ __forceinline__ void store_charge(const ArrayDesc& a, long long idx, int v,
                                             unsigned& flags) {
  if (a.out_n16) {
    if (v > 32767) { v = 32767; flags |= kFlagOverflow; }
    a.out_n16[idx] = (int16_t)v;
  } else {
    if (v > 127) { v = 127; flags |= kFlagOverflow; }
    a.out_n[idx] = (int8_t)v;
  }
}

// number of k-subsets of size w (k <= 16), 0 outside 0 <= w <= k: 16-bit
// entries (C(16, 8) = 12870), by rows (a loop of 64-bit divisions, run by one
// lane of a team while the others wait, took a fifth of a closed pixel's
// prep)
__constant__ unsigned short kBinom[17][17] = {
    {1},
    {1, 1},
    {1, 2, 1},
    {1, 3, 3, 1},
    {1, 4, 6, 4, 1},
    {1, 5, 10, 10, 5, 1},
    {1, 6, 15, 20, 15, 6, 1},
    {1, 7, 21, 35, 35, 21, 7, 1},
    {1, 8, 28, 56, 70, 56, 28, 8, 1},
    {1, 9, 36, 84, 126, 126, 84, 36, 9, 1},
    {1, 10, 45, 120, 210, 252, 210, 120, 45, 10, 1},
    {1, 11, 55, 165, 330, 462, 462, 330, 165, 55, 11, 1},
    {1, 12, 66, 220, 495, 792, 924, 792, 495, 220, 66, 12, 1},
    {1, 13, 78, 286, 715, 1287, 1716, 1716, 1287, 715, 286, 78, 13, 1},
    {1, 14, 91, 364, 1001, 2002, 3003, 3432, 3003, 2002, 1001, 364, 91, 14, 1},
    {1, 15, 105, 455, 1365, 3003, 5005, 6435, 6435, 5005, 3003, 1365, 455, 105, 15, 1},
    {1, 16, 120, 560, 1820, 4368, 8008, 11440, 12870, 11440, 8008, 4368, 1820, 560, 120, 16, 1}};
__device__ __forceinline__ unsigned long long binom(int k, int w) {
  return (w < 0 || w > k) ? 0ull : (unsigned long long)kBinom[k][w];
}

// The descriptor of a list entry's array.
__device__ __forceinline__ const ArrayDesc& desc_of(const GsLaunch& L, int array) {
  return L.table ? L.table[array] : L.one;
}

// ---------------------------------------------------------------------------
// (a0) raster constants of a block: c(ix, iy) = c0 + ix du + iy dw with
// c0 = s Cgd (V0 + x0 u + y0 w), du = s Cgd u dx, dw = s Cgd w dy, formed in
// double-float FP32 from FP64 inputs (one FP64 rounding per input, no FP64
// dependency chains: FP64 issues at a small fraction of the FP32 rate here).
// Used when the host could not precompute them (model updated on the GPU).
// ---------------------------------------------------------------------------
__device__ inline void raster_consts(const ModelData* md, int n, int ng, const Scan& sc,
                                     double carrier, df* sV, df* sU, df* sW, df* c0,
                                     df* du, df* dw) {
  for (int g = threadIdx.x; g < ng; g += blockDim.x) {
    sV[g] = df_from_double(sc.V0[g] + sc.x0 * sc.u[g] + sc.y0 * sc.w[g]);
    sU[g] = df_from_double(sc.u[g] * sc.dx);
    sW[g] = df_from_double(sc.w[g] * sc.dy);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 3 * n; e += blockDim.x) {
    const int i = e % n, which = e / n;
    const df* vec = which == 0 ? sV : (which == 1 ? sU : sW);
    df acc = {0.f, 0.f};
    for (int g = 0; g < ng; ++g)
      acc = df_add(acc, df_mul(df_from_double(carrier * md->Cgd[i * ng + g]), vec[g]));
    (which == 0 ? c0 : (which == 1 ? du : dw))[i] = acc;
  }
}

// Block sum of per-thread counts (all threads must call; result in thread 0).
template <typename U>
__device__ __forceinline__ U block_sum(U v, U* red) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(kFull, v, off);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  U t = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
  return t;
}

// Launch with programmatic stream serialisation (the kernel waits for its
// predecessor's results with grid_dep_wait).
template <typename... KArgs>
inline cudaError_t launch_dependent(void (*kern)(KArgs...), unsigned grid, unsigned block,
                                    cudaStream_t st, KArgs... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// ---------------------------------------------------------------------------
// prep stage: shared state of a block and the per-array set-up
// ---------------------------------------------------------------------------
// Point lists with at most this many gates take c from a staged s Cgd and
// voltages converted once per pixel by the team (one gate per lane).
constexpr int kPointGates = 16;
struct PrepShared {
  ModelConsts cs;
  df sc0[kMaxDot], sdu[kMaxDot], sdw[kMaxDot];
  df sG[kMaxDot][kPointGates];     // point lists of <= kPointGates gates: s Cgd
  __align__(16) float qK[kPrepThreads][kQPRow];  // team QP: factor rows, active lists, unknowns, c
  int qa[kPrepThreads];
  float qz[kPrepThreads];
  float qzl[kPrepThreads];
  float qx[kPrepThreads];
  float qc[kPrepThreads];
  unsigned long long red64[kPrepThreads / 32];
  unsigned red32[kPrepThreads / 32];
  float th0;  // the threshold test's half-width t / 2 in FP32
  int tlt1;   // t < 1
};

// Stage an array's FP32 model constants and raster constants (all threads);
// one thread converts the FP64 threshold for the whole block.
__device__ inline void prep_stage_array(const ArrayDesc& a, PrepShared& sh) {
  stage_consts(&a.md->k, &sh.cs);
  if (threadIdx.x == 0) {
    sh.th0 = __double2float_rn(0.5 * a.mt.t);
    sh.tlt1 = a.mt.t < 1.0 ? 1 : 0;
  }
  if (a.sc.kind == 1 && a.ng <= kPointGates && a.prep_team >= a.ng) {
    for (int e = threadIdx.x; e < a.n * a.ng; e += blockDim.x) {
      const int i = e / a.ng, g = e - i * a.ng;
      sh.sG[i][g] = df_from_double(a.mt.carrier * a.md->Cgd[i * a.ng + g]);
    }
  }
  if (a.sc.kind == 0) {
    bool form = a.rk.gen == 0u;  // on the device
    if (!form) {
      if (threadIdx.x < kMaxDot) {
        sh.sc0[threadIdx.x] = a.rk.c0[threadIdx.x];
        sh.sdu[threadIdx.x] = a.rk.du[threadIdx.x];
        sh.sdw[threadIdx.x] = a.rk.dw[threadIdx.x];
      }
      // of another host copy than the model's?  (The load costs a call 0.6 - 1.5
      // us: only where the model may have changed.)
      if (!a.rk.current) form = a.rk.gen != a.md->k.gen;
    }
    if (form) {
      // (its voltage vectors in the QP rows, which no pixel uses yet)
      static_assert(sizeof(sh.qK) >= 3 * kMaxGate * sizeof(df), "room for V0, u, w");
      df* v = reinterpret_cast<df*>(&sh.qK[0][0]);
      raster_consts(a.md, a.n, a.ng, a.sc, a.mt.carrier, v, v + kMaxGate, v + 2 * kMaxGate,
                    sh.sc0, sh.sdu, sh.sdw);
    }
  }
  __syncthreads();
}

// c of a point-list pixel by its team (out of line: the raster kernels carry
// only the call): lane g converts V_g to double-float once for the team,
// through the team's scratch rows, and each live lane sums its dot's row of
// the staged s Cgd, the same operations in the same order as point_c.
// Every lane of tmask must call; ng <= the team's lanes.
static __device__ __noinline__ df point_c_team(const double* Vp, int ng, bool active, bool live,
                                               int lt, unsigned tmask,
                                               const df (*sG)[kPointGates], float* qx,
                                               float* qz) {
  const int tq = (int)threadIdx.x - lt;
  df vg = {0.f, 0.f};
  if (active && lt < ng) vg = df_from_double(Vp[lt]);
  qx[threadIdx.x] = vg.hi;
  qz[threadIdx.x] = vg.lo;
  __syncwarp(tmask);
  df acc = {0.f, 0.f};
  if (live)
    for (int g = 0; g < ng; ++g) acc = df_add(acc, df_mul(sG[lt][g], df{qx[tq + g], qz[tq + g]}));
  __syncwarp(tmask);
  return acc;
}

// Per-block totals of the prep stage (thread 0's copy is the block's).
struct PrepAcc {
  unsigned long long candidates = 0;
  unsigned qp = 0, doubled = 0;
};

// ---------------------------------------------------------------------------
// (a1)-(a4) for one pixel: induced charge, continuous minimum and candidate
// set (prep_set), h = M (base - c) and S (prep_h).  A team of TP lanes (a power of two >= N, at most 16)
// prepares one pixel, lane i owning dot i; team-wide sums, ballots and gathers
// use shuffles restricted to the team's lanes, so teams of one warp may
// diverge.  Every lane of the team must call; a team without a pixel passes
// active = false.  Per lane: c, x and base of its dot (and whether the dot is
// live); per team: the rest.
// ---------------------------------------------------------------------------
struct PrepPixel {
  df c, x;
  int base;
  bool live;
  unsigned mask;   // ambiguous dots
  int w;           // closed: candidate weight; open: -1
  unsigned flags;
  unsigned qp_set; // QP pixels: the active set the QP settled on
};

template <bool CLOSED, int W = 0>
__device__ __forceinline__ PrepPixel prep_set(const ArrayDesc& a, PrepShared& sh, long long p,
                                              bool active) {
  const int n = a.n;
  const float bx_qp_scale = a.bx_qp_scale > 0.f ? a.bx_qp_scale : sh.cs.bx_qp_scale;
  const bool model_bad = sh.cs.model_bad != 0;

  const int TP = W ? W : a.prep_team;  // W: the team width where it is known
  const int lt = threadIdx.x & (TP - 1);
  const int lane = threadIdx.x & 31;
  const int tbase = lane & ~(TP - 1);                   // team's first lane
  const unsigned tmask = (TP == 32 ? 0xffffffffu : ((1u << TP) - 1u)) << tbase;
  const bool live = active && lt < n;
  const int nhat = a.mt.n_charges;

  // team reductions over lanes (dead lanes contribute zero)
  auto tmax_f = [&](float v) {
    for (int off = 1; off < TP; off <<= 1) v = fmaxf(v, __shfl_xor_sync(tmask, v, off, TP));
    return v;
  };
  auto tsum_i = [&](int v) {
    for (int off = 1; off < TP; off <<= 1) v += __shfl_xor_sync(tmask, v, off, TP);
    return v;
  };
  auto tsum_df = [&](df v) {
    for (int off = 1; off < TP; off <<= 1) {
      df o;
      o.hi = __shfl_xor_sync(tmask, v.hi, off, TP);
      o.lo = __shfl_xor_sync(tmask, v.lo, off, TP);
      v = df_add(v, o);
    }
    return v;
  };
  auto tballot = [&](bool pred) { return (__ballot_sync(tmask, pred) & tmask) >> tbase; };

  // (a1) c_i; a point list of at most one gate per lane: lane g converts the
  // pixel's V_g to double-float once for the team (the team's scratch rows),
  // then each lane sums its dot's row of the staged s Cgd -- the same
  // operations in the same order as point_c, without the per-lane FP64
  // conversions
  df c = {0.f, 0.f};
  if (a.sc.kind == 1 && a.ng <= kPointGates && TP >= a.ng) {
    c = point_c_team(a.sc.V + (active ? p : 0) * a.ng, a.ng, active, live, lt, tmask, sh.sG,
                     sh.qx, sh.qz);
  } else if (live) {
    if (a.sc.kind == 0) {
      int ix, iy;
      if (a.sc.P <= 0xffffffffLL) {  // 32-bit division when the raster allows it
        const unsigned pu = (unsigned)p, width = (unsigned)a.sc.W;
        iy = (int)(pu / width);
        ix = (int)(pu - (unsigned)iy * width);
      } else {
        ix = (int)(p % a.sc.W);
        iy = (int)(p / a.sc.W);
      }
      c = raster_c(sh.sc0[lt], sh.sdu[lt], sh.sdw[lt], ix, iy);
    } else {
      c = point_c(&a.md->Cgd[lt * a.ng], &a.sc.V[p * a.ng], a.ng, a.mt.carrier);
    }
  }
  // (a2) analytic continuous minimum (Appendix C / D)
  df x = c;
  if (CLOSED) {
    const df csum = tsum_df(c);
    const df lam = df_sub({(float)nhat, 0.f}, csum);  // N_hat <= 2^24
    if (live) x = df_add(c, df_mul(lam, sh.cs.vs[lt]));
  }
  const unsigned A =
      tballot(live && (x.hi < 0.f || (x.hi == 0.f && x.lo < 0.f)));
  unsigned flags = 0u;
  unsigned qp_set = 0u;
  float bx = a.bx_analytic;
  // (a3) QP where the analytic minimum is infeasible, by the pixel's team
  const bool need = A != 0u && !(CLOSED && nhat == 0);  // team-uniform
  const int tb = threadIdx.x - lt;
  float scale = 1.f;
  if (A) {
    flags |= kFlagQP;
    const float cmax = tmax_f(live ? fabsf(c.hi + c.lo) : 0.f);
    if (need) {
      scale = 1.f + cmax + (float)nhat;
      bx = fmaxf(bx, bx_qp_scale * scale);
    } else {
      x = {0.f, 0.f};
    }
  }
  float xf = 0.f;
  unsigned Af = 0u;
  int st = 0;
  // open array with one negative c_a (every QP pixel of the 16-dot diagram):
  // the active set {a} solved in place -- z_a = -c_a / Cdd_aa through the
  // same reciprocal square root, x_i = c_i + Cdd_ia z_a -- with the same
  // operations, results and shared state (factor, active list, multiplier)
  // as the team QP's first iteration; it stands when no other x_i is below
  // -tol, else the team QP runs from {a}
  bool solved = false;
  if (!CLOSED && need && __popc(A) == 1) {
    const int ad = __ffs(A) - 1;
    const float cl = live ? c.hi + c.lo : 0.f;
    const float ca = __shfl_sync(tmask, cl, ad, TP);
    const float caa = sh.cs.Cdd[ad * kLdM + ad];
    const float r = caa > 0.f ? rsqrtf(caa) : 0.f;
    const float zf = (-ca * r) * r;
    float xi = 0.f;
    if (live && lt != ad) xi = cl + sh.cs.Cdd[lt * kLdM + ad] * zf;
    const float tolq = 0.25f * bx_qp_scale * scale;
    solved = r > 0.f && tballot(live && lt != ad && xi < -tolq) == 0u;
    if (solved) {
      if (lt == 0) {
        sh.qa[tb] = ad;
        sh.qz[tb] = zf;
        sh.qK[tb][0] = caa * r;
        sh.qK[tb][kQPRow - 1] = r;
      }
      xf = (live && lt != ad) ? (xi > 0.f ? xi : 0.f) : 0.f;
      Af = A;
      __syncwarp(tmask);
    }
  }
  if (need && !solved)
    st = qp_team<float, CLOSED>(n, lt, TP, tmask, tb, sh.cs.Cdd, kLdM, sh.cs.sv, sh.cs.s_s,
                                live ? c.hi + c.lo : 0.f, (float)nhat, A,
                                0.25f * bx_qp_scale * scale, 4 * n + 4, sh.qK, sh.qa, sh.qz,
                                sh.qc, xf, Af);
  if (need) {
    // the FP32 solution stands when its active set is certain at FP32
    // precision (every free x_i and every multiplier more than twice the
    // FP32 margin above zero) and no floor or threshold decision lies
    // within that margin; otherwise one double-float refinement follows
    bool sure = st == 0;
    if (sure && live) {
      if ((Af >> lt) & 1u) {
        sure = sh.qz[tb + __popc(Af & ((1u << lt) - 1u))] > 2.f * bx;
      } else {
        const float fr = xf - floorf(xf);
        sure = xf > 2.f * bx && !(xf >= 0.5f - bx && fminf(fr, 1.f - fr) < bx) &&
               !(sh.tlt1 && fabsf(fabsf(fr - 0.5f) - sh.th0) < bx);
      }
    }
    sure = tballot(!sure) == 0u;
    if (st != 0) {
      flags |= kFlagQPCap;
      if (live) x = {xf, 0.f};
    } else if (sure) {
      if (live) x = {xf, 0.f};
      qp_set = Af;
    } else {
      // one double-float refinement: the margin shrinks to the square of
      // the FP32 one; a multiplier or free x_i below -margin at that
      // precision leaves the active set (and x) to the FP64 recheck
      const float bx2 = fmaxf(a.bx_analytic, sh.cs.bx_qp_scale2 * scale);
      df xr;
      unsigned flip = 0u;
      int bad = qp_team_refine<CLOSED>(n, lt, TP, tmask, tb, sh.cs.Cdd, sh.cs.CddLo, sh.cs.sv2,
                                       live ? c : df{0.f, 0.f}, (float)nhat, Af, 0.25f * bx2,
                                       sh.qK, sh.qa, sh.qz, sh.qzl, sh.qx, xr, flip);
      // a sign violation below FP32 resolution (a nearly degenerate vertex:
      // a multiplier or free x_i within rounding of zero): one more round
      // with those constraints toggled -- the FP32 factor and solve of that
      // active set, and its double-float refinement -- before the FP64
      // recheck is left to settle the pixel
      const unsigned A2 = (Af ^ flip) & ((n < 32 ? (1u << n) : 0u) - 1u);
      if (bad && flip && A2 != Af && !(CLOSED && __popc(A2) == n)) {
        float xf2 = 0.f;
        unsigned Af2 = 0u;
        const int st2 = qp_team<float, CLOSED>(n, lt, TP, tmask, tb, sh.cs.Cdd, kLdM, sh.cs.sv,
                                               sh.cs.s_s, live ? c.hi + c.lo : 0.f, (float)nhat,
                                               A2, 0.25f * bx_qp_scale * scale, 1, sh.qK, sh.qa,
                                               sh.qz, sh.qc, xf2, Af2);
        if (st2 == 0) {
          Af = Af2;
          bad = qp_team_refine<CLOSED>(n, lt, TP, tmask, tb, sh.cs.Cdd, sh.cs.CddLo, sh.cs.sv2,
                                       live ? c : df{0.f, 0.f}, (float)nhat, Af, 0.25f * bx2,
                                       sh.qK, sh.qa, sh.qz, sh.qzl, sh.qx, xr, flip);
        }
      }
      if (live) x = xr;
      if (bad) flags |= kFlagBoundary;
      else bx = bx2;
      // closed with every dot but one active: the sum constraint makes the
      // relaxed minimum the vertex N_hat e_j exactly, so once every
      // multiplier is certainly positive no rounding error is left in x
      // and the floor decisions need no margin
      if (CLOSED && !bad && __popc(Af) == n - 1) {
        const bool zpos = lt >= n - 1 || sh.qz[tb + lt] + sh.qzl[tb + lt] > 0.25f * bx2;
        if (tballot(!zpos) == 0u) {
          if (live) x = ((Af >> lt) & 1u) ? df{0.f, 0.f} : df{(float)nhat, 0.f};
          bx = 0.f;
        }
      }
      qp_set = Af;
    }
    __syncwarp(tmask);
  }

  // (a4) candidate set; the closed doubling loop is team-uniform (its first
  // pass takes t / 2 and t < 1 from the block's staging, later ones double t
  // in FP64)
  double tt = a.mt.t;
  float th = sh.th0;
  bool tlt1 = sh.tlt1 != 0;
  unsigned mask = 0u;
  int w = -1, base = 0;
  bool amb = false;
  for (int iter = 0; iter < 40; ++iter) {
    bool bnd = false;
    if (live) {
      df xi = x;
      if (xi.hi < 0.f || (xi.hi == 0.f && xi.lo < 0.f)) xi = {0.f, 0.f};
      float fl = floorf(xi.hi);
      if (xi.hi == fl && xi.lo < 0.f) fl -= 1.f;
      const float fr = __fadd_rn(__fsub_rn(xi.hi, fl), xi.lo);
      amb = fabsf(fr - 0.5f) <= th;
      base = (int)fl + ((!amb && fr >= 0.5f) ? 1 : 0);
      bnd = (xi.hi >= 0.5f - bx && fminf(fr, 1.f - fr) < bx) ||
            (tlt1 && fabsf(fabsf(fr - 0.5f) - th) < bx);
    }
    if (tballot(bnd)) flags |= kFlagBoundary;
    mask = tballot(live && amb);
    if (!CLOSED) break;
    const int sum = tsum_i(live ? base : 0);
    w = nhat - sum;
    if (w >= 0 && w <= __popc(mask)) break;
    if (!tlt1) {  // t = 1 and still infeasible: impossible in exact arithmetic, settle in FP64
      flags |= kFlagBoundary;
      w = w < 0 ? 0 : __popc(mask);
      break;
    }
    tt = (tt <= 0.0) ? 1.0 : fmin(2.0 * tt, 1.0);
    th = __double2float_rn(0.5 * tt);
    tlt1 = tt < 1.0;
    flags |= kFlagDoubled;
  }
  if (model_bad) flags |= kFlagUnresolved;
  return {c, x, base, live, mask, w, flags, qp_set};
}

// The second half: h of the lane's dot (returned) and S, the sum of the
// magnitudes entering a candidate's energy (per team).
template <int W = 0>
__device__ __forceinline__ float prep_h(const ArrayDesc& a, PrepShared& sh, const PrepPixel& q,
                                        float& S) {
  const int n = a.n;
  const float* sMhi = sh.cs.Mhi;
  const float* sMlo = sh.cs.Mlo;
  const int TP = W ? W : a.prep_team;
  const int lt = threadIdx.x & (TP - 1);
  const int tbase = threadIdx.x & 31 & ~(TP - 1);
  const unsigned tmask = (TP == 32 ? 0xffffffffu : ((1u << TP) - 1u)) << tbase;
  const bool live = q.live, amb = q.live && ((q.mask >> lt) & 1u);
  const unsigned mask = q.mask;
  // h_i = (M (base - c))_i, r = base - c in double-float staged in the
  // team's rows of qx / qz (free after the QP); the products' high parts are
  // summed error-free and their low parts and rounding errors in plain FP32
  // (error O(u^2) of sum |M_ij r_j|, far below the final rounding of h to
  // FP32).  Four columns per step with their loads issued together and two
  // independent sums (even and odd columns), joined error-free at the end.
  const df r = df_sub({(float)q.base, 0.f}, q.c);
  const int tb0 = threadIdx.x - lt;
  __syncwarp(tmask);
  sh.qx[threadIdx.x] = r.hi;
  sh.qz[threadIdx.x] = r.lo;
  __syncwarp(tmask);
  const float* Mrow = sMhi + lt * kLdM;
  const float* Mrowl = sMlo + lt * kLdM;
  float h = 0.f;
  if (live) {
    float shi[2] = {0.f, 0.f}, slo[2] = {0.f, 0.f};
    for (int j0 = 0; j0 < n; j0 += 4) {
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        const int j = j0 + jj;
        const bool on = j < n;
        const int jc = on ? j : 0;
        const float mh = on ? Mrow[jc] : 0.f, ml = on ? Mrowl[jc] : 0.f;
        const float xh = sh.qx[tb0 + jc], xl = sh.qz[tb0 + jc];
        const df pr = two_prod(mh, xh);
        const float small = __fmaf_rn(mh, xl, __fmaf_rn(ml, xh, pr.lo));
        const df sm = two_sum(shi[jj & 1], pr.hi);
        shi[jj & 1] = sm.hi;
        slo[jj & 1] = __fadd_rn(slo[jj & 1], __fadd_rn(sm.lo, small));
      }
    }
    const df st = two_sum(shi[0], shi[1]);
    h = st.hi + (st.lo + (slo[0] + slo[1]));
  }
  // S_i = |h_i| + M_ii / 2 + sum over the ambiguous j < i of |M_ij|: the
  // row's precomputed prefix when every j < i is ambiguous, else four columns
  // per step with two independent sums
  float Si = 0.f;
  const unsigned below = mask & ((1u << lt) - 1u);
  if (live && amb && below == (1u << lt) - 1u) {
    Si = fabsf(h) + sh.cs.absl[lt];
  } else if (live && amb) {
    float sp[2] = {fabsf(h) + 0.5f * Mrow[lt], 0.f};
    for (int j0 = 0; j0 < n; j0 += 4) {
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        const int j = j0 + jj;
        sp[jj & 1] += ((below >> j) & 1u) ? fabsf(Mrow[j < n ? j : 0]) : 0.f;
      }
    }
    Si = sp[0] + sp[1];
  }
  for (int off = 1; off < TP; off <<= 1) Si += __shfl_xor_sync(tmask, Si, off, TP);
  S = Si;
  return h;
}

// The FP32 gap below which a pixel's best two candidates are a near tie.
__device__ __forceinline__ float pixel_bound(const ArrayDesc& a, float S, int k) {
  // the pruned search walks a shallower middle level than the resolve's
  // re-walk (kCheckL2), which shortlists by this bound, and forms each
  // rest state from up to kBnbItBits + 2 more table sums
  return bnb_search(a.cfg.L1, a.cfg.L2)
             ? near_tie_bound(S, k, max(a.cfg.L2, kCheckL2), kBnbItBits + 2)
             : near_tie_bound(S, k, a.cfg.L2);
}

// The pixel's record, for the search and the list kernels (lane lt its dot).
template <bool CLOSED>
__device__ __forceinline__ void store_record(PixRec* rec, const PrepPixel& q, int lt, float h,
                                             float bound) {
  if (q.live) {
    rec->h[lt] = h;
    rec->chi[lt] = q.c.hi;
    rec->clo[lt] = q.c.lo;
    rec->base[lt] = (short)q.base;
  }
  if (lt == 0) {
    rec->mask = (unsigned short)q.mask;
    rec->k = (unsigned char)__popc(q.mask);
    rec->w = (signed char)(CLOSED ? q.w : -1);
    rec->flags = (unsigned char)q.flags;
    rec->qpA = (unsigned short)q.qp_set;
    rec->bound = bound;
  }
}

// prep_set and prep_h for one block's pixels team_base + threadIdx.x / TP below p_end,
// their records and counts.  All threads of the block must call (block
// reductions at the end).
template <bool CLOSED>
__device__ inline void prep_tile(const ArrayDesc& a, PrepShared& sh, long long team_base,
                                 long long p_end, PrepAcc& tot) {
  const int TP = a.prep_team;
  const int lt = threadIdx.x & (TP - 1);
  const long long p = team_base + threadIdx.x / TP;
  const bool active = p < p_end;
  const PrepPixel q = prep_set<CLOSED>(a, sh, p, active);
  float S;
  const float h = prep_h(a, sh, q, S);
  const int k = __popc(q.mask);
  if (active) store_record<CLOSED>(a.recs + p, q, lt, h, pixel_bound(a, S, k));
  unsigned long long my_cand = 0;
  unsigned my_qp = 0, my_doubled = 0;
  if (active && lt == 0) {
    my_cand = CLOSED ? binom(k, q.w) : (1ull << k);
    my_qp = (q.flags & kFlagQP) ? 1u : 0u;
    my_doubled = (q.flags & kFlagDoubled) ? 1u : 0u;
  }
  __syncwarp();
  // one block sum of the three counts packed in 64 bits: candidates in the
  // low 32 (a block prepares 128 / TP pixels of at most 2^N candidates with
  // TP >= N, below 2^20 in all), QP and doubled pixels (<= 128) above
  const unsigned long long packed = block_sum(
      my_cand | ((unsigned long long)my_qp << 32) | ((unsigned long long)my_doubled << 48),
      sh.red64);
  if (threadIdx.x == 0) {
    tot.candidates += packed & 0xffffffffull;
    tot.qp += (unsigned)((packed >> 32) & 0xffffu);
    tot.doubled += (unsigned)(packed >> 48);
  }
}

// ---------------------------------------------------------------------------
// search stage: shared state of a block
// ---------------------------------------------------------------------------
// Three layouts share the space: teams narrower than kTeamFinishMin keep a
// slot table per thread; block-level teams one per team with their walk
// tables; the pruned search (teams of kBnbMinT+ lanes) its bound tables.
constexpr int kTeamsTF = kSearchThreads / kTeamFinishMin;
constexpr int kTeamsBnb = kSearchThreads / kBnbMinT;
struct SearchShared {
  ModelConsts cs;
  union {
    struct {
      int sdot[kSearchThreads][kMaxDot];
      float sh[kSearchThreads][kMaxDot];
    } lane;
    struct {
      int sdot[kTeamsTF][kMaxDot];
      float sh[kTeamsTF][kMaxDot];
      __align__(16) float colt[kTeamsTF][4 * kColStride];
      __align__(16) float itab[kTeamsTF][(1 << kItMax) * kItStride];
      __align__(16) float cslot[kSearchThreads][kItMax];
    } team;
    struct {
      int sdot[kTeamsBnb][kMaxDot];
      float sh[kTeamsBnb][kMaxDot];
      int slot_of[kTeamsBnb][kMaxDot];  // slot of each ambiguous dot
      float pm[kTeamsBnb][kMaxDot * kLdM];
      float vv[kTeamsBnb][kMaxDot];
      __align__(16) float itab[kTeamsBnb][(1 << kBnbItBits) * kBnbStride];
      __align__(16) float ltab[kSearchThreads][kBnbLane];
      __half lb[kTeamsBnb][kBnbStates];
      unsigned short rbuf[kTeamsBnb][kBnbBuf];
      float rlb[kTeamsBnb][kBnbBuf];
      __align__(16) float ptab[kTeamsBnb][1 << kBnbL1];
    } bnb;
  } u;
  unsigned long long red64[kSearchThreads / 32];
  unsigned red32[kSearchThreads / 32];
};

struct SearchAcc {
  unsigned long long evaluated = 0;
  unsigned near_tie = 0, boundary = 0, overflow = 0;
};

// A block that prepares and then searches its own tile holds the two stages'
// scratch in one place; the model constants, first in both, are staged once.
union GsShared {
  PrepShared p;
  SearchShared s;
};
static_assert(offsetof(PrepShared, cs) == 0 && offsetof(SearchShared, cs) == 0,
              "the model constants open both stages' shared state");
static_assert(kPrepThreads == kSearchThreads, "one block size for both stages");

// ---------------------------------------------------------------------------
// (a5)-(a6), (a8) for one tile: candidate search, top-two selection, outputs.
// A team of T lanes (the array's cfg.T) searches one pixel; pixels
// team_base + threadIdx.x / T below p_end.  Pixels whose candidate set is in
// doubt go on the FP64 recheck list, near ties on the resolve list.  All
// threads of the block must call.
// ---------------------------------------------------------------------------
template <int L1, int L2, bool CLOSED, bool TF>
__device__ inline void search_tile(const GsLaunch& L, const ArrayDesc& a, SearchShared& sh,
                                   int array, long long team_base, long long p_end,
                                   SearchAcc& acc) {
  const int n = a.n;
  const float* sM = sh.cs.Mhi;
  const float* sMlo = sh.cs.Mlo;

  const int T = a.cfg.T;
  const int team = threadIdx.x / T, lt = threadIdx.x % T;
  const long long p = team_base + team;
  const bool active = p < p_end;
  const PixRec* rec = a.recs + (active ? p : 0);
  const unsigned mask = active ? rec->mask : 0u;
  const int k = __popc(mask);
  // BNB: the pruned search (5 + 2 split, teams of kBnbMinT+ lanes, which
  // the host guarantees for this split)
  constexpr bool BNB = TF && bnb_search(L1, L2);
  int* sdot = BNB ? sh.u.bnb.sdot[team] : TF ? sh.u.team.sdot[team] : sh.u.lane.sdot[team];
  float* sht = BNB ? sh.u.bnb.sh[team] : TF ? sh.u.team.sh[team] : sh.u.lane.sh[team];
  int* slot_of = BNB ? sh.u.bnb.slot_of[team] : nullptr;
  if (BNB) {
    // slot s = the ambiguous dot of rank s by |h_i + M_ii / 2|, ascending
    // (ties by dot index): the least certain dots are walked, the most
    // certain ones are the outer slots the bounds prune
    if (active)
      for (int i = lt; i < n; i += T)
        sht[i] = ((mask >> i) & 1u) ? fabsf(rec->h[i] + 0.5f * sM[i * kLdM + i]) : 0.f;
    __syncwarp();
    int rank = -1;
    if (active && lt < n && ((mask >> lt) & 1u)) {
      const float key = sht[lt];
      rank = 0;
      for (int j = 0; j < n; ++j) {
        const float kj = sht[j];
        rank += (((mask >> j) & 1u) && (kj < key || (kj == key && j < lt))) ? 1 : 0;
      }
    }
    __syncwarp();
    if (rank >= 0) {
      sdot[rank] = lt;
      sht[rank] = rec->h[lt];
      slot_of[lt] = rank;
    }
  } else if (active) {
    // slot table of the pixel: slot s = the s-th ambiguous dot (lanes in parallel)
    for (int i = lt; i < n; i += T)
      if ((mask >> i) & 1u) {
        const int s = __popc(mask & ((1u << i) - 1u));
        sdot[s] = i;
        sht[s] = rec->h[i];
      }
  }
  __syncwarp();
  float m1 = kInf, m2 = kInf;
  unsigned b1 = 0u;
  unsigned long long ev = 0;
  const SlotView sv{sdot, sht, active ? k : 0, active ? (int)rec->w : -1};
  // TF (teams of 8 or more lanes): search at block level and finish the
  // winning block together; smaller teams finish each lane's best block in
  // the lane.
  float* colt = (TF && !BNB) ? sh.u.team.colt[team] : nullptr;
  float* itab = (TF && !BNB) ? sh.u.team.itab[team] : nullptr;
  if (TF && !BNB) {
    static_assert(L2 <= 4 && L1 + L2 <= kColStride, "column table layout");
    if (active) {
      col_build<L1, L2>(sM, sv, lt, T, colt);
      if (L1 + L2 >= 9) iter_build<L1, L2>(sM, sv, lt, T, itab);
    }
    __syncwarp();
  }
  if (active) {
    if constexpr (BNB) {
      const unsigned wl = threadIdx.x & 31u;
      const unsigned tmask =
          T >= 32 ? kFull : (((1u << T) - 1u) << (wl & ~(unsigned)(T - 1)));
      search_bnb<CLOSED>(sM, sv, lt, T, tmask, rec->bound, sh.cs.qneg, sh.u.bnb.pm[team],
                 sh.u.bnb.vv[team], sh.u.bnb.itab[team],
                 sh.u.bnb.ltab[team * T], sh.u.bnb.lb[team], sh.u.bnb.rbuf[team],
                 sh.u.bnb.rlb[team], sh.u.bnb.ptab[team], m1, b1, m2, ev);
    } else {
      search_lane<L1, L2, CLOSED, false, TF>(sM, sv, lt, T, 0.f, nullptr, nullptr, 0u, m1, b1,
                                             m2, ev, colt, itab,
                                             TF ? sh.u.team.cslot[threadIdx.x] : nullptr);
    }
  }
  // best (block or candidate) with its id, and the second-best minimum
  for (int off = 1; off < T; off <<= 1) {
    const float om1 = __shfl_xor_sync(kFull, m1, off);
    const unsigned ob1 = __shfl_xor_sync(kFull, b1, off);
    const float om2 = __shfl_xor_sync(kFull, m2, off);
    top2_merge(m1, b1, m2, om1, ob1, om2);
  }
  // candidate level inside the winning block, by the whole team; every lane
  // of the warp takes part (the finish shuffles over the full warp), teams
  // without a pixel or without a block keep their result
  if (TF) {
    float e1, e2;
    unsigned bits;
    team_finish<L1, L2, CLOSED>(sM, sv, lt, T, kFull, m1 < kInf ? b1 : 0u, e1, bits, e2);
    if (m1 < kInf) {
      m1 = e1;
      b1 = bits;
      m2 = fminf(m2, e2);
    }
  }

  // epilogue: n* = base + bits and r = n* - c in double-float, one lane per
  // dot, kept in the team's slot-table rows (dead after the finish: r.hi in
  // sh, the bits of r.lo in sdot); then U(n*) = 1/2 r^T M r with the team's
  // lanes splitting the rows.  A row's products M_ij r_j are summed with
  // error-free sums of their high parts and plain FP32 sums of the rounding
  // errors and low-order parts, whose own error is O(u^2) of the row's
  // magnitude, then renormalised to double-float.
  df u = {0.f, 0.f};
  unsigned flags = 0u;
  __syncwarp();
  float* rhi = sht;
  int* rlo = sdot;
  // int8 maps of 4, 8 or 16 dots with a lane per dot: the team's charges go
  // out as one 4-, 8- or 16-byte store per pixel (the same for every team of
  // the launch, so the shuffles below are warp-uniform)
  const bool vec = !a.out_n16 && (n == 4 || n == 8 || n == 16) && T >= n &&
                   (reinterpret_cast<uintptr_t>(a.out_n) & (uintptr_t)(n - 1)) == 0;
  unsigned word = 0u;
  // the record's flags and bound, and the lane's dots' base and c, four dots
  // at a time: their loads are issued together (one round trip to L2)
  const unsigned rflags = active ? rec->flags : 0u;
  const float rbound = active ? rec->bound : 0.f;
  if (active) {
    for (int i0 = lt; i0 < n; i0 += 4 * T) {
      int bq[4];
      float chq[4], clq[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = i0 + q * T;
        const int ic = i < n ? i : i0;
        bq[q] = rec->base[ic];
        chq[q] = rec->chi[ic];
        clq[q] = rec->clo[ic];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = i0 + q * T;
        if (i >= n) continue;
        int ni = bq[q];
        if ((mask >> i) & 1u) {
          const int si = BNB ? slot_of[i] : __popc(mask & ((1u << i) - 1u));
          ni += (int)((b1 >> si) & 1u);
        }
        const df ri = df_sub({(float)ni, 0.f}, {chq[q], clq[q]});
        rhi[i] = ri.hi;
        rlo[i] = __float_as_int(ri.lo);
        if (vec) {
          if (ni > 127) { ni = 127; flags |= kFlagOverflow; }
          word = (unsigned)ni << (8 * (lt & 3));
        } else {
          store_charge(a, p * n + i, ni, flags);
        }
      }
    }
  }
  if (vec) {
    // bytes of lanes 4q .. 4q + 3 into word q (held by all four), then lane 0
    // of the team gathers the words and stores them
    word |= __shfl_xor_sync(kFull, word, 1);
    word |= __shfl_xor_sync(kFull, word, 2);
    const int tb = (int)(threadIdx.x & 31u) & ~(T - 1);
    const unsigned w1 = __shfl_sync(kFull, word, (tb + 4) & 31);
    const unsigned w2 = __shfl_sync(kFull, word, (tb + 8) & 31);
    const unsigned w3 = __shfl_sync(kFull, word, (tb + 12) & 31);
    if (active && lt == 0) {
      int8_t* dst = a.out_n + p * n;
      if (n == 16) *reinterpret_cast<int4*>(dst) = make_int4((int)word, (int)w1, (int)w2, (int)w3);
      else if (n == 8) *reinterpret_cast<int2*>(dst) = make_int2((int)word, (int)w1);
      else *reinterpret_cast<int*>(dst) = (int)word;
    }
  }
  __syncwarp();
  // U = r^T M r.  The pruned search's wide teams (a row per lane) sum full
  // rows, M_ij r_j over j, scaled by r_i.  Narrower teams, whose lanes take
  // several rows each, use the symmetry: U = sum_i r_i S_i with
  // S_i = M_ii r_i + 2 sum_{j > i} M_ij r_j (the upper triangle, 136 products
  // at N = 16 instead of 256); rows i and N - 1 - i pair up to N + 1
  // products, one pair per task, or half a pair when the team has lanes for
  // that; a task's part of each row is summed, scaled by r_i and added to
  // the lane's u.  (Measured: the shorter sums do not pay at 16 lanes, where
  // the pair tasks' extra code costs more than the products they save.)
  if (active && BNB) {
    const int nc = T >= 2 * n ? T / n : 1;
    const int cw = (n + nc - 1) / nc;
    for (int task = lt; task < n * nc; task += T) {
      const int i = task / nc, j0 = (task % nc) * cw, j1 = min(n, j0 + cw);
      float shi = 0.f, slo = 0.f;
      for (int j = j0; j < j1; ++j) {
        const float mh = sM[i * kLdM + j], ml = sMlo[i * kLdM + j];
        const float xh = rhi[j], xl = __int_as_float(rlo[j]);
        const df pr = two_prod(mh, xh);
        const float small = __fmaf_rn(mh, xl, __fmaf_rn(ml, xh, pr.lo));
        const df sm = two_sum(shi, pr.hi);
        shi = sm.hi;
        slo = __fadd_rn(slo, __fadd_rn(sm.lo, small));
      }
      const df acc = fast_two_sum(shi, slo);
      u = df_add(u, df_mul(acc, {rhi[i], __int_as_float(rlo[i])}));
    }
  } else if (active) {
    const int npair = (n + 1) >> 1;
    const int nt = T >= 2 * npair ? 2 : 1;
    for (int task = lt; task < npair * nt; task += T) {
      const int pp = task / nt, hh = task - pp * nt;
      const int q = n - 1 - pp;
      const int len1 = n - pp, len = len1 + (q != pp ? pp + 1 : 0);
      const int mid = (len + 1) >> 1;
      const int e0 = (nt == 2 && hh) ? mid : 0;
      const int e1 = (nt == 2 && !hh) ? mid : len;
      for (int seg = 0; seg < 2; ++seg) {
        const int i = seg ? q : pp;
        const int sa = seg ? max(e0 - len1, 0) : e0;
        const int sb = seg ? e1 - len1 : min(e1, len1);
        if (sb <= sa) continue;
        const int ja = i + sa, jb = i + sb;
        // four columns per step with their loads issued together and two
        // independent sums (even and odd columns), joined error-free at the
        // end; a column past the range adds exact zeros, the off-diagonal
        // ones count twice (an exact scaling)
        float shi[2] = {0.f, 0.f}, slo[2] = {0.f, 0.f};
        for (int jb4 = ja; jb4 < jb; jb4 += 4) {
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const int j = jb4 + jj;
            const bool on = j < jb;
            const int jc = on ? j : ja;
            const float wt = !on ? 0.f : (j == i ? 1.f : 2.f);
            const float mh = wt * sM[i * kLdM + jc], ml = wt * sMlo[i * kLdM + jc];
            const float xh = rhi[jc], xl = __int_as_float(rlo[jc]);
            const df pr = two_prod(mh, xh);
            const float small = __fmaf_rn(mh, xl, __fmaf_rn(ml, xh, pr.lo));
            const df sm = two_sum(shi[jj & 1], pr.hi);
            shi[jj & 1] = sm.hi;
            slo[jj & 1] = __fadd_rn(slo[jj & 1], __fadd_rn(sm.lo, small));
          }
        }
        const df st = two_sum(shi[0], shi[1]);
        const df acc = two_sum(st.hi, __fadd_rn(st.lo, __fadd_rn(slo[0], slo[1])));
        u = df_add(u, df_mul(acc, {rhi[i], __int_as_float(rlo[i])}));
      }
    }
  }
  for (int off = 1; off < T; off <<= 1) {
    df o;
    o.hi = __shfl_xor_sync(kFull, u.hi, off);
    o.lo = __shfl_xor_sync(kFull, u.lo, off);
    u = df_add(u, o);
    flags |= __shfl_xor_sync(kFull, flags, off);
  }
  unsigned my_nt = 0, my_bd = 0, my_ov = 0;
  if (active) {
    flags |= rflags;
    if (!(m2 - m1 > rbound)) flags |= kFlagNearTie;
    if (lt == 0) {
      if (a.out_U) a.out_U[p] = 0.5 * df_to_double(u);
      if (flags & (kFlagBoundary | kFlagQPCap | kFlagUnresolved)) {
        // the candidate set itself may be wrong: FP64 recheck
        const unsigned at = atomicAdd(&L.cnt->n_flag, 1u);
        L.flag_list[at] = ListEntry{array, (int)p, m1, (flags & kFlagNearTie) ? 1 : 0};
        my_bd = 1;
      } else if (flags & kFlagNearTie) {
        // right set, uncertain order: exact energies of the close candidates
        const unsigned at = atomicAdd(&L.cnt->n_tie, 1u);
        L.tie_list[at] = ListEntry{array, (int)p, m1, 0};
        my_nt = 1;
      }
      my_ov = (flags & kFlagOverflow) ? 1u : 0u;
      if (a.out_flags) a.out_flags[p] = (uint8_t)flags;
    }
  }
  // one block sum of the four counts packed in 64 bits: evaluated slots in
  // the low 32 (at most 128 pixels of 2^16 slots per block, 2^23), near-tie,
  // recheck and overflow pixels (<= 128 each) in 10 bits apiece above
  const unsigned long long packed = block_sum(
      ev | ((unsigned long long)my_nt << 32) | ((unsigned long long)my_bd << 42) |
          ((unsigned long long)my_ov << 52),
      sh.red64);
  if (threadIdx.x == 0) {
    acc.evaluated += packed & 0xffffffffull;
    acc.near_tie += (unsigned)((packed >> 32) & 0x3ffu);
    acc.boundary += (unsigned)((packed >> 42) & 0x3ffu);
    acc.overflow += (unsigned)(packed >> 52);
  }
}

// U = r^T M r of the lane's charges ni: a row per lane, as in search_tile's
// wide teams, summed over the team (every lane of tmask calls; rhi, rlo: the
// team's scratch rows).
template <int W>
__device__ __forceinline__ df team_energy(const ModelConsts& cs, int n, int lt, unsigned tmask,
                                          bool live, int ni, df c, float* rhi, float* rlo) {
  const df r = live ? df_sub({(float)ni, 0.f}, c) : df{0.f, 0.f};
  __syncwarp(tmask);
  rhi[lt] = r.hi;
  rlo[lt] = r.lo;
  __syncwarp(tmask);
  df u = {0.f, 0.f};
  if (live) {
    const float* Mh = cs.Mhi + lt * kLdM;
    const float* Ml = cs.Mlo + lt * kLdM;
    float shi = 0.f, slo = 0.f;
    for (int j = 0; j < n; ++j) {
      const float mh = Mh[j], ml = Ml[j];
      const float xh = rhi[j], xl = rlo[j];
      const df pr = two_prod(mh, xh);
      const float small = __fmaf_rn(mh, xl, __fmaf_rn(ml, xh, pr.lo));
      const df sm = two_sum(shi, pr.hi);
      shi = sm.hi;
      slo = __fadd_rn(slo, __fadd_rn(sm.lo, small));
    }
    u = df_mul(fast_two_sum(shi, slo), r);
  }
#pragma unroll
  for (int off = 1; off < W; off <<= 1) {
    df o;
    o.hi = __shfl_xor_sync(tmask, u.hi, off, W);
    o.lo = __shfl_xor_sync(tmask, u.lo, off, W);
    u = df_add(u, o);
  }
  return u;
}

// ---------------------------------------------------------------------------
// (a1)-(a6), (a8) in one pass: a team of W = 4, 8 or 16 lanes, lane i owning
// dot i, prepares a pixel, searches its candidate set and writes its outputs;
// c and the candidate set stay in the lanes.  The search is the sphere search
// where many dots are expected ambiguous, else the enumeration below.  A pixel
// with candidates too close to call, or whose search does not end, gets its
// record and goes on the close list (settle_entry); one whose candidate set is
// in doubt gets its record and goes on the FP64 list.
// What bounds it: instruction issue (1,430 warp instructions per 16-dot pixel
// of the sphere search, 2.4 - 3 a cycle; the tile kernels' 3,061, three
// quarters of them in the FP32 search).  Whole calls, tiles / so: 16 dots
// 100 x 100 60 / 43 us (closed 94 / 52), 16-dot list of 10^4 vectors 76 / 57
// us, 12 dots 400 x 301 243 / 168 us.
// ---------------------------------------------------------------------------
template <int W>
struct PixelShared {
  static constexpr int kTeams = kPrepThreads / W;
  PrepShared p;
  unsigned long long cand[kTeams], ev[kTeams];
  unsigned qp[kTeams], doubled[kTeams], boundary[kTeams], overflow[kTeams];
};
struct SphereShared : PixelShared<kSphT> {
  SphereModel m;
  float4 lev[kTeams][kMaxDot / 2];
};
// The search of a kernel's pixels: the enumeration, the sphere search, or the
// one that a pixel's ambiguous dots call for (a warp's pixels alike: the
// sphere search from kMixedDots on, where the enumeration's 2^k / 256 blocks
// cost more).
enum : int { kPixDense = 0, kPixSphere = 1, kPixMixed = 2 };
constexpr int kMixedDots = 12;
template <int W, int MODE>
struct PixelSharedOf { typedef PixelShared<W> type; };
template <>
struct PixelSharedOf<kSphT, kPixSphere> { typedef SphereShared type; };
template <>
struct PixelSharedOf<kSphT, kPixMixed> { typedef SphereShared type; };
static_assert(kSphT * sizeof(float) * kQPRow >= kSphStack * sizeof(uint2),
              "the team's QP rows hold its waiting nodes");

// Block set-up (all threads), once per array.
__device__ inline void pixel_stage_search(const ArrayDesc& a, SphereShared& sh) {
  sphere_stage(a.md->s, sh.m);
}
template <int W>
__device__ inline void pixel_stage_search(const ArrayDesc&, PixelShared<W>&) {}
template <typename SH>
__device__ inline void pixel_stage_array(const ArrayDesc& a, SH& sh) {
  pixel_stage_search(a, sh);
  prep_stage_array(a, sh.p);  // ends with a barrier
}
template <int W>
__device__ inline void pixel_zero_counts(PixelShared<W>& sh) {
  if (threadIdx.x < sh.kTeams) {
    sh.cand[threadIdx.x] = sh.ev[threadIdx.x] = 0ull;
    sh.qp[threadIdx.x] = sh.doubled[threadIdx.x] = 0u;
    sh.boundary[threadIdx.x] = sh.overflow[threadIdx.x] = 0u;
  }
}
// The block's counts (thread 0 after a barrier).
template <int W>
__device__ inline void pixel_counts(const PixelShared<W>& sh, BlockCounts& prep,
                                    BlockCounts& search) {
  PrepAcc p;
  SearchAcc s;
  for (int t = 0; t < sh.kTeams; ++t) {
    p.candidates += sh.cand[t];
    p.qp += sh.qp[t];
    p.doubled += sh.doubled[t];
    s.evaluated += sh.ev[t];
    s.boundary += sh.boundary[t];
    s.overflow += sh.overflow[t];
  }
  prep.candidates = p.candidates;
  prep.qp = p.qp;
  prep.doubled = p.doubled;
  search.evaluated = s.evaluated;
  search.near_tie = 0u;
  search.boundary = s.boundary;
  search.overflow = s.overflow;
}

// The enumeration: the candidate energies relative to the base,
//     E(b) = sum_{s in b} v_s + sum_{s < s' in b} M_ss',  v = h + M_ss / 2,
// of one pixel by its team.  The first kIn slots are inner (2^kIn energies at
// a time by doubling), the next log2 W the lane's, further ones a loop of the
// whole team; a state of the lane and loop slots is summed from scratch.  Two
// passes: the minimum, then the patterns within G of it (by each lane's best
// block alone unless another block of some lane is that close).  The same
// arguments and results as sphere_search, patterns over the dots; v: the
// dot's single-flip energy; sd, sv, lst: W (lst: 16) words of scratch each.
// What bounds it: instruction issue, about 140 warp instructions a pixel at
// up to kIn + log2 W slots against 320 of the tile kernels' thread per pixel
// or two, which hold 32 pair terms in registers (four blocks per SM).
template <int W, bool CLOSED>
__device__ __forceinline__ unsigned dense_search(const float* sM, int n, int lt, bool active,
                                                 float v, unsigned mask, int w, float G, int* sd,
                                                 float* sv, unsigned* lst, int& close,
                                                 unsigned& evaluated) {
  constexpr int LB = W == 16 ? 4 : W == 8 ? 3 : 2;
  constexpr int kIn = dense_inner(W), NI = 1 << kIn;
  const unsigned hw = threadIdx.x & 31u & ~(unsigned)(W - 1);
  constexpr unsigned kW = W == 32 ? 0xffffffffu : (1u << W) - 1u;
  auto team = [&](bool pred) { return (__ballot_sync(kFull, pred) >> hw) & kW; };
  const int k = active ? __popc(mask) : 0;
  const bool amb = active && ((mask >> lt) & 1u);
  const int slot = __popc(mask & ((1u << lt) - 1u));
  __syncwarp();
  sd[lt] = 0;
  sv[lt] = 0.f;
  __syncwarp();
  if (amb) {
    sd[slot] = lt;
    sv[slot] = v;
  }
  __syncwarp();
  const int nlb = min(max(k - kIn, 0), LB), nout = max(k - kIn - LB, 0);
  // the lane's state: A, q; the inner pair terms P
  int dI[kIn];  // inner dots (as columns)
  float q0[kIn], P[NI], A0 = 0.f, wl[LB];
  int rl[LB];
#pragma unroll
  for (int j = 0; j < kIn; ++j) {
    dI[j] = sd[j];
    q0[j] = j < k ? sv[j] : kBig;
  }
#pragma unroll
  for (int b = 0; b < NI; ++b) P[b] = 0.f;
#pragma unroll
  for (int j = 1; j < kIn; ++j) {
    const float* row = sM + sd[j] * kLdM;
#pragma unroll
    for (int l = 0; l < j; ++l) {
      const float m = row[dI[l]];
#pragma unroll
      for (int b = 0; b < NI; ++b)
        if (((b >> j) & 1) && ((b >> l) & 1)) P[b] += m;
    }
  }
#pragma unroll
  for (int i = 0; i < LB; ++i) {
    rl[i] = sd[kIn + i];
    wl[i] = (i < nlb && ((lt >> i) & 1)) ? 1.f : 0.f;
    const float* row = sM + rl[i] * kLdM;
    float add = sv[kIn + i];
#pragma unroll
    for (int l = 0; l < i; ++l) add = fmaf(wl[l], row[rl[l]], add);
    A0 = fmaf(wl[i], add, A0);
#pragma unroll
    for (int j = 0; j < kIn; ++j) q0[j] = fmaf(wl[i], row[dI[j]], q0[j]);
  }
  const bool own = active && (lt >> nlb) == 0;
  const int r0 = w - __popc((unsigned)lt);  // closed: weight left
  // the energies of one block: loop pattern o
  auto block = [&](unsigned o, float* e) {
    float A = A0, q[kIn];
#pragma unroll
    for (int j = 0; j < kIn; ++j) q[j] = q0[j];
    for (unsigned m = o; m; m &= m - 1u) {
      const int s1 = kIn + LB + __ffs(m) - 1;
      const float* row = sM + sd[s1] * kLdM;
      float add = sv[s1];
#pragma unroll
      for (int i = 0; i < LB; ++i) add = fmaf(wl[i], row[rl[i]], add);
      for (unsigned l = o & ((m & (0u - m)) - 1u); l; l &= l - 1u)
        add += row[sd[kIn + LB + __ffs(l) - 1]];
      A += add;
#pragma unroll
      for (int j = 0; j < kIn; ++j) q[j] += row[dI[j]];
    }
    e[0] = A;
#pragma unroll
    for (int j = 0; j < kIn; ++j)
#pragma unroll
      for (int b = 0; b < (1 << j); ++b) e[b + (1 << j)] = e[b] + q[j];
    const int r = r0 - __popc(o);
#pragma unroll
    for (int b = 0; b < NI; ++b) {
      e[b] += P[b];
      if (CLOSED && popc_c((unsigned)b) != r) e[b] = kInf;
    }
  };
  float g1 = kInf, g2 = kInf;
  unsigned o1 = 0u;
  const unsigned no = own ? 1u << nout : 0u;
#pragma unroll 1
  for (unsigned o = 0; o < no; ++o) {
    float e[NI];
    block(o, e);
    float m = e[0];
#pragma unroll
    for (int b = 1; b < NI; ++b) m = fminf(m, e[b]);
    g2 = fminf(g2, fmaxf(g1, m));
    if (m < g1) {
      g1 = m;
      o1 = o;
    }
  }
  evaluated += no * (unsigned)NI;
  __syncwarp();
  float m1 = g1;
#pragma unroll
  for (int off = W / 2; off > 0; off >>= 1) m1 = fminf(m1, __shfl_xor_sync(kFull, m1, off));
  const float thr = m1 + G;
  // the patterns within the margin: inner bits of a block at a time
  const bool wide = __any_sync(kFull, own && g2 <= thr);
  int nl = 0;
  unsigned b1 = 0u;
#pragma unroll 1
  for (unsigned o = 0;; ++o) {
    const unsigned oo = wide ? o : o1;
    unsigned hit = 0u;
    if (own && oo < no && (wide || g1 <= thr)) {
      float e[NI];
      block(oo, e);
#pragma unroll
      for (int b = 0; b < NI; ++b) hit |= e[b] <= thr ? 1u << b : 0u;
    }
    __syncwarp();
    while (true) {  // one candidate of each lane at a time
      const unsigned has = team(hit != 0u);
      if (!__any_sync(kFull, hit != 0u)) break;
      if (hit) {
        const unsigned sb = (unsigned)(__ffs(hit) - 1) | ((unsigned)lt << kIn) | (oo << (kIn + LB));
        const int at = nl + __popc(has & ((1u << lt) - 1u));
        // slots to dots
        unsigned db = 0u;
        for (unsigned m = sb; m; m &= m - 1u) db |= 1u << sd[__ffs(m) - 1];
        if (at < kSphList) lst[at] = db;
        hit &= hit - 1u;
      }
      nl += __popc(has);
    }
    if (!wide || !__any_sync(kFull, own && o + 1 < no)) break;
  }
  __syncwarp();
  b1 = nl > 0 ? lst[0] : 0u;
  close = (!(m1 < kBig) || nl > kSphList || nl < 1) ? 0 : nl;
  return b1;
}

// One warp's pixels, p its team's (active: below the end).
template <int W, bool CLOSED, int MODE>
__device__ inline void search_pixel(const GsLaunch& L, const ArrayDesc& a,
                                    typename PixelSharedOf<W, MODE>::type& sh, int array,
                                    long long p, bool active) {
  const int n = a.n;
  const int lt = threadIdx.x & (W - 1);
  const int tq = threadIdx.x & ~(W - 1);
  const int team = threadIdx.x / W;
  const unsigned hw = threadIdx.x & 31u & ~(unsigned)(W - 1);
  constexpr unsigned kW = (1u << W) - 1u;
  const PrepPixel q = prep_set<CLOSED, W>(a, sh.p, p, active);
  const bool amb = q.live && ((q.mask >> lt) & 1u);
  const int k = __popc(q.mask);
  const bool qp = (q.flags & kFlagQP) != 0u;
  constexpr float u24 = 5.9604645e-8f;
  // the centre f = x - base
  const float f = q.live ? __fadd_rn(__fsub_rn(q.x.hi, (float)q.base), q.x.lo) : 0.f;
  // A bound of the near-tie bound: S as in prep_h but with a plain FP32 h,
  // whose error (17 roundings of 16 products) is added.  The record's h, in
  // double-float, is formed for the few pixels that need their record; h was
  // an eighth of this kernel's instructions.
  const float r0 = q.live ? __fadd_rn(__fsub_rn((float)q.base, q.c.hi), -q.c.lo) : 0.f;
  const float* Mrow = sh.p.cs.Mhi + lt * kLdM;
  __syncwarp();
  sh.p.qx[threadIdx.x] = r0;
  sh.p.qz[threadIdx.x] = q.live ? __fadd_rn(__fsub_rn(q.x.hi, q.c.hi), q.x.lo - q.c.lo) : 0.f;
  __syncwarp();
  float S = 0.f, v = 0.f;
  {
    float h0 = 0.f, h1 = 0.f;
#pragma unroll
    for (int j = 0; j < W; j += 4) {
      const float4 r4 = *reinterpret_cast<const float4*>(&sh.p.qx[tq + j]);
      h0 = fmaf(Mrow[j], r4.x, h0);
      h1 = fmaf(Mrow[j + 1], r4.y, h1);
      h0 = fmaf(Mrow[j + 2], r4.z, h0);
      h1 = fmaf(Mrow[j + 3], r4.w, h1);
    }
    const unsigned below = q.mask & ((1u << lt) - 1u);
    v = (h0 + h1) + 0.5f * Mrow[lt];
    if (amb) {
      S = fabsf(h0 + h1);
      if (below == (1u << lt) - 1u) {
        S += sh.p.cs.absl[lt];
      } else {
        S += 0.5f * Mrow[lt];
#pragma unroll
        for (int j = 0; j < W; ++j) S += ((below >> j) & 1u) ? fabsf(Mrow[j]) : 0.f;
      }
    }
  }
#pragma unroll
  for (int off = W / 2; off > 0; off >>= 1) S += __shfl_xor_sync(kFull, S, off);
  const unsigned any_qp = __any_sync(kFull, qp);
  int close = 0;
  unsigned ev = 0, bits = 0u;
  const bool sphere =
      MODE == kPixSphere || (MODE == kPixMixed && __any_sync(kFull, active && k >= kMixedDots));
  // max_j |base_j - c_j| (and |x_j - c_j| for the gradient below), which scales
  // the rounding of M r: at most 1 on an open pixel without active constraints
  // (x = c), but a closed one moves every dot by lambda v.  (The sphere search
  // with active constraints takes it along with the gradient's sums.)
  float rmax = 1.f;
  if (sphere ? CLOSED && !any_qp : CLOSED || any_qp) {
    rmax = fmaxf(fabsf(r0), 1.f);
#pragma unroll
    for (int off = W / 2; off > 0; off >>= 1)
      rmax = fmaxf(rmax, __shfl_xor_sync(kFull, rmax, off));
  }
  if constexpr (MODE != kPixDense) if (sphere) {
    // the gradient M (x - c) where a constraint is active (else zero, closed: a
    // multiple of 1)
    float a1 = 0.f, neg = 0.f;
    if (any_qp) {
      float z = 0.f;
      rmax = fmaxf(rmax, fmaxf(fabsf(r0), fabsf(sh.p.qz[threadIdx.x])));
#pragma unroll
      for (int j = 0; j < W; ++j) z = fmaf(Mrow[j], sh.p.qz[tq + j], z);
      if (CLOSED) {  // the multiple of 1: the least entry, a free dot's
        float zm = q.live ? z : kInf;
#pragma unroll
        for (int off = W / 2; off > 0; off >>= 1) zm = fminf(zm, __shfl_xor_sync(kFull, zm, off));
        z -= zm;
      }
      a1 = (qp && amb) ? fmaxf(z, 0.f) : 0.f;
      neg = (qp && amb) ? fmaxf(-z, 0.f) : 0.f;
#pragma unroll
      for (int off = W / 2; off > 0; off >>= 1) {
        neg += __shfl_xor_sync(kFull, neg, off);
        rmax = fmaxf(rmax, __shfl_xor_sync(kFull, rmax, off));
      }
    }
    const float ez = u24 * a.md->s.msum * rmax;  // u sum |M| |r|
    const float bound = pixel_bound(a, S * 1.00001f + 20.f * ez, k);
    neg += (qp ? 24.f : 2.f) * ez;
    // no factor, or a centre outside [-1, 1] (an unsettled QP): left to the
    // FP32 search.  (The mark is read here: held in shared memory the kernel
    // spilled registers, 4 % of 10^4 voltage vectors' time.)
    const bool far = ((__ballot_sync(kFull, !(fabsf(f) <= 1.f)) >> hw) & kW) != 0u;
    bits = sphere_search<CLOSED>(a.md->s, sh.m, n, lt, active && a.md->s.valid && !far, f, a1, q.mask,
                                 q.w, bound, neg, &sh.p.qx[tq], &sh.p.qz[tq], sh.lev[team],
                                 reinterpret_cast<uint2*>(&sh.p.qK[tq][0]), close, ev);
  }
  // (the candidates within the margin: level patterns of the sphere search,
  // dot patterns of the enumeration)
  unsigned* lst =
      reinterpret_cast<unsigned*>(MODE == kPixDense ? &sh.p.qK[tq][0] : &sh.p.qz[tq]);
  if constexpr (MODE != kPixSphere) if (!sphere) {
    const float msum = a.md->s.msum, ez = u24 * msum * rmax;
    // twice the near-tie bound as in the sphere search, once more for this
    // search's own sums (at most 2 k + 8 additions), and the error of the
    // plain h on both sides
    const float G = 3.f * pixel_bound(a, S * 1.00001f + 20.f * ez, k) + 40.f * ez;
    bits = dense_search<W, CLOSED>(sh.p.cs.Mhi, n, lt, active && msum < kInf, v, q.mask, q.w, G,
                                   &sh.p.qa[tq], &sh.p.qc[tq], lst, close, ev);
  }
  const bool done = active && close == 1;
  // candidates too close to tell apart: left, with their patterns over the
  // dots, to the list kernel; so is a search that did not end
  if (__any_sync(kFull, active && close != 1)) {
    int pos = lt;
    if constexpr (MODE != kPixDense) pos = sphere ? sh.m.pos[lt] : lt;
    const bool leave = active && close != 1 && lt == 0;
    CloseEntry* ce = nullptr;
    if (leave) {
      ce = L.close_list + atomicAdd(&L.cnt->n_close, 1u);
      ce->array = array;
      ce->p = (int)p;
      ce->nl = close <= kCloseMax ? close : 0;
    }
#pragma unroll 1
    for (int e = 0; e < kCloseMax; e += 2) {
      const unsigned b0 = __ballot_sync(
          kFull, lt < n && e < close && ((lst[e] >> pos) & 1u));
      const unsigned b1 = __ballot_sync(
          kFull, lt < n && e + 1 < close && ((lst[e + 1] >> pos) & 1u));
      if (leave) ce->pat[e >> 1] = ((b0 >> hw) & kW) | (((b1 >> hw) & kW) << 16);
    }
    __syncwarp();
  }

  // n* = base + bits and U(n*) = 1/2 r^T M r
  int ni = q.base + (int)((bits >> lt) & 1u);
  const df u = team_energy<W>(sh.p.cs, n, lt, kFull, q.live, ni, q.c, &sh.p.qx[tq], &sh.p.qz[tq]);
  unsigned flags = q.flags, ov = 0u;
  // int8 maps of W dots: the team's charges as one W-byte store
  const bool vec =
      !a.out_n16 && n == W && (reinterpret_cast<uintptr_t>(a.out_n) & (W - 1)) == 0;
  if (vec) {
    if (ni > 127) {
      ni = 127;
      ov = kFlagOverflow;
    }
    unsigned w0 = ((unsigned)ni & 0xffu) << (8 * (lt & 3));
    w0 |= __shfl_xor_sync(kFull, w0, 1);
    w0 |= __shfl_xor_sync(kFull, w0, 2);
    int8_t* dst = a.out_n + p * n;
    if constexpr (W == 16) {
      const unsigned w1 = __shfl_sync(kFull, w0, hw + 4), w2 = __shfl_sync(kFull, w0, hw + 8);
      const unsigned w3 = __shfl_sync(kFull, w0, hw + 12);
      if (done && lt == 0)
        *reinterpret_cast<int4*>(dst) = make_int4((int)w0, (int)w1, (int)w2, (int)w3);
    } else if constexpr (W == 8) {
      const unsigned w1 = __shfl_sync(kFull, w0, hw + 4);
      if (done && lt == 0) *reinterpret_cast<int2*>(dst) = make_int2((int)w0, (int)w1);
    } else {
      if (done && lt == 0) *reinterpret_cast<int*>(dst) = (int)w0;
    }
  } else if (done && q.live) {
    store_charge(a, p * n + lt, ni, ov);
  }
  if ((__ballot_sync(kFull, ov != 0u) >> hw) & kW) flags |= kFlagOverflow;
  const unsigned evw = __reduce_add_sync(kFull, ev);
  if (active && lt == 0) {
    sh.cand[team] += CLOSED ? binom(k, q.w) : (1ull << k);
    sh.qp[team] += qp ? 1u : 0u;
    sh.doubled[team] += (q.flags & kFlagDoubled) ? 1u : 0u;
    if (hw == 0u) sh.ev[team] += evw;
  }
  const bool listed = done && (flags & (kFlagBoundary | kFlagQPCap | kFlagUnresolved)) != 0u;
  if (active && (close != 1 || listed)) {
    float Sx;
    const float h = prep_h<W>(a, sh.p, q, Sx);
    store_record<CLOSED>(a.recs + p, q, lt, h, pixel_bound(a, Sx, k));
  }
  if (done && lt == 0) {
    if (a.out_U) a.out_U[p] = 0.5 * df_to_double(u);
    if (a.out_flags) a.out_flags[p] = (uint8_t)flags;
    if (listed) {
      L.flag_list[atomicAdd(&L.cnt->n_flag, 1u)] = ListEntry{array, (int)p, 0.f, 0};
      ++sh.boundary[team];
    }
    if (flags & kFlagOverflow) ++sh.overflow[team];
  }
}

// ---------------------------------------------------------------------------
// Pixels that search_pixel left (the close list): the FP32 search's
// near-tie flag and, where it is set, the argmin by exact energies.
// ---------------------------------------------------------------------------
// The pruned FP32 search's minimum of one block (an outer pattern with its
// middle pattern): the tables' entries, sums and middle walk of search_bnb,
// formed for that block alone.  pm, vv: its slot pairs and single-flip
// energies; ptab: its inner pair table; nlb: the lane bits of its team.
template <bool CLOSED>
__device__ __forceinline__ float bnb_block_min(const float* pm, const float* vv, const float* ptab,
                                               int k, int w, int nlb, unsigned blk) {
  constexpr int L1 = kBnbL1, L2 = kBnbL2, kLB = 5;
  static_assert(L2 == 2, "two middle slots");
  const int nmid = min(max(k - L1, 0), L2), nout = max(k - kBnbIn, 0), nit = nout - nlb;
  const unsigned o = blk >> L2, li = o & ((1u << nlb) - 1u), it = o >> nlb;
  const int s0 = kBnbIn + nlb;
  float wO[kLB], wI[kBnbItBits], L[kBnbIn], At = 0.f, Ai = 0.f, x = 0.f;
#pragma unroll
  for (int i = 0; i < kLB; ++i) wO[i] = (i < nlb && ((li >> i) & 1u)) ? 1.f : 0.f;
#pragma unroll
  for (int i = 0; i < kBnbItBits; ++i) wI[i] = (i < nit && ((it >> i) & 1u)) ? 1.f : 0.f;
#pragma unroll
  for (int i = 0; i < kLB; ++i) {
    const float* prow = pm + min(kBnbIn + i, kMaxDot - 1) * kLdM;
    float add = vv[min(kBnbIn + i, kMaxDot - 1)];
#pragma unroll
    for (int i2 = 0; i2 < i; ++i2) add = fmaf(wO[i2], prow[kBnbIn + i2], add);
    At = fmaf(wO[i], add, At);
  }
#pragma unroll
  for (int j = 0; j < kBnbIn; ++j) {
    float a = vv[j], b = 0.f;
#pragma unroll
    for (int i = 0; i < kLB; ++i) a = fmaf(wO[i], pm[min(kBnbIn + i, kMaxDot - 1) * kLdM + j], a);
#pragma unroll
    for (int i = 0; i < kBnbItBits; ++i) b = fmaf(wI[i], pm[j * kLdM + min(s0 + i, kMaxDot - 1)], b);
    L[j] = a + b;
  }
#pragma unroll
  for (int ii = 0; ii < kBnbItBits; ++ii) {
    const int si = min(s0 + ii, kMaxDot - 1);
    float add = vv[si], cr = 0.f;
#pragma unroll
    for (int i2 = 0; i2 < ii; ++i2)
      add = fmaf(wI[i2], pm[si * kLdM + min(s0 + i2, kMaxDot - 1)], add);
    Ai = fmaf(wI[ii], add, Ai);
#pragma unroll
    for (int i = 0; i < kLB; ++i) cr = fmaf(wO[i], pm[min(kBnbIn + i, kMaxDot - 1) * kLdM + si], cr);
    x = fmaf(wI[ii], cr, x);
  }
  float A = (At + x) + Ai, g0 = L[L1], g1 = L[L1 + 1];
  const unsigned mid = blk & 3u;
  const float mm = nmid > 1 ? pm[(L1 + 1) * kLdM + L1] : 0.f;
  auto flip = [&](int m, float g, bool up) {
    A = up ? A + g : A - g;
#pragma unroll
    for (int j = 0; j < L1; ++j) {
      const float d = m < nmid ? pm[j * kLdM + L1 + m] : 0.f;
      L[j] = up ? L[j] + d : L[j] - d;
    }
  };
  if (mid) {  // the walk's middle patterns: 0, 1, 3, 2
    flip(0, g0, true);
    g1 += mm;
    if (mid & 2u) {
      flip(1, g1, true);
      g0 += mm;
      if (mid == 2u) flip(0, g0, false);
    }
  }
  return CLOSED ? inner_min_closed_smem<L1>(A, L, ptab, w - __popc(o) - __popc(mid))
                : inner_min_open_smem<L1>(A, L, ptab);
}

// A warp's scratch for an entry of the close list.
struct SettleScratch {
  int sdot[kMaxDot];
  float sh[kMaxDot];
  unsigned lst[kCloseMax];
  float rhi[2][kMaxDot], rlo[2][kMaxDot];
  __align__(16) float ptab[1 << kBnbL1];  // the pruned search's tables
  float pm[kMaxDot * kLdM];
  float vv[kMaxDot];
};

// The exhaustive search's sums for a block (a pattern of the outer and middle
// slots), by a warp: lane c < in keeps the coefficient of walked slot c, every
// lane the block's energy A, and lane b forms inner pattern b.  The terms are
// added in search_lane's order, so the results are its to the bit; rolled
// loops over the set slots, because an entry's code runs once per launch on
// cold instruction caches (search_lane itself, unrolled for registers, took
// the list kernel of the 16-dot 257 x 193 diagram at t = 0.5 26.6 us, this
// 16.0).
struct SettleWarp {
  const float* sM;
  const int* dot;   // of each slot
  const float* h;
  int k, L1, in;    // slots; inner, inner + middle slots
  int lane, mydot;
  float v0;         // h + M / 2 of the lane's walked slot (a slot beyond k: never wins)

  __device__ __forceinline__ void init(const float* M, const SlotView& sv, int l1, int l2) {
    sM = M;
    dot = sv.dot;
    h = sv.h;
    k = sv.k;
    L1 = l1;
    in = l1 + l2;
    lane = threadIdx.x & 31;
    mydot = lane < min(in, k) ? dot[lane] : 0;
    v0 = lane < min(in, k) ? h[lane] + 0.5f * sM[mydot * (kLdM + 1)] : (lane < L1 ? kBig : 0.f);
  }
  // A and the lane's coefficient after the slots `bits` (each with its pair
  // terms with those of `bits` below it)
  __device__ __forceinline__ void add_slots(unsigned bits, float& A, float& val) const {
#pragma unroll 1
    for (unsigned m = bits; m; m &= m - 1u) {
      const int s = __ffs(m) - 1;
      const float* row = sM + dot[s] * kLdM;
      float add = h[s] + 0.5f * row[dot[s]];
#pragma unroll 1
      for (unsigned l = bits & ((1u << s) - 1u); l; l &= l - 1u) add += row[dot[__ffs(l) - 1]];
      A += add;
      if (lane < min(in, k)) val += row[mydot];
    }
  }
  // The inner pair terms of pattern `lane`, summed dot by dot.
  __device__ __forceinline__ float pairs() const {
    float P = 0.f;
#pragma unroll 1
    for (int j = 1; j < min(L1, k); ++j) {
      if (!((lane >> j) & 1)) continue;
      float r = 0.f;
#pragma unroll 1
      for (int l = 0; l < j; ++l)
        if ((lane >> l) & 1) r += sM[dot[j] * kLdM + dot[l]];
      P += r;
    }
    return P;
  }
  // The energy of inner pattern `lane` (+inf: not a candidate).
  __device__ __forceinline__ float inner(float A, float val, float P, int r) const {
    float e = A;
#pragma unroll 1
    for (int j = 0; j < L1; ++j) {
      const float q = __shfl_sync(kFull, val, j);
      if ((lane >> j) & 1) e += q;
    }
    e += P;
    return (lane >> L1) != 0 || (r >= 0 && __popc((unsigned)lane) != r) ? kInf : e;
  }
  // The block's minimum as the walk finds it.  split: the outer slots' sums
  // in two groups, those of the team's nlb lane bits and the others.
  __device__ __forceinline__ float walk_min(unsigned blk, int nlb, bool split, float P,
                                            int w) const {
    const int L2 = in - L1;
    const unsigned o = blk >> L2, mid = blk & ((1u << L2) - 1u);
    const unsigned lm = split ? o & ((1u << nlb) - 1u) : o, im = o & ~lm;
    float A = 0.f, val = v0;
    add_slots(lm << in, A, val);
    if (split) {
      float A2 = 0.f, val2 = 0.f, x = 0.f;
      add_slots(im << in, A2, val2);
#pragma unroll 1
      for (unsigned m = im; m; m &= m - 1u) {
        const float* row = sM + dot[in + __ffs(m) - 1] * kLdM;
        float c = 0.f;
#pragma unroll 1
        for (unsigned l = lm; l; l &= l - 1u) c += row[dot[in + __ffs(l) - 1]];
        x += c;
      }
      A = (A + x) + A2;
      val += val2;
    }
#pragma unroll 1
    for (unsigned s = 1, g = 0; g != mid; ++s) {  // the Gray walk to the middle pattern
      const int mb = __ffs(s) - 1;
      g = s ^ (s >> 1);
      const bool up = (g >> mb) & 1u;
      const float gm = __shfl_sync(kFull, val, L1 + mb);
      A = up ? A + gm : A - gm;
      if (lane < min(in, k) && lane != L1 + mb) {
        const float d = sM[mydot * kLdM + dot[L1 + mb]];
        val = up ? val + d : val - d;
      }
    }
    float e = inner(A, val, P, w < 0 ? -1 : max(w - __popc(blk), 0));
    if (w >= 0 && w < __popc(blk)) e = kInf;
    for (int off = 16; off > 0; off >>= 1) e = fminf(e, __shfl_xor_sync(kFull, e, off));
    return e;
  }
};

template <int N>
struct SplitSize { static constexpr int value = N; };
// The exhaustive search of a pixel without a list, by a warp: the same kind of
// results over all its candidates.
template <bool CLOSED>
static __device__ __noinline__ void full_top2(const ArrayDesc& a, const float* sM, const SlotView sv,
                                              const SettleWarp& sw, int nlb, bool split, float P,
                                              float& m1, unsigned& b1, float& m2) {
  const int lane = threadIdx.x & 31, T = a.cfg.T, k = sv.k, L1 = a.cfg.L1, L2 = a.cfg.L2;
  m1 = m2 = kInf;
  b1 = 0u;
  if (T >= kTeamFinishMin) {
    const unsigned nmid = 1u << min(max(k - L1, 0), L2), no = 1u << max(k - L1 - L2, 0);
#pragma unroll 1
    for (unsigned o = 0; o < no; ++o)
#pragma unroll 1
      for (unsigned mid = 0; mid < nmid; ++mid) {
        const unsigned blk = (o << L2) | mid;
        const float e = sw.walk_min(blk, nlb, split, P, sv.w);
        if (lane == 0) {
          m2 = fminf(m2, fmaxf(m1, e));
          if (e < m1) {
            m1 = e;
            b1 = blk;
          }
        }
      }
    return;
  }
  unsigned long long ev = 0;
  auto lanes = [&](auto l1, auto l2) {
    search_lane<decltype(l1)::value, decltype(l2)::value, CLOSED, false, false, 5>(
        sM, sv, lane, T, 0.f, nullptr, nullptr, 0u, m1, b1, m2, ev);
  };
  if (lane < T) {
    if (L2 == 0) lanes(SplitSize<4>{}, SplitSize<0>{});
    else if (L2 == 3) lanes(SplitSize<4>{}, SplitSize<3>{});
    else lanes(SplitSize<5>{}, SplitSize<4>{});
  }
}

// The FP32 search's best candidate (m1, pattern over the slots b1) and
// runner-up m2 among the blocks of the nl listed candidates (slot patterns in
// t.lst), or among all of them (nl = 0), with the sums that the array's search
// takes: its split and team width say which.
template <bool CLOSED>
__device__ __forceinline__ void listed_top2(const ArrayDesc& a, const float* sM, const SlotView sv,
                                            SettleScratch& t, int nl, float& m1, unsigned& b1,
                                            float& m2) {
  const int lane = threadIdx.x & 31, T = a.cfg.T, L1 = a.cfg.L1, L2 = a.cfg.L2, k = sv.k;
  const bool bnb = bnb_search(L1, L2), tf = T >= kTeamFinishMin;
  const int nlb = min(__ffs(T) - 1, max(k - L1 - L2, 0));  // the team's lane bits
  unsigned blk = lane < nl ? t.lst[lane] >> L1 : 0u;
  bool own = lane < nl;  // lane e holds block e, each block once
  for (int e = 0; e < nl; ++e) own = own && (e >= lane || (t.lst[e] >> L1) != blk);
  m1 = m2 = kInf;
  b1 = 0u;
  if (bnb) {
    // the tables of bnb_pair_build, an element per lane, and the inner pairs;
    // a block per lane
#pragma unroll
    for (int e = lane; e < kMaxDot * kMaxDot; e += 32) {
      const int r = e >> 4, c = e & 15;
      t.pm[r * kLdM + c] = (r < k && c < k) ? sM[sv.dot[r] * kLdM + sv.dot[c]] : 0.f;
    }
    if (lane < kMaxDot)
      t.vv[lane] = lane < k ? sv.h[lane] + 0.5f * sM[sv.dot[lane] * (kLdM + 1)]
                            : (lane < kBnbL1 ? kBig : 0.f);
    __syncwarp();
    float r = 0.f;
#pragma unroll
    for (int j = 1; j < kBnbL1; ++j)
#pragma unroll
      for (int l = 0; l < j; ++l)
        r = fmaf((((lane >> j) & 1) && ((lane >> l) & 1)) ? 1.f : 0.f, t.pm[j * kLdM + l], r);
    t.ptab[lane] = r;
    __syncwarp();
    // (a middle pattern beyond the k slots holds no block)
    const unsigned midmax = 1u << min(max(k - kBnbL1, 0), kBnbL2);
    const unsigned nblk = nl > 0 ? (own ? 1u : 0u) : 1u << (max(k - kBnbIn, 0) + kBnbL2);
#pragma unroll 1
    for (unsigned q = nl > 0 ? 0u : (unsigned)lane; q < nblk; q += 32u) {
      const unsigned b = nl > 0 ? blk : q;
      if ((b & 3u) >= midmax) continue;
      const float e = bnb_block_min<CLOSED>(t.pm, t.vv, t.ptab, k, sv.w, nlb, b);
      m2 = fminf(m2, fmaxf(m1, e));
      if (e < m1) {
        m1 = e;
        b1 = b;
      }
    }
  } else {
    const bool split = tf && L1 + L2 >= 9;
    SettleWarp sw;
    sw.init(sM, sv, L1, L2);
    const float P = sw.pairs();
    if (nl == 0) full_top2<CLOSED>(a, sM, sv, sw, nlb, split, P, m1, b1, m2);
#pragma unroll 1
    for (int e = 0; e < nl; ++e) {
      const float m = sw.walk_min(__shfl_sync(kFull, blk, e), nlb, split, P, sv.w);
      if (lane == e && own) m1 = m;
    }
    if (nl > 0) b1 = blk;
    if (!tf && nl > 0) {
      // narrow teams: the best block of each of the team's lanes (v) candidate
      // by candidate, of its other blocks the minimum
      const unsigned v = (blk >> L2) & ((1u << nlb) - 1u);
      bool first = own;
      const float g = m1;
#pragma unroll 1
      for (int e = 0; e < nl; ++e) {
        const float ge = __shfl_sync(kFull, g, e);
        const unsigned ve = __shfl_sync(kFull, v, e);
        if (__shfl_sync(kFull, own ? 1 : 0, e) && e != lane && ve == v &&
            (ge < g || (ge == g && e < lane)))
          first = false;
      }
      if (own && !first) {
        m2 = m1;
        m1 = kInf;
      }
#pragma unroll 1
      for (int e = 0; e < nl; ++e) {
        if (!__shfl_sync(kFull, first ? 1 : 0, e)) continue;
        const unsigned S = __shfl_sync(kFull, blk, e) << L1;
        float A = 0.f, val = sw.v0;
        sw.add_slots(S, A, val);
        const int r = CLOSED ? sv.w - __popc(S) : -1;
        float x1 = sw.inner(A, val, P, r), x2 = kInf;
        if (CLOSED && r < 0) x1 = kInf;
        unsigned xb = (unsigned)lane;
        for (int off = 16; off > 0; off >>= 1) {
          const float o1 = __shfl_xor_sync(kFull, x1, off), o2 = __shfl_xor_sync(kFull, x2, off);
          const unsigned ob = __shfl_xor_sync(kFull, xb, off);
          x2 = fminf(fminf(x2, o2), fmaxf(x1, o1));
          if (o1 < x1 || (o1 == x1 && ob < xb)) {
            x1 = o1;
            xb = ob;
          }
        }
        if (lane == e) {
          m1 = x1;
          m2 = x2;
          b1 = S | xb;
        }
      }
    }
  }
#pragma unroll 1
  for (int off = 1; off < 32; off <<= 1) {
    const float o1 = __shfl_xor_sync(kFull, m1, off), o2 = __shfl_xor_sync(kFull, m2, off);
    const unsigned ob = __shfl_xor_sync(kFull, b1, off);
    top2_merge(m1, b1, m2, o1, ob, o2);
  }
  if (!tf) return;
  float e1, e2;
  unsigned fb;
  const unsigned best = m1 < kInf ? b1 : 0u;
  if (bnb) team_finish<kBnbL1, kBnbL2, CLOSED>(sM, sv, lane & (T - 1), T, kFull, best, e1, fb, e2);
  else team_finish<5, 4, CLOSED>(sM, sv, lane & (T - 1), T, kFull, best, e1, fb, e2);
  if (m1 < kInf) {
    m1 = e1;
    b1 = fb;
    m2 = fminf(m2, e2);
  }
}

// One entry of the close list, by a warp: the argmin by the exact energies of
// the listed candidates, the near-tie flag by the FP32 search's energies of the
// same candidates (any other is further than the bound from the minimum in
// every FP32 sum, so the flag and the charges are those of the FP32 search
// and the resolve).  Without a list (nl = 0): the FP32 search over all of
// them.  Returns 0 when the pixel is done, 1 when the resolve has to follow
// (energies too close for double-float, or no list and a near tie), 2 for
// the FP64 recheck (e: the entry for either).
// What bounds it: latency, on cold instruction caches.  With the whole FP32
// search as a kernel of its own and the resolve behind it, these few pixels
// took 26 us of the 16-dot 100 x 100 diagram's 52; settled inside the sphere
// search's warps they lengthened its tail by 23 us.
template <bool CLOSED>
__device__ inline int settle_entry(const GsLaunch& L, const ArrayDesc& a, const ModelConsts& cs,
                                   SettleScratch& t, const CloseEntry& ce, ListEntry& e) {
  const int n = a.n;
  const int lane = threadIdx.x & 31, lt = lane & 15, half = lane >> 4;
  const PixRec* rec = a.recs + ce.p;
  const bool live = lt < n;
  const int base = live ? rec->base[lt] : 0;
  const df c = live ? df{rec->chi[lt], rec->clo[lt]} : df{0.f, 0.f};
  const float h = live ? rec->h[lt] : 0.f;
  const unsigned mask = rec->mask;
  const float bound = rec->bound;
  const int w = rec->w;
  unsigned flags = rec->flags;
  const int k = __popc(mask);
  const bool amb = live && ((mask >> lt) & 1u);
  const int nl = ce.nl;
  // slots: dots in order, or (pruned search) by |h + M_ii / 2|
  int slot = __popc(mask & ((1u << lt) - 1u));
  if (bnb_search(a.cfg.L1, a.cfg.L2)) {
    const float key = amb ? fabsf(h + 0.5f * cs.Mhi[lt * kLdM + lt]) : 0.f;
    int rank = 0;
#pragma unroll
    for (int j = 0; j < kMaxDot; ++j) {
      const float kj = __shfl_sync(kFull, key, j);
      rank += (((mask >> j) & 1u) && (kj < key || (kj == key && j < lt))) ? 1 : 0;
    }
    slot = rank;
  }
  __syncwarp();
  if (amb && half == 0) {
    t.sdot[slot] = lt;
    t.sh[slot] = h;
  }
  // exact energies, two candidates at a time (2 U)
  df best = {kInf, 0.f}, second = {kInf, 0.f};
  unsigned bbits = 0u;
  auto take = [&](df u, unsigned b) {
    const bool better = u.hi < best.hi || (u.hi == best.hi && u.lo < best.lo);
    const df lose = better ? best : u;
    if (lose.hi < second.hi || (lose.hi == second.hi && lose.lo < second.lo)) second = lose;
    if (better) {
      best = u;
      bbits = b;
    }
  };
  auto pattern = [&](int i) { return (ce.pat[i >> 1] >> (16 * (i & 1))) & 0xffffu; };
#pragma unroll 1
  for (int i = 0; i < nl; i += 2) {
    const unsigned b = pattern(i + half);  // (zero past the list)
    const df u = team_energy<kMaxDot>(cs, n, lt, kFull, live, base + (int)((b >> lt) & 1u), c, t.rhi[half],
                             t.rlo[half]);
    const unsigned sb =
        __reduce_or_sync(half ? 0xffff0000u : 0xffffu, (amb && ((b >> lt) & 1u)) ? 1u << slot : 0u);
    if (lt == 0 && i + half < nl) t.lst[i + half] = sb;
    df u0, u1;
    u0.hi = __shfl_sync(kFull, u.hi, 0);
    u0.lo = __shfl_sync(kFull, u.lo, 0);
    u1.hi = __shfl_sync(kFull, u.hi, 16);
    u1.lo = __shfl_sync(kFull, u.lo, 16);
    take(u0, pattern(i));
    if (i + 1 < nl) take(u1, pattern(i + 1));
  }
  __syncwarp();
  const SlotView sv{t.sdot, t.sh, k, CLOSED ? w : -1};
  float m1, m2;
  unsigned b1;
  listed_top2<CLOSED>(a, cs.Mhi, sv, t, nl, m1, b1, m2);
  const bool near = !(m2 - m1 > bound);
  const bool boundary = (flags & (kFlagBoundary | kFlagQPCap | kFlagUnresolved)) != 0u;
  // the resolve decides gaps of the energies below 1e-10 (1 + |U(base)|):
  // leave it four times that (U(base) <= U + S, and the bound is at least
  // 24 2^-24 S; a wider margin would send a near tie in a hundred through the
  // resolve, 18 us of latency in most diagrams)
  const df gap2 = df_sub(second, best);
  const bool exact = nl > 1 && 0.5f * gap2.hi > 4e-10f * (1.f + best.hi + bound * (16777216.f / 24.f));
  const int next = boundary ? 2 : (near && !exact) ? 1 : 0;
  // the FP32 search's candidate stands until what follows
  const bool bit = amb && ((nl == 0 || (near && next != 0)) ? (b1 >> slot) & 1u
                                                            : (bbits >> lt) & 1u);
  const int ni = base + (bit ? 1 : 0);
  if (nl == 0) best = team_energy<kMaxDot>(cs, n, lt, kFull, live, ni, c, t.rhi[half], t.rlo[half]);
  if (near) flags |= kFlagNearTie | (next == 0 ? kFlagRechecked : 0u);
  unsigned ov = 0u;
  if (live && half == 0) store_charge(a, (long long)ce.p * n + lt, ni, ov);
  if (__any_sync(kFull, ov != 0u)) flags |= kFlagOverflow;
  if (lane == 0) {
    if (a.out_U) a.out_U[ce.p] = 0.5 * df_to_double(best);
    if (a.out_flags) a.out_flags[ce.p] = (uint8_t)flags;
    if (boundary) atomicAdd(&L.cnt->boundary, 1ull);
    else if (near) atomicAdd(&L.cnt->near_tie, 1ull);
    if (near && next == 0) {
      atomicAdd(&L.cnt->resolved, 1ull);
      atomicMax(&L.cnt->shortlist_max, (unsigned long long)nl);
    }
    if (flags & kFlagOverflow) atomicAdd(&L.cnt->overflow, 1ull);
  }
  e = ListEntry{ce.array, ce.p, m1, (next == 2 && near) ? 1 : 0};
  __syncwarp();
  return next;
}

// ---------------------------------------------------------------------------
// (a7, near ties) for one list entry: a pixel whose candidate set is certain
// but whose FP32 best/runner-up gap is under the error bound.  The block
// re-walks the candidates collecting every block of the split whose FP32
// minimum is within the bound of the search's minimum (the exact argmin is
// guaranteed to be among them) and evaluates those candidates exactly,
// relative to the base state,
//     E(b) = sum_{s in b} (h_s + M_ss / 2) + sum_{s < s' in b} M_ss',
// in double-float arithmetic with h = M (base - c) in double-float (about
// 1e-13 absolute).  No FP64 instructions: GB300's FP64 rate is a small
// fraction of its FP32 rate.  A pixel whose two best exact energies are
// within 1e-10 (a true tie) or whose list overflows goes on to the FP64
// recheck, which also applies the lexicographic tie rule.  The resolve split
// is kCheckL1 / kCheckL2 for every array; the search's bound covers it (it
// was derived for a middle level at least as deep).  A block runs an entry's
// code once per launch, on cold instruction caches, so the small reductions
// and sums below stay rolled loops: their bodies are fetched once.
// ---------------------------------------------------------------------------
struct ResolveShared {
  ModelConsts cs;
  int sdot[kMaxDot];
  float sh[kMaxDot];
  df shd[kMaxDot];
  df sui[kMaxDot];
  float pk[kMaxDot][kMaxDot + 1];   // pair terms of the pixel's slots, M_{dot(s) dot(s2)}
  float pkl[kMaxDot][kMaxDot + 1];  // ... and their low parts
  unsigned blist[128];
  unsigned bcnt;
  df rbest[kResolveThreads / 32], rsec[kResolveThreads / 32];
  unsigned rbits[kResolveThreads / 32];
  unsigned dbits;   // the decision of warp 0, for the whole block
  int dok;
  unsigned dflags;
  df ub;            // U(base)
};

template <bool CLOSED>
__device__ inline void resolve_entry(const GsLaunch& L, const ArrayDesc& a, ResolveShared& S,
                                     ListEntry te, unsigned& my_res, unsigned& my_slmax) {
  constexpr int L1 = kCheckL1, L2 = kCheckL2;
  constexpr int NI = 1 << L1;
  constexpr int NM = 1 << L2;
  constexpr int NW = kResolveThreads / 32;
  constexpr unsigned kCap = 128;
  const float* sM = S.cs.Mhi;
  const float* sMlo = S.cs.Mlo;
  const int n = a.n;
  const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
  int* sdot = S.sdot;
  float* sh = S.sh;
  df* shd = S.shd;
  df* sui = S.sui;
  unsigned* blist = S.blist;
  unsigned& bcnt = S.bcnt;
  df* rbest = S.rbest;
  df* rsec = S.rsec;
  unsigned* rbits = S.rbits;
  const long long p = te.p;
  const PixRec* rec = a.recs + p;
  const unsigned mask = rec->mask;
  const int k = __popc(mask);
  const int w = rec->w;
  // the pixel's flags, read while the walk runs
  const unsigned char flags0 = (tid == 0 && a.out_flags) ? a.out_flags[p] : 0;
  // h_i = (M (base - c))_i in double-float, and U(base) = r0 . h / 2: one
  // product M_ij r_j per thread of the first 256 (row i = tid / 16), summed
  // over the row's 16 threads
  {
    static_assert(kResolveThreads >= kMaxDot * kMaxDot, "one thread per matrix entry");
    const int i = tid >> 4, j = tid & 15;
    df prod = {0.f, 0.f};
    if (i < n && j < n) {
      const df rj = df_sub({(float)rec->base[j], 0.f}, {rec->chi[j], rec->clo[j]});
      prod = df_mul({sM[i * kLdM + j], sMlo[i * kLdM + j]}, rj);
    }
#pragma unroll 1
    for (int off = 1; off < 16; off <<= 1) {
      df o;
      o.hi = __shfl_xor_sync(kFull, prod.hi, off, 16);
      o.lo = __shfl_xor_sync(kFull, prod.lo, off, 16);
      prod = df_add(prod, o);
    }
    if (j == 0 && i < n) {
      const df hi = prod;
      const df r0 = df_sub({(float)rec->base[i], 0.f}, {rec->chi[i], rec->clo[i]});
      sui[i] = df_mul(hi, r0);
      if ((mask >> i) & 1u) {
        const int s = __popc(mask & ((1u << i) - 1u));
        sdot[s] = i;
        sh[s] = rec->h[i];
        shd[s] = df_add(hi, df_mul_f({sM[i * kLdM + i], sMlo[i * kLdM + i]}, 0.5f));
      }
    }
  }
  if (tid == 0) bcnt = 0u;
  __syncthreads();
  // U(base) = sum_i r0_i h_i / 2, a 16-lane double-float sum in warp 0
  if (wid == 0) {
    df u = (lane < n) ? sui[lane] : df{0.f, 0.f};
#pragma unroll 1
    for (int off = 8; off > 0; off >>= 1) {
      df o;
      o.hi = __shfl_xor_sync(kFull, u.hi, off, 16);
      o.lo = __shfl_xor_sync(kFull, u.lo, off, 16);
      u = df_add(u, o);
    }
    if (lane == 0) S.ub = df_mul_f(u, 0.5f);
  }
  // the slots' pair terms, one per thread (zero outside the k slots), for
  // the shortlist's sums
  {
    const int s1 = tid >> 4, s2 = tid & 15;
    if (s1 < kMaxDot) {
      const bool on = s1 < k && s2 < k;
      const int e = on ? sdot[s1] * kLdM + sdot[s2] : 0;
      S.pk[s1][s2] = on ? sM[e] : 0.f;
      S.pkl[s1][s2] = on ? sMlo[e] : 0.f;
    }
  }
  // every block whose FP32 minimum is within the bound of the search's
  const SlotView sv{sdot, sh, k, w};
  const float thr = te.m1 + rec->bound;
  float d1, d2;
  unsigned db;
  unsigned long long ev = 0;
  static_assert(kResolveThreads <= 512, "the walk's team is the block: at most 9 lane bits");
  // (outer patterns whose lower bound is above the threshold plus the FP32
  // margin hold no block within the threshold)
  search_lane<L1, L2, CLOSED, true, false, 9>(sM, sv, tid, kResolveThreads, thr, blist, &bcnt,
                                    kCap, d1, db, d2, ev, nullptr, nullptr, nullptr,
                                    thr + 2.0f * rec->bound, S.cs.qneg);
  __syncthreads();
  const unsigned nb = bcnt;
  const bool fits = nb <= kCap;
  df best = {kInf, 0.f}, second = {kInf, 0.f};
  unsigned bbits = 0xffffffffu;
  if (fits) {
    // sixteen threads per shortlisted candidate, thread `sub` taking slot
    // sub when it is set: h_s + M_ss / 2 plus the pair terms with the set
    // slots below s, over a fixed range of slots with zero terms for the
    // others (no data-dependent chains); the high parts are summed
    // error-free, the low parts and rounding errors in plain FP32 (their own
    // error is O(u^2) of the magnitudes); the group then sums its slots
    constexpr int kSub = kMaxDot;
    const int sub = tid & (kSub - 1), grp = tid / kSub;
    const unsigned ncand = nb * NI;
    for (unsigned base_idx = 0; base_idx < ncand; base_idx += kResolveThreads / kSub) {
      const unsigned idx = base_idx + (unsigned)grp;
      bool ok = idx < ncand;
      unsigned bits = 0u;
      if (ok) {
        const unsigned id = blist[idx / NI];
        const unsigned b = idx % NI;
        bits = ((id >> L2) << (L1 + L2)) | ((id & (NM - 1)) << L1) | b;
        ok = (bits >> k) == 0u && (!CLOSED || __popc(bits) == w);
      }
      df E = {0.f, 0.f};
      if (ok && ((bits >> sub) & 1u)) {
        const float* Pr = S.pk[sub];
        const float* Pl = S.pkl[sub];
        const unsigned below = bits & ((1u << sub) - 1u);
        float hi = shd[sub].hi, lo = shd[sub].lo;
#pragma unroll 1
        for (int s2 = 0; s2 < kMaxDot - 1; ++s2) {
          const bool on = (below >> s2) & 1u;
          const df t = two_sum(hi, on ? Pr[s2] : 0.f);
          hi = t.hi;
          lo = __fadd_rn(lo, __fadd_rn(t.lo, on ? Pl[s2] : 0.f));
        }
        E = two_sum(hi, lo);
      }
#pragma unroll 1
      for (int off = 1; off < kSub; off <<= 1) {
        df o;
        o.hi = __shfl_xor_sync(kFull, E.hi, off, kSub);
        o.lo = __shfl_xor_sync(kFull, E.lo, off, kSub);
        E = df_add(E, o);
      }
      if (!ok || sub != 0) continue;
      const bool better = E.hi < best.hi || (E.hi == best.hi && E.lo < best.lo) ||
                          (E.hi == best.hi && E.lo == best.lo && __brev(bits) < __brev(bbits));
      if (better) { second = best; best = E; bbits = bits; }
      else if (E.hi < second.hi || (E.hi == second.hi && E.lo < second.lo)) { second = E; }
    }
  }
  auto less = [](df x, df y) { return x.hi < y.hi || (x.hi == y.hi && x.lo < y.lo); };
  auto merge = [&](df ob, df os, unsigned obb) {
    const bool take = less(ob, best) ||
                      (ob.hi == best.hi && ob.lo == best.lo && __brev(obb) < __brev(bbits));
    const df lose = take ? best : ob;
    const df s2 = less(os, second) ? os : second;
    second = less(lose, s2) ? lose : s2;
    if (take) { best = ob; bbits = obb; }
  };
  // only the group leaders (sub = 0: lanes 0 and 16) hold candidates, so
  // one exchange merges a warp
  static_assert(kMaxDot == 16, "two candidate groups of kMaxDot threads per warp");
  {
    df ob, os;
    ob.hi = __shfl_xor_sync(kFull, best.hi, 16);
    ob.lo = __shfl_xor_sync(kFull, best.lo, 16);
    os.hi = __shfl_xor_sync(kFull, second.hi, 16);
    os.lo = __shfl_xor_sync(kFull, second.lo, 16);
    merge(ob, os, __shfl_xor_sync(kFull, bbits, 16));
  }
  if (lane == 0) { rbest[wid] = best; rsec[wid] = second; rbits[wid] = bbits; }
  __syncthreads();
  // warp 0 merges the warps' results as a shuffle tree (the order by energy,
  // then by the reversed bits, is total, so any merge order gives the same
  // best and second); lane 0 decides
  static_assert((NW & (NW - 1)) == 0 && NW <= 32, "warps of the block: a power of two");
  if (wid == 0) {
    const bool have = lane < NW;
    best = have ? rbest[lane] : df{kInf, 0.f};
    second = have ? rsec[lane] : df{kInf, 0.f};
    bbits = have ? rbits[lane] : 0xffffffffu;
#pragma unroll 1
    for (int off = NW / 2; off > 0; off >>= 1) {
      df ob, os;
      ob.hi = __shfl_xor_sync(kFull, best.hi, off);
      ob.lo = __shfl_xor_sync(kFull, best.lo, off);
      os.hi = __shfl_xor_sync(kFull, second.hi, off);
      os.lo = __shfl_xor_sync(kFull, second.lo, off);
      merge(ob, os, __shfl_xor_sync(kFull, bbits, off));
    }
  }
  if (tid == 0) {
    const df ub = S.ub;
    // exact-tie test in double-float: second - best against
    // 1e-10 (1 + |U(base)|) (no FP64 instructions on this path)
    const float gap = second.hi < kInf ? df_add(second, df_neg(best)).hi : kInf;
    const float eps = 1e-10f * (1.f + fabsf(ub.hi));
    const bool ok = fits && bbits != 0xffffffffu && gap > eps;
    S.dok = ok ? 1 : 0;  // not ok: the caller rechecks the pixel in FP64 next
    S.dbits = bbits;
    S.dflags = 0u;
    if (ok && a.out_U) a.out_U[p] = df_to_double(df_add(ub, best));
    // the shortlist length goes to the counters once per block, at the end
    // of the kernel (an atomic here would hold up the barrier below)
    my_slmax = nb > my_slmax ? nb : my_slmax;
  }
  __syncthreads();
  // the charges, one dot per thread
  if (S.dok) {
    unsigned fl = 0u;
    if (tid < n) {
      int ni = rec->base[tid];
      if ((mask >> tid) & 1u) ni += (int)((S.dbits >> __popc(mask & ((1u << tid) - 1u))) & 1u);
      store_charge(a, p * n + tid, ni, fl);
      if (fl) atomicOr(&S.dflags, fl);
    }
    __syncthreads();
    if (tid == 0) {
      if (a.out_flags) a.out_flags[p] = (uint8_t)(flags0 | kFlagRechecked | S.dflags);
      my_res += 1;
    }
  }
}

// ---------------------------------------------------------------------------
// (a7) FP64 recheck of one list entry (one block per pixel):
//   1. c, the continuous minimum and the candidate set again, in FP64
//      (c and h by N threads in parallel, the minimum by one thread); when
//      that set is the one the FP32 path searched and the FP32 order of the
//      best two was certain, the search's result stands and the pixel is
//      done;
//   2. the FP32 search over that set with all threads -> m1;
//   3. the same search collecting every block whose minimum is within the
//      near-tie bound of m1 (the exact argmin is guaranteed to be there);
//   4. exact FP64 energies of those candidates, ties to the
//      lexicographically smallest charge vector.
// ---------------------------------------------------------------------------
struct RecheckShared {
  __align__(16) double qK[32][kQPRow];  // FP64 team QP of warp 0
  int qa[32];
  double qz[32], qc[32], v64[kMaxDot], sx64[kMaxDot];
  int sqp;
  float sM[kMaxDot * kLdM];
  int sdot[kMaxDot];
  float sh[kMaxDot];
  double sh64[kMaxDot], sc64[kMaxDot];
  int sbase[kMaxDot];
  int sk, sw, sstatus;
  unsigned smask, sflags;
  float sbound;
  float rm1[kRecheckThreads / 32];
  double re[kRecheckThreads / 32];
  unsigned rbits[kRecheckThreads / 32];
  unsigned blist[kBcap];
  unsigned bcount;
};

template <bool CLOSED>
__device__ inline void recheck_entry(const GsLaunch& L, const ArrayDesc& a, RecheckShared& S,
                                     ListEntry fe) {
  constexpr int L1 = kCheckL1, L2 = kCheckL2;
  constexpr int NI = 1 << L1;
  constexpr int NM = 1 << L2;
  constexpr int NW = kRecheckThreads / 32;
  const int n = a.n;
  const int tid = threadIdx.x, wid = tid >> 5, lane = tid & 31;
  const float* sM = S.sM;
  int* sdot = S.sdot;
  float* sh = S.sh;
  double* sh64 = S.sh64;
  double* sc64 = S.sc64;
  int* sbase = S.sbase;
  int& sk = S.sk;
  int& sw = S.sw;
  int& sstatus = S.sstatus;
  unsigned& smask = S.smask;
  unsigned& sflags = S.sflags;
  float& sbound = S.sbound;
  float* rm1 = S.rm1;
  double* re = S.re;
  unsigned* rbits = S.rbits;
  unsigned* blist = S.blist;
  unsigned& bcount = S.bcount;
  const long long p = fe.p;
  if (tid < n) sc64[tid] = pixel_c_f64(a.md, a.ng, a.sc, a.mt.carrier, p, tid);
  __syncthreads();
  if (tid < 32) {
    // continuous minimum in FP64 by warp 0, lane i owning dot i: analytic
    // (Appendix C / D), else the team active-set QP
    const int lt = tid;
    const bool live = lt < n;
    const double ci = live ? sc64[lt] : 0.0;
    double csum = ci, cmax = live ? fabs(ci) : 0.0;
    for (int off = 1; off < 32; off <<= 1) {
      csum += __shfl_xor_sync(kFull, csum, off);
      cmax = fmax(cmax, __shfl_xor_sync(kFull, cmax, off));
    }
    const double nh = (double)a.mt.n_charges;
    double x = CLOSED ? ci + (nh - csum) * (live ? a.md->vs[lt] : 0.0) : ci;
    const unsigned A = __ballot_sync(kFull, live && x < 0.0);
    int st = 0;
    if (A) {
      if (CLOSED && a.mt.n_charges == 0) {
        x = 0.0;
      } else {
        double vi = 0.0;
        if (live)
          for (int j = 0; j < n; ++j) vi += a.md->Cdd[lt * n + j];
        if (lt < kMaxDot) S.v64[lt] = vi;
        double s = vi;
        for (int off = 1; off < 32; off <<= 1) s += __shfl_xor_sync(kFull, s, off);
        __syncwarp();
        unsigned Af = 0u;
        const double tol = 1e-12 * (fmax(cmax, 1.0) + nh);
        // warm start from the active set the FP32 QP settled on, if any
        const unsigned A0 = a.recs[p].qpA ? (unsigned)a.recs[p].qpA : A;
        st = qp_team<double, CLOSED>(n, lt, 32, kFull, 0, a.md->Cdd, n, S.v64, s, ci, nh, A0,
                                     tol, 8 * n + 8, S.qK, S.qa, S.qz, S.qc, x, Af);
      }
    }
    if (live) S.sx64[lt] = x;
    if (lt == 0) S.sqp = (A ? 1 : 0) | (st != 0 ? 2 : 0);
  }
  __syncthreads();
  if (wid == 0) {
    // the candidate set in FP64 (the rules of candidate_set_f64), lane i
    // deciding dot i, the closed doubling loop warp-uniform
    const bool live = lane < n;
    unsigned fl = (S.sqp & 1) ? kFlagQP : 0u;
    unsigned mask = 0u;
    int st = -1, w = -1, bi = 0;
    if (a.md->status == 0 && !(S.sqp & 2)) {
      const double xl = live ? S.sx64[lane] : 0.0;
      const double xi = xl > 0.0 ? xl : 0.0;
      const double fli = floor(xi);
      const double fr = xi - fli;
      double tt = a.mt.t;
      for (int iter = 0; iter < 40; ++iter) {
        const bool am = live && fabs(fr - 0.5) <= 0.5 * tt;
        bi = live ? (int)fli + ((!am && fr >= 0.5) ? 1 : 0) : 0;
        mask = __ballot_sync(kFull, am);
        if (!CLOSED) { st = 0; break; }
        int sum = bi;
        for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(kFull, sum, off);
        w = a.mt.n_charges - sum;
        if (w >= 0 && w <= __popc(mask)) { st = 0; break; }
        if (tt >= 1.0) break;
        tt = (tt <= 0.0) ? 1.0 : fmin(2.0 * tt, 1.0);
        fl |= kFlagDoubled;
      }
    }
    if (live) sbase[lane] = bi;
    // same candidate set as the FP32 search and a certain order: keep its result
    const PixRec* rec = a.recs + p;
    const bool same = st == 0 && fe.tie == 0 && mask == (unsigned)rec->mask &&
                      (!CLOSED || w == (int)rec->w) &&
                      __all_sync(kFull, !live || bi == (int)rec->base[lane]);
    if (lane == 0) {
      sflags = fl;
      smask = mask;
      sw = CLOSED ? w : -1;
      bcount = 0u;
      sstatus = st;
      if (same) {
        if (a.out_flags) a.out_flags[p] = (uint8_t)(a.out_flags[p] | fl | kFlagRechecked);
        sstatus = 1;
      }
    }
  }
  __syncthreads();
  if (sstatus == 1) return;
  if (sstatus != 0) {
    if (tid == 0) {
      if (a.out_flags) a.out_flags[p] |= (uint8_t)kFlagUnresolved;
      atomicAdd(&L.cnt->unresolved, 1ull);
    }
    return;
  }
  const unsigned mask = smask;
  if (tid < n && ((mask >> tid) & 1u)) {
    double h = 0.0;
    for (int j = 0; j < n; ++j) h += a.md->M[tid * n + j] * ((double)sbase[j] - sc64[j]);
    const int s = __popc(mask & ((1u << tid) - 1u));
    sdot[s] = tid;
    sh64[s] = h;
    sh[s] = __double2float_rn(h);
  }
  __syncthreads();
  if (tid == 0) {
    const int k = __popc(mask);
    float S = 0.f;
    for (int s = 0; s < k; ++s) {
      S += fabsf(sh[s]) + 0.5f * sM[sdot[s] * kLdM + sdot[s]];
      for (int q = 0; q < s; ++q) S += fabsf(sM[sdot[s] * kLdM + sdot[q]]);
    }
    sk = k;
    sbound = near_tie_bound(S, k, L2);
  }
  __syncthreads();
  const SlotView sv{sdot, sh, sk, sw};
  float m1, m2;
  unsigned b1;
  unsigned long long ev = 0;
  static_assert(kRecheckThreads <= 512, "the walk's team is the block: at most 9 lane bits");
  search_lane<L1, L2, CLOSED, false, false, 9>(sM, sv, tid, kRecheckThreads, 0.f, nullptr,
                                     nullptr, 0u, m1, b1, m2, ev);
  for (int off = 16; off > 0; off >>= 1) m1 = fminf(m1, __shfl_xor_sync(kFull, m1, off));
  if (lane == 0) rm1[wid] = m1;
  __syncthreads();
  m1 = kInf;
  for (int i = 0; i < NW; ++i) m1 = fminf(m1, rm1[i]);
  const float thr = m1 + sbound;
  float d1, d2;
  unsigned db;
  search_lane<L1, L2, CLOSED, true, false, 9>(sM, sv, tid, kRecheckThreads, thr, blist,
                                    &bcount, kBcap, d1, db, d2, ev, nullptr, nullptr, nullptr,
                                    thr + 2.0f * sbound, a.md->k.qneg);
  __syncthreads();
  const unsigned nb = bcount;
  const bool overflowed = nb > kBcap;
  const unsigned nbl = overflowed ? kBcap : nb;
  // exact FP64 energies of the shortlisted candidates
  double best = 1.0e300;
  unsigned bbits = 0xffffffffu;
  const int k = sk;
  for (unsigned idx = tid; idx < nbl * NI; idx += kRecheckThreads) {
    const unsigned id = blist[idx / NI];
    const unsigned b = idx % NI;
    const unsigned bits = ((id >> L2) << (L1 + L2)) | ((id & (NM - 1)) << L1) | b;
    if ((bits >> k) != 0u) continue;
    if (CLOSED && __popc(bits) != sw) continue;
    double E = 0.0;
    for (unsigned m = bits; m; m &= m - 1u) {
      const int s = __ffs(m) - 1;
      const int d = sdot[s];
      E += sh64[s] + 0.5 * a.md->M[d * n + d];
      for (unsigned q = bits & ((1u << s) - 1u); q; q &= q - 1u)
        E += a.md->M[d * n + sdot[__ffs(q) - 1]];
    }
    if (E < best || (E == best && __brev(bits) < __brev(bbits))) {
      best = E;
      bbits = bits;
    }
  }
  for (int off = 16; off > 0; off >>= 1) {
    const double oe = __shfl_xor_sync(kFull, best, off);
    const unsigned ob = __shfl_xor_sync(kFull, bbits, off);
    if (oe < best || (oe == best && __brev(ob) < __brev(bbits))) { best = oe; bbits = ob; }
  }
  if (lane == 0) { re[wid] = best; rbits[wid] = bbits; }
  __syncthreads();
  if (tid == 0) {
    for (int i = 1; i < NW; ++i)
      if (re[i] < best || (re[i] == best && __brev(rbits[i]) < __brev(bbits))) {
        best = re[i];
        bbits = rbits[i];
      }
    unsigned flags = (a.out_flags ? a.out_flags[p] : 0u) | sflags | kFlagRechecked;
    const bool settled = !overflowed && bbits != 0xffffffffu;
    if (!settled) {
      flags |= kFlagUnresolved;
      atomicAdd(&L.cnt->unresolved, 1ull);
      if (a.out_flags) a.out_flags[p] = (uint8_t)flags;
    }
    sflags = flags;
    rbits[0] = bbits;
    sstatus = settled ? 2 : 3;
    atomicMax(&L.cnt->shortlist_max, (unsigned long long)nb);
  }
  __syncthreads();
  // the charges and U(n*) = 1/2 r^T M r, r = n* - c, by warp 0: lane i its
  // dot's charge and row of M r, then a shuffle sum
  if (sstatus == 2 && wid == 0) {
    const unsigned bb = rbits[0];
    const bool live = lane < n;
    int ni = live ? sbase[lane] : 0;
    if (live && ((mask >> lane) & 1u)) ni += (int)((bb >> __popc(mask & ((1u << lane) - 1u))) & 1u);
    double row = 0.0;
    for (int j = 0; j < n; ++j) {
      const int nj = __shfl_sync(kFull, ni, j);
      if (live) row += a.md->M[lane * n + j] * ((double)nj - sc64[j]);
    }
    double u = live ? ((double)ni - sc64[lane]) * row : 0.0;
    for (int off = 16; off > 0; off >>= 1) u += __shfl_xor_sync(kFull, u, off);
    unsigned fl = 0u;
    if (live) store_charge(a, p * n + lane, ni, fl);
    fl = __reduce_or_sync(kFull, fl);
    if (lane == 0) {
      if (a.out_U) a.out_U[p] = 0.5 * u;
      if (a.out_flags) a.out_flags[p] = (uint8_t)(sflags | fl);
    }
  }
}

}  // namespace qa
