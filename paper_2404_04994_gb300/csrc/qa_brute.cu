// qa_brute.cu -- brute-force ground state (Table I, brute-force row): the
// argmin of U(n) = 1/2 (n - c)^T M (n - c) over every n in [0, n_max]^N
// (open) or every n >= 0 with sum n = N_hat (closed), exact in FP64.  It is
// the reference the default and thresholded methods are measured against
// (Sec. VII, Fig. 4) and an on-device exactness check of their maps.
//
// With R the digit range, the free dots (all N open; the first N - 1 closed,
// the last taking N_hat minus the rest) form a mixed-radix number, dot 0 most
// significant, so numeric order of the code is lexicographic order of n.
//
// Every state is covered, in FP32 first.  In the free digits y the energy is
// E(y) = 1/2 y^T M' y - d' . y (closed arrays eliminate the last dot, M' and
// d' below), so along a line of the last free digit it is a parabola and the
// line's minimum over its range is the integer nearest the vertex, clamped:
// about fifteen FP32 operations for R states.  A team of lanes splits the
// leading digits ("hi states"), each lane walks the lines of the last digit
// but one.  FP32 settles a pixel only when the gap between its best two
// states exceeds twice a bound of the FP32 error (and FP64's near-tie
// margin); otherwise the lines within that threshold are collected and
// their states evaluated in FP64 from scratch, which gives the argmin, the
// near-tie flag and the lexicographic order of equal energies.  A pixel whose
// list overflows, or whose bound is not a number, is walked in FP64 state by
// state (brute_walk_f64).  U(n*) is always formed in FP64.
//
// What bounds it: FP32 issue, in the lines and the per-pixel merge; the FP64
// set-up (GB300 issues two FP64 operations per SM and clock) is spread over
// full warps, one (pixel, dot) pair per thread.  4 dots, n_max = 7, 200 x 200
// pixels: 67 us; the walk of every state in FP64 took 4000 us, and hi states
// rebuilt from their digits for every pixel instead of the table 101 us.
#include "qa_launch.h"
#include "qa_prep.cuh"

namespace qa {

constexpr int kBruteThreads = 128;
constexpr int kBrutePix = 128;      // pixels per block at most
constexpr int kBruteVec = 512;      // ... times dots (or 32 pixels of 16 dots)
constexpr int kBruteTab = 2048;     // floats of the hi-state table
constexpr int kBruteList = 8;       // shortlisted lines per lane of a team
constexpr float kBruteInf = __builtin_huge_valf();

struct BruteShared {
  double M[kMaxDot * kMaxDot];
  double c[kBruteVec];                 // per pixel and dot (stride N): c,
  double d[kBruteVec];                 // M c, at the end the rows of M (n* - c)
  float Mr[kMaxDot][kMaxDot + 1];      // M' of the free digits
  float dr[kBruteVec];                 // d' of the free digits (stride N)
  float ca[kBruteVec];                 // |c_i d_i| / 2: the energy's dropped constant
  float hi[kBruteTab];                 // hi states: Q, t, s, rem, then the digits
  float sumM;                          // sum |M'_ij| (open), max |M'_ij| (closed)
  unsigned long long code[kBrutePix];  // the answer
  unsigned char tie[kBrutePix];        // 1: near tie, 2: no state
  int nv[kBruteVec];                   // its charges
  unsigned long long list[kBruteThreads * kBruteList];  // per team: shortlisted lines (from
                                                        // bit 8), the minimum's digit below
  unsigned cnt[kBruteThreads];
};

// Digits of code (mixed radix R, nfree digits, dot 0 most significant).
__device__ __forceinline__ void brute_digits(unsigned long long code, int R, int nfree,
                                             int* nv) {
  for (int i = nfree - 1; i >= 0; --i) {
    if (code <= 0xffffffffull) {
      const unsigned c32 = (unsigned)code, q = c32 / (unsigned)R;
      nv[i] = (int)(c32 - q * (unsigned)R);
      code = q;
    } else {
      const unsigned long long q = code / (unsigned long long)R;
      nv[i] = (int)(code - q * (unsigned long long)R);
      code = q;
    }
  }
}

__device__ __forceinline__ void brute_keep(double E, unsigned long long code, double& e1,
                                           unsigned long long& c1, double& e2) {
  if (E < e1 || (E == e1 && code < c1)) {
    e2 = e1;
    e1 = E;
    c1 = code;
  } else if (E < e2) {
    e2 = E;
  }
}

// Every state of one pixel in FP64 by the T lanes of its team (lane lt): the
// lanes split the leading digits, each walks the trailing `ni` digits in
// reflected mixed-radix Gray order, one digit +-1 per step, updating
//     E(n) = 1/2 n^T M n - n^T d,  d = M c,  y = M n,
//     E(n + s e_i) = E(n) + s (y_i - d_i) + M_ii / 2,   y += s M e_i,
// and rebuilds E and y from scratch at every outer state.
__device__ __noinline__ void brute_walk_f64(const BruteLaunch& L, const double* M,
                                            const double* d, int lt, int T, double& e1,
                                            unsigned long long& c1, double& e2) {
  const int n = L.a.n;
  const bool closed = L.a.mt.closed != 0;
  const int R = L.radix, nfree = L.nfree, ni = L.ni;
  const int last = n - 1;
  const int nhat = L.a.mt.n_charges;
  unsigned long long rpow_in = 1;  // R^ni
  for (int j = 0; j < ni; ++j) rpow_in *= (unsigned long long)R;
  for (unsigned long long o = lt; o < L.nouter; o += T) {
    int nv[kMaxDot];
    brute_digits(o * rpow_in, R, nfree, nv);
    if (closed) {
      int s = 0;
      for (int j = 0; j < nfree; ++j) s += nv[j];
      nv[last] = nhat - s;
    }
    double y[kMaxDot];
    double E = 0.0;
    for (int i = 0; i < n; ++i) {
      double r = 0.0;
      for (int j = 0; j < n; ++j) r += M[i * n + j] * (double)nv[j];
      y[i] = r;
    }
    for (int i = 0; i < n; ++i) E += (double)nv[i] * (0.5 * y[i] - d[i]);
    int dir[kMaxDot];
    for (int j = 0; j < ni; ++j) dir[j] = 1;
    unsigned long long code = o * rpow_in;
    for (;;) {
      if (!closed || nv[last] >= 0) brute_keep(E, code, e1, c1, e2);
      // next state: lowest trailing digit that can move in its direction
      int j = 0;
      unsigned long long place = 1;
      while (j < ni) {
        const int i = nfree - 1 - j;
        const int v = nv[i] + dir[j];
        if (v >= 0 && v < R) break;
        dir[j] = -dir[j];
        place *= (unsigned long long)R;
        ++j;
      }
      if (j == ni) break;
      const int i = nfree - 1 - j;
      const int sg = dir[j];
      E += (double)sg * (y[i] - d[i]) + 0.5 * M[i * n + i];
      for (int q = 0; q < n; ++q) y[q] += (double)sg * M[q * n + i];
      nv[i] += sg;
      code = sg > 0 ? code + place : code - place;
      if (closed) {  // the last dot gives the unit back
        E += (double)(-sg) * (y[last] - d[last]) + 0.5 * M[last * n + last];
        for (int q = 0; q < n; ++q) y[q] -= (double)sg * M[q * n + last];
        nv[last] -= sg;
      }
    }
  }
}

// E of one state in FP64 from scratch (the same sums as the walk's rebuild).
__device__ __noinline__ double brute_energy_f64(const BruteLaunch& L, const double* M,
                                                const double* d, unsigned long long code) {
  const int n = L.a.n;
  int nv[kMaxDot];
  brute_digits(code, L.radix, L.nfree, nv);
  if (L.a.mt.closed) {
    int s = 0;
    for (int j = 0; j < L.nfree; ++j) s += nv[j];
    nv[n - 1] = L.a.mt.n_charges - s;
  }
  double E = 0.0;
  for (int i = 0; i < n; ++i) {
    double r = 0.0;
    for (int j = 0; j < n; ++j) r += M[i * n + j] * (double)nv[j];
    E += (double)nv[i] * (0.5 * r - d[i]);
  }
  return E;
}

// FP32 constants of a hi state (the digits above the last two): its energy
// A, the linear coefficients t of the last digit but one and s of the last,
// and what the digits leave of N_hat (closed; negative: no state).  All but
// the terms in d' belong to the array: where they fit, the block tabulates
// them (Q = 1/2 y^T M' y, the couplings to the last two digits, rem and the
// digits as floats), so that a pixel's hi state costs a 16-byte load and one
// product per digit.
struct BruteHi {
  float A, t, s;
  int rem;
};

// The array's part from scratch; the digits go to dig (a byte each).
template <typename ID>
__device__ __forceinline__ BruteHi brute_hi_scratch(const BruteShared& sh, ID hs, int R,
                                                    int nfree, int nhat,
                                                    unsigned long long (&dig)[2]) {
  const int nh = nfree > 2 ? nfree - 2 : 0;
  BruteHi h = {0.f, 0.f, 0.f, nhat};
  dig[0] = dig[1] = 0;
  for (int i = nh - 1; i >= 0; --i) {
    const ID qt = hs / (ID)R;
    const unsigned v = (unsigned)(hs - qt * (ID)R);
    hs = qt;
    const float* Mi = sh.Mr[i];
    const float fv = (float)v;
    float acc = 0.5f * Mi[i] * fv;
    for (int j = i + 1; j < nh; ++j)
      acc = fmaf(Mi[j], (float)(unsigned)((dig[j >> 3] >> (8 * (j & 7))) & 255u), acc);
    h.A = fmaf(fv, acc, h.A);
    h.t = fmaf(Mi[nfree - 2], fv, h.t);
    h.s = fmaf(Mi[nfree - 1], fv, h.s);
    h.rem -= (int)v;
    dig[i >> 3] |= (unsigned long long)v << (8 * (i & 7));
  }
  return h;
}

template <typename ID>
__device__ __forceinline__ BruteHi brute_hi(const BruteShared& sh, const float* dr, ID hs, int R,
                                            int nfree, int nhat, bool tab) {
  const int nh = nfree > 2 ? nfree - 2 : 0;
  BruteHi h;
  if (tab) {
    const float* row = sh.hi + (unsigned)hs * (unsigned)(4 + nh);
    h = {row[0], row[1], row[2], (int)row[3]};
    for (int i = 0; i < nh; ++i) h.A = fmaf(-dr[i], row[4 + i], h.A);
  } else {
    unsigned long long dig[2];
    h = brute_hi_scratch<ID>(sh, hs, R, nfree, nhat, dig);
    for (int i = 0; i < nh; ++i)
      h.A = fmaf(-dr[i], (float)(unsigned)((dig[i >> 3] >> (8 * (i & 7))) & 255u), h.A);
  }
  if (nfree >= 2) h.t -= dr[nfree - 2];
  if (nfree >= 1) h.s -= dr[nfree - 1];
  return h;
}

// A line's minimum over the last digit, 0 <= q <= hi: the integer nearest the
// vertex of b + s q + Mll / 2 q^2.
__device__ __forceinline__ float brute_line(float b, float s, float hi, float halfM, float ninv,
                                            float& q) {
  constexpr float kRound = 12582912.f;  // 1.5 2^23: adding it rounds to an integer
  q = fminf(fmaxf(s * ninv, 0.f), hi);
  q = __fsub_rn(__fadd_rn(q, kRound), kRound);
  return fmaf(q, fmaf(q, halfM, s), b);
}

// ID: the type that holds a line's number (hi state times R plus the last
// digit but one).
template <typename ID>
__global__ void __launch_bounds__(kBruteThreads, 6) k_brute(BruteLaunch L) {
  __shared__ BruteShared sh;
  const ArrayDesc& a = L.a;
  const int n = a.n;
  const bool closed = a.mt.closed != 0;
  const int R = L.radix, nfree = L.nfree;
  const int last = n - 1;
  const int nhat = a.mt.n_charges;
  const int PB = L.pix;
  const long long p0 = (long long)blockIdx.x * PB;
  const int np = (int)(a.sc.P - p0 < PB ? a.sc.P - p0 : PB);
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) sh.M[e] = a.md->M[e];
  // c and d = M c in FP64, one (pixel, dot) per thread
  for (int e = threadIdx.x; e < np * n; e += blockDim.x) {
    const int q = e / n, i = e - q * n;
    sh.c[q * n + i] = pixel_c_f64(a.md, a.ng, a.sc, a.mt.carrier, p0 + q, i);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < np * n; e += blockDim.x) {
    const int q = e / n, i = e - q * n;
    double s = 0.0;
    for (int j = 0; j < n; ++j) s += sh.M[i * n + j] * sh.c[q * n + j];
    sh.d[q * n + i] = s;
    sh.ca[q * n + i] = 0.5f * fabsf((float)s * (float)sh.c[q * n + i]);
  }
  // M' of the free digits: M itself (open), or with n_last = N_hat - sum y,
  // M'_ij = M_ij - M_il - M_jl + M_ll
  for (int e = threadIdx.x; e < nfree * nfree; e += blockDim.x) {
    const int i = e / nfree, j = e - i * nfree;
    double m = sh.M[i * n + j];
    if (closed) m = (m - sh.M[i * n + last]) - (sh.M[j * n + last] - sh.M[last * n + last]);
    sh.Mr[i][j] = (float)m;
  }
  __syncthreads();
  // d' = d (open) or d_i - d_l - N_hat (M_il - M_ll)
  for (int e = threadIdx.x; e < np * nfree; e += blockDim.x) {
    const int q = e / nfree, i = e - q * nfree;
    double v = sh.d[q * n + i];
    if (closed)
      v = (v - sh.d[q * n + last]) - (double)nhat * (sh.M[i * n + last] - sh.M[last * n + last]);
    sh.dr[q * n + i] = (float)v;
  }
  if (threadIdx.x < 32) {
    float s = 0.f, m = 0.f;
    for (int e = threadIdx.x; e < nfree * nfree; e += 32) {
      const float v = fabsf(sh.Mr[e / nfree][e % nfree]);
      s += v;
      m = fmaxf(m, v);
    }
    for (int off = 16; off > 0; off >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, off);
      m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    }
    if (threadIdx.x == 0) sh.sumM = closed ? m : s;
  }
  const ID nh = (ID)L.nhi;  // hi states
  const int nhd = nfree > 2 ? nfree - 2 : 0;
  const bool tab = L.nhi * (unsigned)(4 + nhd) <= (unsigned)kBruteTab;
  if (tab) {
    for (unsigned hs = threadIdx.x; hs < (unsigned)nh; hs += blockDim.x) {
      unsigned long long dig[2];
      const BruteHi h = brute_hi_scratch<unsigned>(sh, hs, R, nfree, nhat, dig);
      float* row = sh.hi + hs * (unsigned)(4 + nhd);
      row[0] = h.A;
      row[1] = h.t;
      row[2] = h.s;
      row[3] = (float)h.rem;
      for (int i = 0; i < nhd; ++i)
        row[4 + i] = (float)(unsigned)((dig[i >> 3] >> (8 * (i & 7))) & 255u);
    }
  }
  __syncthreads();

  const int T = L.team;
  const int team = threadIdx.x / T, lt = threadIdx.x % T;
  const int wl = threadIdx.x & 31;
  const unsigned tmask = T >= 32 ? 0xffffffffu : (((1u << T) - 1u) << (wl & ~(T - 1)));
  const float Mll = nfree >= 1 ? sh.Mr[nfree - 1][nfree - 1] : 1.f;
  const float Mmm = nfree >= 2 ? sh.Mr[nfree - 2][nfree - 2] : 0.f;
  const float Mml = nfree >= 2 ? sh.Mr[nfree - 2][nfree - 1] : 0.f;
  const float halfM = 0.5f * Mll, ninv = -1.f / Mll;
  const int Rm = nfree >= 2 ? R : 1;        // values of the last digit but one
  const int topl = nfree >= 1 ? R - 1 : 0;  // largest last digit
  unsigned long long* list = sh.list + team * T * kBruteList;

  for (int q = team; q < np; q += kBruteThreads / T) {
    const float* dr = sh.dr + q * n;
    float m1 = kBruteInf, m2 = kBruteInf;
    ID best = 0;  // best line
    for (ID hs = lt; hs < nh; hs += T) {
      const BruteHi h = brute_hi<ID>(sh, dr, hs, R, nfree, nhat, tab);
      if (closed && h.rem < 0) continue;
      const int vtop = closed ? (h.rem < Rm - 1 ? h.rem : Rm - 1) : Rm - 1;
      float l1 = kBruteInf;
      int lv = 0;
      float fv = 0.f, top = (float)(closed ? min(h.rem, topl) : topl);
#pragma unroll 4
      for (int v = 0; v <= vtop; ++v) {
        float qq;
        const float E = brute_line(fmaf(fmaf(0.5f * Mmm, fv, h.t), fv, h.A),
                                   fmaf(Mml, fv, h.s), top, halfM, ninv, qq);
        m2 = fminf(m2, fmaxf(l1, E));
        lv = E < l1 ? v : lv;
        l1 = fminf(l1, E);
        fv += 1.f;
        if (closed) top -= 1.f;
      }
      m2 = fminf(m2, fmaxf(m1, l1));
      best = l1 < m1 ? hs * (ID)Rm + (ID)lv : best;
      m1 = fminf(m1, l1);
    }
    for (int off = 1; off < T; off <<= 1) {
      const float o1 = __shfl_xor_sync(tmask, m1, off);
      const float o2 = __shfl_xor_sync(tmask, m2, off);
      const ID ob = __shfl_xor_sync(tmask, best, off);
      const bool take = o1 < m1 || (o1 == m1 && ob < best);
      m2 = fminf(fminf(m2, o2), take ? m1 : o1);
      if (take) { m1 = o1; best = ob; }
    }
    // the winning line's digit and its neighbours on the line
    const ID bh = best / (ID)Rm;
    const int bv = (int)(best - bh * (ID)Rm);
    const BruteHi hb = brute_hi<ID>(sh, dr, bh, R, nfree, nhat, tab);
    const float fb = (float)bv;
    const float sb = fmaf(Mml, fb, hb.s);
    const float topb = (float)(closed ? min(hb.rem - bv, topl) : topl);
    const float bb = fmaf(fmaf(0.5f * Mmm, fb, hb.t), fb, hb.A);
    float qb;
    brute_line(bb, sb, topb, halfM, ninv, qb);
    if (qb >= 1.f) m2 = fminf(m2, fmaf(qb - 1.f, fmaf(qb - 1.f, halfM, sb), bb));
    if (qb + 1.f <= topb) m2 = fminf(m2, fmaf(qb + 1.f, fmaf(qb + 1.f, halfM, sb), bb));
    // the FP32 error of an energy: rounded M' and d' and at most 2 nfree + 12
    // roundings of partial sums, each at most S = sum of the terms' magnitudes
    // over the box; and FP64's near-tie margin 1e-9 max(1, |U|), |U| at most
    // |E| + the dropped constant
    float sd = 0.f, cst = 0.f;
    for (int i = 0; i < n; ++i) cst += sh.ca[q * n + i];
    for (int i = 0; i < nfree; ++i) sd = closed ? fmaxf(sd, fabsf(dr[i])) : sd + fabsf(dr[i]);
    const float rr = (float)(R - 1);
    const float S = fmaf(0.5f * rr * rr, sh.sumM, rr * sd);
    if (closed) {
      const float fn = (float)nhat;
      cst += fabsf(0.5f * fn * fn * (float)sh.M[last * n + last]) +
             fabsf(fn * (float)sh.d[q * n + last]);
    }
    const float thr = 2.f * (float)(2 * nfree + 12) * 5.9604645e-8f * S +
                      2e-9f * (1.f + fabsf(m1) + cst);
    unsigned long long code = (unsigned long long)best * (unsigned long long)(topl + 1) +
                              (unsigned long long)(int)qb;
    unsigned char tie = 0;
    // (the vertex picks the line's minimum while Mll is well above the error)
    const bool sane = Mll > 2.f * thr;
    if (!(m2 - m1 > thr && sane)) {  // the same for every lane of the team
      // the lines within the threshold, then their states in FP64: the
      // line's minimum and its neighbours (the states beyond lie at least
      // Mll above the minimum, hence above the threshold)
      if (lt == 0) sh.cnt[team] = 0u;
      __syncwarp(tmask);
      const float lim = m1 + thr;
      bool ok = lim < kBruteInf && sane;
      if (ok) {
        for (ID hs = lt; hs < nh; hs += T) {
          const BruteHi h = brute_hi<ID>(sh, dr, hs, R, nfree, nhat, tab);
          if (closed && h.rem < 0) continue;
          const int vtop = closed ? (h.rem < Rm - 1 ? h.rem : Rm - 1) : Rm - 1;
          for (int v = 0; v <= vtop; ++v) {
            const float fv = (float)v;
            float qq;
            const float E = brute_line(
                fmaf(fmaf(0.5f * Mmm, fv, h.t), fv, h.A), fmaf(Mml, fv, h.s),
                (float)(closed ? min(h.rem - v, topl) : topl), halfM, ninv, qq);
            if (E <= lim) {
              const unsigned at = atomicAdd(&sh.cnt[team], 1u);
              const unsigned long long line = (unsigned long long)(hs * (ID)Rm) + (unsigned)v;
              if (at < (unsigned)(T * kBruteList)) list[at] = (line << 8) | (unsigned)(int)qq;
            }
          }
        }
      }
      __syncwarp(tmask);
      const unsigned cnt = sh.cnt[team];
      ok = ok && cnt >= 1 && cnt <= (unsigned)(T * kBruteList);
      double e1 = 1.0e300, e2 = 1.0e300;
      unsigned long long c1 = ~0ull;
      if (ok) {
        for (unsigned e = lt; e < 3 * cnt; e += T) {
          const unsigned long long cc = list[e / 3] >> 8;
          const int qd = (int)(list[e / 3] & 255u) + (int)(e % 3) - 1;
          // the line's range: its other digits leave the last one nhat - sum
          int top = topl;
          if (closed) {
            ID w = (ID)cc;
            int s = 0;
            for (int j = 0; j < nfree - 1; ++j) {
              const ID q1 = w / (ID)R;
              s += (int)(w - q1 * (ID)R);
              w = q1;
            }
            top = min(top, nhat - s);
          }
          if (qd < 0 || qd > top) continue;
          const unsigned long long cs =
              cc * (unsigned long long)(topl + 1) + (unsigned long long)qd;
          brute_keep(brute_energy_f64(L, sh.M, sh.d + q * n, cs), cs, e1, c1, e2);
        }
      } else {
        brute_walk_f64(L, sh.M, sh.d + q * n, lt, T, e1, c1, e2);
      }
      // team: best (energy, then smaller code), second-best energy
      for (int off = 1; off < T; off <<= 1) {
        const double oe1 = __shfl_xor_sync(tmask, e1, off);
        const double oe2 = __shfl_xor_sync(tmask, e2, off);
        const unsigned long long oc1 = __shfl_xor_sync(tmask, c1, off);
        const bool take = oe1 < e1 || (oe1 == e1 && oc1 < c1);
        const double lose = take ? e1 : oe1;
        e2 = fmin(fmin(e2, oe2), lose);
        if (take) { e1 = oe1; c1 = oc1; }
      }
      code = c1;
      // |U| for the margin: E plus the constant dropped from it
      double U = e1;
      for (int i = 0; i < n; ++i) U += 0.5 * sh.c[q * n + i] * sh.d[q * n + i];
      if (!(e2 - e1 > 1e-9 * fmax(1.0, fabs(U)))) tie = 1;
      if (c1 == ~0ull) tie = 2;
      __syncwarp(tmask);
    }
    if (lt == 0) {
      sh.code[q] = code;
      sh.tie[q] = tie;
    }
  }
  __syncthreads();
  // the charges, then the rows of M (n* - c), one (pixel, dot) per thread, then
  // U(n*) and the flags, one pixel per thread
  for (int q = threadIdx.x; q < np; q += blockDim.x) {
    if (sh.tie[q] == 2) continue;
    brute_digits(sh.code[q], R, nfree, sh.nv + q * n);
    if (closed) {
      int s = 0;
      for (int j = 0; j < nfree; ++j) s += sh.nv[q * n + j];
      sh.nv[q * n + last] = nhat - s;
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < np * n; e += blockDim.x) {
    const int q = e / n, i = e - q * n;
    if (sh.tie[q] == 2) {  // no admissible state (cannot happen for valid input)
      a.out_n[p0 * n + e] = 0;
      continue;
    }
    double r = 0.0;
    for (int j = 0; j < n; ++j) r += sh.M[i * n + j] * ((double)sh.nv[q * n + j] - sh.c[q * n + j]);
    sh.d[e] = r;  // M c is done with
    a.out_n[p0 * n + e] = (int8_t)sh.nv[e];
  }
  __syncthreads();
  for (int q = threadIdx.x; q < np; q += blockDim.x) {
    unsigned flags = sh.tie[q] == 1 ? kBruteNearTie : sh.tie[q] == 2 ? kBruteNone : 0u;
    double U = 0.0;
    if (sh.tie[q] != 2) {
      for (int i = 0; i < n; ++i) {
        U += ((double)sh.nv[q * n + i] - sh.c[q * n + i]) * sh.d[q * n + i];
        if (!closed && sh.nv[q * n + i] == L.n_max) flags |= kBruteAtBox;
      }
      U *= 0.5;
    }
    if (a.out_U) a.out_U[p0 + q] = U;
    if (a.out_flags) a.out_flags[p0 + q] = (uint8_t)flags;
  }
}

cudaError_t launch_brute(const BruteLaunch& L0, cudaStream_t st) {
  if (L0.a.sc.P == 0) return cudaSuccess;
  BruteLaunch L = L0;
  // lanes per pixel: one per hi state, as many as a warp has at most
  L.nhi = 1;
  for (int j = 2; j < L.nfree; ++j) L.nhi *= (unsigned long long)L.radix;
  L.team = 1;
  while (L.team < 32 && (unsigned long long)(2 * L.team) <= L.nhi) L.team *= 2;
  // pixels per block: eight per team where the shared arrays hold them, fewer
  // where that leaves SMs without a block
  L.pix = kBruteThreads / L.team * 8;
  while (L.pix > kBrutePix || L.pix * L.a.n > kBruteVec) L.pix /= 2;
  while (L.pix > 4 && (L.a.sc.P + L.pix - 1) / L.pix < 4LL * L.num_sms) L.pix /= 2;
  // a block's threads beyond its pixels' teams help the shortlist: one lane of
  // a 1- or 2-dot array otherwise forms its up to 3 x 8 states in FP64 one
  // after another, and the one block in a hundred with such a pixel sets the
  // call's time (2 dots closed, 40 x 30 pixels, 12 or 30 charges: 16.1 ->
  // 14.2 us, the shortlist's entries by shifts instead of 64-bit divisions
  // included)
  while (L.team < 32 && 2 * L.team * L.pix <= kBruteThreads) L.team *= 2;
  const long long blocks = (L.a.sc.P + L.pix - 1) / L.pix;
  if (L.nhi * (unsigned long long)L.radix < 0x7fffffffull)
    k_brute<unsigned><<<(unsigned)blocks, kBruteThreads, 0, st>>>(L);
  else
    k_brute<unsigned long long><<<(unsigned)blocks, kBruteThreads, 0, st>>>(L);
  return cudaGetLastError();
}

}  // namespace qa
