// qa_sensor.cu -- charge-sensor response (Sec. IV.A), fused per pixel after
// the ground state of the non-sensing dots:
//   1. with the dots' charges n_D fixed, each sensor takes the charge that
//      minimises the full energy: the best floor / floor + 1 value around the
//      continuous sensor minimum x_S = c_S - (M_SS)^-1 M_SD (n_D - c_D)
//      (2^S candidates, S <= 4; ties to the lexicographically smaller);
//   2. the sensor potential V_S = (M (n - c))_S, Eq. "potential";
//   3. the line shape around the nearest Coulomb peak, eps = M_ss / 2 - |V_s|:
//      Lorentzian 1 / (1 + (eps / gamma)^2) or Gaussian exp(-eps^2 / 2 gamma^2);
//   4. noise along the fast axis: white, 1/f (Voss-McCartney octaves) and a
//      random telegraph, from a counter-based generator (Philox4x32-10,
//      Salmon et al. 2011), so every value is a pure function of (seed,
//      sensor, row, column).
// FP64 throughout.  A block takes a run of one raster row in chunks of 64
// columns, a pixel per thread.  What bounds it: the FP64 pipe (two operations
// per SM and clock), so nothing is formed twice: the induced charges are
// affine along a row (one multiply-add per dot and pixel), and an octave of
// the 1/f noise has one value per 2^k columns, drawn once into shared memory
// (about three normals per pixel and sensor with the white noise, not one per
// octave).  Rows are split into runs only while the GPU has SMs to spare,
// since every run draws its row's telegraph gaps from the start (32 a step).
// 200 x 200 pixels, 4 dots and a sensor with all noises: 118 us with a
// block per row, every normal drawn per pixel and c formed gate by gate;
// about 43 us so.
#include <algorithm>

#include "qa_launch.h"
#include "qa_prep.cuh"

namespace qa {

constexpr int kSensorThreads = 64;
constexpr int kSensorChunk = kSensorThreads;  // columns a block takes at a time
constexpr int kSensorOctaves = 14;            // 2^13 = kSensorMaxW
constexpr int kSensorMaxW = 8192;
constexpr int kSensorMax = 4;

// Philox4x32-10: ten rounds; each multiplies words 0 and 2 by the two round
// constants, mixes the high halves with words 1 / 3 and the key, and bumps
// the key by the two Weyl increments between rounds.
__device__ __forceinline__ uint4 philox10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k.x += 0x9E3779B9u;
      k.y += 0xBB67AE85u;
    }
    const unsigned lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const unsigned lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
  }
  return c;
}

__device__ __forceinline__ uint4 sensor_bits(unsigned long long seed, unsigned tag,
                                             unsigned row, unsigned idx) {
  return philox10(make_uint4(tag, row, idx, 0u),
                  make_uint2((unsigned)seed, (unsigned)(seed >> 32)));
}

// Box-Muller normal from the first two words.
__device__ __forceinline__ double sensor_gauss(unsigned long long seed, unsigned tag,
                                               unsigned row, unsigned idx) {
  const uint4 b = sensor_bits(seed, tag, row, idx);
  const double u1 = ((double)b.x + 1.0) * 2.3283064365386963e-10;  // (0, 1]
  const double u2 = (double)b.y * 2.3283064365386963e-10;          // [0, 1)
  return sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2);
}

// Entries of octave k's values in a chunk (it may straddle one boundary), and
// of all octaves.
__host__ __device__ constexpr int octave_room(int k) { return (kSensorChunk >> k) + 1; }
__host__ __device__ constexpr int octaves_room(int K) {
  int r = 0;
  for (int k = 0; k < K; ++k) r += octave_room(k);
  return r;
}

struct SensorShared {
  double M[kMaxDot * kMaxDot];
  double Mssi[kSensorMax * kSensorMax];
  double c0[kMaxDot], cu[kMaxDot];       // c(x) = carrier (c0 + x cu) in this row
  double white[kSensorMax][kSensorChunk];
  double pink[kSensorMax][octaves_room(kSensorOctaves)];
  unsigned flips[kSensorMax][kSensorMaxW / 32];  // the run's telegraph switch points
  int par0[kSensorMax];                          // parity of those before it
  int status;
};

// S: sensors.  Known when compiled, because an FP64 operation whose predicate
// is off takes the pipe all the same: with loops over the four possible places
// 2 dots and a sensor on 601 x 700 pixels took 87 us without noise (76 with a
// block per row and c formed gate by gate), 49 so.
template <int S>
__global__ void __launch_bounds__(kSensorThreads) k_sensor(SensorLaunch L) {
  __shared__ SensorShared sh;
  const ArrayDesc& a = L.a;
  const int nf = a.n, nd = nf - S;
  const int W = a.sc.W;
  const unsigned row = blockIdx.x;
  const int first = (int)blockIdx.y * L.run;
  const int last = min(first + L.run, W);  // the run's columns
  const int words = (last - first + 31) / 32;
  for (int e = threadIdx.x; e < nf * nf; e += blockDim.x) sh.M[e] = a.md->M[e];
  for (int e = threadIdx.x; e < S * words; e += blockDim.x) sh.flips[e / words][e % words] = 0u;
  if (threadIdx.x >= 32 && threadIdx.x < 32 + nf) {
    const int i = threadIdx.x - 32;
    const double ys = a.sc.y0 + (int)row * a.sc.dy;
    double c0 = 0.0, cu = 0.0;
    for (int g = 0; g < a.ng; ++g) {
      const double G = a.md->Cgd[i * a.ng + g];
      c0 += G * (a.sc.V0[g] + ys * a.sc.w[g]);
      cu += G * a.sc.u[g];
    }
    sh.c0[i] = c0;
    sh.cu[i] = cu;
  }
  __syncthreads();
  if (threadIdx.x == kSensorThreads - 1) {
    // (M_SS)^-1 by Cholesky (S <= 4), column by column
    double Lm[kSensorMax * kSensorMax] = {};
    int ok = 1;
    for (int j = 0; j < S && ok; ++j) {
      double d = sh.M[(nd + j) * nf + nd + j];
      for (int q = 0; q < j; ++q) d -= Lm[j * S + q] * Lm[j * S + q];
      if (!(d > 0.0)) { ok = 0; break; }
      Lm[j * S + j] = sqrt(d);
      for (int i = j + 1; i < S; ++i) {
        double e = sh.M[(nd + i) * nf + nd + j];
        for (int q = 0; q < j; ++q) e -= Lm[i * S + q] * Lm[j * S + q];
        Lm[i * S + j] = e / Lm[j * S + j];
      }
    }
    for (int col = 0; col < S && ok; ++col) {
      double y[kSensorMax];
      for (int i = 0; i < S; ++i) {
        double e = (i == col) ? 1.0 : 0.0;
        for (int q = 0; q < i; ++q) e -= Lm[i * S + q] * y[q];
        y[i] = e / Lm[i * S + i];
      }
      for (int i = S - 1; i >= 0; --i) {
        double e = y[i];
        for (int q = i + 1; q < S; ++q) e -= Lm[q * S + i] * sh.Mssi[q * S + col];
        sh.Mssi[i * S + col] = e / Lm[i * S + i];
      }
    }
    sh.status = ok;
  }
  if (threadIdx.x < 32 && L.jump_prob > 0.0) {
    // switch points in this row, geometric gaps from its first column on: lane
    // j of warp 0 draws the j-th of the next 32 and a scan places them
    const double lq = log(1.0 - L.jump_prob);
    const int lane = threadIdx.x;
    for (int s = 0; s < S; ++s) {
      int pos = -1, before = 0;
      for (unsigned j = 0; pos < last; j += 32) {
        const uint4 b = sensor_bits(L.seed, 2u | ((unsigned)s << 4), row, j + (unsigned)lane);
        const double u = ((double)b.x + 1.0) * 2.3283064365386963e-10;
        const double g = 1.0 + floor(log(u) / lq);
        // a longer gap ends the row as well (as does one that is no number, for a
        // switching probability that vanishes against 1)
        int at = g >= 1.0 && g <= (double)W ? (int)g : W + 1;
        for (int off = 1; off < 32; off <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, at, off);
          if (lane >= off) at += y;
        }
        at += pos;
        before += __popc(__ballot_sync(0xffffffffu, at < first));
        if (at >= first && at < last)
          atomicXor(&sh.flips[s][(at - first) >> 5], 1u << ((at - first) & 31));
        pos = __shfl_sync(0xffffffffu, at, 31);
      }
      if (lane == 0) sh.par0[s] = before & 1;
    }
  }
  __syncthreads();
  if (!sh.status) {  // M_SS of a positive definite M is positive definite: unreachable
    for (int col = first + threadIdx.x; col < last; col += blockDim.x)
      for (int s = 0; s < S; ++s) L.out_signal[((long long)row * W + col) * S + s] = __int_as_float(0x7fc00000);
    return;
  }
  const bool white = L.white_sigma > 0.0, pink = L.pink_sigma > 0.0;
  // (without noise the chunks share nothing, and need no barriers)
  const bool noise = white || pink, jump = L.jump_prob > 0.0;
  const int room = kSensorChunk + octaves_room(L.K);
  for (int b0 = first; b0 < last; b0 += kSensorChunk) {
    const int b1 = min(b0 + kSensorChunk, last);
    // the chunk's normals: white, then the octaves' values
    if (noise)
      for (int e = threadIdx.x; e < S * room; e += blockDim.x) {
        const int s = e / room;
        int r = e - s * room;
        if (r < kSensorChunk) {
          if (white && b0 + r < b1)
            sh.white[s][r] = sensor_gauss(L.seed, (unsigned)s << 4, row, (unsigned)(b0 + r));
        } else if (pink) {
          r -= kSensorChunk;
          const int at = r;
          int k = 0;
          while (r >= octave_room(k)) r -= octave_room(k++);
          if ((b0 >> k) + r <= (b1 - 1) >> k)
            sh.pink[s][at] = sensor_gauss(L.seed, 1u | ((unsigned)s << 4) | ((unsigned)k << 8), row,
                                          (unsigned)((b0 >> k) + r));
        }
      }
    if (noise) __syncthreads();
    const int col = b0 + threadIdx.x;
    if (col < b1) {
      const long long p = (long long)row * W + col;
      const double x = a.sc.x0 + col * a.sc.dx;
      // g_s = (M_SD (n_D - c_D))_s, the dots one after another
      double g[S] = {};
      for (int j = 0; j < nd; ++j) {
        const double r = (double)L.n_dots[p * nd + j] - a.mt.carrier * (sh.c0[j] + x * sh.cu[j]);
#pragma unroll
        for (int s = 0; s < S; ++s) g[s] += sh.M[(nd + s) * nf + j] * r;
      }
      double cs[S], bvec[S], xs[S];
#pragma unroll
      for (int s = 0; s < S; ++s) cs[s] = a.mt.carrier * (sh.c0[nd + s] + x * sh.cu[nd + s]);
      // b_s = g_s - (M_SS c_S)_s : E(n_S) = 1/2 n_S M_SS n_S + n_S . b
#pragma unroll
      for (int s = 0; s < S; ++s) {
        double mc = 0.0, acc = 0.0;
#pragma unroll
        for (int t = 0; t < S; ++t) {
          mc += sh.M[(nd + s) * nf + nd + t] * cs[t];
          acc += sh.Mssi[s * S + t] * g[t];
        }
        bvec[s] = g[s] - mc;
        xs[s] = cs[s] - acc;
      }
      int best[S] = {};
      double bestE = 0.0;
      for (int m = 0; m < (1 << S); ++m) {
        int cand[S];
#pragma unroll
        for (int s = 0; s < S; ++s)
          cand[s] = (int)floor(xs[s] > 0.0 ? xs[s] : 0.0) + ((m >> s) & 1);
        double E = 0.0;
#pragma unroll
        for (int s = 0; s < S; ++s) {
          double q = 0.0;
#pragma unroll
          for (int t = 0; t < S; ++t) q += sh.M[(nd + s) * nf + nd + t] * (double)cand[t];
          E += (double)cand[s] * (0.5 * q + bvec[s]);
        }
        bool better = (m == 0) || E < bestE;
        if (m && E == bestE) {
          // ties to the lexicographically smaller charges
          better = false;
          bool equal = true;
#pragma unroll
          for (int s = 0; s < S; ++s) {
            if (equal && cand[s] != best[s]) {
              better = cand[s] < best[s];
              equal = false;
            }
          }
        }
        if (better) {
          bestE = E;
#pragma unroll
          for (int s = 0; s < S; ++s) best[s] = cand[s];
        }
      }
#pragma unroll
      for (int s = 0; s < S; ++s) {
        const int q = nd + s;
        double V = g[s];  // the dots' part of (M (n - c))_s
#pragma unroll
        for (int t = 0; t < S; ++t) V += sh.M[q * nf + nd + t] * ((double)best[t] - cs[t]);
        const double y = (0.5 * sh.M[q * nf + q] - fabs(V)) / L.width;
        double v = L.shape == 1 ? exp(-0.5 * y * y) : 1.0 / (1.0 + y * y);
        if (white) v += L.white_sigma * sh.white[s][threadIdx.x];
        if (pink) {
          double acc = 0.0;
          int at = 0;
          for (int k = 0; k < L.K; ++k) {
            acc += sh.pink[s][at + (col >> k) - (b0 >> k)];
            at += octave_room(k);
          }
          v += L.pink_sigma * acc / sqrt((double)L.K);
        }
        if (jump) {
          // telegraph state = parity of the switch points at or before col
          unsigned par = (unsigned)sh.par0[s];
          const int rel = col - first, wlast = rel >> 5;
          for (int w = (b0 - first) >> 5; w < wlast; ++w) par ^= __popc(sh.flips[s][w]) & 1u;
          const unsigned keep = (rel & 31) == 31 ? 0xffffffffu : ((2u << (rel & 31)) - 1u);
          par ^= __popc(sh.flips[s][wlast] & keep) & 1u;
          if (par) v += L.jump_amplitude;
        }
        L.out_signal[p * S + s] = (float)v;
        if (L.out_n_sensor) L.out_n_sensor[p * S + s] = (int8_t)(best[s] > 127 ? 127 : best[s]);
        if (L.out_potential) L.out_potential[p * S + s] = V;
      }
    }
    if (noise || jump) __syncthreads();
    // the next chunk starts from this one's parity
    if (threadIdx.x < S && jump) {
      int par = sh.par0[threadIdx.x];
      const int w0 = (b0 - first) >> 5;
      for (int w = w0; w < w0 + kSensorChunk / 32 && w < words; ++w)
        par ^= __popc(sh.flips[threadIdx.x][w]) & 1;
      sh.par0[threadIdx.x] = par;
    }
    if (jump) __syncthreads();
  }
}

cudaError_t launch_sensor(const SensorLaunch& L0, cudaStream_t st) {
  if (L0.a.sc.P == 0) return cudaSuccess;
  SensorLaunch L = L0;
  // one run per row, or several while there are fewer than four blocks per SM
  const int W = L.a.sc.W, H = L.a.sc.H;
  const long long want = (4LL * L.num_sms + H - 1) / H;
  const int runs = (int)std::min<long long>((W + kSensorChunk - 1) / kSensorChunk, want);
  L.run = ((W + runs - 1) / runs + kSensorChunk - 1) / kSensorChunk * kSensorChunk;
  const unsigned cols = (unsigned)((W + L.run - 1) / L.run);
  const dim3 grid((unsigned)H, cols);
  if (L.S == 1) k_sensor<1><<<grid, kSensorThreads, 0, st>>>(L);
  else if (L.S == 2) k_sensor<2><<<grid, kSensorThreads, 0, st>>>(L);
  else if (L.S == 3) k_sensor<3><<<grid, kSensorThreads, 0, st>>>(L);
  else k_sensor<4><<<grid, kSensorThreads, 0, st>>>(L);
  return cudaGetLastError();
}

}  // namespace qa
