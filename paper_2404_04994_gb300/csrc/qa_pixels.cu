// qa_pixels.cu -- the one-pass ground state (search_pixel) of one array: prep,
// search and outputs of each pixel by its team.
#include <algorithm>

#include "qa_gs_tiles.cuh"

namespace qa {

// A persistent grid whose warps take groups of 32 / W pixels one at a time (no
// barrier between a block's warps, so a slow pixel holds up its own warp only).
template <int W, bool CLOSED, int MODE>
__global__ void __launch_bounds__(kPrepThreads, kPixelBlocks)
k_pixels(const __grid_constant__ GsLaunch L) {
  __shared__ typename PixelSharedOf<W, MODE>::type sh;
  const ArrayDesc& a = L.one;
  grid_dep_signal();
  if (blockIdx.x == 0) zero_accumulators(L.cnt);
  pixel_zero_counts(sh);
  pixel_stage_array(a, sh);
  // whole rounds of groups by the warp's place, what is left over from a
  // counter (a counter for all of them cost two microseconds of 24)
  constexpr unsigned kGroup = 32 / W;
  const unsigned groups = (unsigned)((a.sc.P + kGroup - 1) / kGroup);
  const unsigned warps = gridDim.x * (kPrepThreads / 32);
  const unsigned rounds = (groups < warps ? 1u : groups / warps) * warps;
  for (unsigned q = blockIdx.x * (kPrepThreads / 32) + (threadIdx.x >> 5);;) {
    if (q >= rounds || q >= groups) {
      if (rounds >= groups) break;
      if ((threadIdx.x & 31) == 0) q = rounds + atomicAdd(&L.cnt->next, 1u);
      q = __shfl_sync(kFull, q, 0);
      if (q >= groups) break;
    }
    const long long p = (long long)q * kGroup + (threadIdx.x & 31) / W;
    search_pixel<W, CLOSED, MODE>(L, a, sh, 0, p, p < a.sc.P);
    if (q < rounds) q += warps;
  }
  __syncthreads();
  if (threadIdx.x == 0) pixel_counts(sh, L.bc_prep[blockIdx.x], L.bc_search[blockIdx.x]);
}

int pixel_blocks(const GsLaunch& L) {
  const long long teams = kPrepThreads / L.one.prep_team;
  const long long full = (L.one.sc.P + teams - 1) / teams;
  return (int)std::min(full, (long long)L.num_sms * kPixelBlocks);
}

cudaError_t launch_pixels(const GsLaunch& L, cudaStream_t st) {
  const int blocks = pixel_blocks(L);
  const bool cl = L.one.mt.closed != 0;
  typedef void (*Kernel)(GsLaunch);
  Kernel k = nullptr;
  if (L.one.search == kSearchSphere)
    k = cl ? k_pixels<16, true, kPixSphere> : k_pixels<16, false, kPixSphere>;
  else if (L.one.search == kSearchMixed)
    k = cl ? k_pixels<16, true, kPixMixed> : k_pixels<16, false, kPixMixed>;
  else if (L.one.prep_team == 16)
    k = cl ? k_pixels<16, true, kPixDense> : k_pixels<16, false, kPixDense>;
  else if (L.one.prep_team == 8)
    k = cl ? k_pixels<8, true, kPixDense> : k_pixels<8, false, kPixDense>;
  else if (L.one.prep_team == 4)
    k = cl ? k_pixels<4, true, kPixDense> : k_pixels<4, false, kPixDense>;
  if (!k) return cudaErrorInvalidValue;
  k<<<blocks, kPrepThreads, 0, st>>>(L);
  return cudaGetLastError();
}

}  // namespace qa
