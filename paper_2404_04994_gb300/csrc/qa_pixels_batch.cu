// qa_pixels_batch.cu -- the one-pass ground state (search_pixel) of a batch's
// arrays: a persistent grid per team width, form and search, whose blocks take
// work units from a queue.
#include "qa_gs_tiles.cuh"

namespace qa {

// The open and the closed arrays have a kernel each: with both forms' code in
// one kernel its warps miss the instruction cache (10 stalls per issue; 1,600
// us against 550 + 590 us for the 65 arrays of 12 to 16 dots of a batch of
// 192).  A unit's pixels go round the block's warps.
template <int W, bool CLOSED, int MODE>
__global__ void __launch_bounds__(kPrepThreads, kPixelBlocks)
k_pixels_batch(const __grid_constant__ GsLaunch L, int v) {
  __shared__ typename PixelSharedOf<W, MODE>::type sh;
  __shared__ int s_unit;
  int staged = -1;
  grid_dep_signal();
  pixel_zero_counts(sh);
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_unit = (int)atomicAdd(&L.cnt->q_pixel[v], 1u);
    __syncthreads();
    const int u = s_unit;
    if (u >= L.pix_count[v]) break;
    const WorkUnit wu = L.pixel_units[L.pix_first[v] + u];
    const ArrayDesc& a = L.table[wu.array];
    if (wu.array != staged) {
      pixel_stage_array(a, sh);
      staged = wu.array;
    }
    const long long end = wu.first + wu.count;
    for (long long q = wu.first + (threadIdx.x >> 5) * (32 / W); q < end; q += kPrepThreads / W) {
      const long long p = q + (threadIdx.x & 31) / W;
      search_pixel<W, CLOSED, MODE>(L, a, sh, wu.array, p, p < end);
    }
  }
  if (threadIdx.x == 0) {
    const int b = L.pix_bc[v] + blockIdx.x;
    pixel_counts(sh, L.bc_prep[L.grid_prep + b], L.bc_search[L.grid_search + b]);
  }
  grid_dep_wait();  // ends after the grids before it
}

// The search grids and the one-pass grids of a batch share nothing but their
// lists, so each starts while the one before is still running (and ends after
// it: what waits for the last waits for all).  One after another, each with a
// tail of its own, they made batches of a few unlike arrays slower than tiles
// for all: 5 arrays of 2 to 6 dots, 64 x 64 pixels, 137 us against 93; 83 so
// (160 arrays of 2 to 16 dots 913 -> 800).
// Variant 2 s + closed: s = 0 sphere search, 1 either, 2 to 4 the enumeration
// by 16, 8 and 4 lanes.
cudaError_t launch_pixels_batch(const GsLaunch& L, cudaStream_t st) {
  typedef void (*Kernel)(GsLaunch, int);
  static const Kernel table[kPixelVariants] = {
      k_pixels_batch<16, false, kPixSphere>, k_pixels_batch<16, true, kPixSphere>,
      k_pixels_batch<16, false, kPixMixed>,  k_pixels_batch<16, true, kPixMixed>,
      k_pixels_batch<16, false, kPixDense>,  k_pixels_batch<16, true, kPixDense>,
      k_pixels_batch<8, false, kPixDense>,   k_pixels_batch<8, true, kPixDense>,
      k_pixels_batch<4, false, kPixDense>,   k_pixels_batch<4, true, kPixDense>};
  bool first = L.n_search_units == 0;  // (nothing of the batch before it)
  for (int v = 0; v < kPixelVariants; ++v) {
    if (L.pix_count[v] == 0) continue;
    if (first) {
      table[v]<<<L.pix_grid[v], kPrepThreads, 0, st>>>(L, v);
    } else {
      const cudaError_t e = launch_dependent(table[v], (unsigned)L.pix_grid[v], kPrepThreads, st, L, v);
      if (e != cudaSuccess) {
        cudaGetLastError();
        return e;
      }
    }
    first = false;
  }
  return cudaGetLastError();
}

}  // namespace qa
