// spots_split.cu -- the FP32-mixed Bragg-spot sum for Gaussian lattice
// shapes, one warp per pixel (the per-pixel step reduction of Sec. III-B's
// nanoBraggSpots, split across lanes, with the fused addArray accumulate).
//
// Why a second variant: with a Gaussian F_latt only a few percent of the
// (subpixel, layer, phi x mosaic, source) steps of a pixel carry a term that
// does not underflow in FP32, and each such term needs the structure factor
// (64 gathers for tricubic interpolation).  With one thread per pixel those
// terms are scattered over lanes and a warp serialises them.  Here:
//   1. a warp takes B = 32 / U pixels at a time (one when it gets fewer
//      than 256 pixels in all); its lanes set up the
//      U = os^2 x layers sub-pixel units of all B pixels (position,
//      direction, solid angle, capture, polarization; in FP64, for one or two
//      units per pixel in double-float) into shared memory, then the warp
//      sums the pixels one after another;
//   2. lanes take (unit, phi x mosaic) items 32 at a time and form G and r
//      in double-float.  h_x = G_x delta + r_x is linear in a source's
//      delta = 1/lambda - u0, so for each lattice point near the item's
//      sweep the sources whose exponent sum N^2 f^2 / 0.63 can stay below
//      the underflow cut form one interval of the sorted delta table (a
//      quadratic in delta, then a short search); where that does not
//      apply, blocks of 8 sources are pruned by their delta range.  Each
//      non-empty interval becomes one entry of a per-warp ring in shared
//      memory, holding a copy of its item's state;
//   3. whenever the ring holds 32 (entry, source) pairs, each lane takes
//      one pair, forms the step's exact fractional offset and, if the step
//      survives the cut, its term (exp, F_cell from the cell's tricubic
//      polynomial in a per-warp shared-memory cache, or from the table)
//      into its own Kahan sum;
//      In shots of many sources and steps (split_form) a lane takes a whole
//      segment of an entry instead, on which F_cell is a polynomial of degree
//      9 in delta and the exponent a parabola: ~15 instructions per step in
//      place of ~8 per lane and step of the pair queue (sum_tasks).  Large
//      shot: 164.5 -> 107.1 ms; the 512^2 pixels at its centre, where the
//      batches of items without a lattice point in reach end early, 5.0 -> 2.7;
//      In shots of few items and steps per pixel (split_form) each half of the
//      warp takes a pixel of its own: with 10 items a pixel's pass over its
//      items left 22 lanes idle;
//   4. a pixel's lane sums are reduced with warp shuffles in float-float.
// The order of every operation depends only on the pixel's own inputs, so
// a pixel's value does not depend on what else is in the launch.
// Pixels are handed to warps through an atomic counter in a scratch word.
#include "split_kernel.cuh"

namespace nbgb {

extern template SplitKernel pick_split<true>(const SpotArgs &);
template SplitKernel pick_split<false>(const SpotArgs &);

size_t split_smem_bytes(const SpotArgs &a) {
  return split_smem_layout(a.PM, a.S);
}

bool split_supported(const SpotArgs &a) {
  return a.shape == 1 && a.os * a.os * a.T <= kMaxUnits &&
         split_smem_bytes(a) <= 200 * 1024;
}

cudaError_t launch_spots_split(const SpotArgs &a, unsigned long long *work,
                               int sm_count, cudaStream_t st) {
  size_t smem = split_smem_bytes(a);
  auto kern = split_ff(a) ? pick_split<true>(a) : pick_split<false>(a);
  cudaError_t e = cudaFuncSetAttribute(
      kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern,
                                                    kSplitThreads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  long long n_work = a.pixlist ? a.n_list : a.npix;
  long long blocks = (long long)sm_count * per_sm;
  long long need = (n_work + kSplitWarps - 1) / kSplitWarps;
  if (blocks > need) blocks = need;
  if (blocks < 1) return cudaSuccess;
  kern<<<(unsigned)blocks, kSplitThreads, smem, st>>>(a, work);
  return cudaGetLastError();
}

}  // namespace nbgb
