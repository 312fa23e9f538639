// split_kernel.cuh -- the stand-alone warp-per-pixel kernel (spots_split.cu has
// the method) and the choice among its instantiations.  Those of double-float
// and of FP64 unit geometry are compiled in a file each: in one they took 40 s.
#pragma once

#include "split_pixel.cuh"

namespace nbgb {

// COUNT: also count the pairs, intervals and block tests (a.wstats)
template <int INTERP, int HASDIV, int COUNT, bool FF, int FORM>
__global__ void __launch_bounds__(kSplitThreads, FORM == kLines ? kLineBlocks : 5)
    spots_split_kernel(SpotArgs a, unsigned long long *work) {
  extern __shared__ float sms[];
  SplitBlock b;
  split_stage(b, sms, a, a.axh, a.axl, a.src32, a.PM, a.S, a.u0h, a.u0l);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long n_work = a.pixlist ? a.n_list : a.npix;
  SplitCounts cnt;  // work of this warp
  // a warp takes B pixels at a time and sets up all their sub-pixel units
  // in one pass, so the FP64 geometry fills up to 32 lanes
  // (one pixel at a time when a warp gets few pixels of many steps: pixels
  // differ in cost, and grabbing several near the end of a launch leaves a
  // tail; with few steps the geometry of single pixels would cost more: 512^2
  // pixels of 1 unit and 99 steps 1.09 -> 0.22 ms, 8 units and 4800 steps
  // 1.45 -> 1.20 ms, but 4 units and 20000 steps 2.81 -> 3.51 ms)
  const int U = a.os * a.os * a.T;
  const long long per_warp = n_work / ((long long)gridDim.x * kSplitWarps);
  const long long most =
      per_warp >= 256 ? kMaxUnits
      : (long long)U * a.PM * a.S <= 8192 ? per_warp / 16 : 1;
  // (as many as the warp sums side by side where it gets so many)
  constexpr int W = kLanes<FORM>;
  const long long least = per_warp >= 32 / W ? 32 / W : 1;
  const int B =
      (int)max(1ll, min((long long)(kMaxUnits / U), max(most, least)));
  float *unit = b.unit_base + warp * kMaxUnits * kUnitFloats;
  while (true) {
    long long first = 0;
    if (lane == 0) first = (long long)atomicAdd(work, (unsigned long long)B);
    first = __shfl_sync(0xffffffffu, first, 0);
    if (first >= n_work) break;
    const int nb = (int)min((long long)B, n_work - first);
    if (lane < nb * U) {
      const int bi = lane / U;
      const long long gp = a.pixlist ? a.pixlist[first + bi] : first + bi;
      const DevPanel &P = a.panels[panel_of_pixel(a, gp)];
      const long long local = gp - P.pix0;
      const int s = (int)(local / P.nfast);
      const int f = (int)(local - (long long)s * P.nfast);
      split_unit<HASDIV, FF>(a, P, s, f, lane - bi * U, unit + lane * kUnitFloats);
    }
    __syncwarp();
    double mine = 0.0;  // lane bi keeps the sum of pixel bi
    for (int bi = 0; bi < nb; bi += 32 / W) {
      const int pi = bi + (W == 32 ? 0 : lane / W);  // this lane's pixel
      const bool ok = W == 32 || pi < nb;
      const double v = split_sum<INTERP, HASDIV, FORM, COUNT>(
          a, b, unit + (ok ? pi : bi) * U * kUnitFloats, cnt, ok);
      if (W == 32) {
        if (lane == bi) mine = v;
      } else {
        const double got =
            __shfl_sync(0xffffffffu, v, (lane - bi) * W & 31);
        if (lane >= bi && lane < bi + 32 / W) mine = got;
      }
    }
    // fused accumulate into the image: lanes 0 .. nb-1 add the batch's
    // pixels, consecutive in the image, in one coalesced access
    if (lane < nb) {
      const long long gp = a.pixlist ? a.pixlist[first + lane] : first + lane;
      a.image[nb_idx(a.check, NB_SITE_IMAGE, gp, a.npix)] +=
          a.prefactor * mine;
    }
    __syncwarp();  // the next batch rewrites the units
  }
  if (lane == 0 && a.stats && cnt.terms) atomicAdd(a.stats, cnt.terms);
  if (COUNT && lane == 0 && a.wstats) {
    atomicAdd(a.wstats, cnt.pairs);
    atomicAdd(a.wstats + 1, cnt.ivals);
    atomicAdd(a.wstats + 2, cnt.blocks);
  }
}

using SplitKernel = void (*)(SpotArgs, unsigned long long *);

template <int INTERP, int COUNT, bool FF>
static SplitKernel pick_split(const SpotArgs &a) {
  if (a.has_div) return spots_split_kernel<INTERP, 1, COUNT, FF, kPairs>;
  switch (split_form(a, a.PM, a.S, a.span)) {
    case kLines: return spots_split_kernel<INTERP, 0, COUNT, FF, kLines>;
    case kHalves: return spots_split_kernel<INTERP, 0, COUNT, FF, kHalves>;
    // (the early test changes no sum and no count: not built with counters)
    case kPairsEarly:
      if (!COUNT)
        return spots_split_kernel<INTERP, 0, COUNT, FF,
                                  COUNT ? kPairs : kPairsEarly>;
  }
  return spots_split_kernel<INTERP, 0, COUNT, FF, kPairs>;
}

template <bool FF>
SplitKernel pick_split(const SpotArgs &a) {
  if (a.wstats)
    return a.interp ? pick_split<1, 1, FF>(a) : pick_split<0, 1, FF>(a);
  return a.interp ? pick_split<1, 0, FF>(a) : pick_split<0, 0, FF>(a);
}

}  // namespace nbgb
