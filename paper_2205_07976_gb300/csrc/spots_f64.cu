// spots_f64.cu -- the plain FP64 form of the per-pixel Bragg-spot sum
// (nanoBraggSpots, Sec. III-B), one thread per pixel, with the fused
// double accumulate of addArray (Listing 1).
//
// Loop nest per pixel: subpixel x sensor layer -> source -> phi x mosaic.
// Everything is FP64 and this file is compiled without FMA contraction.
// The Miller indices and the fractional offsets are evaluated in the order the
// definition is written, so they are bitwise those of any other uncontracted
// FP64 evaluation (the sinc at N = 200 multiplies h's rounding by pi N).  The
// rest, which is not sensitive to the last bits, is arranged for the FP64
// pipe, which on this part issues at 1/64 of the FP32 rate and so sets the
// kernel's time:
//   * the nearest lattice point comes from an addition that rounds up at the
//     units' place; its integer is then the low word of the sum (a ceil and
//     three conversions less);
//   * the sinc's sines are sin(pi x) for |x| <= 1/2 from one polynomial
//     (sinpi_half); the numerator's argument N f is reduced exactly by one
//     FMA, and its sign drops out;
//   * the Gaussian exponent (summed in explicit FMAs) and the Lagrange
//     weights multiply by 1/0.63 and 1/6 instead of dividing, and the sinc
//     multiplies by one reciprocal per step (a division is a sequence of
//     about ten FP64 instructions; sweep of 30.8 ms: 31.3 with it);
//   * the tricubic sum is nested per axis in explicit FMAs, sum_i w_i
//     sum_j w_j sum_k w_k F_ijk: 84 FP64 operations instead of 256 for the
//     flat triple product sum (the rounding differs at the 1e-15 level);
//   * the table is read from an FP64 copy (a float-to-double conversion
//     is an FP64-pipe instruction too), and the cell's first node comes
//     from the nearest lattice point instead of a floor;
//   * the step's weight, capture, polarization and solid angle are one
//     factor per source.
// 307 x 211 pixels of the precision sweep at N = 200: 42.3 -> 33.3 ms with the
// lattice point, sines and reciprocal above (about 170 -> 110 FP64-pipe
// instructions per sinc step, the pipe 85 % busy).
// Only loop invariants are hoisted (pixel position, solid angle, capture
// fraction per subpixel/layer; scattering vector, polarization and that
// factor per source).  The rotated axes and the source table are staged in
// shared memory per block.
#include "mixed_common.cuh"

namespace nbgb {

__device__ __forceinline__ double dot3d(const double *a, const double *b) {
  return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

// sin(pi x) for |x| <= 1/2: x p(x^2), p the degree-8 minimax polynomial of
// sin(pi x)/x in x^2 on [0, 1/4] (Remez exchange in 60 digits; relative error
// 2.6e-19, 4.0e-17 with the coefficients rounded to FP64): 10 FP64
// operations and an ulp or two of rounding
__device__ __forceinline__ double sinpi_half(double x) {
  const double t = x * x;
  double p = fma(7.6947273844559142e-07, t, -2.1903185429548639e-05);
  p = fma(p, t, 0.00046629968877916672);
  p = fma(p, t, -0.0073704304787646294);
  p = fma(p, t, 0.082145886569893037);
  p = fma(p, t, -0.5992645293187383);
  p = fma(p, t, 2.550164039877294);
  p = fma(p, t, -5.1677127800499694);
  p = fma(p, t, 3.1415926535897931);
  return x * p;
}

// 1.5 * 2^52: adding it rounds to an integer, which the low word then holds
constexpr double kRoundBias = 6755399441055744.0;

// The lattice point n nearest to h (ties down: ceil(h - 1/2)) and the offset
// f = h - n (exact)
__device__ __forceinline__ void nearest_ceil(const double h[3], long long n[3],
                                             double f[3]) {
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    const double c = ceil(h[x] - 0.5);
    n[x] = (long long)c;
    f[x] = h[x] - c;
  }
}
// the same by an addition where |h| allows it
__device__ __forceinline__ void nearest_f64(const double h[3], long long n[3],
                                            double f[3]) {
  // |h| < 2^30 on all axes (integer compares of the high words; a double
  // compare is one more FP64-pipe instruction)
  const int big = max(max(__double2hiint(h[0]) & 0x7fffffff,
                          __double2hiint(h[1]) & 0x7fffffff),
                      __double2hiint(h[2]) & 0x7fffffff);
  if (big < 0x41d00000) {
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const double s = __dadd_ru(h[x] - 0.5, kRoundBias);
      n[x] = __double2loint(s);
      f[x] = h[x] - (s - kRoundBias);
    }
  } else {
    nearest_ceil(h, n, f);
  }
}

// F_latt (up to its sign) at the fractional offset f
template <int SHAPE>
__device__ __forceinline__ double flatt_f64(const SpotArgs &a,
                                            const double f[3]) {
  // sinc: sin(pi N h)/sin(pi h) = +-sin(pi N f)/sin(pi f); the three
  // numerators and the three denominators are multiplied separately and
  // divided once; an axis with |f| below 1e-100 (f = 0 in practice: h is a
  // sum of products of order-one values) contributes its limit N, so the
  // product of denominators cannot underflow
  double num = 1.0, den = 1.0, rad2 = 0.0;
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    if (SHAPE == 0) {
      const double N = a.N64[x];
      double sn;
      if (N < 1e12) {
        // r = N f - round(N f), exact
        const double m = fma(N, f[x], kRoundBias) - kRoundBias;
        sn = sinpi_half(fma(N, f[x], -m));
      } else {
        sn = sin(M_PI * N * f[x]);
      }
      // |f| < 1e-100 from the high word of its bit pattern
      const bool zero =
          (__double2hiint(f[x]) & 0x7fffffff) < __double2hiint(1e-100);
      sn = zero ? N : sn;
      const double sd = zero ? 1.0 : sinpi_half(f[x]);
      num = x ? num * sn : sn;
      den = x ? den * sd : sd;
    } else {
      // sum N^2 f^2 / 0.63 in explicit FMAs (N^2 / 0.63 is loop-invariant)
      rad2 = fma(a.N64[x] * a.N64[x] * (1.0 / 0.63) * f[x], f[x], rad2);
    }
  }
  if (SHAPE == 1) return a.N64[0] * a.N64[1] * a.N64[2] * exp(-rad2);
  return num * __drcp_rn(den);
}

__device__ __forceinline__ bool in_table(const SpotArgs &a, long long i,
                                         long long j, long long k) {
  return (unsigned long long)i < (unsigned long long)a.hn[0] &&
         (unsigned long long)j < (unsigned long long)a.hn[1] &&
         (unsigned long long)k < (unsigned long long)a.hn[2];
}

// The tricubic sum over the 4x4x4 stencil whose first node has flat index
// off: nested per axis in explicit FMAs, sum_i w_i sum_j w_j sum_k w_k
// F_ijk (84 FP64 operations; a flat triple-product sum takes 256).  T is
// double (the FP64 copy of the table) or float (each read converted).
template <typename T>
__device__ __forceinline__ double tricubic_sum(const SpotArgs &a,
                                               const T *tab, long long off,
                                               const double w[3][4]) {
  double sum = 0.0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    double si = 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const T *row = tab + off + ((long long)i * a.hn[1] + j) * a.hn[2];
      double sj = w[2][0] * (double)__ldg(row);
      sj = fma(w[2][1], (double)__ldg(row + 1), sj);
      sj = fma(w[2][2], (double)__ldg(row + 2), sj);
      sj = fma(w[2][3], (double)__ldg(row + 3), sj);
      si = j ? fma(w[1][j], sj, si) : w[1][0] * sj;
    }
    sum = i ? fma(w[0][i], si, sum) : w[0][0] * si;
  }
  return sum;
}

// F_cell at the offset f from lattice point n (ties down, nearest_f64): the
// cell's first node is floor(h) = n - 1 where f < 0, else n, so no floor and
// no second float-to-integer conversion per axis are needed
template <int INTERP>
__device__ __forceinline__ double fcell_f64(const SpotArgs &a,
                                            const double f[3],
                                            const long long n[3]) {
  long long nn[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) nn[c] = n[c] - a.hmin[c];
  if (INTERP == 1) {
    long long fl[3];
    double x[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      // f = h - n is exact (h and n lie within 1/2), and so is h - floor(h)
      // for f < 0: f + 1 holds no bit below h's last one
      // f < 0 from the sign bit (an integer test; f is never -0)
      const bool below = __double_as_longlong(f[c]) < 0;
      fl[c] = nn[c] - (below ? 1 : 0);
      x[c] = below ? f[c] + 1.0 : f[c];
    }
    if (in_table(a, fl[0] - 1, fl[1] - 1, fl[2] - 1) &&
        in_table(a, fl[0] + 2, fl[1] + 2, fl[2] + 2)) {
      // 4-point Lagrange weights on nodes -1, 0, 1, 2, from the shared
      // products t (t - 1) / 6 and (t + 1)(t - 2) / 2 (11 operations per
      // axis; the negations are free operand modifiers)
      double w[3][4];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const double t = x[c], tm1 = t - 1.0, tm2 = t - 2.0, tp1 = t + 1.0;
        const double p6 = t * tm1 * (1.0 / 6.0), q2 = tp1 * tm2 * 0.5;
        w[c][0] = -(p6 * tm2);
        w[c][1] = q2 * tm1;
        w[c][2] = -(q2 * t);
        w[c][3] = p6 * tp1;
      }
      long long off =
          ((long long)(fl[0] - 1) * a.hn[1] + (fl[1] - 1)) * a.hn[2] +
          (fl[2] - 1);
      {
        const long long last = off + (3ll * a.hn[1] + 3) * a.hn[2] + 3;
        if (nb_idx(a.check, NB_SITE_STENCIL, last, table_size(a)) != last)
          off = 0;
      }
      return a.F64t ? tricubic_sum(a, a.F64t, off, w)
                    : tricubic_sum(a, a.F, off, w);
    }
  }
  if (in_table(a, nn[0], nn[1], nn[2])) {
    const long long idx = nb_idx(a.check, NB_SITE_F,
                                 (nn[0] * a.hn[1] + nn[1]) * a.hn[2] + nn[2],
                                 table_size(a));
    return a.F64t ? __ldg(a.F64t + idx) : (double)__ldg(a.F + idx);
  }
  return a.defF64;
}

// F as doubles, for the NB_F64 kernel's reads
__global__ void f64_table_kernel(const float *F, long long n, double *F64t) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    F64t[i] = (double)F[i];
}

cudaError_t build_f64_table(const float *F, long long n, double *F64t,
                            cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  f64_table_kernel<<<1216, 256, 0, st>>>(F, n, F64t);
  return cudaGetLastError();
}

// 2^(lu + lk + lm) neighbouring lanes share a pixel (f64_split): each takes
// every 2^lu-th unit, of those every 2^lk-th source, and of those every 2^lm-th
// orientation
struct F64Split {
  int lu, lk, lm;
};
template <int SHAPE, int INTERP>
__global__ void __launch_bounds__(kTileThreads, 4)
    spots_f64_kernel(SpotArgs a, F64Split sp) {
  extern __shared__ double sm[];
  double *s_ax = sm;
  double *s_src = sm + a.PM * 9;
  for (int i = threadIdx.x; i < a.PM * 9; i += blockDim.x) s_ax[i] = a.ax64[i];
  for (int i = threadIdx.x; i < a.S * SRC64_STRIDE; i += blockDim.x)
    s_src[i] = a.src64[i];
  __syncthreads();

  const int lsplit = sp.lu + sp.lk + sp.lm;
  const long long slot =
      ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> lsplit;
  const int part = threadIdx.x & ((1 << lsplit) - 1);
  const int du = 1 << sp.lu, dk = 1 << sp.lk, dm = 1 << sp.lm;
  const int u0 = part & (du - 1), k0 = (part >> sp.lu) & (dk - 1),
            m0 = part >> (sp.lu + sp.lk);
  long long gp = 0;
  int q = 0, s = 0, fp = 0;
  const bool ok =
      a.pixlist ? map_pixel(a, slot, 0, gp, q, s, fp)
                : map_pixel(a, slot / kTileThreads,
                            (int)(slot % kTileThreads), gp, q, s, fp);
  const DevPanel &P = a.panels[q];
  const double px = P.px;
  const int os = a.os;
  double acc = 0.0;
  const int U = ok ? os * os * a.T : 0;
  for (int u = u0; u < U; u += du) {
    const int t = u % a.T, i = u / a.T / os, j = u / a.T % os;
    // (x / 1 is x: a division is ten FP64 instructions)
    const double fi = os == 1 ? i + 0.5 : (i + 0.5) / os,
                 fj = os == 1 ? j + 0.5 : (j + 0.5) / os;
    double cf = (fp + fi) * px, cs = (s + fj) * px, cn = t * a.dt;
    double pos[3], d[3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
      pos[c] = P.origin[c] + cf * P.fdir[c] + cs * P.sdir[c] +
               cn * P.ndir[c];
    double R = sqrt(dot3d(pos, pos));
#pragma unroll
    for (int c = 0; c < 3; ++c) d[c] = pos[c] / R;
    double omega = px * px * dot3d(P.ndir, pos) / (R * R * R);
    double cap = 1.0;
    if (a.thickness > 0.0) {
      double L = a.atten * dot3d(d, P.ndir);
      cap = exp(-t * a.dt / L) - exp(-(t + 1) * a.dt / L);
    }
    for (int k = k0; k < a.S; k += dk) {
      const double *src = s_src + k * SRC64_STRIDE;
      const double lam = src[SRC64_LAM];
      const double *dir = src + SRC64_DIR;
      double Sv[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) Sv[c] = (d[c] - dir[c]) / lam;
      // Kahn: cos 2psi sin^2 2theta = (d.E')^2 - (d.B')^2 for unit d
      double c2 = dot3d(d, dir), x = dot3d(d, src + SRC64_E),
             y = dot3d(d, src + SRC64_B);
      double pol = 0.5 * (1.0 + c2 * c2 - a.kahn64 * (x * x - y * y));
      // the step's factors that do not depend on phi x mosaic
      const double wcpo = src[SRC64_W] * cap * pol * omega;
      for (int pm = m0; pm < a.PM; pm += dm) {
        const double *A = s_ax + pm * 9;
        double h[3] = {dot3d(A, Sv), dot3d(A + 3, Sv), dot3d(A + 6, Sv)};
        long long n[3];
        double f[3];
        // (Gaussian steps: a ceil measured faster than the biased addition, and
        // F_latt before the lookup, whose results are else held across it:
        // 64^2 pixels of 99 steps 695 -> 654 us; the sinc sweep 30.8 -> 30.3 ms)
        if (SHAPE == 1)
          nearest_ceil(h, n, f);
        else
          nearest_f64(h, n, f);
        const double fl = flatt_f64<SHAPE>(a, f);
        const double a_ = fcell_f64<INTERP>(a, f, n) * fl;
        acc = fma(a_ * a_, wcpo, acc);
      }
    }
  }
  for (int o = 1; o < (1 << lsplit); o <<= 1)
    acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (ok && part == 0)
    a.image[nb_idx(a.check, NB_SITE_IMAGE, gp, a.npix)] += a.prefactor * acc;
}

// How many lanes share a pixel (log2).  The FP64 unit is a scheduler's own, so
// a launch takes as long as the scheduler with the most warps: 307 x 211
// pixels one per lane are 3.6 warps for each of the 608 schedulers, so 4 for
// most, and a list of 9216 pixels leaves half of them without a warp.  Units
// are split as far as a power of two divides them, which repeats nothing (that
// list with 8 units of 12 steps: 870 -> 490 us, half of it the list and the
// image copy); sources and orientations while parts keep at least 128 steps, so
// that the repeated geometry (~130 FP64 instructions against 110 per sinc step)
// stays below 1 % (307 x 211 pixels, sinc, 2000 steps: 33.3 -> 30.2 ms).  A
// rule on the shot alone keeps a pixel's value the same in every launch.
static F64Split f64_split(const SpotArgs &a) {
  F64Split s = {0, 0, 0};
  const int U = a.os * a.os * a.T;
  while (s.lu < 5 && U % (2 << s.lu) == 0) ++s.lu;
  int l = 0;
  while (s.lu + l < 5 && ((long long)a.S * a.PM) >> (l + 1) >= 128) ++l;
  while (s.lk < l && 2 << s.lk <= a.S) ++s.lk;  // sources first
  s.lm = l - s.lk;
  return s;
}

cudaError_t launch_spots_f64(const SpotArgs &a, cudaStream_t st) {
  size_t smem = (size_t)(a.PM * 9 + a.S * SRC64_STRIDE) * sizeof(double);
  F64Split split = f64_split(a);
  const long long most = a.pixlist ? a.n_list : (long long)a.n_tiles * kTileThreads;
  if (most > 1ll << 32) split = {0, 0, 0};  // keeps the grid below 2^31
  const int lsplit = split.lu + split.lk + split.lm;
  const long long pixels =
      a.pixlist ? a.n_list : (long long)a.n_tiles * kTileThreads;
  const long long blocks =
      ((pixels << lsplit) + kTileThreads - 1) / kTileThreads;
  if (blocks <= 0) return cudaSuccess;
  void (*kern)(SpotArgs, F64Split) = nullptr;
  int key = a.shape * 2 + a.interp;
  switch (key) {
    case 0: kern = spots_f64_kernel<0, 0>; break;
    case 1: kern = spots_f64_kernel<0, 1>; break;
    case 2: kern = spots_f64_kernel<1, 0>; break;
    default: kern = spots_f64_kernel<1, 1>; break;
  }
  cudaError_t e = cudaFuncSetAttribute(
      kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)blocks, kTileThreads, smem, st>>>(a, split);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------
// Gaussian shapes, one warp per pixel, with the steps that cannot change the
// pixel's sum screened out (the thread-per-pixel kernel above evaluates all
// of them).  A step costs ~140 FP64-pipe instructions, at 1/64 of the FP32
// rate, and nearly all of them are spent on terms many orders below the
// pixel's sum: a term falls as exp(-2 R / 0.63), R = sum N^2 f^2 up to
// 3 N^2 / 4.  So the warp computes R of every step in FP32 (~20
// instructions), and only the steps whose term may matter go, 32 at a time,
// through the FP64 evaluation, which is that of the kernel above, step by
// step.
//
// The bound: |term| <= Fb^2 (Na Nb Nc)^2 exp(-2 R / 0.63) |w_k| |fac_u|,
// Fb = max(2 max|F|, |default_F|) (the weights of the tricubic interpolant
// sum to at most 1.25^3 < 2 in magnitude) and fac_u the unit's solid angle x
// capture x polarization.  With
//   c_u = 0.315 ln(Fb^2 (Na Nb Nc)^2 U PM sum|w| |fac_u| 2^56 / S),
// S the sum so far, all steps with R > c_u together add less than 2^-56 S:
// an eighth of one FP64 rounding of the sum.  The FP32 R is
// compared with sqrt(c_u) widened by the bound on its error (the offsets
// come from double-float G and r, so they are good to a few 1e-7).
//
// Order of the work on a pixel: the least R of the first unit's steps; the
// first unit's steps within a few units of it (so S is close to its final
// size); then every other step that is not screened out, unit by unit.
// It is bound by the FP64 pipe in the evaluation (the median pixel of the
// large shot evaluates 1200 of its 40000 steps, the mean one 4700: pixels
// near a reflection's plane evaluate more).  Large shot, four rows of 3072
// pixels: 255.7 -> 25.0 ms; a 40x40 window: 255.4 -> 7.3 ms (the thread
// kernel gives it 13 blocks).  The
// order depends on the pixel's inputs only.  Where the bound does not exist
// (a table that is not finite; S zero, negative or not finite) nothing is
// screened out.
constexpr int kF64Warps = 4;
constexpr int kF64Threads = kF64Warps * 32;
constexpr int kF64Chunk = 128;  // sources whose vectors a warp holds
constexpr float kF64Near = 4.f;  // R above its least value, first phase

struct F64Warp {
  double2 src[kF64Chunk][2];  // (d - i0) / lambda, w cap pol omega
  double2 unit[32][2];        // d, cap pol omega
  float uf[32][8];            // v = d - i0 (hi, lo), log2 |fac|
  int cand[64];               // steps waiting: source | pm << 8
};

__host__ __device__ inline size_t f64_warp_smem(int PM, int S) {
  // axes as doubles and as float pairs, (lambda, w) and delta per source
  size_t off = (size_t)PM * 9 * (sizeof(double) + sizeof(float2)) +
               (size_t)S * (sizeof(double2) + sizeof(float));
  off = (off + 15) & ~(size_t)15;
  return off + kF64Warps * sizeof(F64Warp);
}

template <int INTERP>
__global__ void __launch_bounds__(kF64Threads, 4)
    spots_f64_warp_kernel(SpotArgs a, unsigned long long *work) {
  extern __shared__ __align__(16) double sm[];
  double2 *s_lw = reinterpret_cast<double2 *>(sm);
  double *s_ax = sm + 2 * a.S;
  float2 *s_axf = reinterpret_cast<float2 *>(s_ax + a.PM * 9);
  float *s_dh = reinterpret_cast<float *>(s_axf + a.PM * 9);
  F64Warp &W = reinterpret_cast<F64Warp *>(
      reinterpret_cast<char *>(sm) + f64_warp_smem(a.PM, a.S) -
      kF64Warps * sizeof(F64Warp))[threadIdx.x >> 5];
  for (int i = threadIdx.x; i < a.PM * 9; i += blockDim.x) {
    s_ax[i] = a.ax64[i];
    s_axf[i] = make_float2(a.axh[i], a.axl[i]);
  }
  for (int k = threadIdx.x; k < a.S; k += blockDim.x) {
    const double *src = a.src64 + (size_t)k * SRC64_STRIDE;
    s_lw[k] = make_double2(src[SRC64_LAM], src[SRC64_W]);
    s_dh[k] = a.src32[(size_t)k * SRC32_STRIDE + SRC32_DH];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  const float inf = __int_as_float(0x7f800000);
  const int PM = a.PM, S = a.S, os = a.os, U = os * os * a.T;
  const float N2[3] = {a.N[0] * a.N[0], a.N[1] * a.N[1], a.N[2] * a.N[2]};
  const float Nmax = fmaxf(a.N[0], fmaxf(a.N[1], a.N[2]));
  const float dabs = fmaxf(fabsf(s_dh[0]), fabsf(s_dh[S - 1]));  // sorted
  // log2 of the bound without the unit's factor and S
  float kb = inf;
  {
    const float Fm = __ldg(a.fmax);
    if (Fm < 1e37f)
      kb = a.screen_kb + 2.f * log2f(fmaxf(2.f * Fm, fabsf(a.defF)));
  }
  constexpr float kPerLog2 = 0.315f * 0.693147181f;
  // phi x mosaic orientations over the lanes: equal batches of at most 32;
  // below 17, several sources at a time
  const int n_b = (PM + 31) / 32, pmb = (PM + n_b - 1) / n_b;
  const int groups = 32 / pmb, grp = lane / pmb, pml = lane - grp * pmb;

  const long long n_work = a.pixlist ? a.n_list : a.npix;
  // A pixel of many steps is shared by the block's warps, each with a part
  // of its units and the sum of that part for its cuts (a lower bound of the
  // pixel's): pixels differ 100-fold in the steps they evaluate, and one warp
  // per pixel left a tail of a third of the launch on a sample of rows.
  // Otherwise a warp takes a pixel of its own, or several that share the pass
  // over their units' geometry (one when a warp gets few pixels).
  __shared__ long long s_first;
  __shared__ double s_part[kF64Warps];
  const int warp = threadIdx.x >> 5;
  const bool shared_px = U >= kF64Warps && (long long)U * PM * S >= 4096;
  const int ulo = shared_px ? warp * U / kF64Warps : 0,
            uhi = shared_px ? (warp + 1) * U / kF64Warps : U;
  const long long per_warp = n_work / ((long long)gridDim.x * kF64Warps);
  const int Bp = !shared_px && U <= 16 && per_warp >= 64 ? 32 / U : 1;
  while (true) {
    long long first = 0;
    if (shared_px) {
      __syncthreads();  // the last pixel's s_part and s_first are read
      if (threadIdx.x == 0) s_first = (long long)atomicAdd(work, 1ull);
      __syncthreads();
      first = s_first;
    } else {
      if (lane == 0)
        first = (long long)atomicAdd(work, (unsigned long long)Bp);
      first = __shfl_sync(0xffffffffu, first, 0);
    }
    if (first >= n_work) break;
    const int nb = (int)min((long long)Bp, n_work - first);
    double acc = 0.0;
    float cq = inf;   // sqrt of the unit's cut (set_cut)
    float lS = -inf;  // log2 of the sum so far
    for (int ub = ulo; ub < uhi; ub += 32) {
      const int nu = min(32, uhi - ub);  // units of a pixel in this pass
      __syncwarp();
      if (lane < nb * nu) {
        const int bi = lane / nu, u = ub + lane - bi * nu;
        const long long gp = a.pixlist ? a.pixlist[first + bi] : first + bi;
        const DevPanel &P = a.panels[panel_of_pixel(a, gp)];
        const long long local = gp - P.pix0;
        const int s = (int)(local / P.nfast);
        const int f = (int)(local - (long long)s * P.nfast);
        const int t = u % a.T, ij = u / a.T, i = ij / os, j = ij % os;
        const double px = P.px;
        double cf = (f + (i + 0.5) / os) * px, cs = (s + (j + 0.5) / os) * px,
               cn = t * a.dt;
        double pos[3], d[3];
#pragma unroll
        for (int c = 0; c < 3; ++c)
          pos[c] = P.origin[c] + cf * P.fdir[c] + cs * P.sdir[c] +
                   cn * P.ndir[c];
        double R = sqrt(dot3d(pos, pos));
#pragma unroll
        for (int c = 0; c < 3; ++c) d[c] = pos[c] / R;
        double omega = px * px * dot3d(P.ndir, pos) / (R * R * R);
        double cap = 1.0;
        if (a.thickness > 0.0) {
          double L = a.atten * dot3d(d, P.ndir);
          cap = exp(-t * a.dt / L) - exp(-(t + 1) * a.dt / L);
        }
        double c2 = dot3d(d, a.i0), x = dot3d(d, a.e0), y = dot3d(d, a.b0);
        double pol = 0.5 * (1.0 + c2 * c2 - a.kahn64 * (x * x - y * y));
        const double fac = cap * pol * omega;
        W.unit[lane][0] = make_double2(d[0], d[1]);
        W.unit[lane][1] = make_double2(d[2], fac);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const double v = d[c] - a.i0[c];
          const float vh = (float)v;
          W.uf[lane][c] = vh;
          W.uf[lane][3 + c] = (float)(v - (double)vh);
        }
        // log2 |fac| from above: exponent and mantissa of the high word,
        // log2(1 + x) <= x + 0.0861
        const int hi = __double2hiint(fac) & 0x7fffffff;
        W.uf[lane][6] = hi < 0x7ff00000
                            ? (float)hi * (1.f / 1048576.f) - 1022.9f
                            : inf;
      }
      __syncwarp();
      for (int bi = 0; bi < nb; ++bi) {
        if (ub == ulo) {
          acc = 0.0;
          lS = -inf;
        }
        float rcut = 0.f;
        // ph -1: the least R of the first unit; 0: its steps near that; 1:
        // the other steps
        for (int uu = 0; uu < nu; ++uu)
          for (int ph = ub + uu == ulo ? -1 : 1; ph < 2; ++ph) {
            const bool first_unit = ub + uu == ulo;
            const float *uf = W.uf[bi * nu + uu];
            const double2 ua = W.unit[bi * nu + uu][0],
                          uc = W.unit[bi * nu + uu][1];
            const float vh[3] = {uf[0], uf[1], uf[2]},
                        vl[3] = {uf[3], uf[4], uf[5]};
            const float lfac = uf[6];
            // the cut of this unit for the sum so far
            auto set_cut = [&]() {
              cq = inf;
              if (lS > -1000.f) {
                const float c = kPerLog2 * (kb + lfac - lS);
                // a NaN (no bound) leaves no cut
                if (c < 3e38f) cq = sqrtf(fmaxf(c, 0.f)) * 1.00001f;
              }
            };
            set_cut();
            float rmin = inf;
            for (int kc = 0; kc < S; kc += kF64Chunk) {
              const int ks = min(kF64Chunk, S - kc);
              if (ph >= 0) {
                __syncwarp();
                const double v[3] = {ua.x - a.i0[0], ua.y - a.i0[1],
                                     uc.x - a.i0[2]};
                for (int k = lane; k < ks; k += 32) {
                  const double2 lw = s_lw[kc + k];
                  W.src[k][0] = make_double2(v[0] / lw.x, v[1] / lw.x);
                  W.src[k][1] = make_double2(v[2] / lw.x, lw.y * uc.y);
                }
                __syncwarp();
              }
              int head = 0, tail = 0;
              // evaluates the next cnt <= 32 waiting steps, one per lane
              auto evaluate = [&](int cnt) {
                if (lane < cnt) {
                  const int c = W.cand[(head + lane) & 63];
                  const int k = (int)nb_idx(a.check, NB_SITE_SOURCE, c & 255,
                                            ks);
                  const double2 s0 = W.src[k][0], s1 = W.src[k][1];
                  const double Sv[3] = {s0.x, s0.y, s1.x};
                  const double *A = s_ax + (c >> 8) * 9;
                  const double h[3] = {dot3d(A, Sv), dot3d(A + 3, Sv),
                                       dot3d(A + 6, Sv)};
                  long long n[3];
                  double f[3];
                  nearest_f64(h, n, f);
                  const double a_ =
                      fcell_f64<INTERP>(a, f, n) * flatt_f64<1>(a, f);
                  acc = fma(a_ * a_, s1.y, acc);
                }
                head += cnt;
                __syncwarp();
                // log2 S from below: the largest lane sum's exponent and
                // mantissa, log2(1 + x) >= x (the high words of positive
                // doubles order like the values)
                const int hi =
                    __reduce_max_sync(0xffffffffu, __double2hiint(acc));
                lS = hi >= 0x00100000 && hi < 0x7ff00000
                         ? (float)hi * (1.f / 1048576.f) - 1023.f
                         : -inf;
                set_cut();
              };
              for (int b = 0; b < n_b; ++b) {
                const int pm = b * pmb + pml;
                const bool pm_ok = grp < groups && pm < PM;
                const float2 *A = s_axf + (pm_ok ? pm : 0) * 9;
                float G[3], r[3], gm = 0.f, am = 0.f;
#pragma unroll
                for (int x = 0; x < 3; ++x) {
                  const float Ah[3] = {A[3 * x].x, A[3 * x + 1].x,
                                       A[3 * x + 2].x};
                  const float Al[3] = {A[3 * x].y, A[3 * x + 1].y,
                                       A[3 * x + 2].y};
                  float gl, qh, qe, rh, rl;
                  ff_dot3(Ah, Al, vh, vl, G[x], gl);
                  two_prod(G[x], a.u0h, qh, qe);
                  const float ql =
                      __fmaf_rn(G[x], a.u0l, __fmaf_rn(gl, a.u0h, qe));
                  two_sum(__fsub_rn(qh, rintf(qh)), ql, rh, rl);
                  r[x] = rh;
                  gm = fmaxf(gm, fabsf(G[x]));
                  am = fmaxf(am, fabsf(Ah[0]) + fabsf(Ah[1]) + fabsf(Ah[2]));
                }
                // bound on the error of sqrt(R): the offsets' error (FP32
                // roundings of G delta + r, and of the double-float G u0)
                // times sqrt(3) N
                const float em = 1.8f * Nmax *
                                 (4e-7f * (1.f + gm * dabs) +
                                  1e-12f * am * a.u0h);
                for (int k0 = 0; k0 < ks; k0 += groups) {
                  const int k = k0 + grp;
                  const bool ok = pm_ok && k < ks;
                  const float dh = s_dh[kc + (ok ? k : 0)];
                  float R = 0.f;
#pragma unroll
                  for (int x = 0; x < 3; ++x) {
                    const float t = __fmaf_rn(G[x], dh, r[x]);
                    const float f = t - rintf(t);
                    R = __fmaf_rn(N2[x] * f, f, R);
                  }
                  if (ph < 0) {
                    rmin = fminf(rmin, ok ? R : inf);
                    continue;
                  }
                  const float lim = cq + em;
                  const bool keep =
                      ok && (ph == 0 ? R <= rcut
                                     : !(R > lim * lim) &&
                                           !(first_unit && R <= rcut));
                  const unsigned m = __ballot_sync(0xffffffffu, keep);
                  if (m) {
                    if (keep)
                      W.cand[(tail + __popc(m & below)) & 63] = k | (pm << 8);
                    tail += __popc(m);
                    __syncwarp();
                    if (tail - head >= 32) evaluate(32);
                  }
                }
              }
              if (tail > head) evaluate(tail - head);
            }
            if (ph < 0) {
              // positive floats order like their bits
              rmin = __uint_as_float(__reduce_min_sync(
                  0xffffffffu, __float_as_uint(rmin)));
              rcut = rmin + kF64Near;
            }
          }
        if (ub + 32 >= uhi) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1)
            acc += __shfl_xor_sync(0xffffffffu, acc, o);
          if (shared_px) {
            if (lane == 0) s_part[warp] = acc;
            __syncthreads();
            acc = s_part[0];
            for (int w = 1; w < kF64Warps; ++w) acc += s_part[w];
          }
          if (shared_px ? threadIdx.x == 0 : lane == 0) {
            const long long gp =
                a.pixlist ? a.pixlist[first + bi] : first + bi;
            a.image[nb_idx(a.check, NB_SITE_IMAGE, gp, a.npix)] +=
                a.prefactor * acc;
          }
        }
      }
    }
    __syncwarp();  // the next batch rewrites the units
  }
}

// Where the warp kernel runs: its fixed cost per pixel (the first unit's
// extra phase, a partial pass per unit, the divisions by lambda) is paid back
// from about 200 steps per unit with one unit, and 64 with four or more.
// 128x128 windows, tricubic, thread -> warp kernel: 1 unit, 80 steps 0.54 ->
// 0.61 ms, 100 steps 0.76 -> 0.73, 300 steps 1.99 -> 0.91; 8 units, 64 steps
// 3.45 -> 2.05; nearest lookup: 1 unit, 100 steps 0.33 -> 0.41, 300 steps
// 0.71 -> 0.44; 8 units, 64 steps 1.25 -> 0.98.
bool f64_warp_supported(const SpotArgs &a) {
  return a.shape == 1 && !a.has_div && a.fmax &&
         (long long)a.PM * a.S * (a.os * a.os * a.T >= 4 ? 4 : 1) >= 256 &&
         f64_warp_smem(a.PM, a.S) <= 200 * 1024;
}

cudaError_t launch_spots_f64_warp(const SpotArgs &a, unsigned long long *work,
                                  int sm_count, cudaStream_t st) {
  const size_t smem = f64_warp_smem(a.PM, a.S);
  void (*kern)(SpotArgs, unsigned long long *) =
      a.interp ? spots_f64_warp_kernel<1> : spots_f64_warp_kernel<0>;
  cudaError_t e = cudaFuncSetAttribute(
      kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern,
                                                    kF64Threads, smem);
  if (e != cudaSuccess) return e;
  const long long n_work = a.pixlist ? a.n_list : a.npix;
  // a block per pixel, or a warp per pixel and at most four times the blocks
  // that it needs
  const long long need = n_work;
  long long blocks = (long long)sm_count * (per_sm > 0 ? per_sm : 1);
  if (blocks > need) blocks = need;
  if (blocks < 1) return cudaSuccess;
  kern<<<(unsigned)blocks, kF64Threads, smem, st>>>(a, work);
  return cudaGetLastError();
}

// largest |F| of the table: the bits of |F| order like the values, with
// infinities and NaN above every finite one
__global__ void fmax_kernel(const float *F, long long n, unsigned *fmax) {
  unsigned m = 0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    m = max(m, __float_as_uint(F[i]) & 0x7fffffffu);
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(fmax, m);
}

cudaError_t build_fmax(const float *F, long long n, float *fmax,
                       cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(fmax, 0, sizeof(float), st);
  if (e != cudaSuccess || n <= 0) return e;
  const long long blocks = (n + 1023) / 1024;
  fmax_kernel<<<(unsigned)(blocks < 608 ? blocks : 608), 256, 0, st>>>(
      F, n, (unsigned *)fmax);
  return cudaGetLastError();
}

}  // namespace nbgb
