// split_pixel.cuh -- the warp-per-pixel FP32-mixed Bragg-spot sum for
// Gaussian shapes, shared by the stand-alone kernel (spots_split.cu) and the
// serving kernel (serve.cu): table staging (split_stage), the FP64 set-up of
// one sub-pixel unit (split_unit) and the per-pixel sum of one warp
// (split_sum).  See spots_split.cu for the method.
#pragma once

#include "mixed_common.cuh"

namespace nbgb {

constexpr int kSplitWarps = 4;
constexpr int kSplitThreads = kSplitWarps * 32;
constexpr int kMaxUnits = 32;
constexpr int kUnitFloats = 10;  // vh[3], vl[3], scal, df[3]
constexpr int kFfUnits = 2;      // double-float geometry up to so many units
inline bool split_ff(const SpotArgs &a) {
  return a.os * a.os * a.T <= kFfUnits;
}
constexpr int kSrcBlock = 8;     // sources per pruning block
// Per-warp ring of source intervals.  An entry is one (item, source range)
// pair that can hold surviving terms, with a copy of its item's state, so
// that entries outlive the item batch that pushed them.  Pending entries
// never exceed 31 (each holds an unconsumed source) plus the 32 a push adds.
constexpr int kEntries = 64;

// Two kinds of entry.  An interval entry belongs to one lattice point m of
// the item's sweep: every surviving step of it has m as its nearest
// integer, so the entry holds r_q - (m - n0) in place of r_q and m's table
// index, and a step's offset needs no rounding.  A block entry (pruning by
// source blocks, or sources of different directions) holds r_q and n0, and
// each step rounds to its nearest integer.
struct SplitEntry {
  float4 a;  // G_hi h, G_hi k, r h, r k      (r = r_q, or r_q - (m - n0))
  float4 b;  // G_lo h, G_lo k, r_lo h, r_lo k
  float4 c;  // G_hi l, r l, G_lo l, r_lo l
  float4 d;  // n0 h, n0 k, n0 l (floats), or for m (int bits) its table
             // index, or with tricubic cell polynomials ci0, the index
             // packed (10 bits per axis, plus 1) and pk (entry_cell_data);
             // and omega cap pol of the unit
  int4 m;    // first source, count, position of the first source in the
             // pixel's sequence of (entry, source) pairs,
             // pm | unit << 16 | interval entry << 31
};
constexpr int kIntervalEntry = 1 << 31;
// Lines: from so many sources and steps per pixel interval entries are summed
// segment by segment (sum_tasks), in tasks of at most kTaskLen steps (even; 16
// cost the large shot 6 % more).  Kernels of this form have 128 registers (4
// blocks per SM): 96 (5) spill 540 bytes, 168 (3) hide less: 13.4, 11.6 and
// 11.8 ms on 1024^2 pixels of the large shot when it was chosen.
constexpr int kLineSources = 32;
constexpr int kLineSteps = 1200;
constexpr float kLineMean = 15.f;
constexpr int kTaskLen = 32;
constexpr int kLineBlocks = 4;
constexpr int SRC32_PAIR = 4;
static_assert(sizeof(SplitEntry) % 16 == 0, "entries stay 16-byte aligned");
static_assert(SRC32_DL == 0 && SRC32_W == 1 && SRC32_DH == 2 &&
                  SRC32_STRIDE % 4 == 0 && kUnitFloats % 2 == 0,
              "one float4 read of (delta_lo, w, delta_hi, .) per source "
              "and float2 reads of the unit rows");

// ff_dot3 (mixed_common.cuh) with the double-float row stored as
// interleaved (hi, lo) pairs: the same operations, half the shared loads
__device__ __forceinline__ void ff_dot3_pairs(const float2 *A,
                                              const float *vh,
                                              const float *vl, float &gh,
                                              float &gl) {
  const float2 a0 = A[0], a1 = A[1], a2 = A[2];
  float p0, e0, p1, e1, p2, e2;
  two_prod(a0.x, vh[0], p0, e0);
  two_prod(a1.x, vh[1], p1, e1);
  two_prod(a2.x, vh[2], p2, e2);
  float s, t, s2, t2;
  two_sum(p0, p1, s, t);
  two_sum(s, p2, s2, t2);
  float lo = e0 + e1 + e2 + t + t2;
  lo = fmaf(a0.x, vl[0], lo);
  lo = fmaf(a1.x, vl[1], lo);
  lo = fmaf(a2.x, vl[2], lo);
  lo = fmaf(a0.y, vh[0], lo);
  lo = fmaf(a1.y, vh[1], lo);
  lo = fmaf(a2.y, vh[2], lo);
  fast_two_sum(s2, lo, gh, gl);
}

// Per-warp cache of cell polynomials in shared memory.  The terms of one
// evaluation pass almost always lie around a single lattice point n, in the
// cells n - {0,1}^3, and those 8 cells have distinct parities (the low bit
// of each corner index).  So the cache has one slot per parity, and chunk k
// (float4) of slot p sits at float4 k * kCellSlots + p: the same chunk of
// every slot lies in one 128-byte row of shared-memory banks, and one
// 16-byte load of chunk k by all lanes is a single shared-memory wavefront
// whatever mix of slots the lanes read (lanes on one slot get a
// broadcast).  A global 16-byte load delivers 128 bytes per wavefront
// whether the lanes' addresses coincide or not, so reading the 256
// coefficient bytes of each term from global memory costs 2 wavefronts per
// term; from the cache it costs 1/2.
constexpr int kCellSlots = 8;
constexpr int kCellChunks = 16;  // float4 per cell polynomial

// A cell's tricubic polynomial at x (cell coordinates in [0, 1)): nested
// Horner in l, k, h, the z and y chains of the powers x^(2P) and x^(2P+1)
// side by side in packed FMAs (30 packed + 3 scalar FMAs for the 63 of
// the scalar form, with the same roundings); chunk q of the coefficients
// (the layout of SpotArgs::C4) at cp[q * stride], read from shared memory
// (SHARED) or through the read-only path.
template <bool SHARED>
__device__ __forceinline__ float cell_horner(const float4 *cp, int stride,
                                             const float x[3]) {
  const float2 z2 = make_float2(x[2], x[2]), y2 = make_float2(x[1], x[1]);
  float2 q[2];
#pragma unroll
  for (int P = 0; P < 2; ++P) {
    float2 pb[4];
#pragma unroll
    for (int ib = 0; ib < 4; ++ib) {
      const int q0 = (P * 4 + ib) * 2;
      const float4 A = SHARED ? cp[q0 * stride] : __ldg(cp + q0 * stride);
      const float4 B =
          SHARED ? cp[(q0 + 1) * stride] : __ldg(cp + (q0 + 1) * stride);
      float2 v = ffma2(make_float2(A.x, A.y), z2, make_float2(A.z, A.w));
      v = ffma2(v, z2, make_float2(B.x, B.y));
      pb[ib] = ffma2(v, z2, make_float2(B.z, B.w));
    }
    q[P] = ffma2(ffma2(ffma2(pb[3], y2, pb[2]), y2, pb[1]), y2, pb[0]);
  }
  // q[P] = (C(x^(2P)) part, C(x^(2P+1)) part); Horner in x
  return fmaf(fmaf(fmaf(q[1].y, x[0], q[1].x), x[0], q[0].y), x[0], q[0].x);
}

// n[2] of a term whose index is still packed (interval entries with cell
// polynomials): n[0] then holds the packed index of SplitEntry::d.y
constexpr int kPackedIndex = -0x40000000;

// The cell of a tricubic term: whether its 4x4x4 stencil lies inside the
// table (tri), the cell's index in the polynomial table (ci), its parity
// slot in the cache (par) and the coordinates x in [0, 1) within the cell.
struct CellRef {
  bool tri;
  int ci, par;
  float x[3];
};

// The cell of a step with fractional offset fr and table-relative nearest
// index n: its stencil starts at fl - 1, fl = n - (fr < 0) per axis.
template <int INTERP>
__device__ __forceinline__ void cell_of(const SpotArgs &a, bool hit,
                                        const float fr[3], const int n[3],
                                        CellRef &c) {
  int fl[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int neg = fr[k] < 0.f;
    fl[k] = n[k] - neg;
    c.x[k] = neg ? 1.f + fr[k] : fr[k];
  }
  // the 4x4x4 stencil fl - 1 .. fl + 2 inside the table
  c.tri = INTERP == 1 && hit && a.C4 &&
          (unsigned)(fl[0] - 1) < (unsigned)(a.hn[0] - 3) &&
          (unsigned)(fl[1] - 1) < (unsigned)(a.hn[1] - 3) &&
          (unsigned)(fl[2] - 1) < (unsigned)(a.hn[2] - 3);
  c.ci = 0;
  c.par = 0;
  if (c.tri) {
    c.ci = ((fl[0] - 1) * (a.hn[1] - 3) + (fl[1] - 1)) * (a.hn[2] - 3) +
           (fl[2] - 1);
    c.par = (fl[0] & 1) | ((fl[1] & 1) << 1) | ((fl[2] & 1) << 2);
  }
}

// Cell data of an interval entry's lattice point m (table-relative index
// nt), computed once per entry: ci0 = the index of the cell whose stencil
// starts at nt - 1; pk = the parity of nt (bits 0-2) and, in bits 3-10,
// for each sign pattern s of a step's offset (bit k: f_k < 0, which moves
// the stencil one node down along axis k) whether that stencil lies inside
// the table.  A step's cell is then ci0 minus the strides its pattern
// selects, with parity pk ^ s.
__device__ __forceinline__ void entry_cell_data(const SpotArgs &a,
                                                const int nt[3], int &ci0,
                                                int &pk) {
  const int H1 = a.hn[1] - 3, H2 = a.hn[2] - 3;
  ci0 = ((nt[0] - 1) * H1 + (nt[1] - 1)) * H2 + (nt[2] - 1);
  // sign pattern s has bit k set when axis k moves down
  const unsigned pos_bits[3] = {0x55u, 0x33u, 0x0Fu};
  unsigned ok = 0xFFu;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const unsigned span = (unsigned)(a.hn[k] - 3);
    const bool up = (unsigned)(nt[k] - 1) < span;    // f_k >= 0
    const bool down = (unsigned)(nt[k] - 2) < span;  // f_k < 0
    ok &= (up ? pos_bits[k] : 0u) | (down ? (~pos_bits[k] & 0xFFu) : 0u);
  }
  pk = (nt[0] & 1) | ((nt[1] & 1) << 1) | ((nt[2] & 1) << 2) | (int)(ok << 3);
}

__device__ __forceinline__ void cell_of_entry(const SpotArgs &a, bool hit,
                                              const float fr[3], int ci0,
                                              int pk, CellRef &c) {
  const int s = (fr[0] < 0.f) | ((fr[1] < 0.f) << 1) | ((fr[2] < 0.f) << 2);
#pragma unroll
  for (int k = 0; k < 3; ++k) c.x[k] = fr[k] < 0.f ? 1.f + fr[k] : fr[k];
  const int H2 = a.hn[2] - 3;
  c.tri = hit && ((pk >> (3 + s)) & 1);
  c.ci = ci0 - ((s & 1) ? (a.hn[1] - 3) * H2 : 0) - ((s & 2) ? H2 : 0) -
         ((s >> 2) & 1);
  c.par = (pk & 7) ^ s;
}

// The term F_cell^2 F_latt^2 w of a lane whose step survived the cut (`hit`),
// given its fractional offset fr, table-relative nearest index n, cell c
// and exponent sum rad2 = sum N^2 fr^2.  Called
// by all 32 lanes of the warp: missing cells are loaded into the cache by
// the whole warp (one coalesced 256-byte read per cell).  A lane whose
// parity slot ends up holding another cell (two lattice points in one pass)
// reads its cell from global memory instead.
template <int INTERP>
__device__ __forceinline__ float term_value(const SpotArgs &a, bool hit,
                                            const CellRef &c,
                                            const float fr[3], const int n[3],
                                            float rad2, float w,
                                            float4 *cache, int *tags) {
  // fast exp: a few ulp for the significant terms (|argument| < ~20)
  const float fl2 = a.N6 * __expf(-2.f * rad2 * (1.f / 0.63f));
  bool cached = false;
  if (INTERP == 1) {
    const int lane = threadIdx.x & 31;
    unsigned miss = __ballot_sync(0xffffffffu, c.tri && tags[c.par] != c.ci);
    if (miss == 0u) {
      cached = c.tri;
    } else {
      unsigned handled = 0u;
      while (miss) {
        // load the cell of the first missing lane into its parity slot; each
        // slot is loaded at most once per pass
        const int src = __ffs(miss) - 1;
        const int sp = __shfl_sync(0xffffffffu, c.par, src);
        const int sci = __shfl_sync(0xffffffffu, c.ci, src);
        const float2 v = __ldg(
            reinterpret_cast<const float2 *>(
                a.C4 + (size_t)nb_idx(a.check, NB_SITE_CELL, sci,
                                      cell_count(a)) *
                           kCellChunks) +
            lane);
        reinterpret_cast<float2 *>(
            cache)[((lane >> 1) * kCellSlots + sp) * 2 + (lane & 1)] = v;
        __syncwarp();
        if (lane == 0) tags[sp] = sci;
        __syncwarp();
        handled |= 1u << sp;
        miss = __ballot_sync(0xffffffffu, c.tri && !((handled >> c.par) & 1u) &&
                                              tags[c.par] != c.ci);
      }
      cached = c.tri && tags[c.par] == c.ci;
    }
  }
  float fc = 0.f;
  if (cached) {
    fc = cell_horner<true>(cache + c.par, kCellSlots, c.x);
  } else if (c.tri) {
    fc = cell_horner<false>(
        a.C4 + (size_t)nb_idx(a.check, NB_SITE_CELL, c.ci, cell_count(a)) *
                   kCellChunks,
        1, c.x);
  } else if (hit) {
    int nn[3] = {n[0], n[1], n[2]};
    if (n[2] == kPackedIndex) {
      nn[0] = (n[0] & 1023) - 1;
      nn[1] = ((n[0] >> 10) & 1023) - 1;
      nn[2] = ((n[0] >> 20) & 1023) - 1;
    }
    fc = fcell_f32<INTERP>(a, nn, fr);
  }
  return fc * fc * fl2 * w;
}

// Per-block view of one shot's staged tables in shared memory and the
// constants derived from them.
struct SplitBlock {
  const float2 *ax2;  // [PM][9] (hi, lo) pairs
  const float *src, *blk, *dh;
  float *unit_base;
  SplitEntry *ent_base;  // [warp][kEntries]
  float4 *cell_cache;    // [warp][kCellChunks][kCellSlots]
  int *cell_tags;        // [warp][kCellSlots], -1 = empty
  int PM, S, nblk, sstep;
  float u0h, u0l, cwide, dmin, dmax, dmarg, inv_step;
  float cmarg[3];
  float umid, dhalf, nmarg[3];  // split_item's early test
  bool iv_ok, even;
};

// Bytes of dynamic shared memory split_stage lays out for PM orientations
// and S sources.
__host__ __device__ inline int split_axes_floats(int PM) {
  return (2 * PM * 9 + 3) & ~3;  // the source rows after it 16-byte aligned
}

__host__ __device__ inline size_t split_smem_layout(int PM, int S) {
  const int nblk = (S + kSrcBlock - 1) / kSrcBlock;
  size_t off = (size_t)(split_axes_floats(PM) + S * SRC32_STRIDE +
                        kSplitWarps * kMaxUnits * kUnitFloats) *
               sizeof(float);
  off = (off + 15) & ~(size_t)15;
  off += (size_t)kSplitWarps * kEntries * sizeof(SplitEntry);
  off += (size_t)kSplitWarps * kCellChunks * kCellSlots * sizeof(float4);
  off += (size_t)(2 * nblk + S) * sizeof(float);
  off += (size_t)kSplitWarps * kCellSlots * sizeof(int);
  return off;
}

// Whether the ellipsoids of neighbouring lattice points at the (widened) cut
// are disjoint, so that a source has one of them at most
__host__ __device__ inline float cut_wide() {
  return kGaussCut * 0.63f * 1.02f + 1e-4f;
}
constexpr float kDisjoint = 0.49f;
__host__ __device__ inline bool lattice_disjoint(const SpotArgs &a) {
  const float m = sqrtf(cut_wide());
  return m / a.N[0] < kDisjoint && m / a.N[1] < kDisjoint &&
         m / a.N[2] < kDisjoint;
}

// Stages a shot's tables (double-float axes [PM][9], interleaved into
// (hi, lo) pairs, and source rows [S][12]) into the dynamic shared memory
// `sms` and derives the pruning constants.  Called by every thread of the
// block.
__device__ __forceinline__ void split_stage(SplitBlock &b, float *sms,
                                            const SpotArgs &a,
                                            const float *axh, const float *axl,
                                            const float *src32, int PM, int S,
                                            float u0h, float u0l) {
  float2 *s_ax2 = reinterpret_cast<float2 *>(sms);
  float *s_src = sms + split_axes_floats(PM);
  float *s_unit = s_src + S * SRC32_STRIDE;  // [warp][unit][kUnitFloats]
  // entries and cache hold float4s: 16-byte aligned base
  const size_t ent_off =
      ((size_t)(s_unit + kSplitWarps * kMaxUnits * kUnitFloats - sms) *
           sizeof(float) + 15) & ~(size_t)15;
  SplitEntry *s_ent = reinterpret_cast<SplitEntry *>(
      reinterpret_cast<char *>(sms) + ent_off);
  float4 *s_cache = reinterpret_cast<float4 *>(s_ent + kSplitWarps * kEntries);
  float *s_blk =
      reinterpret_cast<float *>(s_cache + kSplitWarps * kCellChunks * kCellSlots);
  const int nblk = (S + kSrcBlock - 1) / kSrcBlock;
  float *s_dh = s_blk + 2 * nblk;  // delta_hi of every source, contiguous
  int *s_tags = reinterpret_cast<int *>(s_dh + S);
  for (int i = threadIdx.x; i < kSplitWarps * kCellSlots; i += blockDim.x)
    s_tags[i] = -1;
  for (int i = threadIdx.x; i < PM * 9; i += blockDim.x)
    s_ax2[i] = make_float2(axh[i], axl[i]);
  for (int i = threadIdx.x; i < S * SRC32_STRIDE; i += blockDim.x)
    s_src[i] = src32[i];
  __syncthreads();
  // with one beam direction a row's other columns hold the source and the
  // next one side by side (sum_tasks): (delta_hi x2, delta_lo x2), w x2; the
  // last source is followed by itself with weight 0
  if (!a.has_div)
    for (int k = threadIdx.x; k < S; k += blockDim.x) {
      float *q = s_src + k * SRC32_STRIDE;
      const float *q1 = k + 1 < S ? q + SRC32_STRIDE : q;
      q[SRC32_PAIR] = q[SRC32_DH];
      q[SRC32_PAIR + 1] = q1[SRC32_DH];
      q[SRC32_PAIR + 2] = q[SRC32_DL];
      q[SRC32_PAIR + 3] = q1[SRC32_DL];
      q[SRC32_PAIR + 4] = q[SRC32_W];
      q[SRC32_PAIR + 5] = k + 1 < S ? q1[SRC32_W] : 0.f;
    }
  // delta_hi range of every block of kSrcBlock sources (the pruning test)
  for (int bb = threadIdx.x; bb < nblk; bb += blockDim.x) {
    float mn = 3.0e38f, mx = -3.0e38f;
    for (int k = bb * kSrcBlock; k < S && k < (bb + 1) * kSrcBlock; ++k) {
      float d = s_src[k * SRC32_STRIDE + SRC32_DH];
      mn = fminf(mn, d);
      mx = fmaxf(mx, d);
    }
    s_blk[2 * bb] = mn;
    s_blk[2 * bb + 1] = mx;
  }
  for (int k = threadIdx.x; k < S; k += blockDim.x)
    s_dh[k] = s_src[k * SRC32_STRIDE + SRC32_DH];
  __syncthreads();
  // exact intervals need delta_hi in ascending order (the library sorts the
  // sources; a caller of the allocation-free entry may not)
  int unsorted = 0;
  for (int k = threadIdx.x; k + 1 < S; k += blockDim.x)
    unsorted |= s_dh[k] > s_dh[k + 1];
  const bool dh_sorted = __syncthreads_or(unsorted) == 0;
  b.ax2 = s_ax2;
  b.src = s_src;
  b.blk = s_blk;
  b.dh = s_dh;
  b.unit_base = s_unit;
  b.ent_base = s_ent;
  b.cell_cache = s_cache;
  b.cell_tags = s_tags;
  b.PM = PM;
  b.S = S;
  b.nblk = nblk;
  b.u0h = u0h;
  b.u0l = u0l;
  // a widened cut for the conservative tests: every surviving term has
  // sum N^2 f^2 <= cutg < cwide, so |f_x| <= sqrt(cwide) / N_x
  b.cwide = cut_wide();
  for (int x = 0; x < 3; ++x) b.cmarg[x] = sqrtf(b.cwide) / a.N[x];
  // exact delta-intervals per lattice point need the ellipsoids of
  // neighbouring lattice points to be disjoint: sqrt(cwide)/N < 1/2
  b.iv_ok = dh_sorted && b.cmarg[0] < kDisjoint && b.cmarg[1] < kDisjoint &&
            b.cmarg[2] < kDisjoint;
  b.dmin = S > 0 ? s_dh[0] : 0.f;
  b.dmax = S > 0 ? s_dh[S - 1] : 0.f;
  b.dmarg = 1e-3f * (b.dmax - b.dmin) / (float)(S > 1 ? S - 1 : 1);
  int sstep = 1;
  while (sstep * 2 <= S) sstep *= 2;
  b.sstep = sstep;
  // the early test: 1/lambda = umid +- dhalf; cmarg plus the error of h in
  // plain FP32 (a few roundings of sum |A_i v_i| / lambda, |v| <= 2)
  {
    float am = 0.f;
    for (int r = threadIdx.x; r < PM * 3; r += blockDim.x)
      am = fmaxf(am, fabsf(s_ax2[3 * r].x) + fabsf(s_ax2[3 * r + 1].x) +
                         fabsf(s_ax2[3 * r + 2].x));
    // positive floats order like their bits
    am = __uint_as_float(
        __reduce_max_sync(0xffffffffu, __float_as_uint(am)));
    __shared__ float s_am[kSplitWarps];
    if ((threadIdx.x & 31) == 0) s_am[threadIdx.x >> 5] = am;
    __syncthreads();
    for (int w = 0; w < kSplitWarps; ++w) am = fmaxf(am, s_am[w]);
    b.umid = u0h + 0.5f * (b.dmin + b.dmax);
    b.dhalf = 0.5f * (b.dmax - b.dmin) * 1.00001f;
    for (int x = 0; x < 3; ++x)
      b.nmarg[x] = b.cmarg[x] + 2e-6f * am * (b.umid + b.dhalf) + 1e-5f;
  }
  // nearly even delta spacing (an equispaced spectrum): the position of a
  // bound in the table is then guessed from the spacing and corrected by a
  // step or two, instead of a binary search
  const float step = S > 1 ? (b.dmax - b.dmin) / (float)(S - 1) : 0.f;
  int uneven = !(step > 0.f);
  for (int k = threadIdx.x; k < S && !uneven; k += blockDim.x)
    uneven |= !(fabsf(s_dh[k] - fmaf((float)k, step, b.dmin)) <= step);
  b.even = __syncthreads_or(uneven) == 0;
  b.inv_step = b.even ? 1.f / step : 0.f;
}

// k1 = #{k : delta_k < lo} and k2 = #{k : delta_k <= hi} in the ascending
// table dh[0..S): from a guess, walk down while the entry below is on the
// wrong side, then up while the entry above is.  Exact for any guess in
// [0, S]; the guess only sets the number of steps.
__device__ __forceinline__ int count_below(const float *dh, int S, int k,
                                           float lo) {
  while (k > 0 && dh[k - 1] >= lo) --k;
  while (k < S && dh[k] < lo) ++k;
  return k;
}
__device__ __forceinline__ int count_at_most(const float *dh, int S, int k,
                                             float hi) {
  while (k > 0 && dh[k - 1] > hi) --k;
  while (k < S && dh[k] <= hi) ++k;
  return k;
}
__device__ __forceinline__ int guess_index(float x, float dmin, float inv,
                                           int S) {
  // fmaxf/fminf also map a NaN to 0
  return (int)fminf(fmaxf(ceilf((x - dmin) * inv), 0.f), (float)S);
}

// Geometry of sub-pixel unit u (subpixel i, j, sensor layer t) of pixel
// (s, f) of panel P into ud[kUnitFloats]: v = d - i0 as double-float,
// omega cap (times the polarization for one beam direction), and d in FP32.
// FF: double-float geometry, for shots of up to kFfUnits units (split_ff).
template <int HASDIV, bool FF>
__device__ __forceinline__ void split_unit(const SpotArgs &a,
                                           const DevPanel &P, int s, int f,
                                           int u, float *ud) {
  const int os = a.os;
  const float kahn = a.kahn;
  int t = u % a.T, ij = u / a.T, i = ij / os, j = ij % os;
  float vh[3], vl[3], df[3], omega;
  // Up to kFfUnits units per pixel: double-float (unit_geometry_ff, as the
  // thread-per-pixel kernel).  A pass over the units of one or a few pixels
  // has few lanes at work, and ~110 FP64-pipe instructions at 16 cycles each
  // then cost more than such a pixel's whole sum (128^2 pixels, 1 unit, 99
  // steps: 83 -> 40 us with batches of pixels, below).  With more units: FP64
  // (one rsqrt, products), which overlaps with the FP32 work of their many
  // steps (1500^2 pixels, 4 units, 99 steps: double-float 2.58, FP64 2.40 ms;
  // large shot, 8 units: 220.4 and 216.5 ms at the time).  The choice depends
  // on the shot alone, so a pixel's value does not depend on the launch, and
  // it is a template parameter: both in one kernel cost the large shot 0.4 %.
  if (FF) {
    unit_geometry_ff<true>(a, P, s, f, i, j, t, vh, vl, df, omega);
  } else {
    const double px = P.px, inv_os = 1.0 / os;
    double cf = (f + (i + 0.5) * inv_os) * px,
           cs = (s + (j + 0.5) * inv_os) * px, cn = t * a.dt;
    double pos[3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
      pos[c] = P.origin[c] + cf * P.fdir[c] + cs * P.sdir[c] +
               cn * P.ndir[c];
    const double inv = rsqrt(dot3d_m(pos, pos));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double d = pos[c] * inv, v = d - a.i0[c];
      vh[c] = (float)v;
      vl[c] = (float)(v - (double)vh[c]);
      df[c] = (float)d;
    }
    omega = (float)(px * px * dot3d_m(P.ndir, pos) * (inv * inv * inv));
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    ud[c] = vh[c];
    ud[3 + c] = vl[c];
    ud[7 + c] = df[c];
  }
  float cap = 1.f;
  if (a.dtff[0] > 0.f) {
    float rho = df[0] * P.ffn[0][0] + df[1] * P.ffn[1][0] +
                df[2] * P.ffn[2][0];
    float L = a.attenf * rho, dtf = a.dtff[0];
    cap = expf(-t * dtf / L) - expf(-(t + 1) * dtf / L);
  }
  float scal = omega * cap;
  if (!HASDIV) {
    float c2 = df[0] * a.i0ff[0][0] + df[1] * a.i0ff[1][0] +
               df[2] * a.i0ff[2][0];
    float x = df[0] * a.e0f[0] + df[1] * a.e0f[1] +
              df[2] * a.e0f[2];
    float y = df[0] * a.b0f[0] + df[1] * a.b0f[1] +
              df[2] * a.b0f[2];
    scal *= 0.5f * (1.f + c2 * c2 - kahn * (x * x - y * y));
  }
  ud[6] = scal;
}

// Work one warp performed (warp-uniform counts), for the launch statistics
struct SplitCounts {
  unsigned long long terms = 0;   // terms evaluated
  unsigned long long pairs = 0;   // (entry, source) pairs tested
  unsigned long long ivals = 0;   // lattice-point intervals solved
  unsigned long long blocks = 0;  // source blocks tested
};

// Per-warp queue of (entry, source) pairs: entries [e0, en) of the ring
// are pending, pairs [ch, ct) of the pixel's sequence are not yet summed.
struct PairQueue {
  int e0 = 0, en = 0, ch = 0, ct = 0;
};

// A warp sums one pixel with all its lanes, or one with every W of them: a
// lane's place among its pixel's lanes, the first of them, and their bits of
// a ballot.
template <int W>
struct Lanes {
  static constexpr unsigned mask = W == 32 ? 0xffffffffu : (1u << (W & 31)) - 1u;
  int l, first;
  __device__ __forceinline__ Lanes() {
    const int lane = threadIdx.x & 31;
    l = lane & (W - 1);
    first = lane & ~(W - 1);
  }
  __device__ __forceinline__ unsigned own(unsigned ballot) const {
    return (ballot >> first) & mask;
  }
};
// entries of the ring of a pixel's lanes
template <int W>
constexpr int kRing = kEntries * W / 32;

// Appends one entry per lane with len > 0 pairs (or tasks), in lane order: the
// state of the lane's item (r and d4 as SplitEntry describes) and the words
// of SplitEntry::m.  Called by all lanes.
template <int W = 32>
__device__ __forceinline__ void push_entries(
    SplitEntry *ring, PairQueue &pq, int len, int mx, int my, int mw,
    const float Gh[3], const float r[3], const float Gl[3], const float rl[3],
    float4 d4) {
  const Lanes<W> at;
  const unsigned any = __ballot_sync(0xffffffffu, len > 0);
  if (any == 0u) return;
  const unsigned hm = at.own(any);
  int inc = len;
#pragma unroll
  for (int o = 1; o < W; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o, W);
    if (at.l >= o) inc += t;
  }
  const int tot = __shfl_sync(0xffffffffu, inc, W - 1, W);
  if (len > 0) {
    SplitEntry &E =
        ring[(pq.en + __popc(hm & ((1u << at.l) - 1u))) & (kRing<W> - 1)];
    E.a = make_float4(Gh[0], Gh[1], r[0], r[1]);
    E.b = make_float4(Gl[0], Gl[1], rl[0], rl[1]);
    E.c = make_float4(Gh[2], r[2], Gl[2], rl[2]);
    E.d = d4;
    E.m = make_int4(mx, my, pq.ct + inc - len, mw);
  }
  pq.en += __popc(hm);
  pq.ct += tot;
  __syncwarp();
}

// Sums the next min(W, ct - ch) pairs of the queue, one per lane: the exact
// fractional offset of the step, the cut test, and for a surviving step its
// term (F_cell from the cell cache, F_latt, weight) into the lane's Kahan
// sum; none where `go` (the same in all of a pixel's lanes) is false.  Called
// by all lanes; returns the number of the warp's surviving terms.
template <int INTERP, int HASDIV, int W = 32>
__device__ __forceinline__ unsigned sum_pairs(
    const SpotArgs &a, const SplitBlock &b, const SplitEntry *ring,
    PairQueue &pq, const float *unit, float4 *cache, int *tags, Kahan &acc,
    unsigned &npairs, bool go = true) {
  const Lanes<W> at;
  const int lane = at.l;
  const int np = go ? min(W, pq.ct - pq.ch) : 0;
  // entries e0 .. e0 + W - 1 can overlap the window [ch, ch + W)
  int4 mm = make_int4(0, 0, 0x7fffffff, 0);
  if (pq.e0 + lane < pq.en) mm = ring[(pq.e0 + lane) & (kRing<W> - 1)].m;
  const bool ov = pq.e0 + lane < pq.en && mm.z < pq.ch + np &&
                  mm.z + mm.y > pq.ch;
  // bit j of M: some entry starts at pair ch + j (entry e0 at bit 0)
  const unsigned M = at.own(__reduce_or_sync(
      0xffffffffu, ov ? 1u << (at.first + max(mm.z - pq.ch, 0)) : 0u));
  // (W < 32: a pixel without pairs in this pass reads some entry, unused)
  const int j0 = __popc(M & (at.mask >> (W - 1 - lane))) - 1,
            j = W == 32 ? j0 : max(j0, 0);
  const int k1 = __shfl_sync(0xffffffffu, mm.x, j, W);
  const int pos = __shfl_sync(0xffffffffu, mm.z, j, W);
  const int aux = __shfl_sync(0xffffffffu, mm.w, j, W);
  const unsigned done = at.own(
      __ballot_sync(0xffffffffu, ov && mm.z + mm.y <= pq.ch + np));
  const bool valid = lane < np;
  const int k =
      valid ? (int)nb_idx(a.check, NB_SITE_SOURCE, k1 + (pq.ch + lane - pos),
                          b.S)
            : 0;
  const SplitEntry &E = ring[(pq.e0 + j) & (kRing<W> - 1)];
  const float4 A = E.a, B = E.b, C = E.c, D = E.d;
  const float Gh[3] = {A.x, A.y, C.x}, r[3] = {A.z, A.w, C.y};
  const float Gl[3] = {B.x, B.y, C.z}, rl[3] = {B.z, B.w, C.w};
  const float *src = b.src + k * SRC32_STRIDE;
  // (delta_lo, w, delta_hi) of source k in one load
  const float4 sw = *reinterpret_cast<const float4 *>(src);
  const float dh = sw.z;
  const float2 dlw = make_float2(sw.x, sw.y);
  float fr[3];
  int n[3];
  if (!HASDIV && (aux & kIntervalEntry)) {
    // G_hi d_hi + (r_q - (m - n0)) in one rounding plus the small terms;
    // the nearest integer is m
    // axes h and k in packed FMAs, l in scalar ones (the same roundings)
    const float2 dh2 = make_float2(dh, dh), dl2 = make_float2(dlw.x, dlw.x);
    const float2 f01 =
        fadd2(ffma2(make_float2(A.x, A.y), dh2, make_float2(A.z, A.w)),
              ffma2(make_float2(A.x, A.y), dl2,
                    ffma2(make_float2(B.x, B.y), dh2, make_float2(B.z, B.w))));
    fr[0] = f01.x;
    fr[1] = f01.y;
    fr[2] = fmaf(Gh[2], dh, r[2]) + fmaf(Gh[2], dlw.x, fmaf(Gl[2], dh, rl[2]));
    if (INTERP == 1 && a.C4) {
      // the packed index; unpacked only where a term needs the table
      // itself (term_value's fallback)
      n[0] = __float_as_int(D.y);
      n[1] = n[2] = kPackedIndex;
    } else {
      n[0] = __float_as_int(D.x);
      n[1] = __float_as_int(D.y);
      n[2] = __float_as_int(D.z);
    }
  } else {
    const float n0[3] = {D.x, D.y, D.z};
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      float tq = fmaf(Gh[x], dh, r[x]);
      float e0 = 0.f, e1 = 0.f;
      if (HASDIV) {
        const size_t e = ((size_t)(aux & 0xffff) * b.S + k) * 3 + x;
        e0 = __ldg(a.divh + e);
        e1 = __ldg(a.divl + e);
        tq -= e0;
      }
      float nf = rintf(tq);
      // G_hi d_hi + (r_q - n) in one rounding (r_q on a 2^-21 grid makes
      // r_q - n exact) plus the small terms
      const float sx = fmaf(Gh[x], dh, __fsub_rn(r[x], nf));
      const float c = fmaf(Gh[x], dlw.x, fmaf(Gl[x], dh, rl[x]));
      fr[x] = sx + c;
      if (HASDIV) {
        // the divergence term moves h after the rint: re-centre
        fr[x] -= e0 + e1;
        const float n2 = rintf(fr[x]);
        fr[x] -= n2;
        nf += n2;
      }
      n[x] = __float2int_rn(n0[x] + nf) - a.hmin[x];
    }
  }
  float rad2 = a.N[0] * a.N[0] * fr[0] * fr[0];
  rad2 = fmaf(a.N[1] * a.N[1], fr[1] * fr[1], rad2);
  rad2 = fmaf(a.N[2] * a.N[2], fr[2] * fr[2], rad2);
  const bool hit = valid && rad2 <= kGaussCut * 0.63f;
  float w = dlw.y * D.w;
  if (HASDIV && hit) {
    const float *df = unit + ((aux >> 16) & 31) * kUnitFloats + 7;
    const float *dir = src + SRC32_DIR, *ev = src + SRC32_E,
                *bv = src + SRC32_B;
    const float c2 = df[0] * dir[0] + df[1] * dir[1] + df[2] * dir[2];
    const float xx = df[0] * ev[0] + df[1] * ev[1] + df[2] * ev[2];
    const float yy = df[0] * bv[0] + df[1] * bv[1] + df[2] * bv[2];
    w *= 0.5f * (1.f + c2 * c2 - a.kahn * (xx * xx - yy * yy));
  }
  npairs += valid;
  const unsigned hm = __ballot_sync(0xffffffffu, hit);
  if (hm != 0u) {
    CellRef cr;
    if (INTERP == 1 && !HASDIV && a.C4 && (aux & kIntervalEntry))
      cell_of_entry(a, hit, fr, __float_as_int(D.x), __float_as_int(D.z), cr);
    else
      cell_of<INTERP>(a, hit, fr, n, cr);
    const float t =
        term_value<INTERP>(a, hit, cr, fr, n, rad2, w, cache, tags);
    if (hit) acc.add(t);
  }
  pq.e0 += __popc(done);
  pq.ch += np;
  __syncwarp();  // the ring slots read above may be refilled next
  return __popc(hm);
}

// ------------------------------------------------- lines through a cell
//
// The steps of an interval entry lie on a line: with t = delta - delta_0 their
// offset from the lattice point is f = f0 + G t.  So
//   sum N^2 f^2 = R* + 2 B* (t - t*) + A (t - t*)^2,  A = sum N^2 G^2,
// and, as long as no offset changes its sign, F_cell is one cell's tricubic
// polynomial on a line: a polynomial of degree 9 in t.  A lane that takes such
// a segment makes its ten coefficients once (cell_line: ~180 FMAs, packed where
// two powers of x go side by side) and then spends ~15 instructions on a step,
// two of them shared loads for a pair of steps, where the pair queue spends ~250
// per 32 steps on finding entry, source and cell and on 63 FMAs and 16 shared
// loads per step.

// Coefficients q of F(x0 + g tau), a cell's polynomial (SpotArgs::C4 at cp) on
// a line: shifted and scaled per power of z, then Horner in y and x with
// polynomials in tau as coefficients.
__device__ __forceinline__ void cell_line(const float4 *cp, const float x0[3],
                                          const float g[3], float q[10]) {
  const f32x2 z0 = splat2(x0[2]), y0 = splat2(x0[1]), gy = splat2(g[1]),
              g1 = splat2(g[2]), g2 = splat2(g[2] * g[2]),
              g3 = splat2(g[2] * g[2] * g[2]);
  const ulonglong2 *c2 = reinterpret_cast<const ulonglong2 *>(cp);
  f32x2 Q[2][7];
#pragma unroll
  for (int P = 0; P < 2; ++P) {
    f32x2 V[7];
#pragma unroll
    for (int ib = 3; ib >= 0; --ib) {
      const ulonglong2 A = __ldg(c2 + (P * 4 + ib) * 2),
                       B = __ldg(c2 + (P * 4 + ib) * 2 + 1);
      // c3 z^3 + .. + c0 about z0: repeated synthetic division
      const f32x2 c3 = A.x;
      f32x2 d[4];
      d[2] = ffma2(c3, z0, A.y);
      d[1] = ffma2(d[2], z0, B.x);
      d[0] = ffma2(d[1], z0, B.y);
      d[2] = ffma2(c3, z0, d[2]);
      d[1] = fmul2(ffma2(d[2], z0, d[1]), g1);
      d[2] = fmul2(ffma2(c3, z0, d[2]), g2);
      d[3] = fmul2(c3, g3);
      if (ib == 3) {
#pragma unroll
        for (int i = 0; i < 4; ++i) V[i] = d[i];
      } else {
        // V (y0 + gy tau) + d; V has L coefficients
        const int L = 6 - ib;
        V[L] = fmul2(V[L - 1], gy);
#pragma unroll
        for (int i = 5; i > 0; --i)
          if (i < L)
            V[i] = ffma2(V[i], y0,
                         i < 4 ? ffma2(V[i - 1], gy, d[i])
                               : fmul2(V[i - 1], gy));
        V[0] = ffma2(V[0], y0, d[0]);
      }
    }
#pragma unroll
    for (int i = 0; i < 7; ++i) Q[P][i] = V[i];
  }
  // Q[P] = the pair of x^(2P) and x^(2P+1): Horner in x
#pragma unroll
  for (int i = 0; i < 7; ++i) q[i] = upk2(Q[1][i]).y;
#pragma unroll
  for (int ia = 2; ia >= 0; --ia) {
    const int L = 9 - ia;  // coefficients of q: 7, 8, 9
    q[L] = q[L - 1] * g[0];
#pragma unroll
    for (int i = 8; i >= 0; --i)
      if (i < L) {
        const float2 c2i = i < 7 ? upk2(Q[ia == 2][i]) : make_float2(0.f, 0.f);
        const float c = ia == 1 ? c2i.y : c2i.x;
        q[i] = fmaf(q[i], x0[0],
                    i == 0  ? c
                    : i < 7 ? fmaf(q[i - 1], g[0], c)
                            : q[i - 1] * g[0]);
      }
  }
}

// The segments of an interval entry [k1, k2) between the sources at which an
// offset changes its sign (tricubic lookup), as the words of SplitEntry::m of
// a line entry: k1 | k2 << 11, number of tasks | b3 << 8, (first task,) b1 | b2
// << 11 with k1 <= b1 <= b2 <= b3 <= k2.  S <= 1024 and at most 3 + S /
// kTaskLen tasks keep the fields.
__device__ __forceinline__ int seg_tasks(int len) {
  return (len + kTaskLen - 1) / kTaskLen;
}
template <int INTERP>
__device__ __forceinline__ void line_segments(const SplitBlock &b, int k1,
                                              int k2, const float Gh[3],
                                              const float dx[3],
                                              const float rl[3], int &mx,
                                              int &my, int &mw) {
  int c[3] = {k2, k2, k2};
  if (INTERP == 1) {
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      // the first source beyond the zero of G delta + dx + rl
      const float z = -__fdividef(dx[x] + rl[x], Gh[x]);
      int lo = k1;
      if (b.even) {
        lo = count_below(b.dh, b.S, guess_index(z, b.dmin, b.inv_step, b.S),
                         z);
      } else {
        int hi = k2;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (b.dh[mid] < z)
            lo = mid + 1;
          else
            hi = mid;
        }
      }
      c[x] = min(max(lo, k1), k2);
    }
  }
  const int lo01 = min(c[0], c[1]), hi01 = max(c[0], c[1]);
  const int b1 = min(lo01, c[2]), b3 = max(hi01, c[2]),
            b2 = max(lo01, min(hi01, c[2]));
  const int n = seg_tasks(b1 - k1) + seg_tasks(b2 - b1) + seg_tasks(b3 - b2) +
                seg_tasks(k2 - b3);
  mx = k1 | (k2 << 11);
  my = n | (b3 << 8);
  mw = b1 | (b2 << 11);
}

// The table-relative lattice point of a line entry (entry_data)
template <int INTERP>
__device__ __forceinline__ void entry_index(const float4 &d, int nt[3]) {
  if (INTERP == 1) {
    const int npk = __float_as_int(d.y);
#pragma unroll
    for (int x = 0; x < 3; ++x) nt[x] = ((npk >> (10 * x)) & 1023) - 1;
  } else {
    nt[0] = __float_as_int(d.x);
    nt[1] = __float_as_int(d.y);
    nt[2] = __float_as_int(d.z);
  }
}

// Sums the next min(32, ct - ch) tasks of a queue of line entries, one per
// lane, into the lane's Kahan sum.  Called by all lanes; returns the lane's
// number of steps under the cut and adds its steps to npairs.
template <int INTERP>
__device__ __forceinline__ unsigned sum_tasks(const SpotArgs &a,
                                              const SplitBlock &b,
                                              const SplitEntry *ring,
                                              PairQueue &pq, Kahan &acc,
                                              unsigned &npairs) {
  // a term's base-2 exponent is -kExp R, R = sum N^2 f^2
  constexpr double kExp = 2.0 / 0.63 * 1.4426950408889634;
  constexpr float kExpH = (float)kExp, kExpL = (float)(kExp - (double)kExpH);
  const int lane = threadIdx.x & 31;
  const int np = min(32, pq.ct - pq.ch);
  // the entry of each task, as in sum_pairs
  int4 mm = make_int4(0, 0, 0x7fffffff, 0);
  if (pq.e0 + lane < pq.en) mm = ring[(pq.e0 + lane) & (kEntries - 1)].m;
  const int mt = mm.y & 255;
  const bool ov = pq.e0 + lane < pq.en && mm.z < pq.ch + np &&
                  mm.z + mt > pq.ch;
  const unsigned M = __reduce_or_sync(
      0xffffffffu, ov ? 1u << max(mm.z - pq.ch, 0) : 0u);
  const int j = __popc(M & (0xffffffffu >> (31 - lane))) - 1;
  const int ex = __shfl_sync(0xffffffffu, mm.x, j),
            ey = __shfl_sync(0xffffffffu, mm.y, j),
            pos = __shfl_sync(0xffffffffu, mm.z, j),
            ew = __shfl_sync(0xffffffffu, mm.w, j);
  const unsigned done =
      __ballot_sync(0xffffffffu, ov && mm.z + mt <= pq.ch + np);
  // the task's sources [p, e)
  int p = 0, e = 0;
  if (lane < np) {
    const int bd[5] = {ex & 2047, ew & 2047, (ew >> 11) & 2047, ey >> 8,
                       ex >> 11};
    int rem = pq.ch + lane - pos;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int nt = seg_tasks(bd[q + 1] - bd[q]);
      if (rem >= 0 && rem < nt) {
        p = bd[q] + rem * kTaskLen;
        e = min(p + kTaskLen, bd[q + 1]);
      }
      rem -= nt;
    }
  }
  const int n = e - p;
  npairs += n;
  const int pf = (int)nb_idx(a.check, NB_SITE_SOURCE, p, b.S),
            pl = (int)nb_idx(a.check, NB_SITE_SOURCE, max(e - 1, 0), b.S);
  const SplitEntry &E4 = ring[(pq.e0 + j) & (kEntries - 1)];
  const float4 Ea = E4.a, Eb = E4.b, Ec = E4.c, Ed = E4.d;
  // The origin of the line is the mean of the first and the last source: its
  // offsets' signs name the segment's cell even where rounding put a source at
  // a sign change on the other side of the cut (line_segments compares with
  // an approximate quotient).  A source's own signs would then name the
  // neighbouring cell, and the other sources be extrapolated from it.
  const float4 sf = *reinterpret_cast<const float4 *>(
                   b.src + pf * SRC32_STRIDE),
               sl = *reinterpret_cast<const float4 *>(
                   b.src + pl * SRC32_STRIDE);
  const float dm = 0.5f * (sf.z + sl.z), dml = 0.5f * (sf.x + sl.x);
  const float half = 0.5f * (sl.z - sf.z);
  const float ih = half > 0.f ? __fdividef(1.f, half) : 0.f;
  // axes h and k side by side in packed operations, l in scalar ones; x - y as
  // ffma2(y, -1, x), one rounding
  const f32x2 m1 = splat2(-1.f);
  const f32x2 Gp = pk2(make_float2(Ea.x, Ea.y)),
              Glp = pk2(make_float2(Eb.x, Eb.y)), half2 = splat2(half),
              N2p = pk2(make_float2(a.N[0] * a.N[0], a.N[1] * a.N[1]));
  const float N2l = a.N[2] * a.N[2];
  const f32x2 sp = ffma2(Gp, splat2(dm), pk2(make_float2(Ea.z, Ea.w))),
              cp = ffma2(Gp, splat2(dml),
                         ffma2(Glp, splat2(dm), pk2(make_float2(Eb.z, Eb.w)))),
              f0p = fadd2(sp, cp), flp = ffma2(ffma2(sp, m1, f0p), m1, cp),
              gp = fmul2(Gp, half2), ngp = fmul2(N2p, gp);
  const float sl_ = fmaf(Ec.x, dm, Ec.y),
              cl = fmaf(Ec.x, dml, fmaf(Ec.z, dm, Ec.w)),
              f0l = __fadd_rn(sl_, cl), fll = __fsub_rn(cl, __fsub_rn(f0l, sl_)),
              gl = Ec.x * half, ngl = N2l * gl;
  const float2 A2 = upk2(fmul2(ngp, gp)), B2 = upk2(fmul2(ngp, f0p)),
               f0h = upk2(f0p), g2 = upk2(gp);
  const float A = fmaf(ngl, gl, A2.x + A2.y),
              B = fmaf(ngl, f0l, B2.x + B2.y);
  const float f0[3] = {f0h.x, f0h.y, f0l}, g[3] = {g2.x, g2.y, gl};
  // The exponents about the task's point nearest to the lattice point, tau* in
  // [-1, 1]: with u = tau - tau*
  //   -kExp R = -ei + ef - kExp (2 B* u + A u^2),
  // R and its slope B* formed at tau* from double-float offsets, ei whole.
  // The largest terms, at u near 0, then carry the rounding of a small number
  // even where all of a pixel's terms lie far from their lattice points (R 15
  // to 26, against 64 bits, rms of a task's sum: 5.3e-6 about the vertex of the
  // whole line in FP32, 2.5e-6; pair by pair 3.5e-6).
  const float ts =
      A > 0.f ? fminf(fmaxf(-__fdividef(B, A), -1.f), 1.f) : 0.f;
  const float th = ts * half;
  float R, Rl, Bs;
  {
    const f32x2 th2 = splat2(th);
    // G th, its rounding (negative), and its sum with f0
    const f32x2 p1 = fmul2(Gp, th2), e1 = ffma2(Gp, ffma2(th2, m1, 0ull), p1),
                s1 = fadd2(f0p, p1), bb = ffma2(f0p, m1, s1),
                e2 = fadd2(ffma2(ffma2(bb, m1, s1), m1, f0p),
                           ffma2(bb, m1, p1)),
                lo = fadd2(ffma2(e1, m1, e2), ffma2(Glp, th2, flp)),
                fs = fadd2(s1, lo), fl = ffma2(ffma2(s1, m1, fs), m1, lo),
                t = fmul2(N2p, fs), te = ffma2(fmul2(N2p, m1), fs, t),
                p2 = fmul2(t, fs), e3 = ffma2(fmul2(t, m1), fs, p2);
    // the rests: 2 t fl - te fs - e3 (te and e3 are negative)
    const float2 q = upk2(p2),
                 rest = upk2(ffma2(fadd2(t, t), fl,
                                   ffma2(ffma2(te, fs, e3), m1, 0ull))),
                 b2 = upk2(fmul2(ngp, fs));
    float p1l, e1l, s1l, e2l, fsl, fl_, tl, tel, p2l, e3l, s2, e4, e5;
    two_prod(Ec.x, th, p1l, e1l);
    two_sum(f0l, p1l, s1l, e2l);
    fast_two_sum(s1l, (e1l + e2l) + fmaf(Ec.z, th, fll), fsl, fl_);
    two_prod(N2l, fsl, tl, tel);
    two_prod(tl, fsl, p2l, e3l);
    two_sum(q.x, q.y, s2, e4);
    two_sum(s2, p2l, R, e5);
    Rl = (rest.x + rest.y) + (e3l + (e4 + e5)) + fmaf(tel, fsl, 2.f * tl * fl_);
    Bs = fmaf(ngl, fsl, b2.x + b2.y);
  }
  const float ei = rintf(kExpH * R);
  const float ef = fmaf(-kExpH, R, ei) - fmaf(kExpL, R, kExpH * Rl);
  const float eB = -2.f * kExpH * Bs, eA = -kExpH * A;
  const float ecut = ei - kGaussCut * 0.63f * kExpH;
  float q[10], Fn = 0.f;
  bool line = true;  // the segment's cell lies in the table
  if (INTERP == 1) {
    CellRef c;
    cell_of_entry(a, n > 0, f0, __float_as_int(Ed.x), __float_as_int(Ed.z), c);
    line = c.tri || n == 0;
    if (c.tri)
      cell_line(a.C4 + (size_t)nb_idx(a.check, NB_SITE_CELL, c.ci,
                                      cell_count(a)) * kCellChunks,
                c.x, g, q);
  } else if (n) {
    int nt[3];
    entry_index<INTERP>(Ed, nt);
    Fn = fcell_f32<0>(a, nt, f0);
  }
  unsigned hits = 0;
  // chunks of 16 steps to be summed step by step, from the table: all of them
  // where some lane's cell reaches out of the table; and those whose sum is
  // not finite, as a line multiplies the steps beyond the cut (and beyond an
  // odd end) by zero, which a table entry that is not finite, or whose square
  // is not, does not survive
  unsigned redo = 0;
  const bool lines = __all_sync(0xffffffffu, line);
  if (!lines) {
    redo = ~0u;
  } else {
    const int nmax = (int)__reduce_max_sync(0xffffffffu, (unsigned)n);
    const float *src = b.src + pf * SRC32_STRIDE + SRC32_PAIR;
    const f32x2 ih2 = splat2(ih), rl2 = splat2(-dml * ih),
                rh2 = splat2(-dm), ts2 = splat2(-ts), eA2 = splat2(eA),
                eB2 = splat2(eB), ef2 = splat2(ef);
    f32x2 q2[10];
    if (INTERP == 1) {
#pragma unroll
      for (int d = 0; d < 10; ++d) q2[d] = splat2(q[d]);
    }
    // (nearest lookup: the entry's one structure factor), and 2^-ei in two
    // factors, as ei reaches 130
    const float fac = (INTERP == 1 ? a.N6 * Ed.w : Fn * Fn * (a.N6 * Ed.w)) *
                      5.4210109e-20f;
    const float scale = __int_as_float((127 + 64 - (int)ei) << 23);
    for (int i0 = 0; i0 < nmax; i0 += 16) {
      f32x2 sum2 = splat2(0.f);  // at most 8 terms per lane half
      const int iend = min(i0 + 16, nmax);
      for (int i = i0; i < iend; i += 2) {
        if (i < n) {
          const ulonglong2 sd = *reinterpret_cast<const ulonglong2 *>(
              src + i * SRC32_STRIDE);
          const f32x2 w =
              *reinterpret_cast<const f32x2 *>(src + i * SRC32_STRIDE + 4);
          const f32x2 tau =
              ffma2(fadd2(sd.x, rh2), ih2, ffma2(sd.y, ih2, rl2));
          const f32x2 u = fadd2(tau, ts2);
          const float2 xe = upk2(ffma2(ffma2(eA2, u, eB2), u, ef2));
          float2 Ex;
          asm("ex2.approx.f32 %0, %1;" : "=f"(Ex.x) : "f"(xe.x));
          asm("ex2.approx.f32 %0, %1;" : "=f"(Ex.y) : "f"(xe.y));
          const bool h0 = xe.x >= ecut, h1 = xe.y >= ecut && i + 1 < n;
          Ex.x = h0 ? Ex.x : 0.f;
          Ex.y = h1 ? Ex.y : 0.f;
          hits += h0;
          hits += h1;
          const f32x2 wE = fmul2(w, pk2(Ex));
          if (INTERP == 1) {
            f32x2 F = q2[9];
#pragma unroll
            for (int d = 8; d >= 0; --d) F = ffma2(F, tau, q2[d]);
            sum2 = ffma2(fmul2(F, F), wE, sum2);
          } else {
            sum2 = fadd2(sum2, wE);
          }
        }
      }
      const float2 sum = upk2(sum2);
      const float v = (sum.x + sum.y) * scale * fac;
      if (fabsf(v) <= 3.4e38f)
        acc.add(v);
      else
        redo |= 1u << (i0 >> 4);
    }
  }
  if (__any_sync(0xffffffffu, redo != 0u)) {
    // the entry read again: kept in registers it would cost the loop above
    // (large shot 101.8 -> 105.9 ms)
    asm volatile("" ::: "memory");
    const float4 Ea = E4.a, Eb = E4.b, Ec = E4.c, Ed = E4.d;
    const float Gh[3] = {Ea.x, Ea.y, Ec.x}, dx[3] = {Ea.z, Ea.w, Ec.y};
    const float Gl[3] = {Eb.x, Eb.y, Ec.z}, rl[3] = {Eb.z, Eb.w, Ec.w};
    const float N2[3] = {a.N[0] * a.N[0], a.N[1] * a.N[1], a.N[2] * a.N[2]};
    int nt[3];
    entry_index<INTERP>(Ed, nt);
    for (int i = 0; i < n; ++i) {
      if (!(redo >> (i >> 4) & 1u)) continue;
      const float4 sw = *reinterpret_cast<const float4 *>(
          b.src + (pf + i) * SRC32_STRIDE);
      float fr[3], rad2 = 0.f;
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        fr[x] = fmaf(Gh[x], sw.z, dx[x]) +
                fmaf(Gh[x], sw.x, fmaf(Gl[x], sw.z, rl[x]));
        rad2 = fmaf(N2[x] * fr[x], fr[x], rad2);
      }
      if (rad2 <= kGaussCut * 0.63f) {
        const float F = fcell_f32<INTERP>(a, nt, fr);
        acc.add(F * F * (a.N6 * __expf(-2.f * rad2 * (1.f / 0.63f))) *
                (sw.y * Ed.w));
        hits += !lines;  // (a line has counted its own)
      }
    }
  }
  pq.e0 += __popc(done);
  pq.ch += np;
  __syncwarp();  // the ring slots read above may be refilled next
  return hits;
}

// The lane's item (unit u, orientation pm) of a batch, 32 items further per
// step without a division.
struct ItemWalk {
  int u, pm, du, dpm;
  __device__ __forceinline__ ItemWalk(int lane, int PM) {
    u = lane / PM;
    pm = lane - u * PM;
    du = 32 / PM;
    dpm = 32 - du * PM;
  }
  __device__ __forceinline__ void next(int PM) {
    u += du;
    pm += dpm;
    if (pm >= PM) {
      pm -= PM;
      ++u;
    }
  }
};

// One (unit, phi x mosaic) item of a lane: G and r = u0 G - n0 in
// double-float, r's high part on a 2^-21 grid.
struct SplitItem {
  bool valid;
  int aux;     // pm | unit << 16
  float scal;  // omega cap pol of the unit
  float Gh[3], Gl[3], rq[3], rl[3], n0[3];
};

// Forms the lane's item (u, pm).  EARLY: returns false, with the
// items not formed, where no lane's sweep comes near a lattice point.
template <bool EARLY>
__device__ __forceinline__ bool split_item(const SplitBlock &b,
                                           const float *unit, int u, int pm,
                                           bool valid, SplitItem &t) {
  const float u0h = b.u0h, u0l = b.u0l;
  t.valid = valid;
  t.aux = pm | (u << 16);
  const float *ud = unit + u * kUnitFloats;
  // vh[3], vl[3], scal as four float2 loads (unit rows are 8-byte aligned)
  const float2 *u2 = reinterpret_cast<const float2 *>(ud);
  const float2 p0 = u2[0], p1 = u2[1], p2 = u2[2], p3 = u2[3];
  const float vh[3] = {p0.x, p0.y, p1.x}, vl[3] = {p1.y, p2.x, p2.y};
  t.scal = p3.x;
  if (EARLY && b.iv_ok) {
    // h in plain FP32 at the sweep's middle, the distance to the nearest
    // integer against half the sweep and the margin
    bool near = t.valid;
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const float2 *A3 = b.ax2 + pm * 9 + 3 * x;
      const float g = fmaf(A3[0].x, vh[0], fmaf(A3[1].x, vh[1],
                                                A3[2].x * vh[2]));
      const float h = g * b.umid;
      near = near && !(fabsf(h - rintf(h)) > fmaf(fabsf(g), b.dhalf,
                                                  b.nmarg[x]));
    }
    if (!__any_sync(0xffffffffu, near)) return false;
  }
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    ff_dot3_pairs(b.ax2 + pm * 9 + 3 * x, vh, vl, t.Gh[x], t.Gl[x]);
    float qh, qe;
    two_prod(t.Gh[x], u0h, qh, qe);
    const float ql = fmaf(t.Gh[x], u0l, fmaf(t.Gl[x], u0h, qe));
    t.n0[x] = rintf(qh);
    float rh, rl0;
    two_sum(__fsub_rn(qh, t.n0[x]), ql, rh, rl0);
    // r_hi on a 2^-21 grid: r_hi - n is then exact for |n| < 7
    t.rq[x] = __fmul_rn(rintf(__fmul_rn(rh, 2097152.f)), 1.f / 2097152.f);
    t.rl[x] = rl0 + __fsub_rn(rh, t.rq[x]);
  }
  return true;
}

// The lattice points an item's sweep can come near: per axis the integers
// ml + 0 .. nm - 1 within sqrt(cwide)/N_x of [h(dmin), h(dmax)], in odometer
// order (dg); A = sum N^2 G^2 of the exponent along the sweep.
struct LatticeRange {
  int ncomb, ml[3], nm[3], dg[3];
  float A;
};
__device__ __forceinline__ void lattice_range(const SplitBlock &b,
                                              const float N2[3],
                                              const SplitItem &t,
                                              LatticeRange &L) {
  L.ncomb = 0;
#pragma unroll
  for (int x = 0; x < 3; ++x) L.ml[x] = L.nm[x] = L.dg[x] = 0;
  if (b.iv_ok && t.valid) {
    L.ncomb = 1;
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const float lo = fmaf(t.Gh[x], b.dmin, t.rq[x]),
                  hi = fmaf(t.Gh[x], b.dmax, t.rq[x]);
      L.ml[x] = (int)ceilf(fminf(lo, hi) - b.cmarg[x]);
      L.nm[x] = (int)floorf(fmaxf(lo, hi) + b.cmarg[x]) - L.ml[x] + 1;
      if (L.nm[x] < 0) L.nm[x] = 0;
      L.ncomb *= L.nm[x];
    }
  }
  L.A = N2[0] * t.Gh[0] * t.Gh[0];
  L.A = fmaf(N2[1] * t.Gh[1], t.Gh[1], L.A);
  L.A = fmaf(N2[2] * t.Gh[2], t.Gh[2], L.A);
}

// The next lattice point of the lane's range (the c-th of all lanes): for
// lattice point m the exponent sum along the sweep is A d^2 + 2 B d + C, below
// cwide on one interval [k1, k2) of the sorted delta table.  dx = r_q - (m -
// n0), nt = the table-relative m.
__device__ __forceinline__ void lattice_interval(
    const SpotArgs &a, const SplitBlock &b, const float N2[3],
    const SplitItem &t, LatticeRange &L, int c, int &k1, int &k2, float dx[3],
    int nt[3]) {
  const int S = b.S;
  const float *s_dh = b.dh;
  k1 = k2 = 0;
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    dx[x] = 0.f;
    nt[x] = 0;
  }
  if (c >= L.ncomb) return;
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    // lattice point n0 + mx; its table index nt
    const int mx = L.ml[x] + L.dg[x];
    dx[x] = t.rq[x] - (float)mx;  // exact: r_q on a 2^-21 grid
    nt[x] = (int)t.n0[x] + mx - a.hmin[x];
  }
  if (++L.dg[0] == L.nm[0]) {
    L.dg[0] = 0;
    if (++L.dg[1] == L.nm[1]) {
      L.dg[1] = 0;
      ++L.dg[2];
    }
  }
  float B = N2[0] * t.Gh[0] * dx[0];
  B = fmaf(N2[1] * t.Gh[1], dx[1], B);
  B = fmaf(N2[2] * t.Gh[2], dx[2], B);
  float C0 = N2[0] * dx[0] * dx[0];
  C0 = fmaf(N2[1] * dx[1], dx[1], C0);
  C0 = fmaf(N2[2] * dx[2], dx[2], C0);
  if (L.A > 0.f) {
    const float disc = fmaf(B, B, -L.A * (C0 - b.cwide));
    if (disc >= 0.f) {
      // the bounds carry a relative margin far above the error of the
      // reciprocal
      const float sq = sqrtf(disc), ia = __frcp_rn(L.A);
      float lo = (-B - sq) * ia, hi = (-B + sq) * ia;
      const float mg = 1e-4f * (fabsf(lo) + fabsf(hi)) + b.dmarg;
      lo -= mg;
      hi += mg;
      // k1 = #{delta < lo}, k2 = #{delta <= hi} (sorted table)
      if (b.even) {
        k1 = count_below(s_dh, S, guess_index(lo, b.dmin, b.inv_step, S), lo);
        k2 = count_at_most(s_dh, S, guess_index(hi, b.dmin, b.inv_step, S),
                           hi);
      } else {
        for (int st = b.sstep; st > 0; st >>= 1) {
          if (k1 + st <= S && s_dh[k1 + st - 1] < lo) k1 += st;
          if (k2 + st <= S && s_dh[k2 + st - 1] <= hi) k2 += st;
        }
      }
    }
  } else if (C0 <= b.cwide) {
    k2 = S;  // the sweep does not move: all or nothing
  }
}

// SplitEntry::d of an interval entry at lattice point nt
template <int INTERP>
__device__ __forceinline__ float4 entry_data(const SpotArgs &a, bool any,
                                             const int nt[3], float scal) {
  if (INTERP == 1 && a.C4) {
    // the lattice point's cell data once per entry; the index packed
    // (clamped to [-1, hn]: any index outside the table looks up
    // default_F, and cell tables exist only for hn < 1024)
    int ci0 = 0, pk = 0, npk = 0;
    if (any) {
      entry_cell_data(a, nt, ci0, pk);
#pragma unroll
      for (int x = 0; x < 3; ++x)
        npk |= (min(max(nt[x], -1), a.hn[x]) + 1) << (10 * x);
    }
    return make_float4(__int_as_float(ci0), __int_as_float(npk),
                       __int_as_float(pk), scal);
  }
  return make_float4(__int_as_float(nt[0]), __int_as_float(nt[1]),
                     __int_as_float(nt[2]), scal);
}

// Pruned scan: h_x = G_x delta + r_x is linear in delta, so a block of
// sources whose delta range keeps some axis farther than sqrt(cut)/N_x from
// every integer holds no surviving term.  Pushes block bb of every lane's
// item that may hold one.
template <int W = 32>
__device__ __forceinline__ void push_block(const SplitBlock &b,
                                           SplitEntry *ring, PairQueue &pq,
                                           const SplitItem &t, int bb) {
  bool pass = false;
  if (t.valid) {
    const float dmn = b.blk[2 * bb], dmx = b.blk[2 * bb + 1];
    pass = true;
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const float lo0 = fmaf(t.Gh[x], dmn, t.rq[x]),
                  hi0 = fmaf(t.Gh[x], dmx, t.rq[x]);
      const float lo = fminf(lo0, hi0) - b.cmarg[x],
                  hi = fmaxf(lo0, hi0) + b.cmarg[x];
      pass = pass && floorf(hi) >= ceilf(lo);
    }
  }
  const int st0 = bb * kSrcBlock;
  const int len = pass ? min(kSrcBlock, b.S - st0) : 0;
  push_entries<W>(ring, pq, len, st0, len, t.aux, t.Gh, t.rq, t.Gl, t.rl,
                  make_float4(t.n0[0], t.n0[1], t.n0[2], t.scal));
}

// How split_sum goes through the interval entries: pair by pair; the same
// with split_item's early test; line by line, with that test; pair by pair,
// two pixels at a time with 16 lanes each (split_form)
enum { kPairs = 0, kPairsEarly = 1, kLines = 2, kHalves = 3 };
constexpr int kHalfItems = 16, kHalfSteps = 128;
constexpr float kHalfPairs = 30.f;
template <int FORM>
constexpr int kLanes = FORM == kHalves ? 16 : 32;  // lanes per pixel

// The share of h space within the cut of a lattice point; they are rare where
// it is below kRareShare
constexpr float kRareShare = 0.2f;
constexpr float kEarlyLine = 0.2f;  // least share of the sources on a line
__host__ __device__ inline float lattice_share(const SpotArgs &a) {
  const float m = sqrtf(kGaussCut * 0.63f) * 2.f;
  return m / a.N[0] * (m / a.N[1]) * (m / a.N[2]);
}

// The sources on a line through a lattice point, for S of them over a relative
// range span of 1/lambda: the width of the cut over the movement of h, at the
// outermost h of the table
inline float line_sources(const SpotArgs &a, int S, float span) {
  float nh = 0.f;
  for (int x = 0; x < 3; ++x) {
    const int lo = a.hmin[x], hi = a.hmin[x] + a.hn[x] - 1;
    const float h = (float)(-lo > hi ? -lo : hi);
    nh = fmaxf(nh, a.N[x] * h);
  }
  const float move = nh * span;
  return move > 0.f ? fminf((float)S, 2.f * sqrtf(kGaussCut * 0.63f) / move * S)
                    : (float)S;
}

// The form for a shot of PM orientations and S sources. Lines need enough tasks
// per pixel to fill a pass, and enough steps per line to pay for its
// coefficients (pairs with the early test -> lines, 700^2 pixels: 1 unit, S =
// 100, M = 12 0.605 -> 0.541 ms; S = 60, M = 30 0.750 -> 0.621; S = 30, M = 50
// 0.820 -> 0.816; S = 20, M = 50 0.696 -> 0.777; S = 60, M = 12, 1000^2 0.787
// -> 0.873; large shot, 1024^2: 18.2 -> 10.2). Where the ellipsoids of lattice
// points overlap (N < 15.4) there are no interval entries, and the blocks of
// sources are better summed by the pair kernels and their 20 warps per SM
// (300^2 pixels, N = 8, 10 items of 180 sources: 2.07 -> 1.68 ms). A line of
// few sources does not pay for its coefficients either: 400^2 pixels, pairs ->
// lines, 40 sources, 30 domains, 9 units, spectrum FWHM 2 %, N = 60 (2.3
// sources on a line, line_sources) 0.80 -> 1.07 ms, N = 18 (7.6) 2.85 -> 3.63;
// 100, 25, 4, N = 25 (13.8) 1.25 -> 1.35, but 24^2 pixels 77 -> 53 us; 180, 25,
// 1, N = 40 (15.5) 325 -> 314 us, N = 25 (24.8) 594 -> 504.
// The early test pays where lattice points are rare: N = 25 (0.07 of h space
// lies within the cut) 1.22 -> 1.05 ms on 1500^2 pixels with S = 11, M = 9, but
// at N = 15 (0.34) it finds one in most batches, 1.86 -> 2.11 ms on the
// 64-panel shot, and so it does where a sweep passes several: 400^2 pixels, 100
// sources, 25 domains, 4 units, FWHM 2 % (0.11 of the sources on a line) 1.17
// -> 1.25 ms; 0.5 %, N = 60 (0.23) 784 -> 747 us.
// Halves pay where a pixel's items leave half the lanes idle (64-panel shot, 10
// items of 8 sources, tricubic 1.83 -> 1.29 ms, nearest 1.47 -> 0.96; N = 25, 9
// items of 11 0.337 -> 0.286). A pixel alone then takes its pairs 16 at a time
// with the other half idle, so a list of few pixels waits for the longer chain:
// 1000 pixels, 100 steps at N = 15 (34 pairs expected) 36.4 -> 39.0 us, 480
// steps 45.7 -> 54.1, but 37.3 -> 37.7 with 99 steps at N = 25 (7 pairs); hence
// the limits on steps and on expected pairs.
__host__ __device__ inline bool half_form(const SpotArgs &a, int PM, int S) {
  const long long items = (long long)a.os * a.os * a.T * PM;
  return !a.has_div && items <= kHalfItems && items * S <= kHalfSteps &&
         (float)(items * S) * lattice_share(a) <= kHalfPairs;
}
inline int split_form(const SpotArgs &a, int PM, int S, float span) {
  if (a.has_div) return kPairs;
  if ((a.interp == 0 || a.C4) && S >= kLineSources &&
      (long long)a.os * a.os * a.T * PM * S >= kLineSteps &&
      lattice_disjoint(a) && line_sources(a, S, span) >= kLineMean)
    return kLines;
  if (half_form(a, PM, S)) return kHalves;
  return lattice_share(a) < kRareShare &&
                 line_sources(a, S, span) >= kEarlyLine * S
             ? kPairsEarly
             : kPairs;
}

// The sum, without the prefactor, of the pixel whose U sub-pixel units are
// already in `unit` (split_unit), computed by the calling warp (all 32
// lanes); every lane returns the same value.  Adds the terms it evaluated
// to `cnt` and, with COUNT, the rest of the work it performed.
template <int INTERP, int HASDIV, int FORM, int COUNT = 0>
__device__ __forceinline__ double split_sum(const SpotArgs &a,
                                            const SplitBlock &b,
                                            const float *unit,
                                            SplitCounts &cnt, bool ok = true) {
  constexpr int W = kLanes<FORM>;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  SplitEntry *ring =
      b.ent_base + warp * kEntries + (W == 32 ? 0 : lane / W * kRing<W>);
  float4 *cache = b.cell_cache + warp * kCellChunks * kCellSlots;
  int *tags = b.cell_tags + warp * kCellSlots;
  const int items = a.os * a.os * a.T * b.PM;
  const float N2[3] = {a.N[0] * a.N[0], a.N[1] * a.N[1], a.N[2] * a.N[2]};

  Kahan acc;
  PairQueue pq;
  unsigned nterms = 0, nivals = 0, nblocks = 0;
  unsigned nlines = 0, npairs = 0;  // the lane's own terms and pairs
  SplitItem t;
  LatticeRange L;
  float dx[3];
  int nt[3], k1, k2;
  if (FORM == kLines) {
    // One loop with a single place where the queue is summed and one where
    // each kind of entry is pushed (with the summing inlined at every push
    // the kernel waited for instructions a fifth of its time, large shot
    // 1024^2 11.6 -> 10.2 ms): the queue, then the next lattice point or
    // source block of the current batch of items, then the next batch.
    enum { kItems, kLattice, kScan } state = kItems;
    bool line_q = false;  // the queue holds tasks, not pairs
    bool flush = false;   // sum the queue to its end first
    int base = 0, c = 0, maxc = 0;
    ItemWalk walk(lane, b.PM);
    while (true) {
      if (pq.ct - pq.ch >= 32 || (flush && pq.ct > pq.ch)) {
        if (line_q)
          nlines += sum_tasks<INTERP>(a, b, ring, pq, acc, npairs);
        else
          nterms += sum_pairs<INTERP, HASDIV>(a, b, ring, pq, unit, cache,
                                              tags, acc, npairs);
        continue;
      }
      flush = false;
      if (state != kItems && line_q != (state == kLattice)) {
        // the other kind of entry: the queue first
        if (pq.ct > pq.ch) {
          flush = true;
          continue;
        }
        line_q = state == kLattice;
      }
      if (state == kLattice) {
        if (c == maxc) {
          state = kItems;
          continue;
        }
        lattice_interval(a, b, N2, t, L, c++, k1, k2, dx, nt);
        // no lane has an entry for this lattice point: nothing to push
        if (!__any_sync(0xffffffffu, k2 > k1)) continue;
        int mx = 0, my = 0, mw = 0;
        if (k2 > k1)
          line_segments<INTERP>(b, k1, k2, t.Gh, dx, t.rl, mx, my, mw);
        push_entries(ring, pq, my & 255, mx, my, mw, t.Gh, dx, t.Gl, t.rl,
                     entry_data<INTERP>(a, k2 > k1, nt, t.scal));
        continue;
      }
      if (state == kScan) {
        if (c == b.nblk) {
          state = kItems;
          continue;
        }
        push_block(b, ring, pq, t, c++);
        continue;
      }
      if (base >= items) {
        if (pq.ct == pq.ch) break;
        flush = true;
        continue;
      }
      const bool valid = base + lane < items;
      const int u = valid ? walk.u : 0, pm = valid ? walk.pm : 0;
      base += 32;
      walk.next(b.PM);
      if (!split_item<true>(b, unit, u, pm, valid, t)) continue;
      lattice_range(b, N2, t, L);
      c = 0;
      if (b.iv_ok && __all_sync(0xffffffffu, L.ncomb <= 8)) {
        state = kLattice;
        maxc = (int)__reduce_max_sync(0xffffffffu, (unsigned)L.ncomb);
        if (COUNT) nivals += __reduce_add_sync(0xffffffffu, (unsigned)L.ncomb);
      } else {
        state = kScan;
        if (COUNT)
          nblocks += __popc(__ballot_sync(0xffffffffu, t.valid)) * b.nblk;
      }
    }
  } else if (FORM == kHalves) {
    // Each half of the warp goes through its own pixel: a pixel's items fit
    // its lanes, its pairs are taken 16 at a time when 16 are there (or at
    // the end), whatever the other half holds, so a pixel's sum does not
    // depend on its neighbour.
    const Lanes<W> at;
    const bool valid = ok && at.l < items;
    const int u = valid ? at.l / b.PM : 0;
    auto drain = [&]() {
      while (true) {
        const bool go = pq.ct - pq.ch >= W;
        if (!__any_sync(0xffffffffu, go)) break;
        nterms += sum_pairs<INTERP, 0, W>(a, b, ring, pq, unit, cache, tags,
                                          acc, npairs, go);
      }
    };
    split_item<false>(b, unit, u, valid ? at.l - u * b.PM : 0, valid, t);
    lattice_range(b, N2, t, L);
    const bool lat =
        b.iv_ok && at.own(__ballot_sync(0xffffffffu, L.ncomb > 8)) == 0u;
    const int mine = lat ? L.ncomb : 0;
    const int maxc = (int)__reduce_max_sync(0xffffffffu, (unsigned)mine);
    if (COUNT) nivals += __reduce_add_sync(0xffffffffu, (unsigned)mine);
    for (int c = 0; c < maxc; ++c) {
      lattice_interval(a, b, N2, t, L, c, k1, k2, dx, nt);
      if (c >= mine) k2 = k1;
      if (!__any_sync(0xffffffffu, k2 > k1)) continue;
      push_entries<W>(ring, pq, k2 > k1 ? k2 - k1 : 0, k1, k2 - k1,
                      t.aux | kIntervalEntry, t.Gh, dx, t.Gl, t.rl,
                      entry_data<INTERP>(a, k2 > k1, nt, t.scal));
      drain();
    }
    t.valid = t.valid && !lat;
    const unsigned scan = __ballot_sync(0xffffffffu, t.valid);
    if (scan) {
      if (COUNT) nblocks += __popc(scan) * b.nblk;
      for (int bb = 0; bb < b.nblk; ++bb) {
        push_block<W>(b, ring, pq, t, bb);
        drain();
      }
    }
    if (__any_sync(0xffffffffu, pq.ct > pq.ch))
      nterms += sum_pairs<INTERP, 0, W>(a, b, ring, pq, unit, cache, tags, acc,
                                        npairs);
  } else {
    auto drain = [&]() {
      while (pq.ct - pq.ch >= 32)
        nterms += sum_pairs<INTERP, HASDIV>(a, b, ring, pq, unit, cache, tags,
                                            acc, npairs);
    };
    // items: lanes take (unit, phi x mosaic) items 32 at a time, form G and r,
    // and push their source intervals; the pair queue is summed 32 pairs at a
    // time as it fills
    ItemWalk walk(lane, b.PM);
    for (int base = 0; base < items; base += 32, walk.next(b.PM)) {
      const bool valid = base + lane < items;
      if (!split_item<FORM == kPairsEarly && !HASDIV>(
              b, unit, valid ? walk.u : 0, valid ? walk.pm : 0, valid, t))
        continue;
      if (HASDIV) {
        // sources of different directions: every source of every item
        push_entries(ring, pq, t.valid ? b.S : 0, 0, b.S, t.aux, t.Gh, t.rq,
                     t.Gl, t.rl,
                     make_float4(t.n0[0], t.n0[1], t.n0[2], t.scal));
        drain();
        continue;
      }
      lattice_range(b, N2, t, L);
      if (b.iv_ok && __all_sync(0xffffffffu, L.ncomb <= 8)) {
        const int maxc =
            (int)__reduce_max_sync(0xffffffffu, (unsigned)L.ncomb);
        if (COUNT) nivals += __reduce_add_sync(0xffffffffu, (unsigned)L.ncomb);
        for (int c = 0; c < maxc; ++c) {
          lattice_interval(a, b, N2, t, L, c, k1, k2, dx, nt);
          // no lane has an entry for this lattice point: nothing to push
          if (!__any_sync(0xffffffffu, k2 > k1)) continue;
          push_entries(ring, pq, k2 > k1 ? k2 - k1 : 0, k1, k2 - k1,
                       t.aux | kIntervalEntry, t.Gh, dx, t.Gl, t.rl,
                       entry_data<INTERP>(a, k2 > k1, nt, t.scal));
          drain();
        }
      } else {
        if (COUNT)
          nblocks += __popc(__ballot_sync(0xffffffffu, t.valid)) * b.nblk;
        for (int bb = 0; bb < b.nblk; ++bb) {
          push_block(b, ring, pq, t, bb);
          drain();
        }
      }
    }
    if (pq.ct > pq.ch)
      nterms += sum_pairs<INTERP, HASDIV>(a, b, ring, pq, unit, cache, tags,
                                          acc, npairs);
  }
  cnt.terms += nterms + __reduce_add_sync(0xffffffffu, nlines);
  if (COUNT) {
    cnt.pairs += __reduce_add_sync(0xffffffffu, npairs);
    cnt.ivals += nivals;
    cnt.blocks += nblocks;
  }

  // ---- warp reduction in float-float: each lane's compensated sum is
  // the pair (s, -c); pairs are added with error-free transformations (so
  // the butterfly gives every lane the same pair) and turned into FP64
  // once.  FP64 instructions run at 1/64 of the FP32 rate on this part and
  // issue per warp, so a per-pixel FP64 tree would cost as much as a
  // pixel's sum when the pixel has few steps.
  float hi, lo;
  fast_two_sum(acc.s, -acc.c, hi, lo);
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) {
    const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
    const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
    float sh, se;
    two_sum(hi, h2, sh, se);
    se += lo + l2;
    fast_two_sum(sh, se, hi, lo);
  }
  __syncwarp();
  return (double)hi + (double)lo;
}

}  // namespace nbgb
