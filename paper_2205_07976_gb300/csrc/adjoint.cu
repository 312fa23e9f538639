// adjoint.cu -- gradients of a scalar image loss through the Bragg-spot sum
// (the refinement loop of x-ray tracing, Sec. II: crystal parameters are
// refined until the simulated image matches the measured one), and the
// Poisson image loss itself.
//
// The crystal is parametrised as lab axes = rows of Rx(tx) Ry(ty) Rz(tz) U
// diag(a, b, c) (orthorhombic cell, fixed orientation U, three small
// rotations), Gaussian F_latt with Na, Nb, Nc, an overall scale and the
// structure-factor table (nearest or tricubic lookup).  Given w_p = dL/dI_p for every
// pixel, the kernel recomputes every step of the forward sum (nothing is
// stored between passes) and accumulates
//   dL/dθ_r  = Σ_p w_p K scale Σ_steps term · Σ_x dlog(F_latt^2)/df_x · dh_x/dθ_r
//   dL/dN_x  = Σ_p w_p K scale Σ_steps term · (2/N_x − 4 N_x f_x^2/0.63)
//   dL/dscale = Σ_p w_p I_p / scale
//   dL/dF[h0] += w_p K scale · 2 F_cell F_latt^2 w_k cap pol ω    (scatter-add)
// with dh_x/dθ_r = (∂A_x/∂θ_r) · (d − i)/λ and dlog(F_latt^2)/df_x =
// −4 N_x^2 f_x / 0.63; with tricubic lookup F_cell also depends on h (the
// derivative of the Lagrange weights) and dL/dF is spread over the 64
// stencil entries with the interpolation weights.  The per-step arithmetic
// is the FP32-mixed form of the forward kernel (double-float fractional
// offsets).
//
// The six derivatives of the axes share one pass.  A step's axes are the lab
// axes rotated by M = U_m R_phi, and so are their derivatives: dA_x/dθ_r =
// M (da_x/dθ_r), a_x the lab axis.  With e_x = term · dlog(F_latt^2)/df_x u
// (and F_cell's part) and v = d − i,
//   Σ_x e_x (dA_x/dθ_r) · v = Σ_x,c (da_x/dθ_r)_c e_x v'_c,  v' = M^T v,
// so the kernels sum the nine products Q_xc = e_x v'_c over all steps, and the
// host contracts them once with the six derivatives of the lab axes.  (Forming
// the 18 products dA_x · v of every orientation, and 18 FMAs per term, took
// 54 shared loads and 54 FMAs per orientation.)  The thirteen sums are FP32
// over a limited number of steps (a unit's in the thread kernel, 16 passes of a
// warp in the ring kernel) and FP64 from there on; per block or pixel row they
// go into a partial row, and the rows are added in a fixed order.
#include "mixed_common.cuh"

namespace nbgb {

struct AdjointArgs {
  SpotArgs a;
  const float *rot;      // [PM][9] M = U_m R_phi, row-major
  const double *dLdI;    // [npix]
  double *gradF;         // [nh*nk*nl], accumulated into
  double *partials;      // [blocks][kGradN]
  double kc;             // r_e^2 fluence / (os^2 M Phi)
  double scale;
  // term-ring kernel: rows of 32 pixels handed to warps by a counter;
  // partials holds one row of the sums per pixel row
  unsigned long long *rows_next;
  long long n_rows;
};

// the sums, each step weighted with dL/dI kc: Q_xc (3 x + c), the three dL/dN
// (both without the scale) and dL/dscale
constexpr int kGradN = 13;
static_assert(kGradN == kAdjointSums, "the host contracts these sums");

// v' = M^T v
__device__ __forceinline__ void unrotate(const float *M, const float v[3],
                                         float r[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c)
    r[c] = fmaf(M[c], v[0], fmaf(M[3 + c], v[1], M[6 + c] * v[2]));
}

// Value F and gradient (dF/dx, dF/dy, dF/dz) at x in [0, 1)^3 of a cell's
// tricubic polynomial, its 64 monomial coefficients C[a][b][c] of
// x^a y^b z^c at cp in the layout of SpotArgs::C4: nested Horner in z, y,
// x carrying the derivatives along, the chains of x^(2P) and x^(2P+1)
// side by side in packed two-lane FMAs.
__device__ __forceinline__ void cell_value_grad(const float4 *cp,
                                                const float x[3], float &F,
                                                float dF[3]) {
  const float2 z2 = make_float2(x[2], x[2]), y2 = make_float2(x[1], x[1]);
  float2 q[2], qy[2], qz[2];
#pragma unroll
  for (int P = 0; P < 2; ++P) {
    float2 pb[4], db[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const float4 A = __ldg(cp + (P * 4 + b) * 2);
      const float4 B = __ldg(cp + (P * 4 + b) * 2 + 1);
      // p = ((c3 z + c2) z + c1) z + c0 and its z-derivative
      float2 p = make_float2(A.x, A.y);
      float2 d = p;
      p = ffma2(p, z2, make_float2(A.z, A.w));
      d = ffma2(d, z2, p);
      p = ffma2(p, z2, make_float2(B.x, B.y));
      d = ffma2(d, z2, p);
      p = ffma2(p, z2, make_float2(B.z, B.w));
      pb[b] = p;
      db[b] = d;
    }
    // Horner in y over b = 3 .. 0: value, y-derivative, z-derivative
    float2 v = pb[3], vy = pb[3], vz = db[3];
    v = ffma2(v, y2, pb[2]);
    vz = ffma2(vz, y2, db[2]);
    vy = ffma2(vy, y2, v);
    v = ffma2(v, y2, pb[1]);
    vz = ffma2(vz, y2, db[1]);
    vy = ffma2(vy, y2, v);
    v = ffma2(v, y2, pb[0]);
    vz = ffma2(vz, y2, db[0]);
    q[P] = v;
    qy[P] = vy;
    qz[P] = vz;
  }
  // q[P] = (Q_{2P}, Q_{2P+1}); Horner in x over a = 3 .. 0
  const float xx = x[0];
  float v = q[1].y, vx = q[1].y, vy = qy[1].y, vz = qz[1].y;
  v = fmaf(v, xx, q[1].x);
  vy = fmaf(vy, xx, qy[1].x);
  vz = fmaf(vz, xx, qz[1].x);
  vx = fmaf(vx, xx, v);
  v = fmaf(v, xx, q[0].y);
  vy = fmaf(vy, xx, qy[0].y);
  vz = fmaf(vz, xx, qz[0].y);
  vx = fmaf(vx, xx, v);
  v = fmaf(v, xx, q[0].x);
  vy = fmaf(vy, xx, qy[0].x);
  vz = fmaf(vz, xx, qz[0].x);
  F = v;
  dF[0] = vx;
  dF[1] = vy;
  dF[2] = vz;
}

// derivatives of the 4-point Lagrange weights (nodes -1, 0, 1, 2) at x
__device__ __forceinline__ void lagrange4_deriv(float x, float w[4]) {
  float x2 = x * x;
  w[0] = -(3.f * x2 - 6.f * x + 2.f) * (1.f / 6.f);
  w[1] = (3.f * x2 - 4.f * x - 1.f) * 0.5f;
  w[2] = -(3.f * x2 - 2.f * x - 2.f) * 0.5f;
  w[3] = (3.f * x2 - 1.f) * (1.f / 6.f);
}

// The sums v[0 .. kGradN) over the warp in FP64, sum r in lanes 2 r and 2 r + 1:
// of 16 a lane hands half to a lane 16 away, of the other 8 half to one 8 away,
// ...: 16 additions in place of 65
__device__ __forceinline__ double warp_sums(double v[16]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int n = 8; n > 0; n >>= 1) {
    const bool up = (lane & 2 * n) != 0;
#pragma unroll
    for (int r = 0; r < n; ++r) {
      const double keep = up ? v[r + n] : v[r], give = up ? v[r] : v[r + n];
      v[r] = keep + __shfl_xor_sync(0xffffffffu, give, 2 * n);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// One thread per pixel (nearest lookup, and tricubic lookup in tables too
// long for the ring kernel below).  Bound by instruction issue: per (pixel,
// orientation) about 150 for the double-float G and r, 12 per source for the
// cut test, and the evaluation of the surviving steps with 18 % of them
// surviving.  64-panel shot (S = 8, 10 domains, nearest): 1316 -> 880 us with
// the nine products Q in place of 18 per orientation and each lane taking its
// own surviving steps; -> 795 with the cut tested two sources at a time
// (cut_sums).  A unit's sums are FP32 (dL/dscale compensated), over the units
// double-float in a column of shared memory, with dL/dI and over the pixels
// FP64, which costs 35 us: all of them FP32 over a pixel's 40 000 steps put
// dL/dN and dL/dscale off by 3e-6 to 1.3e-5 in place of 1e-8 to 8e-7.  (Folding
// every unit into FP64: 4 x 128^2 pixels of 9 units of one step 100 us, not 63.)
template <int HASF, int INTERP>
__global__ void __launch_bounds__(kTileThreads, INTERP ? 3 : 4)
    spots_adjoint_kernel(AdjointArgs g) {
  const SpotArgs &a = g.a;
  extern __shared__ __align__(16) float smf[];
  float *s_axh = smf;
  float *s_axl = smf + a.PM * 9;
  float *s_src = smf + 2 * a.PM * 9;
  float *s_rot = s_src + a.S * SRC32_STRIDE;
  for (int i = threadIdx.x; i < a.PM * 9; i += blockDim.x) {
    s_axh[i] = a.axh[i];
    s_axl[i] = a.axl[i];
    s_rot[i] = g.rot[i];
  }
  for (int i = threadIdx.x; i < a.S * SRC32_STRIDE; i += blockDim.x)
    s_src[i] = a.src32[i];
  __syncthreads();
  // tricubic dL/dF: the terms of a thread near one lattice point n use
  // stencils starting at n-2 or n-1 along each axis, all inside the 5x5x5
  // nodes n-2 .. n+2.  The thread sums their weighted contributions there,
  // in its own column of shared memory (FP32), and adds the touched nodes
  // to the FP64 gradient when n changes and at the end: far fewer global
  // atomics than 64 per term.
  // [125][kTileThreads] after the tables (dynamic shared memory)
  float (*s_facc)[kTileThreads] =
      reinterpret_cast<float (*)[kTileThreads]>(s_rot + a.PM * 9);
  long long near_idx = -1;  // nearest lookup: the entry being summed
  // its run of terms, summed in FP32 (an FP64 instruction per term would
  // cost 64 FP32 ones on this part) and added to the FP64 gradient once
  float near_sum = 0.f;
  int held[3] = {0, 0, 0};  // the lattice point held (table-relative)
  bool holding = false;
  auto flush_node = [&]() {
    if (!holding) return;
    for (int e = 0; e < 125; ++e) {
      const float v = s_facc[e][threadIdx.x];
      if (v == 0.f) continue;  // untouched (may lie outside the table)
      s_facc[e][threadIdx.x] = 0.f;
      const int i = e / 25, j = (e / 5) % 5, k = e % 5;
      atomicAdd(g.gradF + nb_idx(a.check, NB_SITE_GRADF,
                                 ((long long)(held[0] - 2 + i) * a.hn[1] +
                                  (held[1] - 2 + j)) * a.hn[2] +
                                     (held[2] - 2 + k),
                                 table_size(a)),
                (double)v);
    }
    holding = false;
  };
  if (INTERP && HASF)
    for (int e = 0; e < 125; ++e) s_facc[e][threadIdx.x] = 0.f;

  long long item = a.pixlist ? (long long)blockIdx.x * blockDim.x + threadIdx.x
                             : (long long)blockIdx.x;
  long long gp = 0;
  int q = 0, s = 0, f = 0;
  const int lane = threadIdx.x & 31;
  double mine = 0.0;  // lanes 2 r and 2 r + 1: the warp's sum r
  // nearest lookup with several units: a pixel's sums over its units, as
  // double-floats in shared memory (behind the tables)
  constexpr bool kColumns = INTERP == 0;
  const int n_units = a.os * a.os * a.T;
  float2 (*s_tot)[kTileThreads] = reinterpret_cast<float2 (*)[kTileThreads]>(
      s_rot + ((a.PM * 27 & 1) ? a.PM * 9 + 1 : a.PM * 9));
  {
    const bool ok = map_pixel(a, item, threadIdx.x, gp, q, s, f);
    const DevPanel &P = a.panels[ok ? q : 0];
    const int os = a.os;
    const float kahn = a.kahn;
    const float cutg = kGaussCut * 0.63f;
    const double wk = ok ? g.dLdI[gp] * g.kc : 0.0;
    const float N2[3] = {a.N[0] * a.N[0], a.N[1] * a.N[1], a.N[2] * a.N[2]};
    const float cn0[3] = {2.f / a.N[0], 2.f / a.N[1], 2.f / a.N[2]},
                cn1[3] = {-4.f * a.N[0] * (1.f / 0.63f),
                          -4.f * a.N[1] * (1.f / 0.63f),
                          -4.f * a.N[2] * (1.f / 0.63f)};
    for (int i = 0; i < os; ++i)
      for (int j = 0; j < os; ++j)
        for (int t = 0; t < a.T; ++t) {
          float scal = 0.f;
          Kahan acc12;
          float acc[12];
#pragma unroll
          for (int r = 0; r < 12; ++r) acc[r] = 0.f;
          if (ok) {
          float vh[3], vl[3], df[3], omega;
          unit_geometry_ff(a, P, s, f, i, j, t, vh, vl, df, omega);
          float cap = 1.f;
          if (a.dtff[0] > 0.f) {
            float rho = df[0] * P.ffn[0][0] + df[1] * P.ffn[1][0] +
                        df[2] * P.ffn[2][0];
            float L = a.attenf * rho, dtf = a.dtff[0];
            cap = expf(-t * dtf / L) - expf(-(t + 1) * dtf / L);
          }
          float c2 = df[0] * a.i0ff[0][0] + df[1] * a.i0ff[1][0] +
                     df[2] * a.i0ff[2][0],
                xe = df[0] * a.e0f[0] + df[1] * a.e0f[1] + df[2] * a.e0f[2],
                ye = df[0] * a.b0f[0] + df[1] * a.b0f[1] + df[2] * a.b0f[2];
          scal = omega * cap * 0.5f *
                 (1.f + c2 * c2 - kahn * (xe * xe - ye * ye));
          const float fscal = HASF ? (float)(wk * (double)scal * g.scale) : 0.f;
          for (int pm = 0; pm < a.PM; ++pm) {
            const float *Ah = s_axh + pm * 9, *Al = s_axl + pm * 9;
            float Gh[3], Gl[3], rq[3], rl[3], n0[3];
#pragma unroll
            for (int x = 0; x < 3; ++x) {
              ff_dot3(Ah + 3 * x, Al + 3 * x, vh, vl, Gh[x], Gl[x]);
              float qh, qe;
              two_prod(Gh[x], a.u0h, qh, qe);
              float ql = fmaf(Gh[x], a.u0l, fmaf(Gl[x], a.u0h, qe));
              n0[x] = rintf(qh);
              float rh, rl0;
              two_sum(__fsub_rn(qh, n0[x]), ql, rh, rl0);
              rq[x] = __fmul_rn(rintf(__fmul_rn(rh, 2097152.f)),
                                1.f / 2097152.f);
              rl[x] = rl0 + __fsub_rn(rh, rq[x]);
            }
            // Σ_k e_x of this orientation's steps
            float E[3] = {0.f, 0.f, 0.f};
            // the steps that survive the cut, 32 sources at a time: every
            // lane then evaluates its own ones one after another, so that the
            // warp goes through the evaluation as often as the lane with the
            // most (4 or 5 of 8 sources) and not once per source that some
            // lane needs
            for (int k0 = 0; k0 < a.S; k0 += 32) {
            unsigned hits = 0;
            const int nk = min(32, a.S - k0);
            for (int j = 0; j < nk; j += 2) {
              const float *src = s_src + (k0 + j) * SRC32_STRIDE;
              const bool two = j + 1 < nk;
              const float2 rad2 = cut_sums(
                  Gh, rq, a.N,
                  make_float2(src[SRC32_DH],
                              src[two ? SRC32_STRIDE + SRC32_DH : SRC32_DH]));
              if (!(rad2.x > cutg)) hits |= 1u << j;
              if (two && !(rad2.y > cutg)) hits |= 2u << j;
            }
            while (hits) {
              const float *src =
                  s_src + (k0 + __ffs(hits) - 1) * SRC32_STRIDE;
              hits &= hits - 1;
              const float dh = src[SRC32_DH], dl = src[SRC32_DL];
              float fr[3];
              int n[3];
#pragma unroll
              for (int x = 0; x < 3; ++x) {
                const float nf = rintf(fmaf(Gh[x], dh, rq[x]));
                const float sx = fmaf(Gh[x], dh, __fsub_rn(rq[x], nf));
                fr[x] = sx + fmaf(Gh[x], dl, fmaf(Gl[x], dh, rl[x]));
                n[x] = __float2int_rn(n0[x] + nf) - a.hmin[x];
              }
              float rad2 = N2[0] * fr[0] * fr[0];
              rad2 = fmaf(N2[1] * fr[1], fr[1], rad2);
              rad2 = fmaf(N2[2] * fr[2], fr[2], rad2);
              float fl2 = a.N6 * expf(-2.f * rad2 * (1.f / 0.63f));
              bool inside = (unsigned)n[0] < (unsigned)a.hn[0] &&
                            (unsigned)n[1] < (unsigned)a.hn[1] &&
                            (unsigned)n[2] < (unsigned)a.hn[2];
              long long fidx =
                  inside ? ((long long)n[0] * a.hn[1] + n[1]) * a.hn[2] + n[2]
                         : -1;
              float fc, dfc[3] = {0.f, 0.f, 0.f};
              // tricubic: value and gradient of the interpolant, and the
              // stencil (its weights feed the structure-factor gradient)
              bool tri = false;
              int fl[3];
              float wv[3][4];
              if (INTERP == 1) {
                float xs[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                  int neg = fr[c] < 0.f;
                  fl[c] = n[c] - neg;
                  xs[c] = neg ? 1.f + fr[c] : fr[c];
                }
                tri = fl[0] >= 1 && fl[0] + 2 < a.hn[0] && fl[1] >= 1 &&
                      fl[1] + 2 < a.hn[1] && fl[2] >= 1 && fl[2] + 2 < a.hn[2];
                if (tri) {
                  float wd[3][4];
#pragma unroll
                  for (int c = 0; c < 3; ++c) {
                    lagrange4(xs[c], wv[c]);
                    lagrange4_deriv(xs[c], wd[c]);
                  }
                  fc = 0.f;
                  for (int i = 0; i < 4; ++i)
                    for (int j = 0; j < 4; ++j) {
                      const float *row = a.F + stencil_row(a, fl, i, j);
#pragma unroll
                      for (int k = 0; k < 4; ++k) {
                        float Fv = __ldg(row + k);
                        float wij = wv[0][i] * wv[1][j];
                        fc = fmaf(wij * wv[2][k], Fv, fc);
                        dfc[0] = fmaf(wd[0][i] * wv[1][j] * wv[2][k], Fv, dfc[0]);
                        dfc[1] = fmaf(wv[0][i] * wd[1][j] * wv[2][k], Fv, dfc[1]);
                        dfc[2] = fmaf(wij * wd[2][k], Fv, dfc[2]);
                      }
                    }
                }
              }
              if (!tri) fc = inside ? __ldg(a.F + nb_idx(a.check, NB_SITE_F, fidx, table_size(a))) : a.defF;
              const float w = src[SRC32_W];
              const float tw = fc * fc * fl2 * w;
              // d term / d h_x = term dlog_x + 2 F dF/dh_x F_latt^2 w
              const float uk = a.u0h + dh, tu = tw * uk,
                          fgu = 2.f * fc * fl2 * w * uk;
#pragma unroll
              for (int x = 0; x < 3; ++x) {
                E[x] += fmaf(tu, -4.f * N2[x] * fr[x] * (1.f / 0.63f),
                             INTERP ? fgu * dfc[x] : 0.f);
                acc[9 + x] = fmaf(tw, fmaf(cn1[x] * fr[x], fr[x], cn0[x]),
                                  acc[9 + x]);
              }
              acc12.add(tw);
              if (HASF) {
                const float gvf = fscal * (2.f * fc * fl2 * w);
                if (tri) {
                  if (!holding || n[0] != held[0] || n[1] != held[1] ||
                      n[2] != held[2]) {
                    flush_node();
                    held[0] = n[0];
                    held[1] = n[1];
                    held[2] = n[2];
                    holding = true;
                  }
                  // the stencil starts at fl - 1 = n - 2 + o, o = 0 or 1
                  const int o0 = fl[0] - n[0] + 1, o1 = fl[1] - n[1] + 1,
                            o2 = fl[2] - n[2] + 1;
#pragma unroll
                  for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                      const float wij = gvf * (wv[0][i] * wv[1][j]);
                      const int row = ((o0 + i) * 5 + (o1 + j)) * 5 + o2;
#pragma unroll
                      for (int k = 0; k < 4; ++k)
                        s_facc[row + k][threadIdx.x] =
                            fmaf(wij, wv[2][k], s_facc[row + k][threadIdx.x]);
                    }
                } else if (inside) {
                  // consecutive terms mostly hit the same entry: add up
                  // in a register, one atomic per run of equal entries
                  if (fidx != near_idx) {
                    if (near_idx >= 0) atomicAdd(g.gradF + nb_idx(a.check, NB_SITE_GRADF, near_idx, table_size(a)), (double)near_sum);
                    near_idx = fidx;
                    near_sum = 0.f;
                  }
                  near_sum += gvf;
                }
              }
            }
            }
            float vr[3];
            unrotate(s_rot + pm * 9, vh, vr);
#pragma unroll
            for (int x = 0; x < 3; ++x)
#pragma unroll
              for (int c = 0; c < 3; ++c)
                acc[3 * x + c] = fmaf(E[x], vr[c], acc[3 * x + c]);
          }
          }
          if (kColumns && n_units > 1) {
            // into the thread's column of double-floats
            const bool first = (i | j | t) == 0;
#pragma unroll
            for (int r = 0; r < kGradN; ++r) {
              float p, e, lo, hi;
              two_prod(scal, r < 12 ? acc[r] : acc12.s, p, e);
              if (r == 12) e = fmaf(scal, -acc12.c, e);
              float2 &col = s_tot[r][threadIdx.x];
              const float2 old = first ? make_float2(0.f, 0.f) : col;
              float s1, e1;
              two_sum(old.x, p, s1, e1);
              lo = old.y + (e1 + e);
              fast_two_sum(s1, lo, hi, lo);
              col = make_float2(hi, lo);
            }
            continue;
          }
          double v[16];
#pragma unroll
          for (int r = 0; r < 16; ++r)
            v[r] = r < 12    ? wk * (double)scal * (double)acc[r]
                   : r == 12 ? wk * (double)scal * acc12.value()
                             : 0.0;
          mine += warp_sums(v);
        }
    if (kColumns && n_units > 1) {
      double v[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        v[r] = 0.0;
        if (r < kGradN && ok) {
          const float2 c = s_tot[r][threadIdx.x];
          v[r] = wk * ((double)c.x + (double)c.y);
        }
      }
      mine = warp_sums(v);
    }
  }
  if (INTERP && HASF) flush_node();
  if (HASF && near_idx >= 0) atomicAdd(g.gradF + nb_idx(a.check, NB_SITE_GRADF, near_idx, table_size(a)), (double)near_sum);
  // the block's sums in FP64, in a fixed order
  __shared__ double red[kTileThreads / 32][kGradN];
  if ((lane & 1) == 0 && lane / 2 < kGradN)
    red[threadIdx.x >> 5][lane / 2] = mine;
  __syncthreads();
  if (threadIdx.x < kGradN) {
    double v = 0.0;
    for (int w = 0; w < kTileThreads / 32; ++w) v += red[w][threadIdx.x];
    g.partials[(size_t)blockIdx.x * kGradN + threadIdx.x] = v;
  }
}

// ---------------------------------------------------------------------
// Term-ring form (used where every table axis is at most 1000 long).  The
// thread-per-pixel kernel above evaluates a surviving term in the lane of
// its pixel, so a warp runs its expensive tricubic terms (64 table reads
// for the value, gradient and weights, 64 column updates) with only the
// lanes whose pixel has a term at that step.  Here the lanes still scan
// their own pixels' steps in lockstep (every pixel has the same steps),
// but a surviving step is pushed as a record into a per-warp ring in
// shared memory, and whenever the ring holds 32 records the warp
// evaluates them one per lane.  A record carries the step's exact offset,
// its lattice point, its (phi x mosaic, source) indices and the lane of
// its pixel, whose unit geometry and weight dL/dI K cap pol omega sit in a
// per-warp table.  Each lane adds what it evaluates into FP32 sums, which
// the warp folds into FP64 every 16 passes with a fixed butterfly, so the
// thirteen scalars stay deterministic.
//
// Bound by latency: 12 warps per SM (168 registers; the columns below take
// 51 KB a block) issue in 47 % of the cycles.  The lanes run through a row of
// sources, or up to a full ring, in one short loop; taking one step per trip
// through the outer states cost 64-panel shot (S = 8, 10 domains, 18 % of
// the steps surviving) 0.3 ms of 2.64.  Flushes of columns were next: a lane
// per float4 of the column and one pass over a group's lanes where a lane
// per float took four, 0.27 ms.  Tried beside it and slower or no faster:
// columns swizzled over the banks (the updates then conflict), records not
// sorted or grouped without an order (more flushes), records given to lanes
// that hold their column (fewer flushes, a longer sort).
constexpr int kAdjRing = 64;  // pending < 32 after a pass, + 32 pushed
constexpr int kAdjFold = 16;  // passes between folds into FP64

__host__ __device__ inline size_t adj_ring_floats(int PM, int S,
                                                  bool f_cache) {
  // the tables, then (F gradient) each thread's 5x5x4 column as 25 float4,
  // then the records: each 16-byte aligned
  const size_t fl = (size_t)3 * PM * 9 + (size_t)S * SRC32_STRIDE;
  return ((fl + 3) & ~(size_t)3) + (f_cache ? (size_t)100 * kTileThreads : 0);
}

__host__ __device__ inline size_t adj_ring_smem_bytes(int PM, int S,
                                                      bool f_cache) {
  const int warps = kTileThreads / 32;
  return adj_ring_floats(PM, S, f_cache) * sizeof(float) +
         (size_t)warps * kAdjRing * (sizeof(float4) + sizeof(int)) +
         (size_t)warps * 32 * (sizeof(float4) + sizeof(int));
}

template <int HASF, int INTERP>
__global__ void __launch_bounds__(kTileThreads, INTERP ? 3 : 4)
    spots_adjoint_ring_kernel(AdjointArgs g) {
  const SpotArgs &a = g.a;
  extern __shared__ __align__(16) float smf[];
  float *s_axh = smf;
  float *s_axl = smf + a.PM * 9;
  float *s_src = smf + 2 * a.PM * 9;
  float *s_rot = s_src + a.S * SRC32_STRIDE;
  for (int i = threadIdx.x; i < a.PM * 9; i += blockDim.x) {
    s_axh[i] = a.axh[i];
    s_axl[i] = a.axl[i];
    s_rot[i] = g.rot[i];
  }
  for (int i = threadIdx.x; i < a.S * SRC32_STRIDE; i += blockDim.x)
    s_src[i] = a.src32[i];
  const bool fcache = INTERP && HASF;
  float4 (*s_col)[kTileThreads] = reinterpret_cast<float4 (*)[kTileThreads]>(
      smf + adj_ring_floats(a.PM, a.S, false));
  float4 *s_rec = reinterpret_cast<float4 *>(
      smf + adj_ring_floats(a.PM, a.S, fcache));
  int *s_recb = reinterpret_cast<int *>(s_rec + (kTileThreads / 32) * kAdjRing);
  float4 *s_unit =
      reinterpret_cast<float4 *>(s_recb + (kTileThreads / 32) * kAdjRing);
  int *s_perm = reinterpret_cast<int *>(s_unit + (kTileThreads / 32) * 32);
  if (fcache)
    for (int r = 0; r < 25; ++r)
      s_col[r][threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float4 *rec_a = s_rec + warp * kAdjRing;
  int *rec_b = s_recb + warp * kAdjRing;
  float4 *unit_w = s_unit + warp * 32;
  int *perm = s_perm + warp * 32;

  // structure-factor gradient state of this lane.  A tricubic term near
  // lattice point n with its cell starting at fl touches nodes
  // fl - 1 .. fl + 2 on each axis: the lane sums them in a column of 5 x 5
  // nodes around (n_h, n_k) by the 4 nodes fl_l - 1 .. fl_l + 2 along l (a
  // float4 per (h, k) node), keyed by (n_h, n_k, fl_l) packed like a
  // record's lattice point (-1: no column)
  long long near_idx = -1;
  double near_sum = 0.0;
  int held_key = -1;
  // Flushes, cooperatively, the columns of the lanes with `need`: lanes
  // with the same key are summed entry by entry (in FP32, in lane order)
  // and each touched node gets one FP64 atomic; lane r < 25 takes row r of
  // the columns.  Called by all lanes.
  auto flush_columns = [&](bool need) {
    unsigned todo = __ballot_sync(0xffffffffu, need && held_key >= 0);
    while (todo) {
      const int key = __shfl_sync(0xffffffffu, held_key, __ffs(todo) - 1);
      const unsigned grp =
          __ballot_sync(0xffffffffu, need && held_key == key && key >= 0);
      todo &= ~grp;
      const int c0 = (key & 1023) - 1, c1 = ((key >> 10) & 1023) - 1,
                c2 = ((key >> 20) & 1023) - 1;
      if (lane < 25) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        for (unsigned m = grp; m; m &= m - 1) {
          float4 *col = &s_col[lane][warp * 32 + __ffs(m) - 1];
          const float4 c = *col;
          v.x += c.x;
          v.y += c.y;
          v.z += c.z;
          v.w += c.w;
          *col = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const long long at = ((long long)(c0 - 2 + lane / 5) * a.hn[1] +
                              (c1 - 2 + lane % 5)) * a.hn[2] + (c2 - 1);
        const float vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          if (vv[kk] != 0.f)
            atomicAdd(g.gradF + nb_idx(a.check, NB_SITE_GRADF, at + kk,
                                       table_size(a)),
                      (double)vv[kk]);
      }
    }
    if (need) held_key = -1;
    __syncwarp();
  };
  // a record's column key: its lattice point with l replaced by the start
  // of its cell along l
  auto column_key = [&](float4 ra) {
    const int npk = __float_as_int(ra.w);
    return (npk & 0xfffff) |
           ((((npk >> 20) & 1023) - (ra.z < 0.f ? 1 : 0)) << 20);
  };

  const float N2[3] = {a.N[0] * a.N[0], a.N[1] * a.N[1], a.N[2] * a.N[2]};
  const float cutg = kGaussCut * 0.63f;
  const float kahn = a.kahn;
  const float scalef = (float)g.scale;
  float acc[kGradN];
#pragma unroll
  for (int r = 0; r < kGradN; ++r) acc[r] = 0.f;
  double dacc = 0.0;  // lane r < kGradN: the warp's folded sum r
  const float cn0[3] = {2.f / a.N[0], 2.f / a.N[1], 2.f / a.N[2]},
              cn1[3] = {-4.f * a.N[0] * (1.f / 0.63f),
                        -4.f * a.N[1] * (1.f / 0.63f),
                        -4.f * a.N[2] * (1.f / 0.63f)};
  int head = 0, tail = 0, passes = 0;

  auto fold = [&]() {
#pragma unroll
    for (int r = 0; r < kGradN; ++r) {
      float v = acc[r];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == r) dacc += (double)v;
      acc[r] = 0.f;
    }
  };
  // evaluates records head .. head + cnt - 1 (cnt <= 32), one per lane
  auto eval_pass = [&](int cnt) {
    const bool v = lane < cnt;
    int slot = (head + lane) & (kAdjRing - 1);
    if (HASF) {
      // the pass's records in the order of their lattice points (ties in
      // ring order): lanes then keep the node of their column across
      // passes more often, and flush it less
      const int key = v ? column_key(rec_a[slot]) : 0x7fffffff;
      bool placed = !v;
      int pos = 0, base = 0;
      while (__any_sync(0xffffffffu, !placed)) {
        const int kmin = __reduce_min_sync(0xffffffffu, placed ? 0x7fffffff : key);
        const unsigned grp = __ballot_sync(0xffffffffu, !placed && key == kmin);
        if (!placed && key == kmin) {
          pos = base + __popc(grp & ((1u << lane) - 1u));
          placed = true;
        }
        base += __popc(grp);
      }
      if (v) perm[pos] = slot;
      __syncwarp();
      if (v) slot = perm[lane];
      __syncwarp();
      // a lane whose record has another column key than its column
      // flushes the column first
      if (INTERP)
        flush_columns(v && held_key >= 0 &&
                      column_key(rec_a[slot]) != held_key);
    }
    head += cnt;
    if (v) {
      const float4 ra = rec_a[slot];
      const int rb = rec_b[slot];
      const float fr[3] = {ra.x, ra.y, ra.z};
      const int npk = __float_as_int(ra.w);
      int n[3];
#pragma unroll
      for (int x = 0; x < 3; ++x) n[x] = ((npk >> (10 * x)) & 1023) - 1;
      const int pm = rb & 2047, k = (rb >> 11) & 1023, sl = (rb >> 21) & 31;
      const float4 uw = unit_w[sl];
      const float v32[3] = {uw.x, uw.y, uw.z};
      const float Wt = uw.w;
      const float *src = s_src + k * SRC32_STRIDE;
      const float dh = src[SRC32_DH], w = src[SRC32_W];
      float rad2 = N2[0] * fr[0] * fr[0];
      rad2 = fmaf(N2[1] * fr[1], fr[1], rad2);
      rad2 = fmaf(N2[2] * fr[2], fr[2], rad2);
      const float fl2 = a.N6 * expf(-2.f * rad2 * (1.f / 0.63f));
      const bool inside = (unsigned)n[0] < (unsigned)a.hn[0] &&
                          (unsigned)n[1] < (unsigned)a.hn[1] &&
                          (unsigned)n[2] < (unsigned)a.hn[2];
      const long long fidx =
          inside ? ((long long)n[0] * a.hn[1] + n[1]) * a.hn[2] + n[2] : -1;
      float fc, dfc[3] = {0.f, 0.f, 0.f};
      bool tri = false;
      int fl[3];
      float wv[3][4];
      if (INTERP == 1) {
        float xs[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const int neg = fr[c] < 0.f;
          fl[c] = n[c] - neg;
          xs[c] = neg ? 1.f + fr[c] : fr[c];
        }
        tri = fl[0] >= 1 && fl[0] + 2 < a.hn[0] && fl[1] >= 1 &&
              fl[1] + 2 < a.hn[1] && fl[2] >= 1 && fl[2] + 2 < a.hn[2];
        if (tri && a.C4) {
          // value and gradient of the cell's polynomial (its 64 monomial
          // coefficients), and the Lagrange weights for the F scatter
#pragma unroll
          for (int c = 0; c < 3; ++c) lagrange4(xs[c], wv[c]);
          const int ci = ((fl[0] - 1) * (a.hn[1] - 3) + (fl[1] - 1)) *
                             (a.hn[2] - 3) +
                         (fl[2] - 1);
          cell_value_grad(
              a.C4 + (size_t)nb_idx(a.check, NB_SITE_CELL, ci, cell_count(a)) * 16,
              xs, fc, dfc);
        } else if (tri) {
          float wd[3][4];
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            lagrange4(xs[c], wv[c]);
            lagrange4_deriv(xs[c], wd[c]);
          }
          fc = 0.f;
          for (int i = 0; i < 4; ++i)
            for (int j = 0; j < 4; ++j) {
              const float *row =
                  a.F + stencil_row(a, fl, i, j);
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) {
                const float Fv = __ldg(row + kk);
                const float wij = wv[0][i] * wv[1][j];
                fc = fmaf(wij * wv[2][kk], Fv, fc);
                dfc[0] = fmaf(wd[0][i] * wv[1][j] * wv[2][kk], Fv, dfc[0]);
                dfc[1] = fmaf(wv[0][i] * wd[1][j] * wv[2][kk], Fv, dfc[1]);
                dfc[2] = fmaf(wij * wd[2][kk], Fv, dfc[2]);
              }
            }
        }
      }
      if (!tri) fc = inside ? __ldg(a.F + nb_idx(a.check, NB_SITE_F, fidx, table_size(a))) : a.defF;
      const float tw = Wt * (fc * fc * fl2 * w);
      const float uk = a.u0h + dh;
      const float tu = tw * uk, fgu = Wt * (2.f * fc * fl2 * w) * uk;
      float vr[3];
      unrotate(s_rot + pm * 9, v32, vr);
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        const float e = fmaf(tu, -4.f * N2[x] * fr[x] * (1.f / 0.63f),
                             fgu * dfc[x]);
#pragma unroll
        for (int c = 0; c < 3; ++c)
          acc[3 * x + c] = fmaf(e, vr[c], acc[3 * x + c]);
        acc[9 + x] = fmaf(tw, fmaf(cn1[x] * fr[x], fr[x], cn0[x]),
                          acc[9 + x]);
      }
      acc[12] += tw;
      if (HASF) {
        const float gvf = Wt * scalef * (2.f * fc * fl2 * w);
        if (tri) {
          // the column was flushed unless it holds this key
          held_key = (npk & 0xfffff) | ((fl[2] + 1) << 20);
          const int o0 = fl[0] - n[0] + 1, o1 = fl[1] - n[1] + 1;
          float4 *col = &s_col[o0 * 5 + o1][threadIdx.x];
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float wij = gvf * (wv[0][i] * wv[1][j]);
              float4 c = col[(i * 5 + j) * kTileThreads];
              c.x = fmaf(wij, wv[2][0], c.x);
              c.y = fmaf(wij, wv[2][1], c.y);
              c.z = fmaf(wij, wv[2][2], c.z);
              c.w = fmaf(wij, wv[2][3], c.w);
              col[(i * 5 + j) * kTileThreads] = c;
            }
        } else if (inside) {
          if (fidx != near_idx) {
            if (near_idx >= 0) atomicAdd(g.gradF + nb_idx(a.check, NB_SITE_GRADF, near_idx, table_size(a)), near_sum);
            near_idx = fidx;
            near_sum = 0.0;
          }
          near_sum += (double)gvf;
        }
      }
    }
    __syncwarp();
    if (++passes % kAdjFold == 0) fold();
  };

  // Each warp takes rows of 32 pixels (a warp's quarter of a 16x8 tile, or
  // 32 entries of the pixel list) from a counter, and per pixel its steps
  // (unit, phi x mosaic, source): one step per iteration, the same
  // sequence in every lane.  The ring is drained before a unit's row of
  // the unit table is rewritten and at the end of a pixel row, whose
  // sums then go to the row's own partial row: the sums do not depend on
  // which warp took which row.
  const int U = a.os * a.os * a.T;
  auto next_row = [&]() {
    unsigned long long r = 0;
    if (lane == 0) r = atomicAdd(g.rows_next, 1ull);
    return (long long)__shfl_sync(0xffffffffu, r, 0);
  };
  long long row = next_row();
  bool row_done = false;
  int u = 0, pm = 0, k = 0;
  bool new_pixel = true, new_unit = true, new_pm = true;
  bool ok = false;
  const DevPanel *P = a.panels;
  int s = 0, f = 0;
  float W0 = 0.f;
  float vh[3], vl[3];
  float Gh[3], Gl[3], rq[3], rl[3], n0[3];
  while (true) {
    const bool finished = row >= g.n_rows;
    if (tail - head >= 32 ||
        ((finished || new_unit || row_done) && tail > head)) {
      eval_pass(min(32, tail - head));
      continue;
    }
    if (row_done) {
      // the row's records are all evaluated: its sums, then the next row
      fold();
      if (lane < kGradN)
        g.partials[(size_t)row * kGradN + lane] = dacc;
      dacc = 0.0;
      passes = 0;
      row = next_row();
      row_done = false;
      new_pixel = new_unit = new_pm = true;
      continue;
    }
    if (finished) break;
    if (new_pixel) {
      long long gp = 0;
      int q = 0;
      ok = a.pixlist
               ? map_pixel(a, row * 32 + lane, lane, gp, q, s, f)
               : map_pixel(a, row / (kTileThreads / 32),
                           (int)(row % (kTileThreads / 32)) * 32 + lane, gp,
                           q, s, f);
      if (!ok) {
        q = 0;
        s = 0;
        f = 0;
      }
      P = a.panels + q;
      W0 = ok ? (float)(g.dLdI[gp] * g.kc) : 0.f;
      new_pixel = false;
    }
    if (new_unit) {
      const int t = u % a.T, ij = u / a.T, i = ij / a.os, j = ij % a.os;
      float df[3], omega;
      unit_geometry_ff(a, *P, s, f, i, j, t, vh, vl, df, omega);
      float cap = 1.f;
      if (a.dtff[0] > 0.f) {
        const float rho = df[0] * P->ffn[0][0] + df[1] * P->ffn[1][0] +
                          df[2] * P->ffn[2][0];
        const float L = a.attenf * rho, dtf = a.dtff[0];
        cap = expf(-t * dtf / L) - expf(-(t + 1) * dtf / L);
      }
      const float c2 = df[0] * a.i0ff[0][0] + df[1] * a.i0ff[1][0] +
                       df[2] * a.i0ff[2][0],
                  xe = df[0] * a.e0f[0] + df[1] * a.e0f[1] + df[2] * a.e0f[2],
                  ye = df[0] * a.b0f[0] + df[1] * a.b0f[1] + df[2] * a.b0f[2];
      const float scal = omega * cap * 0.5f *
                         (1.f + c2 * c2 - kahn * (xe * xe - ye * ye));
      unit_w[lane] = make_float4(vh[0], vh[1], vh[2], W0 * scal);
      __syncwarp();
      new_unit = false;
    }
    if (new_pm) {
      const float *Ah = s_axh + pm * 9, *Al = s_axl + pm * 9;
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        ff_dot3(Ah + 3 * x, Al + 3 * x, vh, vl, Gh[x], Gl[x]);
        float qh, qe;
        two_prod(Gh[x], a.u0h, qh, qe);
        const float ql = fmaf(Gh[x], a.u0l, fmaf(Gl[x], a.u0h, qe));
        n0[x] = rintf(qh);
        float rh, rl0;
        two_sum(__fsub_rn(qh, n0[x]), ql, rh, rl0);
        rq[x] = __fmul_rn(rintf(__fmul_rn(rh, 2097152.f)), 1.f / 2097152.f);
        rl[x] = rl0 + __fsub_rn(rh, rq[x]);
      }
      new_pm = false;
    }
    // steps (u, pm, k ..) until the row of sources ends or the ring holds a
    // pass: the cheap cut test, then the exact offset of a surviving step
    // and its record
    do {
      const float *src = s_src + k * SRC32_STRIDE;
      const float dh = src[SRC32_DH], dl = src[SRC32_DL];
      float fr[3], nf[3];
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        const float tq = fmaf(Gh[x], dh, rq[x]);
        nf[x] = __fsub_rn(__fadd_rn(tq, kRoundAdd), kRoundAdd);  // rint
        fr[x] = tq - nf[x];
      }
      float rad2 = N2[0] * fr[0] * fr[0];
      rad2 = fmaf(N2[1] * fr[1], fr[1], rad2);
      rad2 = fmaf(N2[2] * fr[2], fr[2], rad2);
      const bool hit = ok && rad2 <= cutg;
      const unsigned hm = __ballot_sync(0xffffffffu, hit);
      if (hm) {
        if (hit) {
          int npk = 0;
#pragma unroll
          for (int x = 0; x < 3; ++x) {
            const float sx = fmaf(Gh[x], dh, __fsub_rn(rq[x], nf[x]));
            fr[x] = sx + fmaf(Gh[x], dl, fmaf(Gl[x], dh, rl[x]));
            const int nx = __float2int_rn(n0[x] + nf[x]) - a.hmin[x];
            npk |= (min(max(nx, -1), a.hn[x]) + 1) << (10 * x);
          }
          const int slot =
              (tail + __popc(hm & ((1u << lane) - 1u))) & (kAdjRing - 1);
          rec_a[slot] = make_float4(fr[0], fr[1], fr[2], __int_as_float(npk));
          rec_b[slot] = pm | (k << 11) | (lane << 21);
        }
        tail += __popc(hm);
      }
    } while (++k < a.S && tail - head < 32);
    __syncwarp();
    // advance (u, pm, k); after the last step of the row's pixels the row
    // is done once its records are evaluated
    if (k == a.S) {
      k = 0;
      new_pm = true;
      if (++pm == a.PM) {
        pm = 0;
        new_unit = true;
        if (++u == U) {
          u = 0;
          row_done = true;
        }
      }
    }
  }
  if (fcache) flush_columns(true);
  if (HASF && near_idx >= 0) atomicAdd(g.gradF + nb_idx(a.check, NB_SITE_GRADF, near_idx, table_size(a)), near_sum);
}

// Sums the partial rows [n][kGradN] in a fixed order: block b its share of
// `per` rows into row b of out.  32 threads per column; a thread's loads are
// independent of one another and a row's columns lie side by side.  (One
// block for all rows took 91 us for the 19968 blocks of the 64-panel shot and
// 347 us for its 79872 pixel rows, waiting on one load after another.)
__global__ void reduce_partials_kernel(const double *part, long long n,
                                       long long per, double *out) {
  __shared__ double red[32][kGradN];
  const int r = threadIdx.x, lane = threadIdx.y;
  const long long first = blockIdx.x * per,
                  last = first + per < n ? first + per : n;
  double v = 0.0;
#pragma unroll 4
  for (long long i = first + lane; i < last; i += 32)
    v += part[i * kGradN + r];
  red[lane][r] = v;
  __syncthreads();
  if (lane == 0) {
    double s = 0.0;
    for (int l = 0; l < 32; ++l) s += red[l][r];
    out[(long long)blockIdx.x * kGradN + r] = s;
  }
}

// rows [0, n) of part to one row in out; scratch for kReduceRows rows
constexpr int kReduceRows = 128;
static cudaError_t reduce_partials(const double *part, long long n,
                                   double *scratch, double *out,
                                   cudaStream_t st) {
  const dim3 threads(kGradN, 32);
  if (n > 4 * kReduceRows) {
    const long long per = (n + kReduceRows - 1) / kReduceRows;
    reduce_partials_kernel<<<kReduceRows, threads, 0, st>>>(part, n, per,
                                                            scratch);
    part = scratch;
    n = kReduceRows;
  }
  reduce_partials_kernel<<<1, threads, 0, st>>>(part, n, n, out);
  return cudaGetLastError();
}

// Poisson loss L = sum_p (I_p + bkg - y_p log(I_p + bkg)) and dL/dI_p.
// Bound by the FP64 pipe (1/64 of the FP32 rate), so the logarithm and the
// quotient share what they can.  m = 2^e z, z in [1, 2); a table of 64
// intervals gives c ~ 1/z, and r = z c - 1 (|r| < 2^-7, rounded once) is
// both the argument of log1p, summed as its series to r^9 (remainder below
// 2^-72; after Tang, "Table-driven implementation of the logarithm function",
// 1990), and the first correction of the reciprocal.  About 30 FP64
// instructions per pixel instead of 70: 234 -> 111 us for the 2.3e6 pixels of
// the 64-panel shot.  The table is made per block from log and division, so
// the blocks are few and persistent.
constexpr int kLogTable = 64;

__device__ __forceinline__ void poisson_pixel(double m, double y,
                                              const double2 *tab, double &l,
                                              double &d) {
  const long long bits = __double_as_longlong(m);
  const int ex = (int)(bits >> 52);  // with the sign: negative for m < 0
  if (ex < 523 || ex > 1523 ||
      ((__double2hiint(y) >> 20) & 0x7ff) > 1500) {
    // tiny, huge, negative or not a number
    l += m - y * log(m);
    d = 1.0 - y / m;
    return;
  }
  const double z = __longlong_as_double((bits & 0x000fffffffffffffll) |
                                        0x3ff0000000000000ll);
  const double2 t = tab[(int)(bits >> 46) & (kLogTable - 1)];
  const double r = fma(z, t.x, -1.0), r2 = r * r;
  double q = fma(r, 1.0 / 9.0, -1.0 / 8.0);
  q = fma(q, r, 1.0 / 7.0);
  q = fma(q, r, -1.0 / 6.0);
  q = fma(q, r, 1.0 / 5.0);
  q = fma(q, r, -0.25);
  q = fma(q, r, 1.0 / 3.0);
  q = fma(q, r, -0.5);
  // the exponent as a double: its bits in the last place of 2^52 + 2^51
  const double e = __longlong_as_double(0x4338000000000000ll + (ex - 1023)) -
                   6755399441055744.0;
  const double lg = fma(e, 0.69314718055994530942, t.y) + fma(q, r2, r);
  l += fma(-y, lg, m);
  // 1/z from c: 1/(1 + r) = (1 - r)(1 + r^2)(1 + r^4) ...
  double x = fma(-t.x, r, t.x);
  x = fma(x, fma(r2, r2, r2), x);
  x = x * __hiloint2double((2046 - ex) << 20, 0);  // 2^-e
  const double p = y * x;
  d = 1.0 - fma(fma(-p, m, y), x, p);
}

__global__ void __launch_bounds__(256)
    poisson_loss_kernel(const double *img, const double *y, long long n,
                        double bkg, double *dLdI, double *partials) {
  __shared__ double2 tab[kLogTable];
  __shared__ double red[8];
  for (int i = threadIdx.x; i < kLogTable; i += blockDim.x) {
    const double c = 1.0 / (1.0 + (i + 0.5) / kLogTable);
    tab[i] = make_double2(c, -log(c));
  }
  __syncthreads();
  double l = 0.0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    double d;
    poisson_pixel(img[i] + bkg, y[i], tab, l, d);
    dLdI[i] = d;
  }
  for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = l;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[w];
    partials[blockIdx.x] = s;
  }
}

// the block sums of the loss, in a fixed order
__global__ void loss_sum_kernel(const double *part, int n, double *out) {
  __shared__ double red[32];
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += 1024) v += part[i];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = red[threadIdx.x];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) *out = v;
  }
}

// The term-ring kernel serves tricubic lookup (its terms are the
// expensive ones: value and gradient of the cell polynomial and 64 column
// updates); it packs a table index in 10 bits per axis.  Nearest lookup
// stays on the thread-per-pixel kernel, which measured as fast or faster.
static bool adjoint_ring_ok(const SpotArgs &a) {
  return a.interp == 1 && a.hn[0] <= 1000 && a.hn[1] <= 1000 &&
         a.hn[2] <= 1000;
}

size_t adjoint_smem_bytes(const SpotArgs &a, bool f_cache) {
  if (adjoint_ring_ok(a)) return adj_ring_smem_bytes(a.PM, a.S, f_cache);
  return (size_t)(3 * a.PM * 9 + a.S * SRC32_STRIDE +
                  (f_cache ? 125 * kTileThreads : 0)) *
         sizeof(float);
}

// rows of partial sums the adjoint writes: one per pixel row of 32 (term
// ring) or per block (thread kernel)
long long adjoint_blocks(const SpotArgs &a) {
  if (adjoint_ring_ok(a))
    return a.pixlist ? (a.n_list + 31) / 32
                     : (long long)a.n_tiles * (kTileThreads / 32);
  return a.pixlist ? (a.n_list + kTileThreads - 1) / kTileThreads
                   : a.n_tiles;
}

size_t adjoint_scratch_bytes(const SpotArgs &a) {
  // the partial rows, the row counter, the rows of the first reduction
  return (size_t)(adjoint_blocks(a) + 1 + kReduceRows) * kGradN *
         sizeof(double);
}

// writes the kGradN sums, without the scale, to sums_out
cudaError_t launch_adjoint(const SpotArgs &a, const float *rot,
                           const double *dLdI, double *gradF,
                           double *partials, double kc, double scale,
                           double *sums_out, int sm_count, cudaStream_t st) {
  AdjointArgs g;
  g.a = a;
  g.rot = rot;
  g.dLdI = dLdI;
  g.gradF = gradF;
  g.partials = partials;
  g.kc = kc;
  g.scale = scale;
  g.rows_next = nullptr;
  g.n_rows = 0;
  size_t smem = adjoint_smem_bytes(a, a.interp && gradF);
  // the columns of the pixels' sums, and a float to align them (beside tables
  // of at most 200 KB that are counted with 180 bytes per orientation too many)
  if (a.interp == 0 && a.os * a.os * a.T > 1)
    smem += sizeof(float) + kGradN * kTileThreads * sizeof(float2);
  long long blocks = adjoint_blocks(a);
  if (blocks <= 0) return cudaSuccess;
  void (*kern)(AdjointArgs);
  if (adjoint_ring_ok(a))  // tricubic only
    kern = gradF ? spots_adjoint_ring_kernel<1, 1>
                 : spots_adjoint_ring_kernel<0, 1>;
  else
    kern = a.interp ? (gradF ? spots_adjoint_kernel<1, 1>
                             : spots_adjoint_kernel<0, 1>)
                    : (gradF ? spots_adjoint_kernel<1, 0>
                             : spots_adjoint_kernel<0, 0>);
  cudaError_t e = cudaFuncSetAttribute(
      kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  long long grid = blocks;
  if (adjoint_ring_ok(a)) {
    // persistent blocks; warps take pixel rows from a counter stored after
    // the partial rows (the buffer holds blocks + 1 rows)
    g.n_rows = blocks;
    g.rows_next = reinterpret_cast<unsigned long long *>(partials +
                                                        blocks * kGradN);
    e = cudaMemsetAsync(g.rows_next, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern,
                                                      kTileThreads, smem);
    if (e != cudaSuccess) return e;
    const long long fit = (long long)(sm_count > 0 ? sm_count : 1) *
                          (per_sm > 0 ? per_sm : 1);
    const long long need = (blocks + kTileThreads / 32 - 1) / (kTileThreads / 32);
    grid = fit < need ? fit : need;
  }
  kern<<<(unsigned)grid, kTileThreads, smem, st>>>(g);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return reduce_partials(partials, blocks, partials + (blocks + 1) * kGradN,
                         sums_out, st);
}

// grad (10) from the kGradN sums and the derivatives of the lab axes
void adjoint_gradient(const double *sums, const double daxes[6][9],
                      double scale, double *grad) {
  for (int r = 0; r < 6; ++r) {
    double v = 0.0;
    for (int i = 0; i < 9; ++i) v += daxes[r][i] * sums[i];
    grad[r] = scale * v;
  }
  for (int x = 0; x < 3; ++x) grad[6 + x] = scale * sums[9 + x];
  grad[9] = sums[12];
}

int loss_blocks(long long n) {
  long long b = (n + 255) / 256;
  return (int)(b < 608 ? (b < 1 ? 1 : b) : 608);
}

cudaError_t launch_poisson_loss(const double *img, const double *y,
                                long long n, double bkg, double *dLdI,
                                double *partials, double *loss_out,
                                cudaStream_t st) {
  int blocks = loss_blocks(n);
  poisson_loss_kernel<<<blocks, 256, 0, st>>>(img, y, n, bkg, dLdI, partials);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  loss_sum_kernel<<<1, 1024, 0, st>>>(partials, blocks, loss_out);
  return cudaGetLastError();
}

}  // namespace nbgb
