// Galerkin assembly kernels of the MTF operator (Sec. 2.3, Sec. 3.2).
//
// Per block i the library builds the dense EFIO T_i and MFIO K_i Galerkin
// matrices at k_i, tested with the x-pairing (Eq. 5):
//   T[m,n] = -i k int int G psi_n(y).psi_m(x) - 1/(i k) int int G div psi_n div psi_m
//   K[m,n] = -int int grad_x G(x,y) . (psi_n(y) x psi_m(x))
// (Eq. 7 potentials, Eq. 9 operators; the normal cancels in the pairing).
// Entries are stored row-major per block as (T.re, T.im, K.re, K.im).
//
// Each triangle pair (tau test, sigma trial) contributes a 3x3 block, with RWG
// functions c_a (x - v_a) and c_b (y - u_b):
//   T_ab = c_a c_b [ -ik sum W G (x - v_a).(y - u_b) - 4/(ik) sum W G ]
//   K_ab = -c_a c_b (v_a - u_b) . sum W g (y - u_b) x (x - v_a),
// g = G (i k - 1/r) / r ((x - y).((y - u_b) x (x - v_a)) by the triple
// product).  x and y are linear in their triangles' coordinates, so the kernels
// never form the 9 products per quadrature point: all 18 entries follow from
// the sums of G and of g times (1, s, t) of x and (1, s', t') of y, nine
// complex sums each (k_regular64), or from the monomials in the coordinates of
// the singular rules (k_singular64).
#include <cmath>

#include "common.h"
#include "kernel64.cuh"
#include "pair_tile.cuh"

namespace mtf {

__constant__ double c_tri_s[6], c_tri_t[6], c_tri_w[6];  // 6-point rule
// per orbit (a, a, 1 - 2a): w, w a, w (1 - 3a); per point: w, w s, w t
__constant__ double c_orbit[2][3], c_point[6][3];

struct C2 {
  double re, im;
};
__device__ __forceinline__ C2 cmul(C2 a, C2 b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ C2 cscale(C2 a, double s) { return {a.re * s, a.im * s}; }
__device__ __forceinline__ C2 cadd(C2 a, C2 b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ C2 csub(C2 a, C2 b) { return {a.re - b.re, a.im - b.im}; }

__device__ __forceinline__ void add_entry(double* TK, int64_t idx, C2 T, C2 K) {
  double* e = TK + 4 * idx;
  atomicAdd(e + 0, T.re);
  atomicAdd(e + 1, T.im);
  atomicAdd(e + 2, K.re);
  atomicAdd(e + 3, K.im);
}
__device__ __forceinline__ void add_entry(float* TK, int64_t idx, C2 T, C2 K) {
  atomicAdd(reinterpret_cast<float4*>(TK) + idx, make_float4(float(T.re), float(T.im), float(K.re), float(K.im)));
}

// ---------------------------------------------------------------------------
// regular (vertex-disjoint) pairs, FP64: one thread per unordered pair, CTAs
// over 16 x 16 tiles of a block's triangles (pair_tile.cuh)
//
// What bounds it: the FP64 pipe.  Both orderings of a pair have transposed
// 3 x 3 blocks (the Galerkin forms are symmetric), so each pair is evaluated
// once and added at the upper position (m < n); k_mirror fills the lower
// triangle.  A kernel evaluation takes the reciprocal square root by a
// Householder step and exp(i k (r - r0)) by its Taylor series (r0 the
// centroid distance; the phase exp(i k r0) is applied once per pair), of the
// length the pair's extent asks for.  The 6-point rule's two orbits share
// their weight, so the moments over (1, s, t) take 14 operations per channel
// and 6 points.  Measured on the split sphere of 7 rings (1.04 M ordered
// pairs): 7.95 -> 2.41 ms.
// ---------------------------------------------------------------------------
struct BlockArgs {
  const double* bt_v;
  const double* bt_c;
  const double* bt_area;
  const int32_t* bt_dof;
  const int32_t* bt_vid;
  const int32_t* blk_T;
  const int32_t* blk_N;
  const int64_t* blk_bt_off;
  const int64_t* blk_mat_off;
  const double* k;  // (re, im) per block
  int nblk;
};

// triangles of one side of a tile: quadrature points, vertices, c_a 2 A
struct Side64 {
  double x[18][kPairTile], v[9][kPairTile], cen[3][kPairTile], c[3][kPairTile];
  float rad[kPairTile];
  int dof[3][kPairTile], vid[3][kPairTile];
};

__device__ __forceinline__ void load_side(const BlockArgs& A, int64_t first, int n, Side64& S) {
  for (int t = threadIdx.x; t < kPairTile * 6; t += blockDim.x) {
    const int q = t / 6, p = t % 6;
    if (q >= n) continue;
    const double* v = A.bt_v + 9 * (first + q);
    for (int c = 0; c < 3; ++c)
      S.x[3 * p + c][q] = v[c] + c_tri_s[p] * (v[3 + c] - v[c]) + c_tri_t[p] * (v[6 + c] - v[c]);
  }
  for (int q = threadIdx.x; q < n; q += blockDim.x) {
    const double* v = A.bt_v + 9 * (first + q);
    for (int c = 0; c < 9; ++c) S.v[c][q] = v[c];
    for (int c = 0; c < 3; ++c) {
      S.cen[c][q] = (v[c] + v[3 + c] + v[6 + c]) * (1.0 / 3.0);
      S.c[c][q] = A.bt_c[3 * (first + q) + c] * (2.0 * A.bt_area[first + q]);
      S.dof[c][q] = A.bt_dof[3 * (first + q) + c];
      S.vid[c][q] = A.bt_vid[3 * (first + q) + c];
    }
    float r = 0.f;
    for (int a = 0; a < 3; ++a) {
      float d2 = 0.f;
      for (int c = 0; c < 3; ++c) {
        const float d = float(v[3 * a + c] - S.cen[c][q]);
        d2 = fmaf(d, d, d2);
      }
      r = fmaxf(r, d2);
    }
    S.rad[q] = sqrtf(r) * 1.0001f;
  }
}

__global__ void __launch_bounds__(128) k_regular64(BlockArgs A, const int64_t* __restrict__ cta_prefix,
                                                   double* __restrict__ TK) {
  __shared__ Side64 X, Y;
  const PairTile P = pair_tile(blockIdx.x, cta_prefix, A.nblk);
  const int i = P.blk, T = A.blk_T[i];
  load_side(A, A.blk_bt_off[i] + P.t0, min(kPairTile, T - P.t0), X);
  load_side(A, A.blk_bt_off[i] + P.s0, min(kPairTile, T - P.s0), Y);
  __syncthreads();
  const double k = A.k[2 * i], m4k2 = -4.0 / (k * k);
  const int N = A.blk_N[i];
  double* M = TK + 4 * A.blk_mat_off[i];
  const int b = threadIdx.x & (kPairTile - 1);
#pragma unroll 1
  for (int a = threadIdx.x / kPairTile; a < kPairTile; a += 128 / kPairTile) {
    // unordered pairs, once each; singular ones are k_singular64's
    bool live = P.t0 + a < P.s0 + b && P.s0 + b < T;
    if (live) {
      bool shared = false;
#pragma unroll
      for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int q = 0; q < 3; ++q) shared |= X.vid[p][a] == Y.vid[q][b];
      live = !shared;
    }
    float ext = live ? float(k) * (X.rad[a] + Y.rad[b]) : 0.f;
    ext = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(ext)));
    const int deg = series_degree(ext);
    if (!live) continue;
    const double D[3] = {X.cen[0][a] - Y.cen[0][b], X.cen[1][a] - Y.cen[1][b], X.cen[2][a] - Y.cen[2][b]};
    const double kr0 = k * sqrt(dot3(D, D));
    // sums over the rule of G exp(-i k r0) 4 pi and of -g: [row: 1, s, t of x][1, s, t of y] (re, im)
    double G[3][3][2], H[3][3][2];
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int q = 0; q < 3; ++q) G[p][q][0] = G[p][q][1] = H[p][q][0] = H[p][q][1] = 0.0;
#pragma unroll 1
    for (int p = 0; p < 6; ++p) {
      const double x0 = X.x[3 * p][a], x1 = X.x[3 * p + 1][a], x2 = X.x[3 * p + 2][a];
      double m[3][4], bc[4];  // y moments of (re G, im G, re H, im H); bc: part common to s and t
#pragma unroll
      for (int f = 0; f < 4; ++f) m[0][f] = m[1][f] = m[2][f] = bc[f] = 0.0;
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        double v[3][4], ri[3], ph[3], sn[3], cs[3];
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          const int q = 3 * o + e;
          const double d[3] = {x0 - Y.x[3 * q][b], x1 - Y.x[3 * q + 1][b], x2 - Y.x[3 * q + 2][b]};
          const double r2 = dot3(d, d);
          ri[e] = rsqrt_h(r2);
          ph[e] = fma(k, r2 * ri[e], -kr0);
        }
        if (deg >= 0) {
          double z[3];
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            z[e] = ph[e] * ph[e];
            cs[e] = c_cos[deg];
            sn[e] = c_sin[deg];
          }
#pragma unroll 1
          for (int t = deg - 1; t >= 0; --t)
#pragma unroll
            for (int e = 0; e < 3; ++e) {
              cs[e] = fma(cs[e], z[e], c_cos[t]);
              sn[e] = fma(sn[e], z[e], c_sin[t]);
            }
#pragma unroll
          for (int e = 0; e < 3; ++e) sn[e] *= ph[e];
        } else {
#pragma unroll
          for (int e = 0; e < 3; ++e) sincos(ph[e], &sn[e], &cs[e]);
        }
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          v[e][0] = ri[e] * cs[e];
          v[e][1] = ri[e] * sn[e];
          const double al = k * ri[e], be = ri[e] * ri[e];  // -g = G (1/r - i k) / r
          v[e][2] = fma(be, v[e][0], al * v[e][1]);
          v[e][3] = fma(be, v[e][1], -(al * v[e][0]));
        }
        // orbit o: barycentric coordinates a, a, 1 - 2a; s = 1 - 2a at its point 1, t at its point 2
        const double w = c_orbit[o][0], wa = c_orbit[o][1], wc = c_orbit[o][2];
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          const double sum = v[0][f] + v[1][f] + v[2][f];
          m[0][f] = fma(w, sum, m[0][f]);
          bc[f] = fma(wa, sum, bc[f]);
          m[1][f] = fma(wc, v[1][f], m[1][f]);
          m[2][f] = fma(wc, v[2][f], m[2][f]);
        }
      }
      const double wx[3] = {c_point[p][0], c_point[p][1], c_point[p][2]};
#pragma unroll
      for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          const double t = q == 0 ? m[0][f] : m[q][f] + bc[f];
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            double& dst = f < 2 ? G[r][q][f] : H[r][q][f - 2];
            dst = fma(wx[r], t, dst);
          }
        }
    }
    // the common phase, and 1 / (4 pi)
    double s0, c0;
    sincos(kr0, &s0, &c0);
    s0 *= INV_FOUR_PI;
    c0 *= INV_FOUR_PI;
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const double gr = G[p][q][0], hr = H[p][q][0];
        G[p][q][0] = gr * c0 - G[p][q][1] * s0;
        G[p][q][1] = gr * s0 + G[p][q][1] * c0;
        H[p][q][0] = hr * c0 - H[p][q][1] * s0;
        H[p][q][1] = hr * s0 + H[p][q][1] * c0;
      }
    // x = v_0 + s E_1 + t E_2, y = u_0 + s' F_1 + t' F_2:
    //   T_ab = c_a c_b [-i k sum G (x - v_a).(y - u_b) - 4 / (i k) sum G]
    //   K_ab = -c_a c_b (v_a - u_b) . sum g (y - u_b) x (x - v_a)
    double E[2][3], F[2][3], De[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      De[c] = X.v[c][a] - Y.v[c][b];
      E[0][c] = X.v[3 + c][a] - X.v[c][a];
      E[1][c] = X.v[6 + c][a] - X.v[c][a];
      F[0][c] = Y.v[3 + c][b] - Y.v[c][b];
      F[1][c] = Y.v[6 + c][b] - Y.v[c][b];
    }
    // ef = E_i . F_j, V_ij(a, b) = det(v_a - u_b, F_j, E_i) from D_ij = det(De, F_j, E_i),
    // Av_j = det(E_1, E_2, F_j), Bv_i = det(F_1, F_2, E_i)
    double ef[2][2], Dv[2][2], Av[2], Bv[2], t3[3];
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        ef[p][q] = dot3(E[p], F[q]);
        cross3(F[q], E[p], t3);
        Dv[p][q] = dot3(De, t3);
        if (p == 1) Av[q] = -dot3(E[0], t3);
        if (q == 1) Bv[p] = dot3(F[0], t3);
      }
    // sum over (i, j) of ef G_ij, with the S0 term of T folded in: X_ab = Xs - Hx_b - Hy_a + ef_ab S0
    double Xs[2], Hx[2][2], Hy[2][2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      Xs[c] = m4k2 * G[0][0][c];
#pragma unroll
      for (int q = 0; q < 2; ++q) Hx[q][c] = fma(ef[0][q], G[1][0][c], ef[1][q] * G[2][0][c]);
#pragma unroll
      for (int p = 0; p < 2; ++p) Hy[p][c] = fma(ef[p][0], G[0][1][c], ef[p][1] * G[0][2][c]);
#pragma unroll
      for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 2; ++q) Xs[c] = fma(ef[p][q], G[1 + p][1 + q][c], Xs[c]);
    }
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const int mrow = X.dof[p][a];
      const double cp = X.c[p][a];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        double x2c[2], kk[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          double t = Xs[c];
          if (q > 0) t -= Hx[q - 1][c];
          if (p > 0) t -= Hy[p - 1][c];
          if (p > 0 && q > 0) t = fma(ef[p - 1][q - 1], G[0][0][c], t);
          x2c[c] = t;
        }
        double V[2][2];
#pragma unroll
        for (int ii = 0; ii < 2; ++ii)
#pragma unroll
          for (int jj = 0; jj < 2; ++jj) {
            double t = Dv[ii][jj];
            if (p == 2 - ii) t += ii == 0 ? Av[jj] : -Av[jj];  // v_a = v_0 + E of the other index
            if (q == 2 - jj) t += jj == 0 ? Bv[ii] : -Bv[ii];
            V[ii][jj] = t;
          }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          double s = 0.0;
#pragma unroll
          for (int ii = 0; ii < 2; ++ii)
#pragma unroll
            for (int jj = 0; jj < 2; ++jj) {
              double n = H[1 + ii][1 + jj][c];
              if (q == jj + 1) n -= H[1 + ii][0][c];
              if (p == ii + 1) n -= H[0][1 + jj][c];
              if (p == ii + 1 && q == jj + 1) n += H[0][0][c];
              s = fma(V[ii][jj], n, s);
            }
          kk[c] = s;
        }
        const double cc = cp * Y.c[q][b];
        const int ncol = Y.dof[q][b];
        const int64_t at = mrow < ncol ? int64_t(mrow) * N + ncol : int64_t(ncol) * N + mrow;
        add_entry(M, at, C2{cc * (k * x2c[1]), -(cc * (k * x2c[0]))}, C2{cc * kk[0], cc * kk[1]});
      }
    }
  }
}

struct __align__(16) Entry64 {
  double x, y, z, w;
};

// lower triangle of every block from the upper one (M symmetric), 32 x 32
// entries per CTA through shared memory; with amax, also the block's largest
// |re|, |im| of T and K (float bits), which the FP16 operator tiles scale by;
// with rot, a copy of the whole block as (K - i T, K + i T), the form the FP64
// matvec multiplies with (apply.cu)
template <class V4>
__global__ void __launch_bounds__(256) k_mirror(V4* __restrict__ TK, const int64_t* __restrict__ tile_prefix, int nblk,
                                                const int32_t* __restrict__ blk_N,
                                                const int64_t* __restrict__ blk_mat_off, unsigned* __restrict__ amax,
                                                V4* __restrict__ rot) {
  __shared__ V4 t[32][33];
  const PairTile P = pair_tile(blockIdx.x, tile_prefix, nblk, 32);
  const int N = blk_N[P.blk];
  V4* M = TK + blk_mat_off[P.blk];
  V4* Q = rot ? rot + blk_mat_off[P.blk] : nullptr;
  auto rotated = [](const V4& v) { return V4{v.z + v.y, v.w - v.x, v.z - v.y, v.w + v.x}; };
  const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;
  float mx = 0.f;
#pragma unroll
  for (int y = ly; y < 32; y += 8) {
    const int r = P.t0 + y, c = P.s0 + lx;
    if (r < N && c < N && r <= c) {
      const V4 v = M[int64_t(r) * N + c];
      t[y][lx] = v;
      if (rot) Q[int64_t(r) * N + c] = rotated(v);
      mx = fmaxf(mx, fmaxf(fmaxf(fabsf(float(v.x)), fabsf(float(v.y))), fmaxf(fabsf(float(v.z)), fabsf(float(v.w)))));
    }
  }
  __syncthreads();
#pragma unroll
  for (int y = ly; y < 32; y += 8) {
    const int r = P.s0 + y, c = P.t0 + lx;  // transposed tile
    if (r < N && c < N && c < r) {
      M[int64_t(r) * N + c] = t[lx][y];
      if (rot) Q[int64_t(r) * N + c] = rotated(t[lx][y]);
    }
  }
  if (amax) {
    mx = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mx)));
    if (lx == 0) atomicMax(amax + P.blk, __float_as_uint(mx));
  }
}

// ---------------------------------------------------------------------------
// singular pairs (Sauter-Schwab), FP64: 16 lanes per pair, lanes over the
// angular ("hat") points of the rule (common.h)
//
// What bounds it: the FP64 pipe (about 1/64 of the FP32 rate).  A rule point
// evaluated by itself costs about 118 FP64 instructions (sqrt, reciprocal,
// sincos, 28 moment sums).  Here the n_ss radial points of a hat point share
// everything: with |x - y| = xi rho the pair's moments are
//   sum W xi^3 xi^m G:  re = P_{2+m} / rho,   im = k S_{3+m},      m = 0, 1, 2
//   sum W xi^3 xi^m g:  re = -(P_m / rho^3 + k^2 S_{2+m} / rho),
//                       im = k (P_{1+m} - S_{1+m}) / rho^2,         m = 1, 2
// (m the degree of the moment's monomial in the coordinates), and the radial
// sums P, S are power series in (k rho)^2: 8 Horner chains of 6 to 12 steps
// per hat point instead of n_ss square roots and sincos.  kappa = k rho <= 2
// is carried to FP64 rounding; wider pairs evaluate the sums point by point.
// The moments are monomials x_i y_j in the rule's own coordinates (their
// weights tabulated per hat point), 6 (coincident, halved by the x <-> y
// symmetry, coplanar: K = 0), 9 + 6 (common edge) or 9 + 8 (common vertex)
// complex sums.  Measured: 15.4 -> 3.5 ms for the 2 x 2 x 2 cube's 11,664
// coincident, 17,496 edge and 52,272 vertex pairs (n_ss = 4).
// ---------------------------------------------------------------------------

// hat-table rows, sums per pair of each kind
template <int KIND> struct SingKind;
template <> struct SingKind<0> { static constexpr int rows = 8, sums = 12; };
template <> struct SingKind<1> { static constexpr int rows = 13, sums = 30; };
template <> struct SingKind<2> { static constexpr int rows = 13, sums = 34; };

// hat-table rows of a kind from its rule, value-major (row r of point p at
// [r npts + p]): the coordinates the distance needs, then the weights times
// the monomials of the moments
static std::vector<double> singular_table(int kind, int n_ss, int& npts) {
  std::vector<double> pts;
  sauter_schwab_hat(kind, n_ss, pts);
  npts = int(pts.size() / 5);
  const int rows = kind == 0 ? SingKind<0>::rows : SingKind<1>::rows;
  std::vector<double> t(size_t(rows) * npts);
  for (int p = 0; p < npts; ++p) {
    const double x1 = pts[5 * p], x2 = pts[5 * p + 1], y1 = pts[5 * p + 2], y2 = pts[5 * p + 3], w = pts[5 * p + 4];
    std::vector<double> v;
    if (kind == 0)
      v = {x1 - y1, x2 - y2, 2 * w, w * (x1 + y1), w * (x2 + y2), 2 * w * x1 * y1, 2 * w * x2 * y2, w * (x1 * y2 + x2 * y1)};
    else if (kind == 1)
      v = {x1 - y1, x2, y2, w, w * x1, w * x2, w * y1, w * y2, w * x1 * y1, w * x1 * y2, w * x2 * y1, w * x2 * y2,
           w * (x1 - y1)};
    else
      v = {x1, x2, y1, y2, w, w * x1, w * x2, w * y1, w * y2, w * x1 * y1, w * x1 * y2, w * x2 * y1, w * x2 * y2};
    for (int r = 0; r < rows; ++r) t[size_t(r) * npts + p] = v[size_t(r)];
  }
  return t;
}

template <int KIND, class OutT>
__global__ void __launch_bounds__(128) k_singular64(BlockArgs A, const SingPair* __restrict__ sp, int64_t npairs,
                                                    const double* __restrict__ tab, int npts,
                                                    const __grid_constant__ SingRadial R, OutT* __restrict__ TK) {
  constexpr int NS = SingKind<KIND>::sums;
  __shared__ double sums[8][NS];
  const int slot = threadIdx.x >> 4, lane = threadIdx.x & 15;
  const int64_t w = int64_t(blockIdx.x) * 8 + slot;
  const SingPair P = sp[min(w, npairs - 1)];  // the tail repeats the last pair (not stored)
  const int64_t qt = P.tau, qs = P.sig;
  const double* vt = A.bt_v + 9 * qt;
  const double* vs = A.bt_v + 9 * qs;
  const double* t0 = vt + 3 * ((P.code >> 2) & 3);
  const double* t1 = vt + 3 * ((P.code >> 4) & 3);
  const double* t2 = vt + 3 * ((P.code >> 6) & 3);
  const double* s0 = vs + 3 * ((P.code >> 8) & 3);
  const double* s1 = vs + 3 * ((P.code >> 10) & 3);
  const double* s2 = vs + 3 * ((P.code >> 12) & 3);
  // x = P0 + x1 e1 + x2 e2, y = P0 + y1 f1 + y2 f2 (P0 shared for every kind)
  double e1[3], e2[3], f1[3], f2[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    e1[c] = t1[c] - t0[c];
    e2[c] = t2[c] - t1[c];
    f1[c] = s1[c] - s0[c];
    f2[c] = s2[c] - s1[c];
  }
  const double k = A.k[2 * P.block], k2 = k * k;
  // steps of the series: kappa is at most k times the largest vertex distance
  float zmax = 0.f;
  if (lane < 9) {
    const double* a = vt + 3 * (lane / 3);
    const double* b = vs + 3 * (lane % 3);
    const double d[3] = {a[0] - b[0], a[1] - b[1], a[2] - b[2]};
    zmax = float(k2 * dot3(d, d)) * 1.0001f;
  }
  zmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(zmax)));
  const int deg = zmax <= 0.0625f ? 6 : zmax <= 0.25f ? 7 : zmax <= 1.f ? 9 : zmax <= 2.25f ? 10 : 12;
  const bool series = zmax <= 4.f;

  double acc[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) acc[q] = 0.0;
  for (int p = lane; p < npts; p += 16) {
    const double* tp = tab + p;
    double d[3];
    if (KIND == 0) {
      const double u = tp[0], v = tp[npts];
#pragma unroll
      for (int c = 0; c < 3; ++c) d[c] = fma(u, e1[c], v * e2[c]);
    } else if (KIND == 1) {
      const double u = tp[0], x2 = tp[npts], y2 = tp[2 * npts];
#pragma unroll
      for (int c = 0; c < 3; ++c) d[c] = fma(u, e1[c], fma(x2, e2[c], -(y2 * f2[c])));
    } else {
      const double x1 = tp[0], x2 = tp[npts], y1 = tp[2 * npts], y2 = tp[3 * npts];
#pragma unroll
      for (int c = 0; c < 3; ++c) d[c] = fma(x1, e1[c], x2 * e2[c]) - fma(y1, f1[c], y2 * f2[c]);
    }
    const double r2 = dot3(d, d);
    const double ri = rsqrt_h(r2), ri2 = ri * ri;
    const double z = k2 * r2;
    double v[8];  // P_1..P_4, S_2..S_5
    if (series) {
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = R.c[deg][j];
#pragma unroll 1
      for (int t = deg - 1; t >= 0; --t)
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = fma(v[j], z, R.c[t][j]);
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = 0.0;
      const double kap = k * (r2 * ri);
#pragma unroll 1
      for (int q = 0; q < R.n; ++q) {
        const double x = R.xi[q], a = kap * x;
        double sn, cs;
        sincos(a, &sn, &cs);
        sn = a > 0.0 ? sn / a : 1.0;
        double wq = R.gw[q] * x;
        v[0] = fma(wq, cs, v[0]);
#pragma unroll
        for (int j = 1; j < 4; ++j) {
          wq *= x;
          v[j] = fma(wq, cs, v[j]);
          v[3 + j] = fma(wq, sn, v[3 + j]);
        }
        v[7] = fma(wq * x, sn, v[7]);
      }
    }
    // G moments of degree 0, 1, 2 (the imaginary parts without their factor k)
    const double Gr[3] = {ri * v[1], ri * v[2], ri * v[3]}, Gi[3] = {v[5], v[6], v[7]};
    const double* wt = tp + size_t(KIND == 0 ? 2 : KIND == 1 ? 3 : 4) * npts;
#pragma unroll
    for (int q = 0; q < (KIND == 0 ? 6 : 9); ++q) {
      const int m = q == 0 ? 0 : q <= (KIND == 0 ? 2 : 4) ? 1 : 2;
      const double ww = wt[size_t(q) * npts];
      acc[2 * q] = fma(ww, Gr[m], acc[2 * q]);
      acc[2 * q + 1] = fma(ww, Gi[m], acc[2 * q + 1]);
    }
    if (KIND != 0) {
      // g moments of degree 1, 2 (minus the real part; im without k)
      const double g1r = ri * fma(ri2, v[0], k2 * v[5]), g1i = ri2 * (v[1] - v[4]);
      const double g2r = ri * fma(ri2, v[1], k2 * v[6]), g2i = ri2 * (v[2] - v[5]);
      // edge: u, x2, y2, x1 y2, x2 y1, x2 y2; vertex: x1, x2, y1, y2, x_i y_j
      constexpr int ng = KIND == 1 ? 6 : 8;
#pragma unroll
      for (int q = 0; q < ng; ++q) {
        const int row = KIND == 1 ? (q == 0 ? 9 : q == 1 ? 2 : q == 2 ? 4 : 3 + q) : 1 + q;
        const bool first = q < (KIND == 1 ? 3 : 4);
        const double ww = wt[size_t(row) * npts];
        acc[18 + 2 * q] = fma(ww, first ? g1r : g2r, acc[18 + 2 * q]);
        acc[18 + 2 * q + 1] = fma(ww, first ? g1i : g2i, acc[18 + 2 * q + 1]);
      }
    }
  }
  int base = 0, count = NS;
  halve_sum<NS>(acc, lane, 8, base, count);
#pragma unroll
  for (int q = 0; q < (NS + 15) / 16; ++q)
    if (q < count) sums[slot][base + q] = acc[q];
  __syncwarp();
  if (lane >= 9 || w >= npairs) return;
  // entry (a, b) of the 3 x 3 block: v_a = P0 + al1 e1 + al2 e2 and u_b =
  // P0 + be1 f1 + be2 f2 with (0, 0), (1, 0), (1, 1) for the vertices in rule order
  const double* S = sums[slot];
  const int a = lane / 3, b = lane % 3;
  const double al[2] = {a > 0 ? 1.0 : 0.0, a > 1 ? 1.0 : 0.0}, be[2] = {b > 0 ? 1.0 : 0.0, b > 1 ? 1.0 : 0.0};
  // sums of G: 1 | x_i | y_j | x_i y_j
  auto G = [&](int q, int c) { return S[2 * q + c]; };
  const double ef[4] = {dot3(e1, f1), dot3(e1, f2), dot3(e2, f1), dot3(e2, f2)};
  double X[2] = {0.0, 0.0};  // sum G (x - v_a) . (y - u_b)
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const double mx = G(1 + i, c);
        const double my = KIND == 0 ? G(1 + j, c) : G(3 + j, c);
        const double mxy = KIND == 0 ? (i == j ? G(3 + i, c) : G(5, c)) : G(5 + 2 * i + j, c);
        X[c] = fma(ef[2 * i + j], mxy - be[j] * mx - al[i] * (my - be[j] * G(0, c)), X[c]);
      }
  const int pa = (P.code >> (2 + 2 * a)) & 3, pb = (P.code >> (8 + 2 * b)) & 3;
  const double cc = 4.0 * INV_FOUR_PI * A.bt_area[qt] * A.bt_area[qs] * A.bt_c[3 * qt + pa] * A.bt_c[3 * qs + pb];
  // T = -i k X - 4 / (i k) S0
  const C2 Tv{cc * fma(k2, X[1], -4.0 * G(0, 1)), cc * (4.0 / k * G(0, 0) - k * X[0])};
  C2 Kv{0.0, 0.0};
  if (KIND != 0) {
    // K_ab = -c_a c_b (v_a - u_b) . sum g (y - u_b) x (x - v_a)
    double s[2] = {0.0, 0.0}, t[3];
    auto g = [&](int q, int c) { return S[18 + 2 * q + c]; };
    if (KIND == 1) {
      cross3(e1, e2, t);
      const double A2 = dot3(t, f2);  // f1 = e1
#pragma unroll
      for (int c = 0; c < 2; ++c)
        s[c] = A2 * (al[1] * g(3, c) - be[1] * g(4, c) + (be[0] - al[0]) * g(5, c) - al[1] * be[1] * g(0, c) +
                     al[0] * be[1] * g(1, c) - al[1] * be[0] * g(2, c));
    } else {
      cross3(e1, e2, t);
      const double A1 = dot3(t, f1), A2 = dot3(t, f2);
      cross3(f1, f2, t);
      const double B1 = dot3(t, e1), B2 = dot3(t, e2);
      const double V[4] = {al[1] * A1 + be[1] * B1, al[1] * A2 - be[0] * B1, be[1] * B2 - al[0] * A1,
                           -(al[0] * A2 + be[0] * B2)};
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int c = 0; c < 2; ++c)
            s[c] = fma(V[2 * i + j], g(4 + 2 * i + j, c) - be[j] * g(i, c) - al[i] * g(2 + j, c), s[c]);
    }
    Kv = C2{cc * s[0], -cc * k * s[1]};
  }
  const int N = A.blk_N[P.block];
  const int64_t ra = A.bt_dof[3 * qt + pa], cb = A.bt_dof[3 * qs + pb];
  // upper position (k_mirror fills the lower one).  Both orderings of an
  // adjacent pair have this value at transposed positions: once here, twice on
  // the diagonal; a coincident pair holds every (a, b) with (b, a) itself.
  const int64_t mat = A.blk_mat_off[P.block];
  if (KIND == 0) {
    if (ra <= cb) add_entry(TK, mat + ra * N + cb, Tv, Kv);
  } else {
    const double two = ra == cb ? 2.0 : 1.0;
    add_entry(TK, mat + (ra < cb ? ra * N + cb : cb * N + ra), cscale(Tv, two), cscale(Kv, two));
  }
}

// the three kinds of the mesh's singular pairs (sorted by kind)
template <class OutT>
static void launch_singular(mtf_system sys, const BlockArgs& A, OutT* TK, cudaStream_t s) {
  mtf_mesh m = sys->mesh;
  int64_t at = 0;  // the list is sorted by kind
  for (int kind = 0; kind < 3; ++kind) {
    int64_t end = at;
    while (end < int64_t(m->sing.size()) && (m->sing[size_t(end)].code & 3) == kind) ++end;
    const int64_t np = end - at;
    if (np > 0) {
      const unsigned g = unsigned((np + 7) / 8);
      auto go = [&](auto kernel) {
        MTF_LAUNCH(KID_SINGULAR64, s, kernel<<<g, 128, 0, s>>>(A, m->d_sing.p + at, np, sys->d_ss_pts[kind].p,
                                                               sys->ss_npts[kind], sys->ss_radial, TK));
      };
      if (kind == 0) go(k_singular64<0, OutT>);
      else if (kind == 1) go(k_singular64<1, OutT>);
      else go(k_singular64<2, OutT>);
    }
    at = end;
  }
}

// ---------------------------------------------------------------------------
// transmission Gram values (Eq. 18): one thread per exchange entry
//   G^{ij}[m, n] on triangle t = c_a^i c_b^j int_t n_i . ((x - v_a) x (x - v_b))
// ---------------------------------------------------------------------------
__global__ void k_exchange_values(const XEntry* __restrict__ xe, int64_t nent, const double* __restrict__ bt_v,
                                  const double* __restrict__ bt_c, const double* __restrict__ bt_area,
                                  const int8_t* __restrict__ bt_swap, double* __restrict__ xval) {
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= nent) return;
  const XEntry X = xe[e];
  const int a = X.ab & 3, b = (X.ab >> 2) & 3;
  const double* v = bt_v + 9 * int64_t(X.bt_i);
  double e1[3], e2[3], n[3];
  for (int c = 0; c < 3; ++c) {
    e1[c] = v[3 + c] - v[c];
    e2[c] = v[6 + c] - v[c];
  }
  n[0] = e1[1] * e2[2] - e1[2] * e2[1];
  n[1] = e1[2] * e2[0] - e1[0] * e2[2];
  n[2] = e1[0] * e2[1] - e1[1] * e2[0];
  const double nn = sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
  const double sw = bt_swap[X.bt_i] / nn;
  double acc = 0.0;
  for (int q = 0; q < 6; ++q) {
    double x[3], u[3], w[3];
    for (int c = 0; c < 3; ++c) {
      x[c] = v[c] + c_tri_s[q] * e1[c] + c_tri_t[q] * e2[c];
      u[c] = x[c] - v[3 * a + c];
      w[c] = x[c] - v[3 * b + c];
    }
    const double cr0 = u[1] * w[2] - u[2] * w[1], cr1 = u[2] * w[0] - u[0] * w[2],
                 cr2 = u[0] * w[1] - u[1] * w[0];
    acc += c_tri_w[q] * (n[0] * cr0 + n[1] * cr1 + n[2] * cr2);
  }
  xval[e] = 2.0 * bt_area[X.bt_i] * sw * acc * bt_c[3 * X.bt_i + a] * bt_c[3 * X.bt_j + b];
}

// ---------------------------------------------------------------------------
// incident data (Eq. 22): b_D = 2 int E_inc . psi, b_N = 2 int (d x p) e^{ik0 d.x} . psi
// on Gamma_0 (= -2 <gamma_.,0 E_inc, psi>_x); one thread per (dof of block 0, rhs)
// ---------------------------------------------------------------------------
__global__ void k_rhs(const int32_t* __restrict__ dof_bt, int N0, int nrhs, int64_t n_total,
                      const double* __restrict__ bt_v, const double* __restrict__ bt_c,
                      const double* __restrict__ bt_area, double k0, const double* __restrict__ dirs,
                      const double* __restrict__ pols, double* __restrict__ b) {
  const int64_t tid = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (tid >= int64_t(N0) * nrhs) return;
  const int m = int(tid % N0), col = int(tid / N0);
  const double* d = dirs + 3 * col;
  const double* P = pols + 6 * col;  // complex128 x 3
  const C2 p[3] = {{P[0], P[1]}, {P[2], P[3]}, {P[4], P[5]}};
  C2 dxp[3];
  dxp[0] = csub(cscale(p[2], d[1]), cscale(p[1], d[2]));
  dxp[1] = csub(cscale(p[0], d[2]), cscale(p[2], d[0]));
  dxp[2] = csub(cscale(p[1], d[0]), cscale(p[0], d[1]));
  C2 sE{0, 0}, sN{0, 0};
  for (int e = 0; e < 2; ++e) {
    const int code = dof_bt[2 * m + e];
    const int64_t q = code / 3;
    const int a = code % 3;
    const double* v = bt_v + 9 * q;
    const double ca = bt_c[3 * q + a], A2 = 2.0 * bt_area[q];
    for (int qp = 0; qp < 6; ++qp) {
      double x[3], f[3];
      for (int c = 0; c < 3; ++c) {
        x[c] = v[c] + c_tri_s[qp] * (v[3 + c] - v[c]) + c_tri_t[qp] * (v[6 + c] - v[c]);
        f[c] = ca * (x[c] - v[3 * a + c]);
      }
      double sn, cs;
      sincos(k0 * (d[0] * x[0] + d[1] * x[1] + d[2] * x[2]), &sn, &cs);
      const C2 ph{cs * A2 * c_tri_w[qp], sn * A2 * c_tri_w[qp]};
      C2 pe{0, 0}, pn{0, 0};
      for (int c = 0; c < 3; ++c) {
        pe = cadd(pe, cscale(p[c], f[c]));
        pn = cadd(pn, cscale(dxp[c], f[c]));
      }
      sE = cadd(sE, cmul(ph, pe));
      sN = cadd(sN, cmul(ph, pn));
    }
  }
  double* bc = b + 2 * (int64_t(col) * n_total);
  bc[2 * m] = 2.0 * sE.re;
  bc[2 * m + 1] = 2.0 * sE.im;
  bc[2 * (N0 + m)] = 2.0 * sN.re;
  bc[2 * (N0 + m) + 1] = 2.0 * sN.im;
}

template <class MatT>
__global__ void k_split_block(const MatT* __restrict__ TK, int64_t n, double* __restrict__ T,
                              double* __restrict__ K) {
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= n) return;
  T[2 * e] = TK[4 * e];
  T[2 * e + 1] = TK[4 * e + 1];
  K[2 * e] = TK[4 * e + 2];
  K[2 * e + 1] = TK[4 * e + 3];
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
static void upload_rule_constants(cudaStream_t s) {
  const TriRule& r = triangle_rule6();
  MTF_CUDA(cudaMemcpyToSymbolAsync(c_tri_s, r.s, sizeof(r.s), 0, cudaMemcpyHostToDevice, s));
  MTF_CUDA(cudaMemcpyToSymbolAsync(c_tri_t, r.t, sizeof(r.t), 0, cudaMemcpyHostToDevice, s));
  MTF_CUDA(cudaMemcpyToSymbolAsync(c_tri_w, r.w, sizeof(r.w), 0, cudaMemcpyHostToDevice, s));
  double orbit[2][3], point[6][3];
  for (int o = 0; o < 2; ++o) {
    const double w = r.w[3 * o], a = r.s[3 * o];
    orbit[o][0] = w;
    orbit[o][1] = w * a;
    orbit[o][2] = w * (1.0 - 3.0 * a);
  }
  for (int p = 0; p < 6; ++p) {
    point[p][0] = r.w[p];
    point[p][1] = r.w[p] * r.s[p];
    point[p][2] = r.w[p] * r.t[p];
  }
  MTF_CUDA(cudaMemcpyToSymbolAsync(c_orbit, orbit, sizeof(orbit), 0, cudaMemcpyHostToDevice, s));
  MTF_CUDA(cudaMemcpyToSymbolAsync(c_point, point, sizeof(point), 0, cudaMemcpyHostToDevice, s));
}

static BlockArgs block_args(mtf_system sys) {
  mtf_mesh m = sys->mesh;
  BlockArgs A;
  A.bt_v = m->d_bt_v.p;
  A.bt_c = m->d_bt_c.p;
  A.bt_area = m->d_bt_area.p;
  A.bt_dof = m->d_bt_dof.p;
  A.bt_vid = m->d_bt_vid.p;
  A.blk_T = m->d_blk_T.p;
  A.blk_N = m->d_blk_N.p;
  A.blk_bt_off = m->d_blk_bt_off.p;
  A.blk_mat_off = m->d_blk_mat_off.p;
  A.k = sys->d_k.p;
  A.nblk = m->nd;
  return A;
}

// v[k] -> out[k] = fl(v[k]), out[n + k] = fl(v[k] - fl(v[k]))
__global__ void k_split_pairs(const double* __restrict__ v, int64_t n, float* __restrict__ out) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= n) return;
  const double a = v[t];
  const float h = float(a);
  out[t] = h;
  out[n + t] = float(a - double(h));
}

// room for the rotated copy of the FP64 blocks, where it may be kept
static void alloc_rotated_copy(mtf_system sys) {
  if (sys->d_rot64.p || sys->rot64_off) return;
  const size_t n = size_t(sys->mesh->n_mat) * 4;
  static RotatedBudget budgets[64];  // per device
  int dev = 0;
  size_t free_bytes = 0, total_bytes = 0;
  MTF_CUDA(cudaGetDevice(&dev));
  MTF_CUDA(cudaMemGetInfo(&free_bytes, &total_bytes));
  sys->rot64_off = dev >= 64 || !rotated_copy_fits(n * sizeof(double), free_bytes) ||
                   !sys->rot64_share.take(budgets[dev], n * sizeof(double), total_bytes);
  if (sys->rot64_off) return;
  try {
    sys->d_rot64.alloc(n);
  } catch (const Error& e) {
    if (e.status != MTF_ERR_OOM) throw;
    cudaGetLastError();  // (the matvec does without)
    sys->d_rot64.p = nullptr;
    sys->rot64_share.give();
    sys->rot64_off = true;
  }
}

void launch_assemble(mtf_system sys, cudaStream_t s) {
  mtf_mesh m = sys->mesh;
  upload_rule_constants(s);
  // Sauter-Schwab tables (once per system)
  if (sys->ss_npts[0] == 0) {
    for (int kind = 0; kind < 3; ++kind) {
      const std::vector<double> tab = singular_table(kind, sys->opt.n_ss, sys->ss_npts[kind]);
      sys->d_ss_pts[kind].upload(tab, s);
      MTF_CUDA(cudaStreamSynchronize(s));
    }
    singular_radial(sys->opt.n_ss, sys->ss_radial);
  }
  BlockArgs A = block_args(sys);
  const bool fp64_blocks = sys->opt.precision == MTF_PREC_FP64 || sys->opt.residual_fp64;
  if (fp64_blocks) {
    sys->d_TK64.alloc(size_t(m->n_mat) * 4);
    MTF_CUDA(cudaMemsetAsync(sys->d_TK64.p, 0, size_t(m->n_mat) * 4 * sizeof(double), s));
    if (sys->opt.precision == MTF_PREC_FP64) alloc_rotated_copy(sys);
    const int64_t nct = m->reg_cta_prefix.back();
    MTF_LAUNCH(KID_REGULAR64, s, k_regular64<<<unsigned(nct), 128, 0, s>>>(A, m->d_reg_cta_prefix.p, sys->d_TK64.p));
    launch_singular(sys, A, sys->d_TK64.p, s);
    MTF_LAUNCH(KID_MIRROR, s, k_mirror<Entry64><<<unsigned(m->mirror_cta_prefix.back()), 256, 0, s>>>(
        reinterpret_cast<Entry64*>(sys->d_TK64.p), m->d_mirror_cta_prefix.p, m->nd, m->d_blk_N.p, m->d_blk_mat_off.p,
        nullptr, reinterpret_cast<Entry64*>(sys->d_rot64.p)));
  }
  if (fp64_blocks && sys->opt.precision != MTF_PREC_FP64) {
    // residual_fp64: the FP64 entries split into FP32 pairs once per assembly,
    // for the double-float residual matvec
    const int64_t nv = m->n_mat * 4;
    sys->d_TK64hl.alloc(size_t(nv) * 2);
    MTF_LAUNCH(KID_MISC, s, k_split_pairs<<<unsigned((nv + 255) / 256), 256, 0, s>>>(sys->d_TK64.p, nv,
                                                                                     sys->d_TK64hl.p));
  }
  if (sys->opt.precision != MTF_PREC_FP64) {
    // mixed: FP32 storage; regular pairs in FP32, singular pairs in FP64
    sys->d_TK32.alloc(size_t(m->n_mat) * 4);
    MTF_CUDA(cudaMemsetAsync(sys->d_TK32.p, 0, size_t(m->n_mat) * 4 * sizeof(float), s));
    launch_assemble_regular32(sys, s);
    launch_singular(sys, A, sys->d_TK32.p, s);
    MTF_LAUNCH(KID_MIRROR, s, k_mirror<float4><<<unsigned(m->mirror_cta_prefix.back()), 256, 0, s>>>(
        reinterpret_cast<float4*>(sys->d_TK32.p), m->d_mirror_cta_prefix.p, m->nd, m->d_blk_N.p, m->d_blk_mat_off.p,
        sys->opt.mv_tensor ? tc_operator_amax(sys, s) : nullptr, nullptr));
    if (sys->opt.mv_tensor) tc_build_operator(sys, s);
    else tile_matvec_operator(sys, s);
  }
  launch_exchange_values(sys, s);
}

__global__ void k_d2f(const double* __restrict__ a, int64_t n, float* __restrict__ out) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t < n) out[t] = float(a[t]);
}

void launch_exchange_values(mtf_system sys, cudaStream_t s) {
  mtf_mesh m = sys->mesh;
  const int64_t nent = m->n_rows * 6;
  sys->d_xval.alloc(size_t(nent));
  MTF_LAUNCH(KID_XVALUES, s, k_exchange_values<<<unsigned((nent + 255) / 256), 256, 0, s>>>(
      m->d_xent.p, nent, m->d_bt_v.p, m->d_bt_c.p, m->d_bt_area.p, m->d_bt_swap.p, sys->d_xval.p));
  // FP32 copy for the FP32 epilogues of the mixed inner solver
  sys->d_xval32.alloc(size_t(nent));
  MTF_LAUNCH(KID_XVALUES, s, k_d2f<<<unsigned((nent + 255) / 256), 256, 0, s>>>(sys->d_xval.p, nent, sys->d_xval32.p));
}

void launch_rhs(mtf_system sys, int nrhs, const double* d_dirs, const double* d_pols, double* b,
                cudaStream_t s) {
  mtf_mesh m = sys->mesh;
  upload_rule_constants(s);
  MTF_CUDA(cudaMemsetAsync(b, 0, size_t(m->n_total) * nrhs * 2 * sizeof(double), s));
  const int N0 = m->blk[0].N;
  const int64_t nth = int64_t(N0) * nrhs;
  MTF_LAUNCH(KID_RHS, s, k_rhs<<<unsigned((nth + 127) / 128), 128, 0, s>>>(m->d_dof_bt.p, N0, nrhs, m->n_total, m->d_bt_v.p,
                                                      m->d_bt_c.p, m->d_bt_area.p, sys->k0, d_dirs, d_pols, b));
  MTF_CUDA(cudaGetLastError());
}

void launch_get_block(mtf_system sys, int i, double* t_out, double* k_out, cudaStream_t s) {
  mtf_mesh m = sys->mesh;
  const int64_t n = int64_t(m->blk[i].N) * m->blk[i].N;
  if (sys->opt.precision == MTF_PREC_FP64) {
    const double* src = sys->d_TK64.p + 4 * m->blk[i].mat_off;
    MTF_LAUNCH(KID_SPLIT, s, k_split_block<double><<<unsigned((n + 255) / 256), 256, 0, s>>>(src, n, t_out, k_out));
  } else {
    const float* src = sys->d_TK32.p + 4 * m->blk[i].mat_off;
    MTF_LAUNCH(KID_SPLIT, s, k_split_block<float><<<unsigned((n + 255) / 256), 256, 0, s>>>(src, n, t_out, k_out));
  }
  MTF_CUDA(cudaGetLastError());
}

}  // namespace mtf
