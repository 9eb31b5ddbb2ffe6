// Mixed-precision assembly of the regular (vertex-disjoint) triangle pairs.
//
// Same Galerkin integrals as k_regular64 (Eqs. 7-9 tested with Eq. 5), with
// the Helmholtz kernel evaluated in FP32 except for what FP32 cannot carry.
// With centroids o_tau, o_sigma (FP64), Delta = o_tau - o_sigma, R0 the FP32
// number next to |Delta| and dR2 = |Delta|^2 - R0^2, every point pair has
// r = R0 + dr with
//   dr = (2 Delta.e + e.e + dR2) / (r + R0),   e = x' - y'  (local offsets),
// which is free of cancellation, and
//   exp(i k r) = exp(i k R0) exp(i k dr).
// The per-pair factor exp(i k R0) is formed from an FP64 phase reduced modulo
// 2 pi, the per-point factor exp(i k dr) from the Taylor series of sin and cos
// (|k dr| is bounded by k times the pair's radii; larger arguments fall back
// to sincosf).  Kernel sums are accumulated in FP32 and rotated by
// exp(i k R0) once per pair.
#include <cmath>

#include "common.h"
#include "pair_tile.cuh"

namespace mtf {

// the 6-point rule (own copy in this translation unit)
__constant__ double c_tri_s[6], c_tri_t[6];
// its orbits (a, a, 1 - 2a): w, w (a - 1/3), w (1 - 3a); its points: w,
// w (s - 1/3), w (t - 1/3)
__constant__ float c_orbit32[2][3], c_point32[6][3];

#define INV_SQRT_FOUR_PI 0.28209479177387814347
#define TWO_PI_D 6.283185307179586476925
#define INV_TWO_PI_D 0.159154943091895335769

// sin and cos from their Taylor series (coefficients (-1)^j / (2j+1)! and
// (-1)^j / (2j)!).  NARROW: |x| <= 0.5, 3 and 4 terms beyond the first
// (truncation 6e-9 and 3e-10); otherwise |x| <= 1.6, 6 and 7 terms (below 1e-9).
template <bool NARROW>
__device__ __forceinline__ void sincos_taylor(float x, float* s, float* c) {
  const float x2 = x * x;
  float s_, c_;
  if (NARROW) {
    s_ = -1.0f / 5040.0f;
    c_ = 1.0f / 40320.0f;
  } else {
    s_ = 1.0f / 6227020800.0f;
    s_ = fmaf(s_, x2, -1.0f / 39916800.0f);
    s_ = fmaf(s_, x2, 1.0f / 362880.0f);
    s_ = fmaf(s_, x2, -1.0f / 5040.0f);
    c_ = -1.0f / 87178291200.0f;
    c_ = fmaf(c_, x2, 1.0f / 479001600.0f);
    c_ = fmaf(c_, x2, -1.0f / 3628800.0f);
    c_ = fmaf(c_, x2, 1.0f / 40320.0f);
  }
  s_ = fmaf(s_, x2, 1.0f / 120.0f);
  s_ = fmaf(s_, x2, -1.0f / 6.0f);
  s_ = s_ * x2;
  *s = fmaf(s_, x, x);
  c_ = fmaf(c_, x2, -1.0f / 720.0f);
  c_ = fmaf(c_, x2, 1.0f / 24.0f);
  c_ = fmaf(c_, x2, -0.5f);
  *c = fmaf(c_, x2, 1.0f);
}

// a / b for b > 0 in the normal range: the approximate reciprocal with one
// residual correction
__device__ __forceinline__ float div_corr(float a, float b) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(b));
  const float q = a * r;
  return fmaf(fmaf(-q, b, a), r, q);
}

__device__ __forceinline__ float dot3f(const float* a, const float* b) { return fmaf(a[0], b[0], fmaf(a[1], b[1], a[2] * b[2])); }
__device__ __forceinline__ void cross3f(const float* a, const float* b, float* c) {
  c[0] = fmaf(a[1], b[2], -(a[2] * b[1]));
  c[1] = fmaf(a[2], b[0], -(a[0] * b[2]));
  c[2] = fmaf(a[0], b[1], -(a[1] * b[0]));
}

// Per block-triangle geometry relative to the centroid (FP64): quadrature
// points (6x3), vertices (3x3) and the edges from vertex 0 (2x3), RWG c_a 2 A / sqrt(4 pi) (3) and the largest
// vertex distance in FP32.  The RWG factors scale whole rows and columns, and
// on structured meshes their rounding is the same everywhere: they carry their
// residues (K of a cube of 8 x 8 squares per face: error 1.7e-7 without, 7e-8
// with them), and the rule's weight sum in FP32 over the exact one, 7e-9 that
// every entry would share.
struct Geom32Args {
  const double* bt_v;
  const double* bt_c;
  const double* bt_area;
  int64_t n_bt;
  double wsum;   // sum of the FP32 weights over the exact sum
  double* cen;   // 3 per bt
  float* qx;     // 18 per bt
  float* pv;     // 24 per bt: vertices, v_1 - v_0, v_2 - v_0, the vertices' rounding
  float* cc;     // 8 per bt: c_a 2 A / sqrt(4 pi) (3), radius, the residues of the first three
};

__global__ void k_geom32(Geom32Args G) {
  const int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (q >= G.n_bt) return;
  const double* v = G.bt_v + 9 * q;
  double o[3];
  for (int c = 0; c < 3; ++c) o[c] = (v[c] + v[3 + c] + v[6 + c]) * (1.0 / 3.0);
  for (int c = 0; c < 3; ++c) G.cen[3 * q + c] = o[c];
  for (int p = 0; p < 6; ++p)
    for (int c = 0; c < 3; ++c)
      G.qx[18 * q + 3 * p + c] =
          float(v[c] - o[c] + c_tri_s[p] * (v[3 + c] - v[c]) + c_tri_t[p] * (v[6 + c] - v[c]));
  float rad = 0.f;
  for (int a = 0; a < 3; ++a) {
    float d2 = 0.f;
    for (int c = 0; c < 3; ++c) {
      const float d = float(v[3 * a + c] - o[c]);
      G.pv[24 * q + 3 * a + c] = d;
      if (a > 0) G.pv[24 * q + 6 + 3 * a + c] = float(v[3 * a + c] - v[c]);
      G.pv[24 * q + 15 + 3 * a + c] = float(v[3 * a + c] - o[c] - double(d));
      d2 = fmaf(d, d, d2);
    }
    rad = fmaxf(rad, d2);
    const double ca = G.bt_c[3 * q + a] * (2.0 * INV_SQRT_FOUR_PI * G.bt_area[q]) / G.wsum;
    G.cc[8 * q + a] = float(ca);
    G.cc[8 * q + 4 + a] = float(ca - double(float(ca)));
  }
  G.cc[8 * q + 3] = sqrtf(rad) * 1.0001f;
  G.cc[8 * q + 7] = 0.f;
}

struct Reg32Args {
  const double* cen;
  const float* qx;
  const float* pv;
  const float* cc;
  const int32_t* bt_dof;
  const int32_t* bt_vid;
  const int32_t* blk_T;
  const int32_t* blk_N;
  const int64_t* blk_bt_off;
  const int64_t* blk_mat_off;
  const double* k;
  const float4* k32;  // per block: k, its residue, -4 / k^2, its residue
  int nblk;
};

// triangles of one side of a tile (value-major, so that lanes read
// consecutive words)
struct Side32 {
  double cen[3][kPairTile];
  float x[18][kPairTile], v[24][kPairTile], c[8][kPairTile];
  int dof[3][kPairTile], vid[3][kPairTile];
};

__device__ __forceinline__ void load_side(const Reg32Args& A, int64_t first, int n, Side32& S) {
  for (int t = threadIdx.x; t < n * 18; t += 128) S.x[t % 18][t / 18] = A.qx[18 * first + t];
  for (int t = threadIdx.x; t < n * 24; t += 128) S.v[t % 24][t / 24] = A.pv[24 * first + t];
  for (int t = threadIdx.x; t < n * 8; t += 128) S.c[t % 8][t / 8] = A.cc[8 * first + t];
  for (int t = threadIdx.x; t < n * 3; t += 128) {
    S.cen[t % 3][t / 3] = A.cen[3 * first + t];
    S.dof[t % 3][t / 3] = A.bt_dof[3 * first + t];
    S.vid[t % 3][t / 3] = A.bt_vid[3 * first + t];
  }
}

// the 3 kernel values of one orbit of y points: re, im of G 4 pi exp(-i k r0)
// and of -g
template <bool NARROW>
__device__ __forceinline__ void orbit_values(const float (*yx)[kPairTile], int b, const float* xp, const float* D,
                                             float R0, float dR2, float k, bool wide, float (*v)[4]) {
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const float e0 = xp[0] - yx[3 * e][b], e1 = xp[1] - yx[3 * e + 1][b], e2 = xp[2] - yx[3 * e + 2][b];
    const float u = fmaf(fmaf(2.0f, D[0], e0), e0, fmaf(fmaf(2.0f, D[1], e1), e1, fmaf(fmaf(2.0f, D[2], e2), e2, dR2)));
    const float t2 = fmaf(R0, R0, u);  // r^2
    const float ri = rsqrtf(t2);
    const float ph = k * div_corr(u, fmaf(t2, ri, R0));  // k (r - r0)
    float sn, cs;
    if (NARROW || !wide) sincos_taylor<NARROW>(ph, &sn, &cs);
    else sincosf(ph, &sn, &cs);
    v[e][0] = ri * cs;
    v[e][1] = ri * sn;
    const float al = k * ri, be = ri * ri;  // -g = G (1/r - i k) / r
    v[e][2] = fmaf(be, v[e][0], al * v[e][1]);
    v[e][3] = fmaf(be, v[e][1], -(al * v[e][0]));
  }
}

// Regular pairs of the mixed path: one thread per unordered pair, CTAs over
// 16 x 16 tiles of a block's triangles, added at the upper position as
// k_regular64 does (the same moments, about the centroids).  Bounds:
// FP32 issue, then the FP32x4 atomics (9 per pair).  Measured on the 2 x 2 x 2
// cube (22.5 M ordered pairs): 3.53 -> 1.42 ms.
__global__ void __launch_bounds__(128, 4) k_regular32(Reg32Args A, const int64_t* __restrict__ cta_prefix,
                                                      float* __restrict__ TK) {
  __shared__ Side32 X, Y;
  const PairTile P = pair_tile(blockIdx.x, cta_prefix, A.nblk);
  const int i = P.blk, T = A.blk_T[i];
  load_side(A, A.blk_bt_off[i] + P.t0, min(kPairTile, T - P.t0), X);
  load_side(A, A.blk_bt_off[i] + P.s0, min(kPairTile, T - P.s0), Y);
  __syncthreads();
  const double kr = A.k[2 * i];
  const float4 k32 = A.k32[i];
  const float k = k32.x;
  const int N = A.blk_N[i];
  float4* M = reinterpret_cast<float4*>(TK) + A.blk_mat_off[i];
  const int b = threadIdx.x & (kPairTile - 1);
#pragma unroll 1
  for (int a = threadIdx.x / kPairTile; a < kPairTile; a += 128 / kPairTile) {
    bool live = P.t0 + a < P.s0 + b && P.s0 + b < T;
    if (live) {
      bool shared = false;
#pragma unroll
      for (int p = 0; p < 3; ++p)
#pragma unroll
        for (int q = 0; q < 3; ++q) shared |= X.vid[p][a] == Y.vid[q][b];
      live = !shared;
    }
    // |k (r - r0)| is at most k times the two radii
    float ext = live ? k * (X.c[3][a] + Y.c[3][b]) : 0.f;
    ext = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(ext)));
    if (!live) continue;
    // ---- FP64 per-pair part: Delta, |Delta|^2 - R0^2 and exp(i k R0) for the
    // FP32 number R0 next to |Delta|; the rounding of the reduced phase to
    // FP32 is put back to first order
    const double dD0 = X.cen[0][a] - Y.cen[0][b], dD1 = X.cen[1][a] - Y.cen[1][b], dD2 = X.cen[2][a] - Y.cen[2][b];
    const double R2 = fma(dD0, dD0, fma(dD1, dD1, dD2 * dD2));
    const float R0 = sqrtf(float(R2));
    const float dR2 = float(fma(-double(R0), double(R0), R2));
    const double ph = kr * double(R0), phr = ph - TWO_PI_D * rint(ph * INV_TWO_PI_D);
    const float ph_hi = float(phr), ph_lo = float(phr - double(ph_hi));
    float s0, c0;
    sincosf(ph_hi, &s0, &c0);
    const float s0r = s0;
    s0 = fmaf(ph_lo, c0, s0);
    c0 = fmaf(-ph_lo, s0r, c0);
    const float D[3] = {float(dD0), float(dD1), float(dD2)};

    float G[3][3][2], H[3][3][2];  // [1, s - 1/3, t - 1/3 of x][the same of y] (re, im)
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int q = 0; q < 3; ++q) G[p][q][0] = G[p][q][1] = H[p][q][0] = H[p][q][1] = 0.f;
#pragma unroll 1
    for (int p = 0; p < 6; ++p) {
      const float xp[3] = {X.x[3 * p][a], X.x[3 * p + 1][a], X.x[3 * p + 2][a]};
      float m[3][4], bc[4];
#pragma unroll
      for (int f = 0; f < 4; ++f) m[0][f] = m[1][f] = m[2][f] = bc[f] = 0.f;
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        float v[3][4];
        if (ext <= 0.5f) orbit_values<true>(Y.x + 9 * o, b, xp, D, R0, dR2, k, false, v);
        else orbit_values<false>(Y.x + 9 * o, b, xp, D, R0, dR2, k, ext > 1.6f, v);
        const float w = c_orbit32[o][0], wa = c_orbit32[o][1], wc = c_orbit32[o][2];
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          const float sum = v[0][f] + v[1][f] + v[2][f];
          m[0][f] = fmaf(w, sum, m[0][f]);
          bc[f] = fmaf(wa, sum, bc[f]);
          m[1][f] = fmaf(wc, v[1][f], m[1][f]);
          m[2][f] = fmaf(wc, v[2][f], m[2][f]);
        }
      }
      const float wx[3] = {c_point32[p][0], c_point32[p][1], c_point32[p][2]};
#pragma unroll
      for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          const float t = q == 0 ? m[0][f] : m[q][f] + bc[f];
#pragma unroll
          for (int r = 0; r < 3; ++r) {
            float& dst = f < 2 ? G[r][q][f] : H[r][q][f - 2];
            dst = fmaf(wx[r], t, dst);
          }
        }
    }
    // rotate every moment by exp(i k R0), those of G by k exp(i k R0)
    const float ck0 = fmaf(c0, k, c0 * k32.y), sk0 = fmaf(s0, k, s0 * k32.y);
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const float gr = G[p][q][0], hr = H[p][q][0];
        G[p][q][0] = gr * ck0 - G[p][q][1] * sk0;
        G[p][q][1] = gr * sk0 + G[p][q][1] * ck0;
        H[p][q][0] = hr * c0 - H[p][q][1] * s0;
        H[p][q][1] = hr * s0 + H[p][q][1] * c0;
      }
    // With x' = x - o_tau, y' = y - o_sigma (centroids), p_a = v_a - o_tau,
    // q_b = u_b - o_sigma and the vector moments Sx = sum G x', Hx = sum H x',
    // Hc = sum H x' x y' (H = -g):
    //   X_ab = Sxy - p_a . Sy - q_b . (Sx - p_a S0)
    //   K_ab / (c_a c_b) = kap_a - q_b . Lam_a,  A = D + p_a,
    //   U_a = -Hc - Hy x p_a,  R_a = Hx - H0 p_a,  kap_a = A . U_a,  Lam_a = U_a + R_a x A
    // (moments about the centroids: the FP32 combinations lose little; on
    // structured meshes the rounding of p_a and q_b is the same for every
    // triangle and adds up, so K's leading term H0 D . (q_b x p_a) takes its
    // residue too)
    float E[2][3], F[2][3], q3[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      E[0][c] = X.v[9 + c][a];
      E[1][c] = X.v[12 + c][a];
      F[0][c] = Y.v[9 + c][b];
      F[1][c] = Y.v[12 + c][b];
#pragma unroll
      for (int q = 0; q < 3; ++q) q3[q][c] = Y.v[3 * q + c][b];
    }
    const float Q0[2] = {fmaf(k32.z, G[0][0][0], k32.w * G[0][0][0]), fmaf(k32.z, G[0][0][1], k32.w * G[0][0][1])};
    float Sx[3][2], Sy[3][2], Hx[3][2], Hy[3][2], Hc[3][2], Sxy[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      Sxy[c] = 0.f;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        Sx[d][c] = fmaf(E[0][d], G[1][0][c], E[1][d] * G[2][0][c]);
        Sy[d][c] = fmaf(F[0][d], G[0][1][c], F[1][d] * G[0][2][c]);
        Hx[d][c] = fmaf(E[0][d], H[1][0][c], E[1][d] * H[2][0][c]);
        Hy[d][c] = fmaf(F[0][d], H[0][1][c], F[1][d] * H[0][2][c]);
        Hc[d][c] = 0.f;
      }
    }
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float t3[3];
        cross3f(E[p], F[q], t3);
        const float ef = dot3f(E[p], F[q]);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          Sxy[c] = fmaf(ef, G[1 + p][1 + q][c], Sxy[c]);
#pragma unroll
          for (int d = 0; d < 3; ++d) Hc[d][c] = fmaf(t3[d], H[1 + p][1 + q][c], Hc[d][c]);
        }
      }
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      float pa[3], A3[3], base[2], kap[2], B3[3][2], L3[3][2];
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        pa[d] = X.v[3 * p + d][a];
        A3[d] = D[d] + pa[d];
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const float sy[3] = {Sy[0][c], Sy[1][c], Sy[2][c]}, hy[3] = {Hy[0][c], Hy[1][c], Hy[2][c]};
        base[c] = Sxy[c] - dot3f(pa, sy);
        float U[3], R[3], t[3];
        cross3f(hy, pa, U);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          B3[d][c] = fmaf(-pa[d], G[0][0][c], Sx[d][c]);
          U[d] = -Hc[d][c] - U[d];
          R[d] = fmaf(-X.v[15 + 3 * p + d][a], H[0][0][c], fmaf(-pa[d], H[0][0][c], Hx[d][c]));
        }
        kap[c] = dot3f(A3, U);
        cross3f(R, A3, t);
#pragma unroll
        for (int d = 0; d < 3; ++d) L3[d][c] = U[d] + t[d];
      }
      const int mrow = X.dof[p][a];
      const float cp = X.c[p][a], cpl = X.c[4 + p][a];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        float xc[2], kk[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          xc[c] = base[c] - fmaf(q3[q][0], B3[0][c], fmaf(q3[q][1], B3[1][c], q3[q][2] * B3[2][c]));
          kk[c] = kap[c] - fmaf(q3[q][0], L3[0][c], fmaf(q3[q][1], L3[1][c], q3[q][2] * L3[2][c]));
          kk[c] -= fmaf(Y.v[15 + 3 * q][b], L3[0][c], fmaf(Y.v[16 + 3 * q][b], L3[1][c], Y.v[17 + 3 * q][b] * L3[2][c]));
        }
        // c_a c_b = cc + cl; T = -i c_a c_b (k X - 4 / k S0): the S0 term is the
        // large one, and combinations without divergence cancel it, but not the
        // entries' own roundings.  So it is rounded once per pair (Q0) and each
        // entry once, at the end (with S0 at the head of X's sums: T 2.9e-7
        // and a solve near a resonance 4.7e-6, so 2.3e-7 and 4.2e-6)
        const float cq = Y.c[q][b], cc = cp * cq, cl = fmaf(cp, cq, -cc) + fmaf(cp, Y.c[4 + q][b], cpl * cq);
        float tv[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) tv[c] = fmaf(cc, Q0[c], fmaf(cc, xc[c], fmaf(cl, Q0[c], cl * xc[c])));
        const int ncol = Y.dof[q][b];
        const int64_t at = mrow < ncol ? int64_t(mrow) * N + ncol : int64_t(ncol) * N + mrow;
        atomicAdd(M + at, make_float4(tv[1], -tv[0], fmaf(cc, kk[0], cl * kk[0]), fmaf(cc, kk[1], cl * kk[1])));
      }
    }
  }
}

void launch_assemble_regular32(mtf_system sys, cudaStream_t s) {
  mtf_mesh m = sys->mesh;
  const TriRule& rule = triangle_rule6();
  MTF_CUDA(cudaMemcpyToSymbolAsync(c_tri_s, rule.s, sizeof(rule.s), 0, cudaMemcpyHostToDevice, s));
  MTF_CUDA(cudaMemcpyToSymbolAsync(c_tri_t, rule.t, sizeof(rule.t), 0, cudaMemcpyHostToDevice, s));
  float orbit[2][3], point[6][3];
  for (int o = 0; o < 2; ++o) {
    const double w = rule.w[3 * o], a = rule.s[3 * o];
    orbit[o][0] = float(w);
    orbit[o][1] = float(w * (a - 1.0 / 3.0));
    orbit[o][2] = float(w * (1.0 - 3.0 * a));
  }
  for (int p = 0; p < 6; ++p) {
    point[p][0] = float(rule.w[p]);
    point[p][1] = float(rule.w[p] * (rule.s[p] - 1.0 / 3.0));
    point[p][2] = float(rule.w[p] * (rule.t[p] - 1.0 / 3.0));
  }
  MTF_CUDA(cudaMemcpyToSymbolAsync(c_orbit32, orbit, sizeof(orbit), 0, cudaMemcpyHostToDevice, s));
  MTF_CUDA(cudaMemcpyToSymbolAsync(c_point32, point, sizeof(point), 0, cudaMemcpyHostToDevice, s));
  if (!sys->d_cen.p) {
    sys->d_cen.alloc(size_t(m->n_bt) * 3);
    sys->d_qx.alloc(size_t(m->n_bt) * 18);
    sys->d_pv.alloc(size_t(m->n_bt) * 24);
    sys->d_cc.alloc(size_t(m->n_bt) * 8);
  }
  double wsum = 0.0, w32 = 0.0;
  for (int p = 0; p < 6; ++p) {
    wsum += rule.w[p];
    w32 += double(float(rule.w[p]));
  }
  Geom32Args G{m->d_bt_v.p, m->d_bt_c.p, m->d_bt_area.p, m->n_bt, w32 / wsum, sys->d_cen.p, sys->d_qx.p, sys->d_pv.p, sys->d_cc.p};
  MTF_LAUNCH(KID_MISC, s, k_geom32<<<unsigned((m->n_bt + 127) / 128), 128, 0, s>>>(G));
  Reg32Args A{sys->d_cen.p, sys->d_qx.p, sys->d_pv.p, sys->d_cc.p, m->d_bt_dof.p, m->d_bt_vid.p,
              m->d_blk_T.p, m->d_blk_N.p, m->d_blk_bt_off.p, m->d_blk_mat_off.p, sys->d_k.p,
              reinterpret_cast<const float4*>(sys->d_rho32.p) + m->nd, m->nd};
  const int64_t nct = m->reg_cta_prefix.back();
  MTF_LAUNCH(KID_REGULAR32, s, k_regular32<<<unsigned(nct), 128, 0, s>>>(A, m->d_reg_cta_prefix.p, sys->d_TK32.p));
}

}  // namespace mtf
