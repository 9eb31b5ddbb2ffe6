// Far and near fields of solutions (Stratton-Chu, Eq. 8), FP64.
//
// Both are dense products: for a point p (observation direction, or point in
// Omega_i) the field is linear in the D and N coefficients of the block's
// dofs,
//   far:   z+-(p, c) = sum_m Q+-[p, m] (h u_N +- i u_D)[m, c],
//          E = i k0 h / (4 pi) (E_1 e_1 + E_2 e_2),  z+- = E_1 +- i E_2,
//   near:  U(p, c) = sum_m H[p, m] u_D[m, c] + E[p, m] u_N[m, c],
// whose coefficients do not depend on the right-hand side.  With M the
// integrals of RWG function m over its triangles (6-point rule),
//   Q+- = e_1.M +- i e_2.M,  M = int psi_m exp(-i k0 x^.y),  (e_1, e_2, x^/h)
//         orthonormal, h = |x^| (1 for the unit directions of the interface),
//   H = c_a (X - v_a) x int g (y - v_a)     ((X - y) x (y - v_a) = (X - v_a) x (y - v_a)),
//   E = i c_a / rho [k int G (y - v_a) + (2 / k) int g (X - y)]   (div psi = 2 c_a).
//
// Bound: the FP64 pipe.  A warp per point, lanes over the 32 triangles of a
// chunk, forms the coefficients once (one rsqrt step, one short Taylor phase
// per rule point; moments over the rule's orbits); the two halves of a dof
// whose triangles are both in the chunk are added; then the lanes turn to the
// right-hand sides (up to 32) and slices of the chunk's dofs.  Work items are
// (8 points of one block) x (a range of chunks), about two per SM, times
// passes of up to 32 right-hand sides; fewer points and narrower passes where
// that would leave SMs idle; their sums are added in order by k_field_sum.
// Before, every right-hand side re-evaluated the kernel at every rule point: 16
// right-hand sides on the 2 x 2 x 2 cube (181 directions and 584 points) took 96.0 ms, now 7.5 ms.
#include <algorithm>
#include <cmath>

#include "common.h"
#include "kernel64.cuh"

namespace mtf {

constexpr int kFieldPts = 8;   // points per work item (one per warp), at most
constexpr int kFieldThreads = 32 * kFieldPts;
constexpr int kFieldBatch = 4096;  // point groups per launch (bounds the workspace)

struct FieldRule {
  double s[6], t[6];
  double orbit[2][3];  // w, w a, w (1 - 3a) of the orbit (a, a, 1 - 2a)
};

struct FieldMesh {
  const double* bt_v;
  const double* bt_c;
  const double* bt_area;
  const int2* dofs;      // per chunk: {corner | second corner << 8 (0xff: none), local dof}
  const int32_t* first;  // first entry of every chunk (and the end)
};

struct FieldItem {
  int32_t group, chunk0, chunk1, part;
};
struct FieldGroup {  // points of one block; chunk = first chunk of the block
  int32_t point0, n, chunk, T;
  int64_t bt0, dof0;  // first block-triangle, unknown offset
  int32_t N, item0, items, pad;
  double k, irho;
};

template <bool FAR> struct FieldCfg {
  static constexpr int co = FAR ? 4 : 12;   // doubles per (point, dof)
  static constexpr int out = FAR ? 4 : 6;   // doubles per (point, right-hand side)
};

struct FieldGeom {  // a chunk's triangles: rule points about the centroid, vertices, centroid, c_a 2 A
  double y[18][kFieldTris], v[9][kFieldTris], cen[3][kFieldTris], c[3][kFieldTris];
  float rad[kFieldTris];
};

template <bool FAR>
static size_t field_smem(int L) {
  return sizeof(FieldGeom) + sizeof(double) * (size_t(kFieldPts) * 3 * kFieldTris * FieldCfg<FAR>::co) +
         sizeof(double2) * size_t(3 * kFieldTris) * 2 * L;
}

// e_1, e_2 orthonormal to x^ (e_1 x e_2 = x^ / |x^|), h = |x^|
__device__ __forceinline__ double far_basis(const double* xh, double* e1, double* e2) {
  const double h = sqrt(dot3(xh, xh));
  if (!(h > 0.0)) {
    e1[0] = 1.0; e1[1] = 0.0; e1[2] = 0.0;
    e2[0] = 0.0; e2[1] = 1.0; e2[2] = 0.0;
    return 0.0;
  }
  const double a0 = fabs(xh[0]), a1 = fabs(xh[1]), a2 = fabs(xh[2]);
  const double ax[3] = {a0 <= a1 && a0 <= a2 ? 1.0 : 0.0, a1 < a0 && a1 <= a2 ? 1.0 : 0.0, a2 < a0 && a2 < a1 ? 1.0 : 0.0};
  cross3(ax, xh, e1);
  const double n = 1.0 / sqrt(dot3(e1, e1));
  for (int c = 0; c < 3; ++c) e1[c] *= n;
  cross3(xh, e1, e2);
  for (int c = 0; c < 3; ++c) e2[c] /= h;
  return h;
}

// exp(i x) of three arguments by the series of the given degree (-1: sincos)
__device__ __forceinline__ void phases3(const double* x, int deg, double* cs, double* sn) {
  if (deg >= 0) {
    double z[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      z[e] = x[e] * x[e];
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
    for (int e = 0; e < 3; ++e) sn[e] *= x[e];
  } else {
#pragma unroll
    for (int e = 0; e < 3; ++e) sincos(x[e], &sn[e], &cs[e]);
  }
}

// moments over (1, s, t) of NF real channels from an orbit's three values
template <int NF>
__device__ __forceinline__ void add_orbit(const double* w, const double (*v)[NF], double (*m)[NF], double* bc) {
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    const double sum = v[0][f] + v[1][f] + v[2][f];
    m[0][f] = fma(w[0], sum, m[0][f]);
    bc[f] = fma(w[1], sum, bc[f]);
    m[1][f] = fma(w[2], v[1][f], m[1][f]);
    m[2][f] = fma(w[2], v[2][f], m[2][f]);
  }
}

template <bool FAR>
__global__ void __launch_bounds__(kFieldThreads) k_field(const FieldMesh A, const __grid_constant__ FieldRule R,
                                                         const FieldItem* __restrict__ items,
                                                         const FieldGroup* __restrict__ groups,
                                                         const double* __restrict__ pts, const double* __restrict__ x,
                                                         int64_t n_total, int c0, int nrhs, int L, int group_pts,
                                                         double* __restrict__ part) {
  constexpr int CO = FieldCfg<FAR>::co, OUT = FieldCfg<FAR>::out;
  extern __shared__ __align__(16) unsigned char raw[];
  FieldGeom& S = *reinterpret_cast<FieldGeom*>(raw);
  double* coef = reinterpret_cast<double*>(raw + sizeof(FieldGeom));            // [point][corner][CO]
  double2* u = reinterpret_cast<double2*>(coef + kFieldPts * 3 * kFieldTris * CO);  // [dof][slot][L]
  c0 += int(blockIdx.y) * L;  // the pass
  const int nc = min(L, nrhs - c0);
  const FieldItem it = items[blockIdx.x];
  const FieldGroup g = groups[it.group];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int col = lane % L, slice = lane / L, nslice = 32 / L;
  const bool mine = warp < g.n;
  double P[3] = {0.0, 0.0, 0.0}, e1[3], e2[3], h = 1.0;
  if (mine)
    for (int c = 0; c < 3; ++c) P[c] = pts[3 * (g.point0 + warp) + c];
  if (FAR) h = far_basis(P, e1, e2);
  double acc[OUT];
#pragma unroll
  for (int q = 0; q < OUT; ++q) acc[q] = 0.0;

  for (int ch = it.chunk0; ch < it.chunk1; ++ch) {
    const int t0 = (ch - g.chunk) * kFieldTris, nt = min(kFieldTris, g.T - t0);
    const int d0 = A.first[ch], nd = A.first[ch + 1] - d0;
    __syncthreads();
    for (int t = threadIdx.x; t < nt; t += kFieldThreads) {
      const double* v = A.bt_v + 9 * (g.bt0 + t0 + t);
      double r = 0.0;
      for (int c = 0; c < 3; ++c) S.cen[c][t] = (v[c] + v[3 + c] + v[6 + c]) * (1.0 / 3.0);
      for (int a = 0; a < 3; ++a) {
        double d2 = 0.0;
        for (int c = 0; c < 3; ++c) {
          const double d = v[3 * a + c] - S.cen[c][t];
          S.v[3 * a + c][t] = v[3 * a + c];
          d2 = fma(d, d, d2);
        }
        r = fmax(r, d2);
        S.c[a][t] = A.bt_c[3 * (g.bt0 + t0 + t) + a] * (2.0 * A.bt_area[g.bt0 + t0 + t]);
      }
      S.rad[t] = float(sqrt(r)) * 1.0001f;
      for (int q = 0; q < 6; ++q)
        for (int c = 0; c < 3; ++c)
          S.y[3 * q + c][t] = v[c] - S.cen[c][t] + R.s[q] * (v[3 + c] - v[c]) + R.t[q] * (v[6 + c] - v[c]);
    }
    // the chunk's coefficients of the right-hand sides
    for (int t = threadIdx.x; t < nd * 2 * L; t += kFieldThreads) {
      const int c = t % L, slot = (t / L) & 1, d = t / (2 * L);
      double2 v = make_double2(0.0, 0.0);
      if (c < nc)
        v = reinterpret_cast<const double2*>(x)[int64_t(c0 + c) * n_total + g.dof0 + slot * int64_t(g.N) + A.dofs[d0 + d].y];
      u[t] = v;
    }
    __syncthreads();

    // ---- coefficients: warp = point, lane = triangle ----------------------
    if (mine) {
      const bool live = lane < nt;
      const int t = live ? lane : 0;
      const float kf = float(g.k) * (FAR ? float(h) * 1.0001f : 1.0001f);
      const int deg = series_degree(__uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(live ? kf * S.rad[t] : 0.f))));
      const double cen[3] = {S.cen[0][t], S.cen[1][t], S.cen[2][t]};
      double E[2][3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        E[0][c] = S.v[3 + c][t] - S.v[c][t];
        E[1][c] = S.v[6 + c][t] - S.v[c][t];
      }
      double* out = coef + (size_t(warp) * 3 * kFieldTris + 3 * lane) * CO;
      if constexpr (FAR) {
        const double ph0 = -g.k * dot3(P, cen);
        double m[3][2] = {}, bc[2] = {};
#pragma unroll
        for (int o = 0; o < 2; ++o) {
          double ph[3], cs[3], sn[3], v[3][2];
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            const int q = 3 * (3 * o + e);
            const double y[3] = {S.y[q][t], S.y[q + 1][t], S.y[q + 2][t]};
            ph[e] = -g.k * dot3(P, y);
          }
          phases3(ph, deg, cs, sn);
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            v[e][0] = cs[e];
            v[e][1] = sn[e];
          }
          add_orbit<2>(R.orbit[o], v, m, bc);
        }
        double s0, cc0;
        sincos(ph0, &s0, &cc0);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          const double re = r ? m[r][0] + bc[0] : m[r][0], im = r ? m[r][1] + bc[1] : m[r][1];
          m[r][0] = re * cc0 - im * s0;
          m[r][1] = re * s0 + im * cc0;
        }
        const double a1[2] = {dot3(E[0], e1), dot3(E[1], e1)}, a2[2] = {dot3(E[0], e2), dot3(E[1], e2)};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          double p1[2], p2[2];
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            p1[c] = fma(m[1][c], a1[0], m[2][c] * a1[1]);
            p2[c] = fma(m[1][c], a2[0], m[2][c] * a2[1]);
            if (a > 0) {
              p1[c] = fma(-m[0][c], a1[a - 1], p1[c]);
              p2[c] = fma(-m[0][c], a2[a - 1], p2[c]);
            }
          }
          const double ca = S.c[a][t];
          out[CO * a] = ca * (p1[0] - p2[1]);      // Q+
          out[CO * a + 1] = ca * (p1[1] + p2[0]);
          out[CO * a + 2] = ca * (p1[0] + p2[1]);  // Q-
          out[CO * a + 3] = ca * (p1[1] - p2[0]);
        }
      } else {
        const double D[3] = {P[0] - cen[0], P[1] - cen[1], P[2] - cen[2]};
        const double kr0 = g.k * sqrt(dot3(D, D));
        double m[3][4] = {}, bc[4] = {};  // re, im of G 4 pi exp(-i k r0) and of -g
#pragma unroll
        for (int o = 0; o < 2; ++o) {
          double ri[3], ph[3], cs[3], sn[3], v[3][4];
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            const int q = 3 * (3 * o + e);
            const double d[3] = {D[0] - S.y[q][t], D[1] - S.y[q + 1][t], D[2] - S.y[q + 2][t]};
            const double r2 = dot3(d, d);
            ri[e] = rsqrt_h(r2);
            ph[e] = fma(g.k, r2 * ri[e], -kr0);
          }
          phases3(ph, deg, cs, sn);
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            v[e][0] = ri[e] * cs[e];
            v[e][1] = ri[e] * sn[e];
            const double al = g.k * ri[e], be = ri[e] * ri[e];
            v[e][2] = fma(be, v[e][0], al * v[e][1]);
            v[e][3] = fma(be, v[e][1], -(al * v[e][0]));
          }
          add_orbit<4>(R.orbit[o], v, m, bc);
        }
        double s0, cc0;
        sincos(kr0, &s0, &cc0);
        s0 *= INV_FOUR_PI;
        cc0 *= INV_FOUR_PI;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
          for (int f = 0; f < 4; f += 2) {
            const double re = r ? m[r][f] + bc[f] : m[r][f], im = r ? m[r][f + 1] + bc[f + 1] : m[r][f + 1];
            const double a = re * cc0 - im * s0, b = re * s0 + im * cc0;
            m[r][f] = f ? -a : a;  // G, g
            m[r][f + 1] = f ? -b : b;
          }
        double X0[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) X0[c] = P[c] - S.v[c][t];
        const double k2 = 2.0 / g.k;
#pragma unroll
        for (int c = 0; c < 2; ++c) {  // real, imaginary parts
          double Z0[3], Y0[3], W[3];   // int G (y - v_0), int g (y - v_0), int g (X - y)
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            Z0[d] = fma(m[1][c], E[0][d], m[2][c] * E[1][d]);
            Y0[d] = fma(m[1][2 + c], E[0][d], m[2][2 + c] * E[1][d]);
            W[d] = k2 * fma(X0[d], m[0][2 + c], -Y0[d]);
          }
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            double Xa[3], Ya[3], H[3];
            const double ca = S.c[a][t], ci = ca * g.irho;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              Xa[d] = a ? X0[d] - E[a - 1][d] : X0[d];
              Ya[d] = a ? fma(-m[0][2 + c], E[a - 1][d], Y0[d]) : Y0[d];
            }
            cross3(Xa, Ya, H);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              const double z = a ? fma(-m[0][c], E[a - 1][d], Z0[d]) : Z0[d];
              const double e = ci * fma(g.k, z, W[d]);
              out[CO * a + 2 * d + c] = ca * H[d];
              out[CO * a + 6 + 2 * d + 1 - c] = c ? -e : e;  // times i
            }
          }
        }
      }
    }
    __syncwarp();
    if (!mine) continue;  // (the next chunk's barriers are met at its start)
    double* cw = coef + size_t(warp) * 3 * kFieldTris * CO;
    // the two halves of dofs inside the chunk
    for (int d = lane; d < nd; d += 32) {
      const int e = A.dofs[d0 + d].x;
      if ((e >> 8) != 0xff)
#pragma unroll
        for (int q = 0; q < CO; ++q) cw[CO * (e & 0xff) + q] += cw[CO * (e >> 8) + q];
    }
    __syncwarp();
    // ---- products: lane = (right-hand side, slice of the dofs), the chunk's
    // sum by itself (one running sum over thousands of dofs loses a digit)
    double sum[OUT];
#pragma unroll
    for (int q = 0; q < OUT; ++q) sum[q] = 0.0;
    for (int d = slice; d < nd; d += nslice) {
      const double2* w = reinterpret_cast<const double2*>(cw + CO * (A.dofs[d0 + d].x & 0xff));
      const double2 uD = u[(2 * d) * L + col], uN = u[(2 * d + 1) * L + col];
      if constexpr (FAR) {
        const double pr = fma(h, uN.x, -uD.y), pi = fma(h, uN.y, uD.x);  // h u_N + i u_D
        const double mr = fma(h, uN.x, uD.y), mi = fma(h, uN.y, -uD.x);  // h u_N - i u_D
        const double2 qp = w[0], qm = w[1];
        sum[0] = fma(qp.x, pr, fma(-qp.y, pi, sum[0]));
        sum[1] = fma(qp.x, pi, fma(qp.y, pr, sum[1]));
        sum[2] = fma(qm.x, mr, fma(-qm.y, mi, sum[2]));
        sum[3] = fma(qm.x, mi, fma(qm.y, mr, sum[3]));
      } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const double2 H = w[c], N = w[3 + c];
          sum[2 * c] = fma(H.x, uD.x, fma(-H.y, uD.y, sum[2 * c]));
          sum[2 * c + 1] = fma(H.x, uD.y, fma(H.y, uD.x, sum[2 * c + 1]));
          sum[2 * c] = fma(N.x, uN.x, fma(-N.y, uN.y, sum[2 * c]));
          sum[2 * c + 1] = fma(N.x, uN.y, fma(N.y, uN.x, sum[2 * c + 1]));
        }
      }
    }
#pragma unroll
    for (int q = 0; q < OUT; ++q) acc[q] += sum[q];
  }
  if (!mine) return;
#pragma unroll
  for (int q = 0; q < OUT; ++q)
    for (int o = L; o < 32; o <<= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
  if (lane < nc) {
    double* o = part + (((size_t(blockIdx.y) * gridDim.x + it.part) * group_pts + warp) * L + lane) * OUT;
#pragma unroll
    for (int q = 0; q < OUT; ++q) o[q] = acc[q];
  }
}

// sums of a group's items in order, and the far field's polarisations:
// thread = (point, right-hand side); point order[p] of the call
template <bool FAR>
__global__ void k_field_sum(const double* __restrict__ part, const FieldGroup* __restrict__ groups, int n_groups,
                            const double* __restrict__ pts, const int32_t* __restrict__ order, int n_items, int c0,
                            int nrhs, int L, int group_pts, int npts, double* __restrict__ fout) {
  constexpr int OUT = FieldCfg<FAR>::out;
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  c0 += int(blockIdx.y) * L;
  const int c = int(t % L), p = int((t / L) % group_pts);
  const int64_t gi = t / (int64_t(L) * group_pts);
  if (gi >= n_groups || c0 + c >= nrhs) return;
  const FieldGroup g = groups[gi];
  if (p >= g.n) return;
  double s[OUT];
#pragma unroll
  for (int q = 0; q < OUT; ++q) s[q] = 0.0;
  for (int i = 0; i < g.items; ++i) {
    const double* v = part + (((size_t(blockIdx.y) * n_items + g.item0 + i) * group_pts + p) * L + c) * OUT;
#pragma unroll
    for (int q = 0; q < OUT; ++q) s[q] += v[q];
  }
  double* f = fout + 6 * (int64_t(c0 + c) * npts + order[g.point0 + p]);
  if constexpr (FAR) {
    const double P[3] = {pts[3 * (g.point0 + p)], pts[3 * (g.point0 + p) + 1], pts[3 * (g.point0 + p) + 2]};
    double e1[3], e2[3];
    const double h = far_basis(P, e1, e2), sc = 0.5 * g.k * INV_FOUR_PI * h;
    // i E_1 = i (z+ + z-) / 2, i E_2 = (z+ - z-) / 2
    const double r1 = -sc * (s[1] + s[3]), i1 = sc * (s[0] + s[2]), r2 = sc * (s[0] - s[2]), i2 = sc * (s[1] - s[3]);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      f[2 * d] = fma(r1, e1[d], r2 * e2[d]);
      f[2 * d + 1] = fma(i1, e1[d], i2 * e2[d]);
    }
  } else {
#pragma unroll
    for (int q = 0; q < OUT; ++q) f[q] = s[q];
  }
}

// points (host, 3 per point) in blocks dom (host; null: block 0): groups of 4 or 8
// points of one block, items of about equal chunk counts, in batches
template <bool FAR>
static void run_fields(mtf_system sys, const double* x, int nrhs, const double* pts, const int32_t* dom, int npts,
                       double* f, cudaStream_t s) {
  mtf_mesh m = sys->mesh;
  FieldRule R;
  const TriRule& rule = triangle_rule6();
  for (int q = 0; q < 6; ++q) {
    R.s[q] = rule.s[q];
    R.t[q] = rule.t[q];
  }
  for (int o = 0; o < 2; ++o) {
    const double w = rule.w[3 * o], a = rule.s[3 * o];
    R.orbit[o][0] = w;
    R.orbit[o][1] = w * a;
    R.orbit[o][2] = w * (1.0 - 3.0 * a);
  }
  int dev = 0, sms = 0;
  MTF_CUDA(cudaGetDevice(&dev));
  MTF_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  std::vector<int32_t> order(static_cast<size_t>(npts));
  for (int p = 0; p < npts; ++p) order[size_t(p)] = p;
  if (dom) std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return dom[a] < dom[b]; });
  // Points per item (8 or 4) and right-hand sides per pass (32 to 4): 8 points
  // share a chunk's geometry and fill each quarter of an SM with two warps, and
  // wide passes form the coefficients least often.  A call with fewer items
  // than SMs is a chain of FP64 operations (about 600 a chunk for the
  // coefficients and 36 per right-hand side of the pass, 64 cycles each, times
  // the warps of a quarter): both are halved while the items still fit one per
  // SM.  Near field of 64 solutions at 2 points, 80 triangles: 223 us with 8
  // points and passes of 32 in turn, 84 us so; 100 points, one solution, 20
  // triangles: 115 -> 87 us.
  std::vector<int64_t> count(size_t(m->nd), 0);
  for (int p = 0; p < npts; ++p) ++count[dom ? size_t(dom[p]) : 0];
  const auto n_items = [&](int pts_per) {
    int64_t n = 0;
    for (int i = 0; i < m->nd; ++i)
      n += (count[size_t(i)] + pts_per - 1) / pts_per * (m->fld_chunk[size_t(i) + 1] - m->fld_chunk[size_t(i)]);
    return n;
  };
  const int group_pts = n_items(kFieldPts / 2) <= sms ? kFieldPts / 2 : kFieldPts;
  int L = 1;
  while (L < std::min(nrhs, 32)) L *= 2;
  bool narrow = false;
  while (L > 4 && n_items(group_pts) * ((nrhs + L / 2 - 1) / (L / 2)) <= sms) {
    L /= 2;
    narrow = true;
  }
  const FieldMesh A{m->d_bt_v.p, m->d_bt_c.p, m->d_bt_area.p, m->d_fld_dofs.p, m->d_fld_first.p};
  int at = 0;
  while (at < npts) {
    std::vector<FieldGroup> groups;
    std::vector<double> sorted;
    const int p_begin = at;
    int64_t total = 0;
    while (at < npts && int(groups.size()) < kFieldBatch) {
      const int i = dom ? dom[order[size_t(at)]] : 0;
      FieldGroup g{};
      g.point0 = at - p_begin;
      while (g.n < group_pts && at < npts && (!dom || dom[order[size_t(at)]] == i)) {
        const double* p = pts + 3 * int64_t(order[size_t(at)]);
        sorted.insert(sorted.end(), p, p + 3);
        ++g.n;
        ++at;
      }
      const BlockInfo& B = m->blk[size_t(i)];
      g.chunk = m->fld_chunk[size_t(i)];
      g.T = B.T;
      g.N = B.N;
      g.bt0 = B.bt_off;
      g.dof0 = B.dof_off;
      g.k = sys->k_re[size_t(i)];
      g.irho = 1.0 / sys->rho_re[size_t(i)];
      total += m->fld_chunk[size_t(i) + 1] - g.chunk;
      groups.push_back(g);
    }
    // about two items per SM: a CTA holds most of an SM's shared memory
    const int64_t per = std::max<int64_t>(1, (total + 2 * sms - 1) / (2 * sms));
    std::vector<FieldItem> items;
    for (size_t q = 0; q < groups.size(); ++q) {
      FieldGroup& g = groups[q];
      const int nch = (g.T + kFieldTris - 1) / kFieldTris;
      const int n = int((nch + per - 1) / per);
      g.item0 = int(items.size());
      g.items = n;
      for (int e = 0; e < n; ++e)
        items.push_back({int32_t(q), g.chunk + int(int64_t(nch) * e / n), g.chunk + int(int64_t(nch) * (e + 1) / n),
                         int32_t(items.size())});
    }
    // one allocation per batch: groups | items | order | points | partial sums
    const size_t bg = groups.size() * sizeof(FieldGroup), bi = items.size() * sizeof(FieldItem),
                 bo = (sizeof(int32_t) * size_t(at - p_begin) + 15) / 16 * 16, bp = sorted.size() * sizeof(double);
    const size_t head = (bg + bi + bo + bp + 255) / 256 * 256;
    std::vector<unsigned char> host(head);
    std::copy_n(reinterpret_cast<const unsigned char*>(groups.data()), bg, host.data());
    std::copy_n(reinterpret_cast<const unsigned char*>(items.data()), bi, host.data() + bg);
    std::copy_n(reinterpret_cast<const unsigned char*>(order.data() + p_begin), sizeof(int32_t) * size_t(at - p_begin),
                host.data() + bg + bi);
    std::copy_n(reinterpret_cast<const unsigned char*>(sorted.data()), bp, host.data() + bg + bi + bo);
    // partial sums of a pass; passes per launch within 64 MB
    const size_t pass_doubles = items.size() * size_t(group_pts) * size_t(L) * FieldCfg<FAR>::out;
    const int per_launch = int(std::min({size_t(nrhs + L - 1) / size_t(L), size_t(65535),
                                         std::max<size_t>(1, (size_t(8) << 20) / pass_doubles)}));
    // a workspace of up to 4 MB stays with the system: an allocation that needs
    // new mapped memory takes 0.15 ms, as long as such a call
    const size_t need = head + size_t(per_launch) * pass_doubles * sizeof(double);
    DevBuf<unsigned char> own;
    DevBuf<unsigned char>& ws = need <= kFieldKeep ? sys->d_field : own;
    if (ws.n < need) ws.alloc(need);
    MTF_CUDA(cudaMemcpyAsync(ws.p, host.data(), head, cudaMemcpyHostToDevice, s));
    const auto* dg = reinterpret_cast<const FieldGroup*>(ws.p);
    const auto* di = reinterpret_cast<const FieldItem*>(ws.p + bg);
    const auto* dord = reinterpret_cast<const int32_t*>(ws.p + bg + bi);
    const auto* dp = reinterpret_cast<const double*>(ws.p + bg + bi + bo);
    auto* part = reinterpret_cast<double*>(ws.p + head);
    MTF_CUDA(cudaFuncSetAttribute(k_field<FAR>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(field_smem<FAR>(32))));
    for (int c0 = 0; c0 < nrhs;) {
      // whole passes together, then the rest in a pass of its own width (narrow
      // passes run side by side: the last one may be partly empty)
      int Lq = L, np = narrow ? (nrhs - c0 + L - 1) / L : (nrhs - c0) / L;
      if (np == 0) {
        np = 1;
        while (Lq / 2 >= nrhs - c0) Lq /= 2;
      }
      np = std::min(np, per_launch);
      MTF_LAUNCH(KID_FARFIELD, s,
                 k_field<FAR><<<dim3(unsigned(items.size()), unsigned(np)), kFieldThreads, field_smem<FAR>(Lq), s>>>(
                     A, R, di, dg, dp, x, m->n_total, c0, nrhs, Lq, group_pts, part));
      const int64_t nt = int64_t(groups.size()) * group_pts * Lq;
      MTF_LAUNCH(KID_FARFIELD, s, k_field_sum<FAR><<<dim3(unsigned((nt + 127) / 128), unsigned(np)), 128, 0, s>>>(
          part, dg, int(groups.size()), dp, dord, int(items.size()), c0, nrhs, Lq, group_pts, npts, f));
      c0 += np * Lq;
    }
    MTF_CUDA(cudaStreamSynchronize(s));  // the workspace and the host tables are released
  }
}

void launch_farfield(mtf_system sys, const double* x, int nrhs, const double* obs, int nobs, double* f, cudaStream_t s) {
  run_fields<true>(sys, x, nrhs, obs, nullptr, nobs, f, s);
}

void launch_nearfield(mtf_system sys, const double* x, int nrhs, const double* pts, const int32_t* dom, int npts,
                      double* f, cudaStream_t s) {
  run_fields<false>(sys, x, nrhs, pts, dom, npts, f, s);
}

}  // namespace mtf
