// MTF operator apply y = M x (Problem 2): per block i the dense Calderon
// part 2 A_i u_i = 2 [K u_D + rho^-1 T u_N ; -rho T u_D + K u_N] (Eq. 9)
// fused with the skeleton exchange sum_{j in Lambda_i} G^{ij} u_j applied to
// both trace slots with the same sign (Eqs. 11-13, Remark 2).
//
// The FP64 matvec takes the two traces together: with w = x_N / rho_i and
// u+- = x_D +- i w,
//   (K -+ i T) u+- = (K x_D + T w) +- i (K w - T x_D) =: y+-,
//   y_D = y+ + y-,   y_N = -i rho_i (y+ - y-),
// two complex products per entry and right-hand side instead of the four of
// K x_D, K x_N, T x_D, T x_N.  A row is then exact to 2^-53 of (|K| + |T|)
// (|x_D| + |w|), as with four products where both traces are filled; K x_D
// alone (x_N = 0) is exact to 2^-53 of |T| |x_D| only, about 1 / (k h) more
// (mtf.h; the tensor-core matvec, whose unit is 2^-22, keeps K apart).  FP64 systems keep the entries in this form
// (d_rot64, written with the mirrored blocks) where memory is plentiful
// (rotated_copy.h); otherwise they, and FP32-stored entries (the residual_df =
// 0 residual), are rotated as they are read, with the same results.
//
// Bound: the FP64 pipe (8 instructions per entry and right-hand side; the
// 32-byte entries would stream in an eighth of that time).  A CTA of 8 warps
// takes R rows per warp of one block; tiles of 128 columns of u+- are formed
// once per CTA in shared memory; the exchange entries join the lanes' sums
// before the reduction.  Rows per CTA (8, 16, 32) are chosen for the fewest
// rounds of CTAs over the SMs.  Measured on the split sphere of 11 rings (3
// blocks of 2,178 rows), 2 right-hand sides: 1,503 -> 470 us (588 us without
// the rotated copy).
#include <algorithm>

#include "common.h"
#include "kernel64.cuh"

namespace mtf {

constexpr int kMvCols = 128;

struct MvArgs {
  const void* entries;
  const XEntry* xe;
  const double* xval;
  const int32_t* prefix;  // first CTA of every block
  const int32_t* blk_N;
  const int64_t* blk_dof_off;
  const int64_t* blk_mat_off;
  const int64_t* blk_row_off;
  const double* rho;  // (re, im = 0) per block
  int nblk;
};

// what an entry is stored as: (K - i T, K + i T) or (T, K)
enum class Ent { kRotated64, kBlocks64, kBlocks32 };

template <Ent E>
__device__ __forceinline__ void load_rotated(const void* entries, int64_t e, double* a) {
  if constexpr (E == Ent::kRotated64) {
    const double2 p = __ldg(static_cast<const double2*>(entries) + 2 * e);
    const double2 m = __ldg(static_cast<const double2*>(entries) + 2 * e + 1);
    a[0] = p.x; a[1] = p.y; a[2] = m.x; a[3] = m.y;
  } else {
    double tr, ti, kr, ki;
    if constexpr (E == Ent::kBlocks64) {
      const double2 t = __ldg(static_cast<const double2*>(entries) + 2 * e);
      const double2 k = __ldg(static_cast<const double2*>(entries) + 2 * e + 1);
      tr = t.x; ti = t.y; kr = k.x; ki = k.y;
    } else {
      const float4 v = __ldg(static_cast<const float4*>(entries) + e);
      tr = v.x; ti = v.y; kr = v.z; ki = v.w;
    }
    a[0] = kr + ti; a[1] = ki - tr; a[2] = kr - ti; a[3] = ki + tr;
  }
}

// The end of a warp's R rows: acc (per lane, [row][right-hand side][y+ re, im,
// y- re, im]) with the exchange entries added, summed over the lanes, as y_D
// and y_N; sums: the warp's R NC 4 doubles of shared memory
template <int NC, int R>
__device__ __forceinline__ void mv_finish(const MvArgs& A, int i, int m0, int lane, int64_t off,
                                          const double* __restrict__ x, int64_t ldx, double* __restrict__ y, int64_t ldy,
                                          int c0, double* acc, double* sums) {
  constexpr int NV = R * NC * 4;
  const int N = A.blk_N[i];
  const double rho = A.rho[2 * i], ir = 1.0 / rho;
  // the row's six exchange entries, one per lane: sum_j v x_j in both slots,
  // y+- += (dD +- i dN / rho) / 2
  if (lane < 6) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int64_t e = 6 * (A.blk_row_off[i] + min(m0 + r, N - 1)) + lane;
      const XEntry X = A.xe[e];
      const double v = 0.5 * A.xval[e], vi = v * ir;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const double2* xc = reinterpret_cast<const double2*>(x) + int64_t(c0 + c) * ldx + X.col;
        const double2 d = xc[0], w = xc[X.ab >> 4];
        double* s = acc + 4 * (r * NC + c);
        s[0] += fma(v, d.x, -(vi * w.y));
        s[1] += fma(v, d.y, vi * w.x);
        s[2] += fma(v, d.x, vi * w.y);
        s[3] += fma(v, d.y, -(vi * w.x));
      }
    }
  }
  int base = 0, count = NV;
  halve_sum<NV>(acc, lane, 16, base, count);
#pragma unroll
  for (int q = 0; q < (NV + 31) / 32; ++q)
    if (q < count) sums[base + q] = acc[q];
  __syncwarp();
  if (lane < R * NC) {
    const int r = lane / NC, c = lane % NC;
    if (m0 + r < N) {
      const double* s = sums + 4 * lane;
      double2* yc = reinterpret_cast<double2*>(y) + int64_t(c0 + c) * ldy + off + m0 + r;
      yc[0] = make_double2(s[0] + s[2], s[1] + s[3]);
      yc[N] = make_double2(rho * (s[1] - s[3]), rho * (s[2] - s[0]));
    }
  }
}

// y = M x for right-hand sides c0 .. c0 + NC - 1; R rows per warp
template <Ent E, int NC, int R>
__global__ void __launch_bounds__(256, R * NC >= 4 ? 2 : 4) k_matvec(const MvArgs A, const double* __restrict__ x, int64_t ldx,
                                                double* __restrict__ y, int64_t ldy, int c0) {
  MTF_PDL_WAIT();
  MTF_PDL_TRIGGER();
  constexpr int NV = R * NC * 4;
  __shared__ double2 us[NC][kMvCols][2];  // u+, u- of a tile of columns
  __shared__ double sums[8][NV];
  int lo = 0, hi = A.nblk - 1;
  while (lo < hi) {  // largest block with prefix <= CTA
    const int mid = (lo + hi + 1) >> 1;
    if (A.prefix[mid] <= int(blockIdx.x)) lo = mid; else hi = mid - 1;
  }
  const int i = lo, N = A.blk_N[i];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = (int(blockIdx.x) - A.prefix[i]) * 8 * R + warp * R;
  const int64_t off = A.blk_dof_off[i];
  const double rho = A.rho[2 * i], ir = 1.0 / rho;
  int64_t row[R];  // first entries of the warp's rows (the last one repeated past the block)
  double acc[NV];
#pragma unroll
  for (int r = 0; r < R; ++r) row[r] = A.blk_mat_off[i] + int64_t(min(m0 + r, N - 1)) * N;
#pragma unroll
  for (int q = 0; q < NV; ++q) acc[q] = 0.0;
  for (int n0 = 0; n0 < N; n0 += kMvCols) {
    __syncthreads();
    for (int t = threadIdx.x; t < NC * kMvCols; t += 256) {
      const int c = t / kMvCols, n = n0 + t % kMvCols;
      if (n < N) {
        const double2* xc = reinterpret_cast<const double2*>(x) + int64_t(c0 + c) * ldx + off + n;
        const double2 d = xc[0], w = xc[N];
        us[c][t % kMvCols][0] = make_double2(fma(-ir, w.y, d.x), fma(ir, w.x, d.y));
        us[c][t % kMvCols][1] = make_double2(fma(ir, w.y, d.x), fma(-ir, w.x, d.y));
      }
    }
    __syncthreads();
#pragma unroll 2
    for (int n = lane; n < min(kMvCols, N - n0); n += 32) {
      double a[R][4];
#pragma unroll
      for (int r = 0; r < R; ++r) load_rotated<E>(A.entries, row[r] + n0 + n, a[r]);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const double2 p = us[c][n][0], m = us[c][n][1];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          double* s = acc + 4 * (r * NC + c);
          s[0] = fma(a[r][0], p.x, fma(-a[r][1], p.y, s[0]));
          s[1] = fma(a[r][0], p.y, fma(a[r][1], p.x, s[1]));
          s[2] = fma(a[r][2], m.x, fma(-a[r][3], m.y, s[2]));
          s[3] = fma(a[r][2], m.y, fma(a[r][3], m.x, s[3]));
        }
      }
    }
  }
  mv_finish<NC, R>(A, i, m0, lane, off, x, ldx, y, ldy, c0, acc, sums[warp]);
}

template <Ent E, int NC, int R>
static void mv64_launch(mtf_system sys, const MvArgs& A, unsigned grid, const double* x, int64_t ldx, double* y,
                        int64_t ldy, int c0, cudaStream_t s) {
  MTF_LAUNCH(KID_MATVEC64, s, launch_pdl(k_matvec<E, NC, R>, dim3(grid), dim3(256), 0, s, A, x, ldx, y, ldy, c0));
}

// passes of up to 4 right-hand sides
template <Ent E>
static void matvec64(mtf_system sys, const void* entries, const double* x, int64_t ldx, double* y, int64_t ldy, int nrhs,
                     cudaStream_t s) {
  mtf_mesh m = sys->mesh;
  int dev = 0, sms = 0;
  MTF_CUDA(cudaGetDevice(&dev));
  MTF_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  MvArgs A{entries, m->d_xent.p, sys->d_xval.p, nullptr, m->d_blk_N.p, m->d_blk_dof_off.p, m->d_blk_mat_off.p,
           m->d_blk_row_off.p, sys->d_rho.p, m->nd};
  for (int c0 = 0; c0 < nrhs; c0 += 4) {
    const int nc = std::min(4, nrhs - c0);
    // rounds of CTAs over the SMs times a CTA's work per column: 64 R products
    // and 6 operations of the tile of u (R = 4 only while its sums fit)
    int best = 0;
    int64_t cost = 0;
    for (int q = 0; q < (nc <= 2 ? 3 : 2); ++q) {
      const int64_t rounds = (m->mv_cta_prefix[q].back() + sms - 1) / sms;
      const int64_t t = rounds * ((64 << q) + 6);
      if (q == 0 || t < cost) {
        best = q;
        cost = t;
      }
    }
    A.prefix = m->d_mv_cta_prefix[best].p;
    const unsigned grid = unsigned(m->mv_cta_prefix[best].back());
#define MTF_MV(NCV, RV) mv64_launch<E, NCV, RV>(sys, A, grid, x, ldx, y, ldy, c0, s)
    if (nc == 1) best == 0 ? MTF_MV(1, 1) : best == 1 ? MTF_MV(1, 2) : MTF_MV(1, 4);
    else if (nc == 2) best == 0 ? MTF_MV(2, 1) : best == 1 ? MTF_MV(2, 2) : MTF_MV(2, 4);
    else if (nc == 3) best == 0 ? MTF_MV(3, 1) : MTF_MV(3, 2);
    else best == 0 ? MTF_MV(4, 1) : MTF_MV(4, 2);
#undef MTF_MV
  }
}

// Refinement residual matvec of the mixed path: FP32-stored (T, K), input x
// split into FP32 pairs x = x_hi + x_lo (48 significant bits), and every
// product accumulated in double-float: a x_hi = p + e exactly (e by FMA),
// a x_lo and a_lo x_hi added to e, p added to the running (hi, lo) pair by an
// error-free two-sum.  The sums carry about 2^-46 relative error against a few times
// 2^-53 for FP64 FMAs, at FP32 throughput instead of the narrow FP64 pipe.
// Lanes convert to FP64 for the warp reduction and the FP64 epilogue (rho,
// exchange).
// (the _rn intrinsics keep the compiler from contracting the product into
// the sum, which would break the error-free transformations)
__device__ __forceinline__ void df_mac(float& hi, float& lo, float a, float al, float xh, float xl) {
  const float p = __fmul_rn(a, xh);
  float e = fmaf(a, xh, -p);  // exact: a xh = p + e
  e = fmaf(a, xl, e);
  e = fmaf(al, xh, e);
  const float s = __fadd_rn(hi, p);  // two-sum of hi and p
  const float z = __fsub_rn(s, hi);
  const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, z)), __fsub_rn(p, z));
  hi = s;
  lo = __fadd_rn(lo, __fadd_rn(err, e));
}

// a + b = s + e exactly (Knuth's two-sum)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float z = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
}

// The rotated products of the FP64 matvec in double-float: the entries
// A+- = K -+ i T as exact FP32 pairs (two-sums of the stored parts), the
// inputs u+- as pairs formed once per apply (k_split_pm).  CTA = 8 warps x R
// rows of one block, tiles of 128 columns of u+- in shared memory, NC
// right-hand sides.  Bound: FP32 issue (11 instructions per real product).
// E64: the operator is the FP64 blocks, given as FP32 pairs (TK = fl(v),
// TKlo = fl(v - fl(v)), split once per assembly), so the residual of the
// FP64-assembled system costs FP32 work (residual_fp64).  4 x 4 x 4 cube, 16
// right-hand sides: 12.4 -> 4.7 ms.
template <bool E64, int NC, int R>
__global__ void __launch_bounds__(256) k_matvec_df(const MvArgs A, const float* __restrict__ TKlo,
                                                   const float4* __restrict__ u, const double* __restrict__ x, int64_t ldx,
                                                   double* __restrict__ y, int64_t ldy, int c0, int64_t n_rows) {
  constexpr int NV = R * NC * 4;
  __shared__ float4 us[NC][kMvCols][2];  // (u+, u-) hi, lo of a tile of columns
  __shared__ double sums[8][NV];
  int lo = 0, hi = A.nblk - 1;
  while (lo < hi) {  // largest block with prefix <= CTA
    const int mid = (lo + hi + 1) >> 1;
    if (A.prefix[mid] <= int(blockIdx.x)) lo = mid; else hi = mid - 1;
  }
  const int i = lo, N = A.blk_N[i];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = (int(blockIdx.x) - A.prefix[i]) * 8 * R + warp * R;
  const int64_t off = A.blk_dof_off[i], r0 = A.blk_row_off[i];
  int64_t row[R];
  float ah[NV], al[NV];
#pragma unroll
  for (int r = 0; r < R; ++r) row[r] = A.blk_mat_off[i] + int64_t(min(m0 + r, N - 1)) * N;
#pragma unroll
  for (int q = 0; q < NV; ++q) ah[q] = al[q] = 0.f;
  for (int n0 = 0; n0 < N; n0 += kMvCols) {
    __syncthreads();
    for (int t = threadIdx.x; t < NC * kMvCols * 2; t += 256) {
      const int c = t / (2 * kMvCols), n = n0 + (t >> 1) % kMvCols;
      if (n < N) us[c][(t >> 1) % kMvCols][t & 1] = u[2 * (int64_t(c0 + c) * n_rows + r0 + n) + (t & 1)];
    }
    __syncthreads();
    for (int n = lane; n < min(kMvCols, N - n0); n += 32) {
      float4 h[R], l[R];  // A+ re, im, A- re, im
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float4 v = __ldg(static_cast<const float4*>(A.entries) + row[r] + n0 + n);  // T, K
        two_sum(v.z, v.y, h[r].x, l[r].x);
        two_sum(v.w, -v.x, h[r].y, l[r].y);
        two_sum(v.z, -v.y, h[r].z, l[r].z);
        two_sum(v.w, v.x, h[r].w, l[r].w);
        if constexpr (E64) {
          const float4 w = __ldg(reinterpret_cast<const float4*>(TKlo) + row[r] + n0 + n);
          l[r].x += w.z + w.y;
          l[r].y += w.w - w.x;
          l[r].z += w.z - w.y;
          l[r].w += w.w + w.x;
        }
      }
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const float4 uh = us[c][n][0], ul = us[c][n][1];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          float* H = ah + 4 * (r * NC + c);
          float* Lo = al + 4 * (r * NC + c);
          df_mac(H[0], Lo[0], h[r].x, l[r].x, uh.x, ul.x);
          df_mac(H[0], Lo[0], -h[r].y, -l[r].y, uh.y, ul.y);
          df_mac(H[1], Lo[1], h[r].x, l[r].x, uh.y, ul.y);
          df_mac(H[1], Lo[1], h[r].y, l[r].y, uh.x, ul.x);
          df_mac(H[2], Lo[2], h[r].z, l[r].z, uh.z, ul.z);
          df_mac(H[2], Lo[2], -h[r].w, -l[r].w, uh.w, ul.w);
          df_mac(H[3], Lo[3], h[r].z, l[r].z, uh.w, ul.w);
          df_mac(H[3], Lo[3], h[r].w, l[r].w, uh.z, ul.z);
        }
      }
    }
  }
  double acc[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) acc[q] = double(ah[q]) + double(al[q]);
  mv_finish<NC, R>(A, i, m0, lane, off, x, ldx, y, ldy, c0, acc, sums[warp]);
}

// u+- of every row and right-hand side as FP32 pairs: u[2 (c n_rows + row)] =
// (u+, u-) hi, the next float4 the lo parts
__global__ void k_split_pm(const double* __restrict__ x, int64_t ldx, int64_t n_rows, int nrhs,
                           const int32_t* __restrict__ row_blk, const int64_t* __restrict__ blk_row_off,
                           const int32_t* __restrict__ blk_N, const int64_t* __restrict__ blk_dof_off,
                           const double* __restrict__ rho, float4* __restrict__ u) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= n_rows * nrhs) return;
  const int64_t row = t % n_rows, c = t / n_rows;
  const int i = row_blk[row];
  const double2* xc = reinterpret_cast<const double2*>(x) + c * ldx + blk_dof_off[i] + (row - blk_row_off[i]);
  const double2 d = xc[0], w = xc[blk_N[i]];
  const double ir = 1.0 / rho[2 * i];
  const double v[4] = {fma(-ir, w.y, d.x), fma(ir, w.x, d.y), fma(ir, w.y, d.x), fma(-ir, w.x, d.y)};
  const float4 h = make_float4(float(v[0]), float(v[1]), float(v[2]), float(v[3]));
  u[2 * t] = h;
  u[2 * t + 1] = make_float4(float(v[0] - double(h.x)), float(v[1] - double(h.y)), float(v[2] - double(h.z)),
                             float(v[3] - double(h.w)));
}

// residual matvec with the stored FP32 entries (TKlo null) or their pairs
template <bool E64>
static void matvec_df(mtf_system sys, const float* TK, const float* TKlo, const double* x, int64_t ldx, double* y,
                      int64_t ldy, int nrhs, cudaStream_t s) {
  mtf_mesh m = sys->mesh;
  const size_t nu = size_t(8) * m->n_rows * nrhs;
  if (sys->d_x32.n < nu) sys->d_x32.alloc(nu);
  float4* u = reinterpret_cast<float4*>(sys->d_x32.p);
  MTF_LAUNCH(KID_MISC, s, k_split_pm<<<unsigned((m->n_rows * nrhs + 255) / 256), 256, 0, s>>>(
      x, ldx, m->n_rows, nrhs, m->d_row_blk.p, m->d_blk_row_off.p, m->d_blk_N.p, m->d_blk_dof_off.p, sys->d_rho.p, u));
  const MvArgs A{TK, m->d_xent.p, sys->d_xval.p, m->d_mv_cta_prefix[1].p, m->d_blk_N.p, m->d_blk_dof_off.p,
                 m->d_blk_mat_off.p, m->d_blk_row_off.p, sys->d_rho.p, m->nd};
  const unsigned grid = unsigned(m->mv_cta_prefix[1].back());
  for (int c0 = 0; c0 < nrhs;) {
    const int nc = nrhs - c0 >= 4 ? 4 : nrhs - c0 >= 2 ? 2 : 1;
#define MTF_DF(NCV) \
  MTF_LAUNCH(KID_MATVEC64, s, k_matvec_df<E64, NCV, 2><<<grid, 256, 0, s>>>(A, TKlo, u, x, ldx, y, ldy, c0, m->n_rows))
    if (nc == 4) MTF_DF(4);
    else if (nc == 2) MTF_DF(2);
    else MTF_DF(1);
#undef MTF_DF
    c0 += nc;
  }
}

__global__ void k_to_f32(const double* __restrict__ x, int64_t ldx, int64_t n2, int nrhs, float* __restrict__ out) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= n2 * nrhs) return;
  const int64_t c = t / n2, k = t % n2;
  out[t] = float(x[2 * c * ldx + k]);
}

void launch_matvec_kind(mtf_system sys, int kind, const double* x, int64_t ldx, double* y, int64_t ldy,
                        int nrhs, cudaStream_t s) {
  mtf_mesh m = sys->mesh;
  if (kind == MV_AUTO) kind = sys->opt.precision == MTF_PREC_FP64 ? MV_FP64 : MV_FP32;
  if (kind == MV_FP64 && sys->opt.precision != MTF_PREC_FP64 && sys->d_TK64hl.p) {
    // mixed path with residual_fp64: the FP64 blocks as FP32 pairs, double-float sums
    matvec_df<true>(sys, sys->d_TK64hl.p, sys->d_TK64hl.p + size_t(m->n_mat) * 4, x, ldx, y, ldy, nrhs, s);
  } else if (kind == MV_FP64) {
    if (sys->d_rot64.p) matvec64<Ent::kRotated64>(sys, sys->d_rot64.p, x, ldx, y, ldy, nrhs, s);
    else matvec64<Ent::kBlocks64>(sys, sys->d_TK64.p, x, ldx, y, ldy, nrhs, s);
  } else if (kind == MV_FP32) {
    const int64_t n2 = 2 * m->n_total;
    if (sys->d_x32.n < size_t(n2) * nrhs) sys->d_x32.alloc(size_t(n2) * nrhs);
    MTF_LAUNCH(KID_MISC, s, k_to_f32<<<unsigned((n2 * nrhs + 255) / 256), 256, 0, s>>>(x, ldx, n2, nrhs, sys->d_x32.p));
    launch_matvec_stream64(sys, x, ldx, sys->d_x32.p, m->n_total, y, ldy, nrhs, s);
  } else if (sys->opt.residual_df) {
    // FP32 storage, double-float sums of the split input
    matvec_df<false>(sys, sys->d_TK32.p, nullptr, x, ldx, y, ldy, nrhs, s);
  } else {
    matvec64<Ent::kBlocks32>(sys, sys->d_TK32.p, x, ldx, y, ldy, nrhs, s);
  }
}

// y = M x with the operator as stored: FP64 storage and arithmetic on the FP64
// path and on the mixed path with residual_fp64; FP32 storage with
// double-float accumulation of the FP64 input (the refinement residual) on
// the mixed path otherwise.
void launch_matvec(mtf_system sys, const double* x, int64_t ldx, double* y, int64_t ldy, int nrhs,
                   cudaStream_t s) {
  const bool fp64 = sys->opt.precision == MTF_PREC_FP64 || sys->opt.residual_fp64;
  launch_matvec_kind(sys, fp64 ? MV_FP64 : MV_FP32_ACC64, x, ldx, y, ldy, nrhs, s);
}

}  // namespace mtf
