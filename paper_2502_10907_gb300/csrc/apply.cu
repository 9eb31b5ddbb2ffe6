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
// K x_D, K x_N, T x_D, T x_N.  FP64 systems keep the entries in this form
// (d_rot64, written with the mirrored blocks); FP32-stored entries (the
// residual_df = 0 residual) are rotated as they are read.
//
// Bound: the FP64 pipe (8 instructions per entry and right-hand side; the
// 32-byte entries would stream in an eighth of that time).  A CTA of 8 warps
// takes R rows per warp of one block; tiles of 128 columns of u+- are formed
// once per CTA in shared memory; the exchange entries join the lanes' sums
// before the reduction.  Rows per CTA (8, 16, 32) are chosen for the fewest
// rounds of CTAs over the SMs.  Measured on the split sphere of 11 rings (3
// blocks of 2,178 rows), 2 right-hand sides: 1,503 -> 470 us.
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

template <class MatT>
__device__ __forceinline__ void load_rotated(const void* entries, int64_t e, double* a) {
  if constexpr (sizeof(MatT) == 8) {
    const double2 p = __ldg(static_cast<const double2*>(entries) + 2 * e);
    const double2 m = __ldg(static_cast<const double2*>(entries) + 2 * e + 1);
    a[0] = p.x; a[1] = p.y; a[2] = m.x; a[3] = m.y;
  } else {
    const float4 v = __ldg(static_cast<const float4*>(entries) + e);  // T, K
    const double tr = v.x, ti = v.y, kr = v.z, ki = v.w;
    a[0] = kr + ti; a[1] = ki - tr; a[2] = kr - ti; a[3] = ki + tr;
  }
}

// y = M x for right-hand sides c0 .. c0 + NC - 1; R rows per warp
template <class MatT, int NC, int R>
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
      for (int r = 0; r < R; ++r) load_rotated<MatT>(A.entries, row[r] + n0 + n, a[r]);
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
    if (q < count) sums[warp][base + q] = acc[q];
  __syncwarp();
  if (lane < R * NC) {
    const int r = lane / NC, c = lane % NC;
    if (m0 + r < N) {
      const double* s = sums[warp] + 4 * lane;
      double2* yc = reinterpret_cast<double2*>(y) + int64_t(c0 + c) * ldy + off + m0 + r;
      yc[0] = make_double2(s[0] + s[2], s[1] + s[3]);
      yc[N] = make_double2(rho * (s[1] - s[3]), rho * (s[2] - s[0]));
    }
  }
}

template <class MatT, int NC, int R>
static void mv64_launch(mtf_system sys, const MvArgs& A, unsigned grid, const double* x, int64_t ldx, double* y,
                        int64_t ldy, int c0, cudaStream_t s) {
  MTF_LAUNCH(KID_MATVEC64, s, launch_pdl(k_matvec<MatT, NC, R>, dim3(grid), dim3(256), 0, s, A, x, ldx, y, ldy, c0));
}

// passes of up to 4 right-hand sides
template <class MatT>
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
#define MTF_MV(NCV, RV) mv64_launch<MatT, NCV, RV>(sys, A, grid, x, ldx, y, ldy, c0, s)
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
// a x_lo added to e, p added to the running (hi, lo) pair by an error-free
// two-sum.  The sums carry about 2^-46 relative error against a few times
// 2^-53 for FP64 FMAs, at FP32 throughput instead of the narrow FP64 pipe.
// Lanes convert to FP64 for the warp reduction and the FP64 epilogue (rho,
// exchange).
// (the _rn intrinsics keep the compiler from contracting the product into
// the sum, which would break the error-free transformations)
__device__ __forceinline__ void df_mac(float& hi, float& lo, float a, float xh, float xl) {
  const float p = __fmul_rn(a, xh);
  float e = fmaf(a, xh, -p);  // exact: a xh = p + e
  e = fmaf(a, xl, e);
  const float s = __fadd_rn(hi, p);  // two-sum of hi and p
  const float z = __fsub_rn(s, hi);
  const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, z)), __fsub_rn(p, z));
  hi = s;
  lo = __fadd_rn(lo, __fadd_rn(err, e));
}

// E64: the operator is the FP64 blocks, given as FP32 pairs (TK = fl(v),
// TKlo = fl(v - fl(v)), split once per assembly): every product adds the
// lo part times the input's hi part to the running lo sum, so the residual
// of the FP64-assembled system costs FP32 work (residual_fp64).
template <bool E64>
__global__ void __launch_bounds__(256) k_matvec_df(
    const float* __restrict__ TK, const float* __restrict__ TKlo, const XEntry* __restrict__ xe,
    const double* __restrict__ xval,
    const int32_t* __restrict__ row_blk, const int64_t* __restrict__ blk_row_off,
    const int32_t* __restrict__ blk_N, const int64_t* __restrict__ blk_dof_off,
    const int64_t* __restrict__ blk_mat_off, const double* __restrict__ rho, const double* __restrict__ x,
    int64_t ldx, const float* __restrict__ xh, const float* __restrict__ xl, int64_t ldxv, double* __restrict__ y,
    int64_t ldy, int nrhs, int64_t n_rows) {
  const int64_t r = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (r >= n_rows) return;
  const int i = row_blk[r];
  const int64_t m = r - blk_row_off[i];
  const int N = blk_N[i];
  const int64_t off = blk_dof_off[i];
  const float* row = TK + 4 * (blk_mat_off[i] + m * N);
  const float* rowlo = E64 ? TKlo + 4 * (blk_mat_off[i] + m * N) : nullptr;
  const double rr = rho[2 * i], ri = rho[2 * i + 1];
  const double rn = rr * rr + ri * ri;
  const double ir = rr / rn, ii = -ri / rn;  // 1 / rho
  for (int c0 = 0; c0 < nrhs; c0 += 2) {
    const int nc = min(2, nrhs - c0);
    float ah[2][8], al[2][8];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int q = 0; q < 8; ++q) ah[c][q] = al[c][q] = 0.f;
    constexpr int U = 4;
    for (int n0 = lane; n0 < N; n0 += 32 * U) {
      float4 e[U], el[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int n = n0 + 32 * u;
        if (n < N) {
          e[u] = __ldg(reinterpret_cast<const float4*>(row) + n);
          if constexpr (E64) el[u] = __ldg(reinterpret_cast<const float4*>(rowlo) + n);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int n = n0 + 32 * u;
        if (n >= N) break;
        const float Tr = e[u].x, Ti = e[u].y, Kr = e[u].z, Ki = e[u].w;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if (c < nc) {
            const int64_t o = 2 * (int64_t(c0 + c) * ldxv + off);
            const float2 dh = *reinterpret_cast<const float2*>(xh + o + 2 * n);
            const float2 dl = *reinterpret_cast<const float2*>(xl + o + 2 * n);
            const float2 nh = *reinterpret_cast<const float2*>(xh + o + 2 * (N + n));
            const float2 nl = *reinterpret_cast<const float2*>(xl + o + 2 * (N + n));
            float* H = ah[c];
            float* Lo = al[c];
            // T xd, T xn, K xd, K xn
            df_mac(H[0], Lo[0], Tr, dh.x, dl.x);
            df_mac(H[0], Lo[0], -Ti, dh.y, dl.y);
            df_mac(H[1], Lo[1], Tr, dh.y, dl.y);
            df_mac(H[1], Lo[1], Ti, dh.x, dl.x);
            df_mac(H[2], Lo[2], Tr, nh.x, nl.x);
            df_mac(H[2], Lo[2], -Ti, nh.y, nl.y);
            df_mac(H[3], Lo[3], Tr, nh.y, nl.y);
            df_mac(H[3], Lo[3], Ti, nh.x, nl.x);
            df_mac(H[4], Lo[4], Kr, dh.x, dl.x);
            df_mac(H[4], Lo[4], -Ki, dh.y, dl.y);
            df_mac(H[5], Lo[5], Kr, dh.y, dl.y);
            df_mac(H[5], Lo[5], Ki, dh.x, dl.x);
            df_mac(H[6], Lo[6], Kr, nh.x, nl.x);
            df_mac(H[6], Lo[6], -Ki, nh.y, nl.y);
            df_mac(H[7], Lo[7], Kr, nh.y, nl.y);
            df_mac(H[7], Lo[7], Ki, nh.x, nl.x);
            if constexpr (E64) {
              // the entries' lo parts times the inputs' hi parts
              const float tr = el[u].x, ti = el[u].y, kr = el[u].z, ki = el[u].w;
              Lo[0] = fmaf(tr, dh.x, fmaf(-ti, dh.y, Lo[0]));
              Lo[1] = fmaf(tr, dh.y, fmaf(ti, dh.x, Lo[1]));
              Lo[2] = fmaf(tr, nh.x, fmaf(-ti, nh.y, Lo[2]));
              Lo[3] = fmaf(tr, nh.y, fmaf(ti, nh.x, Lo[3]));
              Lo[4] = fmaf(kr, dh.x, fmaf(-ki, dh.y, Lo[4]));
              Lo[5] = fmaf(kr, dh.y, fmaf(ki, dh.x, Lo[5]));
              Lo[6] = fmaf(kr, nh.x, fmaf(-ki, nh.y, Lo[6]));
              Lo[7] = fmaf(kr, nh.y, fmaf(ki, nh.x, Lo[7]));
            }
          }
        }
      }
    }
    double acc[2][8];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        double v = double(ah[c][q]) + double(al[c][q]);
#pragma unroll
        for (int s2 = 16; s2 > 0; s2 >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s2);
        acc[c][q] = v;
      }
    if (lane < nc) {
      double a[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) a[q] = lane == 0 ? acc[0][q] : acc[1][q];
      const int col = c0 + lane;
      const double* xc = x + 2 * int64_t(col) * ldx;
      // yD = 2 (Kx + Ty / rho), yN = 2 (-rho Tx + Ky)
      double yDr = 2.0 * (a[4] + (a[2] * ir - a[3] * ii));
      double yDi = 2.0 * (a[5] + (a[2] * ii + a[3] * ir));
      double yNr = 2.0 * (a[6] - (a[0] * rr - a[1] * ri));
      double yNi = 2.0 * (a[7] - (a[0] * ri + a[1] * rr));
#pragma unroll
      for (int e2 = 0; e2 < 6; ++e2) {
        const XEntry X = xe[6 * r + e2];
        const double v = xval[6 * r + e2];
        const int Nj = X.ab >> 4;
        yDr += v * xc[2 * int64_t(X.col)];
        yDi += v * xc[2 * int64_t(X.col) + 1];
        yNr += v * xc[2 * (int64_t(X.col) + Nj)];
        yNi += v * xc[2 * (int64_t(X.col) + Nj) + 1];
      }
      double* yc = y + 2 * (int64_t(col) * ldy + off);
      yc[2 * m] = yDr;
      yc[2 * m + 1] = yDi;
      yc[2 * (N + m)] = yNr;
      yc[2 * (N + m) + 1] = yNi;
    }
  }
}

// x (FP64, column stride ldx) -> FP32 pair hi = fl(x), lo = fl(x - hi), n2
// reals per column, columns packed
__global__ void k_split_f32(const double* __restrict__ x, int64_t ldx, int64_t n2, int nrhs, float* __restrict__ hi,
                            float* __restrict__ lo) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t >= n2 * nrhs) return;
  const int64_t c = t / n2, k = t % n2;
  const double v = x[2 * c * ldx + k];
  const float h = float(v);
  hi[t] = h;
  lo[t] = float(v - double(h));
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
  const unsigned blocks = unsigned((m->n_rows * 32 + 255) / 256);
  if (kind == MV_AUTO) kind = sys->opt.precision == MTF_PREC_FP64 ? MV_FP64 : MV_FP32;
  if (kind == MV_FP64 && sys->opt.precision != MTF_PREC_FP64 && sys->d_TK64hl.p) {
    // mixed path with residual_fp64: the FP64 blocks as FP32 pairs, double-float sums
    const int64_t n2 = 2 * m->n_total;
    if (sys->d_x32.n < 2 * size_t(n2) * nrhs) sys->d_x32.alloc(2 * size_t(n2) * nrhs);
    float* xh = sys->d_x32.p;
    float* xl = xh + size_t(n2) * nrhs;
    MTF_LAUNCH(KID_MISC, s, k_split_f32<<<unsigned((n2 * nrhs + 255) / 256), 256, 0, s>>>(x, ldx, n2, nrhs, xh, xl));
    MTF_LAUNCH(KID_MATVEC64, s, k_matvec_df<true><<<blocks, 256, 0, s>>>(
        sys->d_TK64hl.p, sys->d_TK64hl.p + size_t(m->n_mat) * 4, m->d_xent.p, sys->d_xval.p, m->d_row_blk.p,
        m->d_blk_row_off.p, m->d_blk_N.p, m->d_blk_dof_off.p, m->d_blk_mat_off.p, sys->d_rho.p, x, ldx, xh, xl,
        m->n_total, y, ldy, nrhs, m->n_rows));
  } else if (kind == MV_FP64) {
    matvec64<double>(sys, sys->d_rot64.p, x, ldx, y, ldy, nrhs, s);
  } else if (kind == MV_FP32) {
    const int64_t n2 = 2 * m->n_total;
    if (sys->d_x32.n < size_t(n2) * nrhs) sys->d_x32.alloc(size_t(n2) * nrhs);
    MTF_LAUNCH(KID_MISC, s, k_to_f32<<<unsigned((n2 * nrhs + 255) / 256), 256, 0, s>>>(x, ldx, n2, nrhs, sys->d_x32.p));
    launch_matvec_stream64(sys, x, ldx, sys->d_x32.p, m->n_total, y, ldy, nrhs, s);
  } else if (sys->opt.residual_df) {
    // FP32 storage, double-float sums of the split input
    const int64_t n2 = 2 * m->n_total;
    if (sys->d_x32.n < 2 * size_t(n2) * nrhs) sys->d_x32.alloc(2 * size_t(n2) * nrhs);
    float* xh = sys->d_x32.p;
    float* xl = xh + size_t(n2) * nrhs;
    MTF_LAUNCH(KID_MISC, s, k_split_f32<<<unsigned((n2 * nrhs + 255) / 256), 256, 0, s>>>(x, ldx, n2, nrhs, xh, xl));
    MTF_LAUNCH(KID_MATVEC64, s, k_matvec_df<false><<<blocks, 256, 0, s>>>(
        sys->d_TK32.p, nullptr, m->d_xent.p, sys->d_xval.p, m->d_row_blk.p, m->d_blk_row_off.p, m->d_blk_N.p,
        m->d_blk_dof_off.p, m->d_blk_mat_off.p, sys->d_rho.p, x, ldx, xh, xl, m->n_total, y, ldy, nrhs, m->n_rows));
  } else {
    matvec64<float>(sys, sys->d_TK32.p, x, ldx, y, ldy, nrhs, s);
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
