// Restarted flexible GMRES for M u = b (Sec. 5.3: relative tolerance and an
// iteration cap), batched over right-hand sides: every right-hand side has its
// own Krylov basis, all of them advance together so that each operator apply
// is one multi-column matvec.  Orthogonalisation is classical Gram-Schmidt
// applied twice (CGS2) in FP64 on the device; the small Hessenberg least-
// squares problems (Givens rotations) run on the host from the (j+2) new
// Hessenberg entries per right-hand side copied back each iteration, while
// the device runs the next one (an iteration queued past convergence is
// discarded).  A
// restart cycle ends on convergence of every right-hand side, on the restart
// length or on the iteration cap; each cycle starts from the true residual
// b - M x, which is also the stopping test.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdlib>
#include <complex>

#include "common.h"
#include "kernel64.cuh"

namespace mtf {

using cd = std::complex<double>;

struct GmresWork {
  int nrhs = 0, m = 0;
  int64_t n = 0;
  DevBuf<double> V, Z, w, r, b, y;
  // two slots of [hA (m+1) x nrhs][hB (m+1) x nrhs][norm nrhs] complex [sum of
  // squares nrhs]: step j of a cycle uses slot j mod 2 with j + 1 in place of
  // m + 1, the norms outside the steps use slot 0 in full
  DevBuf<double> h;
  double* h_host = nullptr;
  cudaEvent_t ev[2] = {nullptr, nullptr};
  int sms = 0;
  ~GmresWork() {
    if (h_host) cudaFreeHost(h_host);
    for (auto& e : ev)
      if (e) cudaEventDestroy(e);
  }
};

void destroy_gmres(GmresWork* w) { delete w; }

// nrm[c] = ||w^c||, out^c = w^c / nrm[c] (zero if nrm is 0); one CTA per c
__global__ void __launch_bounds__(1024) k_norm_scale(const double* __restrict__ w, int64_t n,
                                                      double* __restrict__ nrm, double* __restrict__ out,
                                                      int64_t out_stride) {
  const int c = blockIdx.x;
  const double2* x = reinterpret_cast<const double2*>(w) + int64_t(c) * n;
  double s = 0;
  for (int64_t k = threadIdx.x; k < n; k += blockDim.x) s += x[k].x * x[k].x + x[k].y * x[k].y;
  __shared__ double red[32];
  __shared__ double tot;
  for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0;
    for (int q = 0; q < int(blockDim.x >> 5); ++q) a += red[q];
    tot = sqrt(a);
    nrm[2 * c] = tot;
    nrm[2 * c + 1] = 0.0;
  }
  __syncthreads();
  const double inv = tot > 0 ? 1.0 / tot : 0.0;
  double2* o = reinterpret_cast<double2*>(out) + int64_t(c) * out_stride;
  for (int64_t k = threadIdx.x; k < n; k += blockDim.x) o[k] = make_double2(x[k].x * inv, x[k].y * inv);
}

__global__ void k_sub(const double* __restrict__ a, const double* __restrict__ b, double* __restrict__ out,
                      int64_t n2) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t < n2) out[t] = a[t] - b[t];
}

static inline unsigned nblk(int64_t n, int t) { return unsigned((n + t - 1) / t); }

// Gram-Schmidt kernels of the FP64 Arnoldi step.  Bound: the FP64 pipe (4
// instructions per entry and basis vector) once every SM has work; on small
// systems (2,000 unknowns) the former kernels ran on 60 to 80 of the 152 SMs.
// Measured there at 300 basis vectors: dots 20 -> 12 us, update 22 -> 12 us (with launch events).

// h[c ldh + i] += sum over a segment of conj(V_i^c) w^c: one warp per (pair of
// basis vectors, segment, right-hand side), the pairs of a segment in
// consecutive warps (w's segment stays in L1); segments so that about 16
// warps per SM run whatever the number of basis vectors is
__global__ void __launch_bounds__(256) k_dots64(const double* __restrict__ V, const double* __restrict__ w, int64_t n,
                                                int ldv, int rows, int nseg, int64_t seg, int nrhs,
                                                double* __restrict__ h, int ldh) {
  MTF_PDL_WAIT();
  MTF_PDL_TRIGGER();
  const int pairs = (rows + 1) / 2;
  const int64_t id = (int64_t(blockIdx.x) * 256 + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (id >= int64_t(pairs) * nseg * nrhs) return;
  const int i0 = 2 * int(id % pairs), g = int(id / pairs % nseg), c = int(id / (int64_t(pairs) * nseg));
  const int64_t k0 = g * seg, k1 = min(n, k0 + seg);
  const double2* v0 = reinterpret_cast<const double2*>(V) + (int64_t(c) * ldv + i0) * n;
  const double2* v1 = i0 + 1 < rows ? v0 + n : v0;
  const double2* x = reinterpret_cast<const double2*>(w) + int64_t(c) * n;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
  for (int64_t k = k0 + lane; k < k1; k += 32) {
    const double2 a = v0[k], b = v1[k], t = x[k];
    v[0] = fma(a.x, t.x, fma(a.y, t.y, v[0]));
    v[1] = fma(a.x, t.y, fma(-a.y, t.x, v[1]));
    v[2] = fma(b.x, t.x, fma(b.y, t.y, v[2]));
    v[3] = fma(b.x, t.y, fma(-b.y, t.x, v[3]));
  }
  int base = 0, count = 4;
  halve_sum<4>(v, lane, 16, base, count);
  if (count > 0 && i0 + base / 2 < rows) atomicAdd(h + 2 * (int64_t(c) * ldh + i0) + base, v[0]);
}

static void launch_dots(const double* V, const double* w, int64_t n, int ldv, int rows, double* h, int ldh, int nrhs,
                        int sms, cudaStream_t s) {
  const int64_t pairs = (rows + 1) / 2;
  const int64_t nseg = std::max<int64_t>(1, std::min<int64_t>((n + 63) / 64, 16 * sms / (pairs * nrhs)));
  const int64_t seg = (n + nseg - 1) / nseg;
  MTF_LAUNCH(KID_DOTS, s, launch_pdl(k_dots64, dim3(nblk(pairs * nseg * nrhs, 8)), dim3(256), 0, s, V, w, n, ldv, rows,
                                     int(nseg), seg, nrhs, h, ldh));
}

// w^c += sign sum_{i<j} V_i^c h_i^c ; optionally ss[c] += ||w^c||^2 (after update).
// CTA = 8 consecutive rows (a 128-byte run of every vector) x 32 groups of
// basis vectors (i = group mod 32): 8 lanes and 4 groups per warp
__global__ void __launch_bounds__(256) k_axpy64(const double* __restrict__ V, const double* __restrict__ h, int j,
                                                int64_t n, int ldv, int ldh, double sign, double* __restrict__ w,
                                                double* __restrict__ ss) {
  MTF_PDL_WAIT();
  MTF_PDL_TRIGGER();
  const int c = blockIdx.y;
  const int r = threadIdx.x & 7, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t k = int64_t(blockIdx.x) * 8 + r;
  __shared__ double2 part[8][8];
  const double2* hc = reinterpret_cast<const double2*>(h) + int64_t(c) * ldh;
  const double2* v = reinterpret_cast<const double2*>(V) + int64_t(c) * ldv * n + min(k, n - 1);
  double sr = 0, si = 0;
#pragma unroll 8
  for (int i = threadIdx.x >> 3; i < j; i += 32) {
    const double2 a = v[int64_t(i) * n], t = hc[i];
    sr = fma(a.x, t.x, fma(-a.y, t.y, sr));
    si = fma(a.x, t.y, fma(a.y, t.x, si));
  }
#pragma unroll
  for (int o = 8; o < 32; o <<= 1) {
    sr += __shfl_xor_sync(0xffffffffu, sr, o);
    si += __shfl_xor_sync(0xffffffffu, si, o);
  }
  if (lane < 8) part[warp][r] = make_double2(sr, si);
  __syncthreads();
  if (threadIdx.x < 8) {
    double sq = 0;
    if (k < n) {
      double tr = 0, ti = 0;
#pragma unroll
      for (int g = 0; g < 8; ++g) {
        tr += part[g][r].x;
        ti += part[g][r].y;
      }
      double2* x = reinterpret_cast<double2*>(w) + int64_t(c) * n + k;
      double2 o = *x;
      o.x = fma(sign, tr, o.x);
      o.y = fma(sign, ti, o.y);
      *x = o;
      sq = fma(o.x, o.x, o.y * o.y);
    }
    if (ss) {
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) sq += __shfl_xor_sync(0xffu, sq, o);
      if (threadIdx.x == 0) atomicAdd(ss + c, sq);
    }
  }
}

static void launch_axpy(const double* V, const double* h, int j, int64_t n, int ldv, int ldh, double sign, double* w,
                        double* ss, int nrhs, cudaStream_t s) {
  MTF_LAUNCH(KID_AXPY, s, launch_pdl(k_axpy64, dim3(nblk(n, 8), unsigned(nrhs)), dim3(256), 0, s, V, h, j, n, ldv, ldh,
                                     sign, w, ss));
}

// out^c = w^c / sqrt(ss[c]) (zero if 0); nrm[c] = (sqrt(ss[c]), 0); clears the
// nclear accumulators of the next step
__global__ void __launch_bounds__(256) k_scale(const double* __restrict__ w, int64_t n, const double* __restrict__ ss,
                                               double* __restrict__ nrm, double* __restrict__ out, int64_t out_stride,
                                               double* __restrict__ clear, int64_t nclear) {
  MTF_PDL_WAIT();
  MTF_PDL_TRIGGER();
  const int c = blockIdx.y;
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (c == 0)
    for (int64_t q = k; q < nclear; q += int64_t(gridDim.x) * blockDim.x) clear[q] = 0.0;
  const double t = sqrt(ss[c]);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    nrm[2 * c] = t;
    nrm[2 * c + 1] = 0.0;
  }
  if (k >= n) return;
  const double inv = t > 0 ? 1.0 / t : 0.0;
  const double2 a = reinterpret_cast<const double2*>(w)[int64_t(c) * n + k];
  reinterpret_cast<double2*>(out)[int64_t(c) * out_stride + k] = make_double2(a.x * inv, a.y * inv);
}

// One restarted GMRES solve of M x = b (x starts at 0) with the given matvec
// flavour.  Per right-hand side: iters[c] += inner iterations, rel[c] = final
// true relative residual (w.r.t. the same flavour).
static mtf_status gmres_core(mtf_system sys, int nrhs, const double* b_dev, double* x_dev, int mvkind,
                             double tol, int max_iter, std::vector<int>& iters, int& restarts,
                             std::vector<double>& rel, cudaStream_t s) {
  mtf_mesh msh = sys->mesh;
  const int64_t n = msh->n_total;
  const int m = std::max(1, sys->opt.restart);
  GmresWork& G = *sys->gw;
  double* hN = G.h.p + 4 * size_t(m + 1) * nrhs;
  double* hostN = G.h_host + 4 * size_t(m + 1) * nrhs;
  const size_t slot = G.h.n / 2;
  const int ldv = m + 1;
  const size_t vec_bytes = size_t(n) * nrhs * 2 * sizeof(double);

  std::vector<double> bnorm(nrhs);
  MTF_LAUNCH(KID_NORM, s, k_norm_scale<<<nrhs, 1024, 0, s>>>(b_dev, n, hN, G.w.p, n));
  MTF_CUDA(cudaMemcpyAsync(hostN, hN, size_t(nrhs) * 2 * sizeof(double), cudaMemcpyDeviceToHost, s));
  MTF_CUDA(cudaStreamSynchronize(s));
  for (int c = 0; c < nrhs; ++c) bnorm[c] = hostN[2 * c] > 0 ? hostN[2 * c] : 1.0;
  MTF_CUDA(cudaMemsetAsync(x_dev, 0, vec_bytes, s));

  std::vector<int> done(nrhs, 0), jc(nrhs, 0);
  std::vector<cd> H(size_t(m + 1) * m * nrhs), g(size_t(m + 1) * nrhs), sn(size_t(m) * nrhs);
  std::vector<double> cs(size_t(m) * nrhs);
  std::vector<double> yhost(size_t(m + 1) * nrhs * 2);
  int total = 0;
  bool first = true;
  mtf_status status = MTF_OK;
  const bool pre = sys->opt.precond == MTF_PRECOND_OSRC;
  if (pre && G.Z.n != size_t(m) * n * nrhs * 2) G.Z.alloc(size_t(m) * n * nrhs * 2);
  while (true) {
    // true residual r = b - M x and its norm; V_0 = r / ||r||
    if (first) {
      MTF_CUDA(cudaMemcpyAsync(G.r.p, b_dev, vec_bytes, cudaMemcpyDeviceToDevice, s));
    } else {
      launch_matvec_kind(sys, mvkind, x_dev, n, G.w.p, n, nrhs, s);
      MTF_LAUNCH(KID_SUB, s, k_sub<<<nblk(n * nrhs * 2, 256), 256, 0, s>>>(b_dev, G.w.p, G.r.p, n * nrhs * 2));
    }
    first = false;
    MTF_LAUNCH(KID_NORM, s, k_norm_scale<<<nrhs, 1024, 0, s>>>(G.r.p, n, hN, G.V.p, int64_t(ldv) * n));
    MTF_CUDA(cudaMemcpyAsync(hostN, hN, size_t(nrhs) * 2 * sizeof(double), cudaMemcpyDeviceToHost, s));
    MTF_CUDA(cudaStreamSynchronize(s));
    bool all = true;
    for (int c = 0; c < nrhs; ++c) {
      rel[c] = hostN[2 * c] / bnorm[c];
      if (!std::isfinite(rel[c])) status = MTF_ERR_NAN;
      done[c] = rel[c] <= tol;
      all = all && done[c];
      jc[c] = 0;
      std::fill(g.begin() + size_t(c) * (m + 1), g.begin() + size_t(c + 1) * (m + 1), cd(0));
      g[size_t(c) * (m + 1)] = hostN[2 * c];
    }
    if (status != MTF_OK) break;
    if (all) break;
    if (total >= max_iter) {
      status = MTF_ERR_NOCONV;
      break;
    }
    ++restarts;
    std::vector<int> active(nrhs);
    for (int c = 0; c < nrhs; ++c) active[c] = !done[c];
    // step j: z_j = P v_j (flexible right preconditioning), w = M z_j, CGS2
    // h_A = V^H w, w -= V h_A, h_B = V^H w, w -= V h_B (with ||w||^2),
    // v_{j+1} = w / ||w||, all on the device; its coefficients go to the
    // pinned slot j mod 2
    auto launch_step = [&](int j) {
      if (pre) {
        launch_osrc_apply(sys, G.V.p + 2 * size_t(j) * n, int64_t(ldv) * n, G.Z.p + 2 * size_t(j) * n,
                          int64_t(m) * n, nrhs, s);
        launch_matvec_kind(sys, mvkind, G.Z.p + 2 * size_t(j) * n, int64_t(m) * n, G.r.p, n, nrhs, s);
      } else {
        launch_matvec_kind(sys, mvkind, G.V.p + 2 * size_t(j) * n, int64_t(ldv) * n, G.r.p, n, nrhs, s);
      }
      const size_t L = size_t(j) + 1;
      double* hA = G.h.p + (j & 1) * slot;
      double* hB = hA + 2 * L * nrhs;
      double* nrm = hB + 2 * L * nrhs;
      double* ss = nrm + 2 * nrhs;  // sum of squares scratch after the norms
      launch_dots(G.V.p, G.r.p, n, ldv, j + 1, hA, j + 1, nrhs, G.sms, s);
      launch_axpy(G.V.p, hA, j + 1, n, ldv, j + 1, -1.0, G.r.p, nullptr, nrhs, s);
      launch_dots(G.V.p, G.r.p, n, ldv, j + 1, hB, j + 1, nrhs, G.sms, s);
      launch_axpy(G.V.p, hB, j + 1, n, ldv, j + 1, -1.0, G.r.p, ss, nrhs, s);
      MTF_LAUNCH(KID_NORM, s, launch_pdl(k_scale, dim3(nblk(n, 256), unsigned(nrhs)), dim3(256), 0, s, G.r.p, n, ss, nrm,
                                         G.V.p + 2 * size_t(j + 1) * n, int64_t(ldv) * n, G.h.p + ((j + 1) & 1) * slot,
                                         int64_t(4 * (L + 1) + 3) * nrhs));
      MTF_CUDA(cudaMemcpyAsync(G.h_host + (j & 1) * slot, hA, (4 * L + 2) * nrhs * sizeof(double),
                               cudaMemcpyDeviceToHost, s));
      MTF_CUDA(cudaEventRecord(G.ev[j & 1], s));
    };
    MTF_CUDA(cudaMemsetAsync(G.h.p, 0, 7 * size_t(nrhs) * sizeof(double), s));  // step 0's accumulators
    launch_step(0);
    for (int j = 0; j < m && total < max_iter; ++j) {
      if (j + 1 < m && total + 1 < max_iter) launch_step(j + 1);
      MTF_CUDA(cudaEventSynchronize(G.ev[j & 1]));
      const double* hostA = G.h_host + (j & 1) * slot;
      const double* hostB = hostA + 2 * size_t(j + 1) * nrhs;
      const double* hostW = hostB + 2 * size_t(j + 1) * nrhs;
      ++total;
      bool all_done = true;
      for (int c = 0; c < nrhs; ++c) {
        if (!active[c]) continue;
        cd* Hc = &H[size_t(c) * (m + 1) * m + size_t(j) * (m + 1)];
        for (int q = 0; q <= j; ++q)
          Hc[q] = cd(hostA[2 * (size_t(c) * (j + 1) + q)] + hostB[2 * (size_t(c) * (j + 1) + q)],
                     hostA[2 * (size_t(c) * (j + 1) + q) + 1] + hostB[2 * (size_t(c) * (j + 1) + q) + 1]);
        Hc[j + 1] = cd(hostW[2 * c], 0.0);
        // previous rotations
        for (int q = 0; q < j; ++q) {
          const double cq = cs[size_t(c) * m + q];
          const cd sq = sn[size_t(c) * m + q];
          const cd t = cq * Hc[q] + sq * Hc[q + 1];
          Hc[q + 1] = -std::conj(sq) * Hc[q] + cq * Hc[q + 1];
          Hc[q] = t;
        }
        // new rotation zeroing H[j+1, j]
        const cd a = Hc[j], bb = Hc[j + 1];
        const double an = std::abs(a), bn = std::abs(bb), tt = std::hypot(an, bn);
        double cj;
        cd sj;
        if (tt == 0) {
          cj = 1.0;
          sj = 0.0;
        } else if (an == 0) {
          cj = 0.0;
          sj = std::conj(bb) / tt;
          Hc[j] = tt;
        } else {
          cj = an / tt;
          sj = (a / an) * std::conj(bb) / tt;
          Hc[j] = (a / an) * tt;
        }
        Hc[j + 1] = 0.0;
        cs[size_t(c) * m + j] = cj;
        sn[size_t(c) * m + j] = sj;
        cd* gc = &g[size_t(c) * (m + 1)];
        gc[j + 1] = -std::conj(sj) * gc[j];
        gc[j] = cj * gc[j];
        jc[c] = j + 1;
        ++iters[c];
        const double est = std::abs(gc[j + 1]) / bnorm[c];
        if (!std::isfinite(est)) status = MTF_ERR_NAN;
        if (est <= tol * 0.5 || hostW[2 * c] == 0.0) active[c] = 0;
        all_done = all_done && !active[c];
      }
      if (status != MTF_OK || all_done) break;
    }
    if (status != MTF_OK) break;
    // x += V y, y = R^{-1} g per right-hand side
    std::fill(yhost.begin(), yhost.end(), 0.0);
    int jmax = 0;
    for (int c = 0; c < nrhs; ++c) {
      const int jj = jc[c];
      jmax = std::max(jmax, jj);
      const cd* Hc = &H[size_t(c) * (m + 1) * m];
      std::vector<cd> yy(jj);
      for (int q = jj - 1; q >= 0; --q) {
        cd acc = g[size_t(c) * (m + 1) + q];
        for (int p = q + 1; p < jj; ++p) acc -= Hc[size_t(p) * (m + 1) + q] * yy[p];
        yy[q] = acc / Hc[size_t(q) * (m + 1) + q];
      }
      for (int q = 0; q < jj; ++q) {
        yhost[2 * (size_t(c) * (m + 1) + q)] = yy[q].real();
        yhost[2 * (size_t(c) * (m + 1) + q) + 1] = yy[q].imag();
      }
    }
    if (jmax > 0) {
      MTF_CUDA(cudaMemcpyAsync(G.y.p, yhost.data(), yhost.size() * sizeof(double), cudaMemcpyHostToDevice, s));
      // x += Z y (flexible) or V y
      launch_axpy(pre ? G.Z.p : G.V.p, G.y.p, jmax, n, pre ? m : ldv, m + 1, 1.0, x_dev, nullptr, nrhs, s);
      MTF_CUDA(cudaStreamSynchronize(s));  // yhost is reused next cycle
    }
  }
  return status;
}

// Fewest right-hand sides for which the block cycle is used.  With 2 waves
// of one incidence direction (the split sphere) the block space needed as
// many steps as each single space (437 against 440) and its per-step host
// synchronisation made the solve slower; with 16 waves of 8 directions (the
// 4 x 4 x 4 cube) it needed 838 block steps where single spaces needed
// about 6,000 iterations.
constexpr int kBlockMinRhs = 4;

__global__ void k_add(double* __restrict__ x, const double* __restrict__ d, int64_t n2) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t < n2) x[t] += d[t];
}

mtf_status solve(mtf_system sys, int nrhs, const double* b_dev, double* x_dev, mtf_solve_stats* st,
                 cudaStream_t s) {
  const auto t0 = std::chrono::steady_clock::now();
  sys->t_launch = sys->t_lsq = sys->t_wait = 0;
  mtf_mesh msh = sys->mesh;
  const int64_t n = msh->n_total;
  const int m = std::max(1, sys->opt.restart);
  if (!sys->gw) sys->gw = new GmresWork();
  GmresWork& G = *sys->gw;
  const bool mixed = sys->opt.precision != MTF_PREC_FP64;
  sys->learned_active = false;  // the learned correction runs in the mixed path only
  if (G.nrhs != nrhs || G.m != m || G.n != n) {
    G.V.alloc(size_t(m + 1) * n * nrhs * 2);
    G.w.alloc(size_t(n) * nrhs * 2);
    G.r.alloc(size_t(n) * nrhs * 2);
    G.y.alloc(size_t(m + 1) * nrhs * 2);
    G.h.alloc(2 * size_t(2 * (m + 1) + 2) * nrhs * 2);
    if (G.h_host) cudaFreeHost(G.h_host);
    G.h_host = nullptr;
    MTF_CUDA(cudaMallocHost(&G.h_host, G.h.n * sizeof(double)));
    for (auto& e : G.ev)
      if (!e) MTF_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    int dev = 0;
    MTF_CUDA(cudaGetDevice(&dev));
    MTF_CUDA(cudaDeviceGetAttribute(&G.sms, cudaDevAttrMultiProcessorCount, dev));
    G.nrhs = nrhs;
    G.m = m;
    G.n = n;
  }
  std::vector<int> iters(nrhs, 0);
  std::vector<double> rel(nrhs, 1.0);
  int restarts = 0, refinements = 0;
  const int max_iter = std::max(1, sys->opt.max_iter);
  mtf_status status = MTF_OK;
  if (!mixed) {
    status = gmres_core(sys, nrhs, b_dev, x_dev, MV_FP64, sys->opt.tol, max_iter, iters, restarts, rel, s);
  } else {
    // FP64 iterative refinement: r = b - M x with FP64 accumulation over the
    // FP32-stored operator; each correction is one FGMRES cycle in FP32
    // (fgmres_cycle32) that adds its update to x.  A cycle that ends on the
    // restart length is a restart (the next one starts from the new FP64
    // residual); one that reaches its tolerance ends a refinement step.
    if (G.b.n != size_t(n) * nrhs * 2) G.b.alloc(size_t(n) * nrhs * 2);  // residual
    const size_t vec_bytes = size_t(n) * nrhs * 2 * sizeof(double);
    double* hN = G.h.p + 4 * size_t(m + 1) * nrhs;
    double* hostN = G.h_host + 4 * size_t(m + 1) * nrhs;
    std::vector<double> bnorm(nrhs);
    MTF_LAUNCH(KID_NORM, s, k_norm_scale<<<nrhs, 1024, 0, s>>>(b_dev, n, hN, G.w.p, n));
    MTF_CUDA(cudaMemcpyAsync(hostN, hN, size_t(nrhs) * 2 * sizeof(double), cudaMemcpyDeviceToHost, s));
    MTF_CUDA(cudaStreamSynchronize(s));
    for (int c = 0; c < nrhs; ++c) bnorm[c] = hostN[2 * c] > 0 ? hostN[2 * c] : 1.0;
    MTF_CUDA(cudaMemsetAsync(x_dev, 0, vec_bytes, s));
    const int max_ref = std::max(1, sys->opt.max_refine);
    int total = 0;
    // learned correction: used while it keeps the FP64 residual falling; a
    // cycle that fails to reduce it by 5% falls back to plain block-OSRC
    sys->learned_active = sys->opt.learned && sys->learned && sys->opt.precond == MTF_PRECOND_OSRC;
    double prev_rmax = -1.0;
    for (int it = 0;; ++it) {
      if (it == 0) {
        MTF_CUDA(cudaMemcpyAsync(G.b.p, b_dev, vec_bytes, cudaMemcpyDeviceToDevice, s));
      } else {
        // b - M x with the FP64 blocks (residual_fp64) or the FP32-stored ones
        launch_matvec_kind(sys, sys->opt.residual_fp64 ? MV_FP64 : MV_FP32_ACC64, x_dev, n, G.w.p, n, nrhs, s);
        MTF_LAUNCH(KID_SUB, s, k_sub<<<nblk(n * nrhs * 2, 256), 256, 0, s>>>(b_dev, G.w.p, G.b.p, n * nrhs * 2));
      }
      MTF_LAUNCH(KID_NORM, s, k_norm_scale<<<nrhs, 1024, 0, s>>>(G.b.p, n, hN, G.w.p, n));
      MTF_CUDA(cudaMemcpyAsync(hostN, hN, size_t(nrhs) * 2 * sizeof(double), cudaMemcpyDeviceToHost, s));
      MTF_CUDA(cudaStreamSynchronize(s));
      double rmax = 0;
      for (int c = 0; c < nrhs; ++c) {
        rel[c] = hostN[2 * c] / bnorm[c];
        if (!std::isfinite(rel[c])) status = MTF_ERR_NAN;
        rmax = std::max(rmax, rel[c]);
      }
      if (status != MTF_OK) break;
      if (rmax <= sys->opt.tol) break;
      if (sys->learned_active && prev_rmax > 0 && rmax > 0.95 * prev_rmax) sys->learned_active = false;
      prev_rmax = rmax;
      if (refinements >= max_ref || total >= max_iter) {
        status = MTF_ERR_NOCONV;
        break;
      }
      // right-hand sides already converged get a zero residual
      for (int c = 0; c < nrhs; ++c)
        if (rel[c] <= sys->opt.tol)
          MTF_CUDA(cudaMemsetAsync(G.b.p + 2 * size_t(c) * n, 0, size_t(n) * 2 * sizeof(double), s));
      const double tol_min = sys->opt.inner_tol_min > 0 ? sys->opt.inner_tol_min : 1e-5;
      // 4 or more right-hand sides share one block space (with or without
      // the learned correction, which both cycles apply after block-OSRC).  A
      // block space gains a digit in a few steps at its end, and near a
      // resonance the solution's error is the residual times about 60, set by
      // the order of the assembly's atomics: aiming at 0.15 tol instead of 0.3
      // halves the error of a batch of cut spheres for 1 or 2 block steps (1 to
      // 2 %); with 4 to 64 right-hand sides it takes 2 to 5 of 98 to 925 steps
      // more on the 2 x 2 x 2 and 4 x 4 x 4 cubes.
      const bool block = sys->opt.block_krylov && nrhs >= kBlockMinRhs;
      const double inner_tol = std::min(0.5, std::max(tol_min, (block ? 0.15 : 0.3) * sys->opt.tol / rmax));
      std::vector<int> it_in(nrhs, 0);
      bool reached = false;
      if (block)
        status = fgmres_block32(sys, nrhs, G.b.p, x_dev, inner_tol, max_iter - total, it_in, reached, s);
      else
        status = fgmres_cycle32(sys, nrhs, G.b.p, x_dev, inner_tol, max_iter - total, it_in, reached, s, it);
      if (status != MTF_OK) break;
      int mx = 0;
      for (int c = 0; c < nrhs; ++c) {
        iters[c] += it_in[c];
        mx = std::max(mx, it_in[c]);
      }
      total += mx;
      ++restarts;
      if (reached) ++refinements;
    }
    MTF_CUDA(cudaStreamSynchronize(s));
  }
  if (st) {
    st->iterations = *std::max_element(iters.begin(), iters.end());
    st->restarts = restarts;
    st->refinements = refinements;
    st->converged = status == MTF_OK;
    st->rel_residual = *std::max_element(rel.begin(), rel.end());
    st->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    st->launch_seconds = sys->t_launch;
    st->lsq_seconds = sys->t_lsq;
    st->wait_seconds = sys->t_wait;
  }
  return status;
}

}  // namespace mtf
