// Physics-based preconditioner P = Id - Lambda* Sigma* (Sect. 5.2) with the
// block-diagonal inner preconditioner of App. F.
//
//  Sigma*: unpolarised, unmagnetised PRD-AA on Stokes I only (K = Q = 0):
//     eps_bar*(z,u) = k [alpha0 sum_g c_g r_AA(u'+s_g, u+s_g) + (beta0-alpha0) phi*(u) phi*(u')] J_bar(u')
//     with J_bar the angle average of the comoving I, r_AA = (1/pi) 1/2 int sin(Theta) Re F dTheta
//     (Eq. R_AA), c_g the J-level weights (2J+1)/(2(2L+1)) and phi* = sum_g c_g H(a,u+s_g)/sqrt(pi);
//     eps* = eps_bar* back in the observer frame.  Lambda*: scalar DELO-linear with eta_I.
//  P^-1 y: m_in Richardson sweeps x <- x + P_hat^-1 (y - P x) from x = 0, with
//     P_hat_i^-1 = Id + Lambda_ii Phi_bar_i (Id - A_i)^-1 Phi^Omega,  A_i = Phi^Omega Lambda_ii Phi_bar_i
//     (App. F, without the frame-change interpolations inside P_hat).
//  Q, U, V pass through unchanged (P is the identity there).
#include <cmath>
#include <vector>
#include <cooperative_groups.h>
#include "prd_internal.h"
#include "device_common.cuh"

namespace prd {

namespace cg = cooperative_groups;

int launch_pc_tiles(Ctx* c, const std::vector<double>& shift_g, std::vector<double>& aa_tiles,
                    std::vector<double>& r3g);

// The sweeps run in FP64 in both modes: the residual y - P x of a later sweep
// cancels almost completely, and the block inverse amplifies whatever rounding
// it carries, so in FP32 it would leave P^-1 neither accurate nor linear.  The
// vectors of P^-1 are Stokes I only and its tables small; the FP32 tables of
// the ctx (K/DELO weights, Lambda_ii) enter as fixed coefficients.

// A sweep is two kernels, all of it on scalar vectors [z][Omega][nu]:
//   pc_local_kernel  everything that stays within a height: x += P_hat^-1 r, then the comoving
//                    angle average of x, V = Phi_bar J and the second derivatives of V's spline
//                    (V does not depend on direction, so one spline serves them all, and its
//                    second derivatives are another product, Q Phi_bar J);
//   pc_ray_kernel    along the rays: eps* = V at the observer's frequencies, scalar DELO-linear,
//                    r = y - x + Lambda* eps*.
// What bounds them: launches and FP64 latency at small sizes, FP64 arithmetic at large ones.
// A height has a cluster of four CTAs that share its directions and matrix rows through
// distributed shared memory, so that tens of heights fill the chip.  Against one kernel per
// step (33 launches of which four frame changes of all Stokes parameters, products with a row
// per thread and their broadcast to every direction): 20 heights x 16 directions x
// 100 frequencies 217 -> 92 us.
constexpr int kPcCluster = 4;
constexpr int kPcThreads = 256;
constexpr int kPcRows = 32;          // directions whose splines a CTA solves side by side

struct PcArgs {
  const double *Mm, *Phi, *QPhi;     // [z][N][N]
  const double *w, *sp, *tin;        // angular weights, spline tables, frame-change points
  const int* iin;
  double *x, *r, *V, *V2;            // [z][o][n] iterate and residual; [z][n] spline of eps* (values, second derivatives)
  int nO, N;
};

// J over the cluster: every CTA's partial sums jp -> the total in j (all CTAs, fixed order)
__device__ __forceinline__ void pc_cluster_sum(cg::cluster_group& cl, double* jp, double* j, int N) {
  cl.sync();
  for (int n = threadIdx.x; n < N; n += kPcThreads) {
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < kPcCluster; ++k) v += *cl.map_shared_rank(jp + n, k);
    j[n] = v;
  }
  __syncthreads();
}
// row . j by 8 lanes (l8 = lane & 7), the sum on all of them
__device__ __forceinline__ double pc_row_dot(const double* __restrict__ row, const double* j, int N, int l8) {
  double s = 0.0;
  for (int m = l8; m < N; m += 8) s += row[m] * j[m];
#pragma unroll
  for (int d = 4; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
  return s;
}
// partial angle sums: thread (part, n) has s; the parts are added in order into jp
__device__ __forceinline__ void pc_part_sum(double s, bool live, int part, int parts, int n, double* red, double* jp, int N) {
  if (live) red[part * N + n] = s;
  __syncthreads();
  for (int i = threadIdx.x; i < N; i += kPcThreads) {
    double v = 0.0;
    for (int k = 0; k < parts; ++k) v += red[k * N + i];
    jp[i] = v;
  }
}

__host__ __device__ inline int pc_parts(int N) { return N >= kPcThreads ? 1 : kPcThreads / N; }
static size_t pc_smem(int N) {
  return sizeof(double) * ((size_t)4 * N + (size_t)pc_parts(N) * N + (size_t)2 * kPcRows * N);
}

template <typename T>
__global__ void __cluster_dims__(kPcCluster, 1, 1) __launch_bounds__(kPcThreads)
    pc_local_kernel(PcArgs a, const T* __restrict__ y, const T* __restrict__ lii, T* __restrict__ out, int first, int last) {
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) double pcs[];
  const int N = a.N, tid = threadIdx.x, l8 = tid & 7;
  const int cr = (int)cl.block_rank(), iz = blockIdx.x / kPcCluster;
  const int o0 = a.nO * cr / kPcCluster, o1 = a.nO * (cr + 1) / kPcCluster;   // directions of this CTA
  const int n0 = N * cr / kPcCluster, n1 = N * (cr + 1) / kPcCluster;         // its matrix rows
  double *jp = pcs, *j = jp + N, *V = j + N, *jp2 = V + N, *red = jp2 + N, *xs = red + pc_parts(N) * N, *g = xs + kPcRows * N;
  const size_t z0 = (size_t)iz * a.nO * N;
  const int parts = pc_parts(N);
  // thread (part, n): node n of the directions o0 + part, o0 + part + parts, ..
  const int part = min(tid / N, parts), nn = tid - part * N;
  auto resid = [&](size_t pt) { return first ? (double)y[pt * 4] : a.r[pt]; };
  // J = sum_o w_o r(o); one node per thread, more where N exceeds the CTA (N <= 256)
  {
    double s = 0.0;
    if (part < parts)
      for (int o = o0 + part; o < o1; o += parts) s += a.w[o] * resid(z0 + (size_t)o * N + nn);
    pc_part_sum(s, part < parts, part, parts, nn, red, jp, N);
  }
  pc_cluster_sum(cl, jp, j, N);
  // V = M J, the rows shared out, every CTA gets all of V
  for (int n = n0 + (tid >> 3); n - (tid >> 3) < n1; n += kPcThreads / 8) {
    const double v = pc_row_dot(a.Mm + ((size_t)iz * N + min(n, n1 - 1)) * N, j, N, l8);
    if (n < n1 && l8 < kPcCluster) *cl.map_shared_rank(V + n, l8) = v;
  }
  cl.sync();
  // x += r + Lambda_ii V, and the comoving angle average of x
  double s2 = 0.0;
  const double* tab = a.sp + (size_t)iz * kSpTabs * N;
  for (int ob = o0; ob < o1; ob += kPcRows) {
    const int nb = min(kPcRows, o1 - ob);
    for (int i = tid; i < nb * N; i += kPcThreads) {
      const size_t pt = z0 + (size_t)ob * N + i;
      const int n = i % N;
      double x = resid(pt) + (double)lii[pt] * V[n];
      if (!first) x = a.x[pt] + x;
      if (last) {
        out[pt * 4] = (T)x;
        out[pt * 4 + 1] = y[pt * 4 + 1];
        out[pt * 4 + 2] = y[pt * 4 + 2];
        out[pt * 4 + 3] = y[pt * 4 + 3];
      } else {
        a.x[pt] = x;
        xs[i] = x;
      }
    }
    if (last) continue;
    __syncthreads();
    // second derivatives of the rows' splines, g[node][row] (the recurrence of the frame change kernel)
    for (int i = tid; i < nb * N; i += kPcThreads) {
      const int row = i / N, n = i - row * N;
      const double* xr = xs + row * N;
      g[n * kPcRows + row] = (n > 0 && n < N - 1)
          ? tab[kSpE1 * N + n - 1] * (xr[n + 1] - xr[n]) - tab[kSpE0 * N + n - 1] * (xr[n] - xr[n - 1]) : 0.0;
    }
    __syncthreads();
    if (tid < nb) {
      double prev = 0.0, next = 0.0;
#pragma unroll 8
      for (int n = 1; n < N - 1; ++n) {
        prev = g[n * kPcRows + tid] - tab[kSpCg * N + n - 1] * prev;
        g[n * kPcRows + tid] = prev;
      }
#pragma unroll 8
      for (int n = N - 2; n >= 1; --n) {
        next = g[n * kPcRows + tid] - tab[kSpCp * N + n - 1] * next;
        g[n * kPcRows + tid] = next;
      }
    }
    __syncthreads();
    if (part < parts)
      for (int row = part; row < nb; row += parts) {
        const size_t pt = z0 + (size_t)(ob + row) * N + nn;
        const int k = a.iin[pt];
        const double* xr = xs + row * N;
        double v;
        if (k < 0) v = xr[0];
        else if (k >= N - 1) v = xr[N - 1];
        else {
          const double t = a.tin[pt], omt = 1.0 - t, k6 = tab[kSpK6 * N + k];
          v = xr[k] + t * (xr[k + 1] - xr[k]) + k6 * (omt * omt * omt - omt) * g[k * kPcRows + row] +
              k6 * (t * t * t - t) * g[(k + 1) * kPcRows + row];
        }
        s2 += a.w[ob + row] * v;
      }
    __syncthreads();
  }
  if (!last) {
    pc_part_sum(s2, part < parts, part, parts, nn, red, jp2, N);
    pc_cluster_sum(cl, jp2, j, N);
    for (int n = n0 + (tid >> 3); n - (tid >> 3) < n1; n += kPcThreads / 8) {
      const size_t row = (size_t)iz * N + min(n, n1 - 1);
      const double v = pc_row_dot(a.Phi + row * N, j, N, l8), m = pc_row_dot(a.QPhi + row * N, j, N, l8);
      if (n < n1 && l8 == 0) {
        a.V[row] = v;
        a.V2[row] = m;
      }
    }
  }
  cl.sync();   // no CTA leaves while another reads its shared memory
}

// 32 rays per CTA (lanes); heights in chunks: the warps evaluate eps* and fetch the DELO weights of
// their heights, then one warp runs the recurrence (three FP64 FMAs a height) and all write r.
constexpr int kPcChunk = 32;
template <typename T>
__global__ void __launch_bounds__(kPcThreads) pc_ray_kernel(PcArgs a, const T* __restrict__ y, const T* __restrict__ kt,
                                                            const double* __restrict__ mu, const int* __restrict__ ibk,
                                                            const double* __restrict__ tbk, int nz) {
  __shared__ double sm[kPcChunk][4][32];               // S, exp(-dtau), alpha, beta; then I in S's place
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nr = a.nO * a.N, N = a.N, ray0 = blockIdx.x * 32 + lane, ray = min(ray0, nr - 1);
  const bool up = mu[ray / N] > 0.0;
  double I = 0.0, Sp = 0.0;
  for (int c0 = 0; c0 < nz; c0 += kPcChunk) {
    const int nc = min(kPcChunk, nz - c0);
    for (int q = warp; q < nc; q += kPcThreads / 32) {
      const int iz = up ? c0 + q : nz - 1 - (c0 + q);
      const size_t pt = (size_t)iz * nr + ray;
      const double *v = a.V + (size_t)iz * N, *m = a.V2 + (size_t)iz * N;
      const int k = ibk[pt];
      double e;
      if (k < 0) e = v[0];
      else if (k >= N - 1) e = v[N - 1];
      else {
        const double t = tbk[pt], omt = 1.0 - t, k6 = a.sp[(size_t)iz * kSpTabs * N + kSpK6 * N + k];
        e = v[k] + t * (v[k + 1] - v[k]) + k6 * (omt * omt * omt - omt) * m[k] + k6 * (t * t * t - t) * m[k + 1];
      }
      const T* w = kt + pt * 10;
      sm[q][0][lane] = e * (double)w[6];
      sm[q][1][lane] = (double)w[7];
      sm[q][2][lane] = (double)w[8];
      sm[q][3][lane] = (double)w[9];
    }
    __syncthreads();
    if (warp == 0)
      for (int q = 0; q < nc; ++q) {
        const double S = sm[q][0][lane], e = sm[q][1][lane], al = sm[q][2][lane], be = sm[q][3][lane];
        if (c0 + q == 0) I = 0.0;
        else if (e <= 0.5) I = S + e * (I - S) + al * (Sp - S);   // thick: photon-exact form
        else I = e * I + al * Sp + be * S;                          // thin: standard form
        sm[q][0][lane] = I;
        Sp = S;
      }
    __syncthreads();
    if (ray0 < nr)
      for (int q = warp; q < nc; q += kPcThreads / 32) {
        const size_t pt = (size_t)(up ? c0 + q : nz - 1 - (c0 + q)) * nr + ray;
        a.r[pt] = ((double)y[pt * 4] - a.x[pt]) + sm[q][0][lane];
      }
    __syncthreads();
  }
}

static int lu_inverse(std::vector<double>& A, int n) {
  std::vector<int> piv(n);
  std::vector<double> inv((size_t)n * n, 0.0);
  for (int k = 0; k < n; ++k) {
    int p = k;
    for (int i = k + 1; i < n; ++i)
      if (std::fabs(A[(size_t)i * n + k]) > std::fabs(A[(size_t)p * n + k])) p = i;
    piv[k] = p;
    if (A[(size_t)p * n + k] == 0.0) return -1;
    if (p != k)
      for (int j = 0; j < n; ++j) std::swap(A[(size_t)k * n + j], A[(size_t)p * n + j]);
    for (int i = k + 1; i < n; ++i) {
      const double f = A[(size_t)i * n + k] / A[(size_t)k * n + k];
      A[(size_t)i * n + k] = f;
      for (int j = k + 1; j < n; ++j) A[(size_t)i * n + j] -= f * A[(size_t)k * n + j];
    }
  }
  for (int col = 0; col < n; ++col) {
    std::vector<double> b(n, 0.0);
    b[col] = 1.0;
    for (int k = 0; k < n; ++k)
      if (piv[k] != k) std::swap(b[k], b[piv[k]]);
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < i; ++j) b[i] -= A[(size_t)i * n + j] * b[j];
    for (int i = n - 1; i >= 0; --i) {
      for (int j = i + 1; j < n; ++j) b[i] -= A[(size_t)i * n + j] * b[j];
      b[i] /= A[(size_t)i * n + i];
    }
    for (int i = 0; i < n; ++i) inv[(size_t)i * n + col] = b[i];
  }
  A.swap(inv);
  return 0;
}

int launch_precond_setup(Ctx* c) {
  const int nz = c->nz, N = c->nnu, nO = c->nO, ng = c->ngrp;
  // J-level shifts at B = 0 and weights
  std::vector<double> sg((size_t)nz * ng), cg(ng);
  const prd_atom& at = c->atom;
  for (int g = 0; g < ng; ++g) {
    const double E = (at.twoS == 0 ? at.E_u_cm[0] : at.E_u_cm[g]) * kCmToHz - c->nu0;
    cg[g] = (at.twoS == 0) ? 1.0 : (g == 0 ? 1.0 / 3.0 : 2.0 / 3.0);
    for (int iz = 0; iz < nz; ++iz) sg[(size_t)iz * ng + g] = E / c->dnuD[iz];
  }
  std::vector<double> aa, r3;   // aa: [z][g][N][2N]; r3: [z][g*g][2N]
  int rc = launch_pc_tiles(c, sg, aa, r3);
  if (rc) return rc;
  std::vector<double> phi((size_t)nz * N * N), Mm((size_t)nz * N * N), qphi((size_t)nz * N * N, 0.0);
  std::vector<int> bad(nz, 0);
#pragma omp parallel for schedule(dynamic)
  for (int iz = 0; iz < nz; ++iz) {
    const double a0 = (1.0 - c->eps[iz]) * (1.0 - c->rE[iz]);
    const double b0 = 1.0 - c->eps[iz];
    std::vector<double> ph(N), rs(N, 0.0);
    for (int n = 0; n < N; ++n) {
      double s = 0.0;
      for (int g = 0; g < ng; ++g)
        s += cg[g] * faddeeva_host(cplx(c->u[(size_t)iz * N + n] + sg[(size_t)iz * ng + g], c->a[iz])).real() / kSqrtPi;
      ph[n] = s;
    }
    for (int g = 0; g < ng; ++g) {
      const double* rr = &r3[((size_t)iz * ng * ng + g * ng + g) * 2 * N];
      for (int m = 0; m < N; ++m) rs[m] += cg[g] * rr[m] / (2.0 * kSqrtPi);
    }
    double* P = &phi[(size_t)iz * N * N];
    for (int n = 0; n < N; ++n)
      for (int m = 0; m < N; ++m) {
        double v = 0.0;
        for (int g = 0; g < ng; ++g) v += cg[g] * aa[(((size_t)iz * ng + g) * N + n) * 2 * N + m] / kPi;
        P[(size_t)n * N + m] = c->k[iz] * (a0 * v + (b0 - a0) * ph[n] * rs[m]);
      }
    // second derivatives of the natural spline through the columns of Phi_bar (zero at the ends)
    const double* Q = &c->Q[(size_t)iz * N * N];
    double* QP = &qphi[(size_t)iz * N * N];
    for (int n = 1; n + 1 < N; ++n)
      for (int k = 0; k < N; ++k) {
        const double qv = Q[(size_t)n * N + k];
        for (int m = 0; m < N; ++m) QP[(size_t)n * N + m] += qv * P[(size_t)k * N + m];
      }
    // lambda_bar(n) = sum_o w_o Lambda_ii(z, o, n)
    std::vector<double> lb(N, 0.0);
    for (int o = 0; o < nO; ++o)
      for (int n = 0; n < N; ++n) lb[n] += c->wang[o] * c->pc_lii_host[((size_t)iz * nO + o) * N + n];
    std::vector<double> A((size_t)N * N);
    for (int n = 0; n < N; ++n)
      for (int m = 0; m < N; ++m) A[(size_t)n * N + m] = (n == m ? 1.0 : 0.0) - lb[n] * P[(size_t)n * N + m];
    if (lu_inverse(A, N)) { bad[iz] = 1; continue; }
    double* Mz = &Mm[(size_t)iz * N * N];
    for (int n = 0; n < N; ++n)
      for (int m = 0; m < N; ++m) {
        double s = 0.0;
        for (int k = 0; k < N; ++k) s += P[(size_t)n * N + k] * A[(size_t)k * N + m];
        Mz[(size_t)n * N + m] = s;
      }
  }
  for (int iz = 0; iz < nz; ++iz)
    if (bad[iz]) return fail(c, PRD_E_ARG, "block-Jacobi matrix (Id - A_i) is singular at height " + std::to_string(iz));
  if ((rc = upload(c, c->pc_phi, phi.data(), phi.size() * 8)) || (rc = upload(c, c->pc_M, Mm.data(), Mm.size() * 8)) ||
      (rc = upload(c, c->pc_qphi, qphi.data(), qphi.size() * 8)))
    return rc;
  DBuf w;
  if ((rc = upload(c, w, c->wang.data(), nO * 8))) return rc;
  c->owned.push_back(w);     // angular weights (double), freed with the ctx
  c->pc_w = w.p;
  const size_t vb = nvec(c) / 4 * sizeof(double);          // Stokes I only
  if ((rc = dalloc(c, c->pc_x, vb)) || (rc = dalloc(c, c->pc_r, vb)) ||
      (rc = dalloc(c, c->pc_v, (size_t)2 * nz * N * sizeof(double))))
    return rc;
  PRD_CUDA_TRY(c, cudaFuncSetAttribute(pc_local_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
  PRD_CUDA_TRY(c, cudaFuncSetAttribute(pc_local_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
  return PRD_OK;
}

template <typename T>
static int precond_T(Ctx* c, const T* y, T* x) {
  const int nz = c->nz, N = c->nnu;
  double* V = (double*)c->pc_v.p;
  const PcArgs a{(const double*)c->pc_M.p, (const double*)c->pc_phi.p, (const double*)c->pc_qphi.p,
                 (const double*)c->pc_w, (const double*)c->sp.p, (const double*)c->tin.p, (const int*)c->iin.p,
                 (double*)c->pc_x.p, (double*)c->pc_r.p, V, V + (size_t)nz * N, c->nO, N};
  for (int sweep = 0; sweep < c->m_in; ++sweep) {
    // r = y - P x on Stokes I (P x = x - Lambda* Sigma* x); the first sweep starts from x = 0
    if (sweep > 0)
      pc_ray_kernel<T><<<ceil_div(c->nO * N, 32), kPcThreads, 0, c->stream>>>(
          a, y, (const T*)c->kt.p, (const double*)c->dmu.p, (const int*)c->ibk.p, (const double*)c->tbk.p, nz);
    // x += P_hat^-1 r, and Sigma* x up to the frame change back
    pc_local_kernel<T><<<nz * kPcCluster, kPcThreads, pc_smem(N), c->stream>>>(
        a, y, (const T*)c->pc_lii.p, x, sweep == 0 ? 1 : 0, sweep == c->m_in - 1 ? 1 : 0);
  }
  PRD_CUDA_TRY(c, cudaPeekAtLastError());
  return PRD_OK;
}

int apply_precond(Ctx* c, const void* y, void* x) {
  if (c->m_in <= 0) {
    PRD_CUDA_TRY(c, cudaMemcpyAsync(x, y, nvec(c) * c->esz, cudaMemcpyDeviceToDevice, c->stream));
    return PRD_OK;
  }
  if (c->prec == PRD_FP64) return precond_T<double>(c, (const double*)y, (double*)x);
  return precond_T<float>(c, (const float*)y, (float*)x);
}

}  // namespace prd
