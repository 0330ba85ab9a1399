// Per-apply kernels of y = (Id - Lambda Sigma) x.
//   S1  frame change observer -> comoving: natural spline of I(z,Omega',.)
//       evaluated at u_m - u_b(z,Omega')                     (Sect. 4.1)
//   S3+S4  R_II contraction over (Theta class, Omega', triple, frequency)
//       with the Stokes-route coefficients folded in          (Eq. RQIIKKp)
//   S5  R_III, separable in incident and outgoing frequency  (Eq. RIIIQKKp)
//   S6  frame change back (u_n + u_b(z,Omega)) and Kirchhoff factor f (App. E)
//   S7+S8  DELO-linear sweep per ray, y = x - Lambda eps      (Sect. 3)
#include <algorithm>
#include <cstdio>
#include <cuda_bf16.h>
#include <type_traits>
#include "prd_internal.h"
#include "device_common.cuh"
#include "ring.h"

namespace prd {

// (s, c) += x (x exact float); error-free two-sum of s and x into s, error into c
__device__ __forceinline__ void dd_add(float& s, float& c, float x) {
  const float t = s + x;
  const float bb = t - s;
  c += (s - (t - bb)) + (x - bb);
  s = t;
}

// ------------------------------------------------------------------ splines
template <typename T> struct V4;
template <> struct V4<float> { using type = float4; };
template <> struct V4<double> { using type = double4_16a; };

// Frame change of R (z, Omega) rows of one height per CTA: the natural spline of
// every Stokes row (its second derivatives M from the tridiagonal system, in FP64)
// evaluated at the tabulated points; the intensity is multiplied by fI (nullable).
//
// What bounds it: the Thomas recurrence, 2 (N - 2) dependent FP64 steps per row,
// on a chip with two FP64 lanes a clock and SM.  So the recurrence is stripped to
// one FP64 FMA a step: the divisions are folded into per-height factors (e0, e1,
// cg, cp of the spline tables), the right-hand sides are formed by the whole CTA
// beforehand, and the rows, right-hand sides and factors sit in shared memory, so
// that no step waits for a global load.  M never leaves the CTA.  Against two
// kernels that walked global memory with a thread per row and divided at every
// step: an FP32 apply of 8 x 64 rows of 200 points 3399 -> 2952 us, of 10 x 16 rows of
// 27 points 262 -> 201 us, a preconditioner apply of 20 x 16 rows of 100 points
// (four FP64 frame changes) 1097 -> 217 us.
// R = 4 rows a CTA (16 recurrences in a warp) where there are more than four rows for
// every SM, R = 1 below that, so that the right-hand sides and evaluations of a
// small problem still spread over the chip.
constexpr int kSplThreads = 128;

template <typename T, int R>
struct SplineSmem {
  // g: [node][chain] FP64 right-hand sides, then second derivatives; ys: [row][node]
  // with an odd row stride (rows fall in different banks); Mt: the second
  // derivatives in T (FP64 reads g itself); cg, cp: recurrence factors
  static __host__ __device__ int stride(int N) { return N | 1; }
  static __host__ __device__ size_t ys_off(int N) { return (size_t)N * 4 * R * 8; }
  static __host__ __device__ size_t mt_off(int N) { return ys_off(N) + (size_t)R * stride(N) * 4 * sizeof(T); }
  static __host__ __device__ size_t tab_off(int N) {
    return mt_off(N) + (sizeof(T) == 8 ? 0 : (size_t)N * 4 * R * sizeof(T));
  }
  static __host__ __device__ size_t bytes(int N) { return tab_off(N) + (size_t)2 * N * 8; }
};

template <typename T, int R>
__global__ void __launch_bounds__(kSplThreads) spline_kernel(const T* __restrict__ y, RowAdds add,
                                                             const int* __restrict__ kidx,
                                                             const double* __restrict__ tt,
                                                             const double* __restrict__ sp,
                                                             const double* __restrict__ fI, T* __restrict__ out,
                                                             int nO, int N) {
  using V = typename V4<T>::type;
  using L = SplineSmem<T, R>;
  constexpr int C = 4 * R;                           // recurrences of the CTA
  extern __shared__ __align__(16) unsigned char spsm[];
  double* g = reinterpret_cast<double*>(spsm);
  V* ys = reinterpret_cast<V*>(spsm + L::ys_off(N));
  T* Mt = sizeof(T) == 8 ? reinterpret_cast<T*>(g) : reinterpret_cast<T*>(spsm + L::mt_off(N));
  double* cg = reinterpret_cast<double*>(spsm + L::tab_off(N));
  double* cp = cg + N;
  const int iz = blockIdx.y, o0 = blockIdx.x * R, nr = min(R, nO - o0), tid = threadIdx.x;
  const int S = L::stride(N);
  const double* tab = sp + (size_t)iz * kSpTabs * N;
  const size_t row0 = (size_t)iz * nO + o0;
  {
    const V* src = reinterpret_cast<const V*>(y) + row0 * N;
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (r < nr)
        for (int i = tid; i < N; i += kSplThreads) {
          V v = src[(size_t)r * N + i];
          if constexpr (sizeof(T) == 4) {
            if (add.ent) {
              // the entries' parts, eight loads at a time, added in order; their rounding errors are kept
              // and added last: the largest error against FP64 over eight grids of 27 to 200 points is
              // 3.3e-7 to 5.3e-7 instead of 4.9e-7 to 7.4e-7, for 1 to 6 us of the frame change
              float4 err = make_float4(0.f, 0.f, 0.f, 0.f);
              auto sum = [&](float4 w) {
                dd_add(v.x, err.x, w.x); dd_add(v.y, err.y, w.y);
                dd_add(v.z, err.z, w.z); dd_add(v.w, err.w, w.w);
              };
              const int e0 = add.ptr[o0 + r], e1 = add.ptr[o0 + r + 1], cnt = gridDim.y * add.nent;
              const int G = i >= add.n0 ? add.G : 1;
              for (int e = e0, p = 0; e < e1;) {
                float4 w[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                  w[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                  if (e < e1) {
                    w[q] = add.ent[add_off(p, iz * add.nent + add.list[e].x, cnt, N, add.n0, i)];
                    if (++p == G) { p = 0; ++e; }
                  }
                }
#pragma unroll
                for (int q = 0; q < 8; ++q) sum(w[q]);
              }
              // and the further parts of this height's split items
              if (add.zs > 1 && (iz + 1) * add.nwork > add.split0) {
                const size_t ps = (size_t)add.nsplit * 32 * (N + (add.G - 1) * (N - add.n0));
                for (int e = e0; e < e1; ++e) {
                  const int l = add.list[e].y, it = iz * add.nwork + (l >> 5) - add.split0;
                  if (it < 0) continue;
                  for (int g = 0; g < G; ++g) {
                    const float4* a = add.tail + add_off(g, it * 32 + (l & 31), add.nsplit * 32, N, add.n0, i);
#pragma unroll 8
                    for (int p = 0; p < add.zs - 1; ++p) sum(a[p * ps]);
                  }
                }
              }
              // (a sum that overflowed has no rounding error: it stays the infinity that it is)
              v.x += err.x == err.x ? err.x : 0.f; v.y += err.y == err.y ? err.y : 0.f;
              v.z += err.z == err.z ? err.z : 0.f; v.w += err.w == err.w ? err.w : 0.f;
            }
          }
          ys[r * S + i] = v;
        }
  }
  for (int i = tid; i < N; i += kSplThreads) {
    cg[i] = tab[kSpCg * N + i];
    cp[i] = tab[kSpCp * N + i];
  }
  __syncthreads();
  // right-hand sides divided by the pivots; end nodes zero (natural spline)
  for (int idx = tid; idx < N * C; idx += kSplThreads) {
    const int i = idx / C, ch = idx - i * C;
    double v = 0.0;
    if (i > 0 && i < N - 1 && (ch >> 2) < nr) {
      const T* yr = reinterpret_cast<const T*>(ys + (ch >> 2) * S) + (ch & 3);
      const double y0 = (double)yr[(i - 1) * 4], y1 = (double)yr[i * 4], y2 = (double)yr[(i + 1) * 4];
      v = tab[kSpE1 * N + i - 1] * (y2 - y1) - tab[kSpE0 * N + i - 1] * (y1 - y0);
    }
    g[idx] = v;
  }
  __syncthreads();
  if (tid < C) {
    // blocks of kB steps: their factors and right-hand sides are read before the
    // dependent FMAs, so a step costs one FMA latency
    constexpr int kB = 8;
    double prev = 0.0;
    int i = 1;
    for (; i + kB <= N - 1; i += kB) {
      double a[kB], f[kB];
#pragma unroll
      for (int q = 0; q < kB; ++q) { a[q] = g[(i + q) * C + tid]; f[q] = cg[i + q - 1]; }
#pragma unroll
      for (int q = 0; q < kB; ++q) { prev = a[q] - f[q] * prev; a[q] = prev; }
#pragma unroll
      for (int q = 0; q < kB; ++q) g[(i + q) * C + tid] = a[q];
    }
    for (; i < N - 1; ++i) {
      prev = g[i * C + tid] - cg[i - 1] * prev;
      g[i * C + tid] = prev;
    }
    if (sizeof(T) != 8) Mt[tid] = Mt[(N - 1) * C + tid] = (T)0;
    double next = 0.0;
    i = N - 2;
    for (; i - kB >= 0; i -= kB) {
      double a[kB], f[kB];
#pragma unroll
      for (int q = 0; q < kB; ++q) { a[q] = g[(i - q) * C + tid]; f[q] = cp[i - q - 1]; }
#pragma unroll
      for (int q = 0; q < kB; ++q) { next = a[q] - f[q] * next; a[q] = next; }
#pragma unroll
      for (int q = 0; q < kB; ++q) Mt[(i - q) * C + tid] = (T)a[q];
    }
    for (; i >= 1; --i) {
      next = g[i * C + tid] - cp[i - 1] * next;
      Mt[i * C + tid] = (T)next;
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (r >= nr) break;
    const size_t p0 = (row0 + r) * N;
    const V* yr = ys + r * S;
    for (int n = tid; n < N; n += kSplThreads) {
      const size_t pt = p0 + n;
      const int k = kidx[pt];
      V v;
      if (k < 0) v = yr[0];
      else if (k >= N - 1) v = yr[N - 1];
      else {
        const double t = tt[pt], omt = 1.0 - t, k6 = tab[kSpK6 * N + k];
        // y_k + t (y_{k+1} - y_k) + ...: reproduces a constant exactly in any precision
        const T c1 = (T)t, c2 = (T)(k6 * (omt * omt * omt - omt)), c3 = (T)(k6 * (t * t * t - t));
        const V a = yr[k], b = yr[k + 1];
        const V ma = *reinterpret_cast<const V*>(Mt + (size_t)k * C + 4 * r);
        const V mb = *reinterpret_cast<const V*>(Mt + (size_t)(k + 1) * C + 4 * r);
        v.x = a.x + c1 * (b.x - a.x) + c2 * ma.x + c3 * mb.x;
        v.y = a.y + c1 * (b.y - a.y) + c2 * ma.y + c3 * mb.y;
        v.z = a.z + c1 * (b.z - a.z) + c2 * ma.z + c3 * mb.z;
        v.w = a.w + c1 * (b.w - a.w) + c2 * ma.w + c3 * mb.w;
      }
      if (fI) v.x *= (T)fI[pt];
      reinterpret_cast<V*>(out)[pt] = v;
    }
  }
}

// Shared memory the dynamic-size kernels of this file may be launched with, set
// once (at setup) to the device's limit: a per-launch value would race between
// contexts of different sizes on different threads.
template <typename K>
static int allow_smem(Ctx* c, K kern) {
  PRD_CUDA_TRY(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
  return PRD_OK;
}

template <typename T>
static void launch_spline(Ctx* c, const T* y, const int* kidx, const double* tt, const double* fI, T* out, int nO,
                          const RowAdds& add = RowAdds(), int z0 = 0, int nz = 0) {
  // all heights, or the nz from z0 on
  if (!nz) nz = c->nz;
  const int N = c->nnu;
  const size_t pt = (size_t)z0 * nO * N;
  const double* sp = (const double*)c->sp.p + (size_t)z0 * kSpTabs * N;
  y += 4 * pt;
  out += 4 * pt;
  kidx += pt;
  tt += pt;
  if (fI) fI += pt;
  if (nz * nO <= 4 * c->nsm)
    spline_kernel<T, 1><<<dim3(nO, nz), kSplThreads, SplineSmem<T, 1>::bytes(N), c->stream>>>(y, add, kidx, tt, sp, fI, out, nO, N);
  else
    spline_kernel<T, 4><<<dim3((nO + 3) / 4, nz), kSplThreads, SplineSmem<T, 4>::bytes(N), c->stream>>>(y, add, kidx, tt, sp, fI, out, nO, N);
}

// ------------------------------------------------------------------ R_III
// J[z][ku kv] += sum_{o', j} rin[z][o'][q][j] * sum_m r3w[z][q][m] I~[z][o'][m][j],  q = (ku kv, l')
// One block per (o', z): the direction's comoving row I~[z][o'][.][.] is staged in
// shared memory and thread q forms S_j = sum_m r3w[q][m] I~_j(m) (arithmetic in A,
// so the FP32 path runs on the FP32 pipe), then adds sum_j rin_j S_j to J in FP64.
template <typename T, typename A>
__global__ void r3_J_kernel(const A* __restrict__ Ic, const T* __restrict__ r3w, const T* __restrict__ rin,
                            double* __restrict__ J, int nO, int N, int nq, int nl) {
  using V = typename V4<A>::type;
  const int o = blockIdx.x, iz = blockIdx.y;
  extern __shared__ __align__(16) unsigned char r3smem[];
  V* row = reinterpret_cast<V*>(r3smem);
  const V* src = reinterpret_cast<const V*>(Ic) + ((size_t)iz * nO + o) * N;
  for (int m = threadIdx.x; m < N; m += blockDim.x) row[m] = src[m];
  __syncthreads();
  for (int q = threadIdx.x; q < nq; q += blockDim.x) {
    const T* w = r3w + ((size_t)iz * nq + q) * 2 * N;
    A sr[4] = {0, 0, 0, 0}, si[4] = {0, 0, 0, 0};
    for (int m = 0; m < N; ++m) {
      const A wr = (A)w[m], wi = (A)w[N + m];
      const V iv = row[m];
      sr[0] += wr * iv.x; sr[1] += wr * iv.y; sr[2] += wr * iv.z; sr[3] += wr * iv.w;
      si[0] += wi * iv.x; si[1] += wi * iv.y; si[2] += wi * iv.z; si[3] += wi * iv.w;
    }
    const T* ri = rin + (((size_t)iz * nO + o) * nq + q) * 8;
    double jr = 0.0, ji = 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double rr = (double)ri[2 * j], rm = (double)ri[2 * j + 1];
      jr += rr * (double)sr[j] - rm * (double)si[j];
      ji += rr * (double)si[j] + rm * (double)sr[j];
    }
    const int uv = q / nl;
    atomicAdd(&J[((size_t)iz * (nq / nl) + uv) * 2], jr);
    atomicAdd(&J[((size_t)iz * (nq / nl) + uv) * 2 + 1], ji);
  }
}

// eps_bar[z][o][n][i] = Re sum_uv ab[uv] J[uv] sum_l' O_i(o; uv, l') prof[uv][l'][n]
// One block per (o, z): C = ab J per uv and the direction's O_i coefficients are
// staged in shared memory; the profile rows are read coalesced along n.  The sum over
// (uv, l') is a chain of loads, so where N is small its terms are shared out between `parts`
// threads per n and added in order (72 terms one after the other took 27 us for 27
// frequencies, shared out 9).  Arithmetic in A.
constexpr int kR3Threads = 256;
template <typename T, typename A>
__global__ void __launch_bounds__(kR3Threads) r3_out_kernel(const double* __restrict__ J, const T* __restrict__ ab,
                                                            const T* __restrict__ rout, const T* __restrict__ prof,
                                                            A* __restrict__ eb, int nO, int N, int nuv, int nl,
                                                            int parts) {
  using V = typename V4<A>::type;
  const int o = blockIdx.x, iz = blockIdx.y;
  const int zo = iz * nO + o;
  extern __shared__ __align__(16) unsigned char r3smem[];
  V* P = reinterpret_cast<V*>(r3smem);                 // [part][n] partial sums (parts > 1)
  A* C = reinterpret_cast<A*>(P + (parts > 1 ? parts * N : 0));   // [uv][2]
  A* R = C + 2 * nuv;                                  // [uv][l'][8]
  for (int uv = threadIdx.x; uv < nuv; uv += kR3Threads) {
    const double jr = J[((size_t)iz * nuv + uv) * 2], ji = J[((size_t)iz * nuv + uv) * 2 + 1];
    const double ar = (double)ab[((size_t)iz * nuv + uv) * 2], ai = (double)ab[((size_t)iz * nuv + uv) * 2 + 1];
    C[2 * uv] = (A)(ar * jr - ai * ji);
    C[2 * uv + 1] = (A)(ar * ji + ai * jr);
  }
  for (int k = threadIdx.x; k < nuv * nl * 8; k += kR3Threads) R[k] = (A)rout[(size_t)zo * nuv * nl * 8 + k];
  __syncthreads();
  const int part = threadIdx.x / N, n = threadIdx.x - part * N, nq = nuv * nl;
  A acc[4] = {0, 0, 0, 0};
  if (part < parts) {
#pragma unroll 4
    for (int q = part; q < nq; q += parts) {
      const int uv = nl == 2 ? q >> 1 : q;             // 1 or 2 lower states
      const A cr = C[2 * uv], ci = C[2 * uv + 1];
      const T* pp = prof + (((size_t)iz * nq + q) * N + n) * 2;
      const A pr = (A)pp[0], pi = (A)pp[1];
      const A dr = cr * pr - ci * pi, di = cr * pi + ci * pr;
      const A* ro = R + q * 8;
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[i] += ro[2 * i] * dr - ro[2 * i + 1] * di;
    }
  }
  if (parts > 1) {
    if (part < parts) { V v; v.x = acc[0]; v.y = acc[1]; v.z = acc[2]; v.w = acc[3]; P[part * N + n] = v; }
    __syncthreads();
    if (part == 0)
      for (int k = 1; k < parts; ++k) {
        const V v = P[k * N + n];
        acc[0] += v.x; acc[1] += v.y; acc[2] += v.z; acc[3] += v.w;
      }
  }
  if (part == 0) {
    V v;
    v.x = acc[0]; v.y = acc[1]; v.z = acc[2]; v.w = acc[3];
    reinterpret_cast<V*>(eb)[(size_t)zo * N + n] = v;
  }
}

// The Sigma tables an apply reads: the ctx precision's, or (FP32 mode, t64) the
// FP64 copies kept for the refinement residuals.
struct SigmaTables {
  const void *tiles, *Y, *r3w, *r3in, *r3out, *r3prof, *r3ab;
  int ld, fmt;
};
static SigmaTables sigma_tables(const Ctx* c, bool t64) {
  if (t64)
    return {c->tiles64.p, c->Y64.p, c->r3w64.p, c->r3in64.p, c->r3out64.p, c->r3prof64.p, c->r3ab64.p, c->ld64(), TILE_PLAIN};
  return {c->tiles.p, c->Y.p, c->r3w.p, c->r3in.p, c->r3out.p, c->r3prof.p, c->r3ab.p, c->ld(), c->tile_fmt()};
}

// launchers (shared by the apply and the line-of-sight paths)
template <typename T, typename A>
static void launch_r3_J(Ctx* c, const A* Ic, double* J, int nO, const SigmaTables& tb) {
  const int nuv = c->nu_st * c->nu_st, nq = nuv * c->nl_st, N = c->nnu;
  r3_J_kernel<T, A><<<dim3(nO, c->nz), 128, (size_t)N * 4 * sizeof(A), c->stream>>>(
      Ic, (const T*)tb.r3w, (const T*)tb.r3in, J, nO, N, nq, c->nl_st);
}
template <typename T, typename A>
static void launch_r3_out(Ctx* c, const double* J, const T* rout, A* eb, int nO, const SigmaTables& tb) {
  const int nuv = c->nu_st * c->nu_st, N = c->nnu;
  const int parts = kR3Threads / N;                    // N <= 256
  const size_t smem = sizeof(A) * ((parts > 1 ? (size_t)4 * parts * N : 0) + (size_t)2 * nuv + (size_t)nuv * c->nl_st * 8);
  r3_out_kernel<T, A><<<dim3(nO, c->nz), kR3Threads, smem, c->stream>>>(
      J, (const T*)tb.r3ab, rout, (const T*)tb.r3prof, eb, nO, N, nuv, c->nl_st, parts);
}

// ------------------------------------------------------------------ R_II (SIMT)
// One CTA per (z, class, chunk of 16 output directions).  Over the triples t
// and blocks of 16 incident frequencies m it builds, in shared memory,
//   Z_t[m][(o,i)] = sum_{o' : Theta(o,o') = class} sum_j Y_t,ij(o,o') I~_j(o', m)
// and accumulates  eps_bar[n][(o,i)] += sum_m Re(T_t[n][m] Z_t[m][(o,i)])
// with the tile T_t of (z, class) streamed from global memory.
constexpr int kCW = 16;      // output directions per CTA
constexpr int kMB = 16;      // incident-frequency block
constexpr int kMaxRows = 16; // rows per thread (N <= 256)

// element (n, k) of the stored tile at t (format fmt)
template <typename T>
__device__ __forceinline__ T tile_get(const unsigned char* t, int n, int k, int N, int ld, int fmt) {
  if (sizeof(T) == 8 || fmt == TILE_PLAIN) return reinterpret_cast<const T*>(t)[(size_t)n * ld + k];
  if (fmt == TILE_F32) return (T)reinterpret_cast<const float*>(t)[tile_off(n, k, N, ld, true)];
  const __nv_bfloat16* b = reinterpret_cast<const __nv_bfloat16*>(t);
  if (fmt == TILE_BF16HI) return (T)__bfloat162float(b[tile_off_hi(n, k, N, ld)]);
  return (T)(__bfloat162float(b[tile_off_split(n, k, N, ld, false)]) + __bfloat162float(b[tile_off_split(n, k, N, ld, true)]));
}

template <typename T, typename A>
__global__ void __launch_bounds__(256) r2_simt_kernel(const unsigned char* __restrict__ tiles, const T* __restrict__ Y,
                                                      const A* __restrict__ Ic, const int* __restrict__ cls,
                                                      A* __restrict__ eb, int ncls, int ntrip, int nO, int N,
                                                      int npairs, int ld, int fmt, int ts) {
  const int chunk = blockIdx.x / ts, part = blockIdx.x - chunk * ts, c = blockIdx.y, iz = blockIdx.z;
  const int* cout_ptr = cls;
  const int* cout_dir = cls + ncls + 1;
  const int ne_tot = cout_ptr[ncls];
  const int* pair_ptr = cout_dir + ne_tot;
  const int* pair_in = pair_ptr + ne_tot + 1;
  const int e0 = cout_ptr[c] + chunk * kCW;
  const int e_end = cout_ptr[c + 1];
  if (e0 >= e_end) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  A (*Zs)[2][kCW * 4] = reinterpret_cast<A (*)[2][kCW * 4]>(smraw);
  T* Asb = reinterpret_cast<T*>(smraw + sizeof(A) * kMB * 2 * kCW * 4);
  // As[h][n][mm] -> Asb[(h * N + n) * (kMB + 1) + mm]
  // columns of this block as a power of two: a block of 8 outputs has twice the threads per
  // column, not half of them idle
  const int tid = threadIdx.x, ne = e_end - e0;
  const int lc = ne <= 4 ? 2 : (ne <= 8 ? 3 : 4), tx = tid & ((1 << lc) - 1), ty = tid >> lc, nty = 256 >> lc;
  const int e_mine = e0 + tx;
  A acc[kMaxRows][4];
#pragma unroll
  for (int r = 0; r < kMaxRows; ++r)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[r][i] = (A)0;
  const int nrows = (N + nty - 1) / nty;
  const size_t tile_sz = (size_t)N * ld * (fmt == TILE_BF16HI ? 2 : sizeof(T));
  const unsigned char* tbase = tiles + ((size_t)iz * ncls + c) * ntrip * tile_sz;
  // Z-building role: thread -> (e = tid & 15, m = tid >> 4)
  const int ze = tid & 15, zm = tid >> 4;
  const int e_z = e0 + ze;
  for (int t = ntrip * part / ts; t < ntrip * (part + 1) / ts; ++t) {
    const unsigned char* tile = tbase + (size_t)t * tile_sz;
    for (int m0 = 0; m0 < N; m0 += kMB) {
      const int mb = min(kMB, N - m0);
      // ---- Z block
      {
        const int m = m0 + zm;
        A zr[4] = {0, 0, 0, 0}, zi[4] = {0, 0, 0, 0};
        if (e_z < e_end && m < N) {
          for (int p = pair_ptr[e_z]; p < pair_ptr[e_z + 1]; ++p) {
            const int op = pair_in[p];
            const A* iv = Ic + (((size_t)iz * nO + op) * N + m) * 4;
            const T* y = Y + (((size_t)iz * npairs + p) * ntrip + t) * 32;
            const A i0 = iv[0], i1 = iv[1], i2 = iv[2], i3 = iv[3];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const T* yi = y + i * 8;
              zr[i] += (A)yi[0] * i0 + (A)yi[2] * i1 + (A)yi[4] * i2 + (A)yi[6] * i3;
              zi[i] += (A)yi[1] * i0 + (A)yi[3] * i1 + (A)yi[5] * i2 + (A)yi[7] * i3;
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          Zs[zm][0][ze * 4 + i] = zr[i];
          Zs[zm][1][ze * 4 + i] = zi[i];
        }
      }
      // ---- tile block: rows n, columns m0..m0+15 (Re and Im halves)
      for (int idx = tid; idx < N * 2 * kMB; idx += 256) {
        const int mm = idx % kMB;
        const int h = (idx / kMB) & 1;
        const int n = idx / (2 * kMB);
        const int m = m0 + mm;
        Asb[(h * N + n) * (kMB + 1) + mm] = (m < N) ? tile_get<T>(tile, n, h * N + m, N, ld, fmt) : (T)0;
      }
      __syncthreads();
#pragma unroll 4
      for (int mm = 0; mm < mb; ++mm) {
        A zr[4], zi[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          zr[i] = Zs[mm][0][tx * 4 + i];
          zi[i] = Zs[mm][1][tx * 4 + i];
        }
#pragma unroll
        for (int r = 0; r < kMaxRows; ++r) {
          if (r < nrows) {
            const int n = ty + nty * r;
            if (n < N) {
              const A ar = Asb[n * (kMB + 1) + mm], ai = Asb[(N + n) * (kMB + 1) + mm];
#pragma unroll
              for (int i = 0; i < 4; ++i) acc[r][i] += ar * zr[i] - ai * zi[i];
            }
          }
        }
      }
      __syncthreads();
    }
  }
  if (e_mine < e_end) {
    const int o = cout_dir[e_mine];
#pragma unroll
    for (int r = 0; r < kMaxRows; ++r) {
      const int n = ty + nty * r;
      if (r < nrows && n < N) {
        A* dst = eb + (((size_t)iz * nO + o) * N + n) * 4;
#pragma unroll
        for (int i = 0; i < 4; ++i) atomicAdd(dst + i, acc[r][i]);
      }
    }
  }
}

// ------------------------------------------------------------------ R_II, double-float
// The same contraction for the FP64 refinement residuals, run on the FP32 pipes
// (GB300's FP64 rate is 1/64 of its FP32 rate).  Every FP64 operand a is split
// into a = hi + lo (two floats, |lo| <= 2^-24 |a|); a product of two operands
// is hi*hi exactly (FMA error term) plus the hi*lo cross terms, and the sum is
// kept as an unevaluated float pair (s, c) with the error-free two-sum of s
// (Dekker / Knuth double-single arithmetic).  Dropped: lo*lo (2^-48 relative)
// and the rounding of c; the result carries ~2^-44 relative error per term,
// far below the 1e-10 residuals the refinement needs.
struct F2 { float hi, lo; };
__device__ __forceinline__ F2 split2(double a) {
  const float h = (float)a;
  return {h, (float)(a - (double)h)};
}

__global__ void __launch_bounds__(256) r2_dd_kernel(const double* __restrict__ tiles, const double* __restrict__ Y,
                                                    const double* __restrict__ Ic, const int* __restrict__ cls,
                                                    double* __restrict__ eb, int ncls, int ntrip, int nO, int N,
                                                    int npairs, int ld, int ts) {
  const int chunk = blockIdx.x / ts, part = blockIdx.x - chunk * ts, c = blockIdx.y, iz = blockIdx.z;
  const int* cout_ptr = cls;
  const int* cout_dir = cls + ncls + 1;
  const int ne_tot = cout_ptr[ncls];
  const int* pair_ptr = cout_dir + ne_tot;
  const int* pair_in = pair_ptr + ne_tot + 1;
  const int e0 = cout_ptr[c] + chunk * kCW;
  const int e_end = cout_ptr[c + 1];
  if (e0 >= e_end) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  float4 (*Zs)[kCW * 4] = reinterpret_cast<float4 (*)[kCW * 4]>(smraw);        // [mm][col]: zr hi/lo, zi hi/lo
  float2* Asb = reinterpret_cast<float2*>(smraw + sizeof(float4) * kMB * kCW * 4);  // [(h N + n)(kMB+1) + mm]
  // columns of this block as a power of two: a block of 8 outputs has twice the threads per
  // column, not half of them idle
  const int tid = threadIdx.x, ne = e_end - e0;
  const int lc = ne <= 4 ? 2 : (ne <= 8 ? 3 : 4), tx = tid & ((1 << lc) - 1), ty = tid >> lc, nty = 256 >> lc;
  const int e_mine = e0 + tx;
  float accs[kMaxRows][4], accc[kMaxRows][4];
#pragma unroll
  for (int r = 0; r < kMaxRows; ++r)
#pragma unroll
    for (int i = 0; i < 4; ++i) { accs[r][i] = 0.f; accc[r][i] = 0.f; }
  const int nrows = (N + nty - 1) / nty;
  const size_t tile_sz = (size_t)N * ld;
  const double* tbase = tiles + ((size_t)iz * ncls + c) * ntrip * tile_sz;
  const int ze = tid & 15, zm = tid >> 4;
  const int e_z = e0 + ze;
  for (int t = ntrip * part / ts; t < ntrip * (part + 1) / ts; ++t) {
    const double* tile = tbase + (size_t)t * tile_sz;
    for (int m0 = 0; m0 < N; m0 += kMB) {
      const int mb = min(kMB, N - m0);
      {
        const int m = m0 + zm;
        double zr[4] = {0, 0, 0, 0}, zi[4] = {0, 0, 0, 0};
        if (e_z < e_end && m < N) {
          for (int p = pair_ptr[e_z]; p < pair_ptr[e_z + 1]; ++p) {
            const double* iv = Ic + (((size_t)iz * nO + pair_in[p]) * N + m) * 4;
            const double* y = Y + (((size_t)iz * npairs + p) * ntrip + t) * 32;
            const double i0 = iv[0], i1 = iv[1], i2 = iv[2], i3 = iv[3];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const double* yi = y + i * 8;
              zr[i] += yi[0] * i0 + yi[2] * i1 + yi[4] * i2 + yi[6] * i3;
              zi[i] += yi[1] * i0 + yi[3] * i1 + yi[5] * i2 + yi[7] * i3;
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const F2 a = split2(zr[i]), b = split2(zi[i]);
          Zs[zm][ze * 4 + i] = make_float4(a.hi, a.lo, b.hi, b.lo);
        }
      }
      for (int idx = tid; idx < N * 2 * kMB; idx += 256) {
        const int mm = idx % kMB;
        const int h = (idx / kMB) & 1;
        const int n = idx / (2 * kMB);
        const int m = m0 + mm;
        const F2 v = split2(m < N ? tile[(size_t)n * ld + h * N + m] : 0.0);
        Asb[(h * N + n) * (kMB + 1) + mm] = make_float2(v.hi, v.lo);
      }
      __syncthreads();
#pragma unroll 2
      for (int mm = 0; mm < mb; ++mm) {
        float4 z[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) z[i] = Zs[mm][tx * 4 + i];
#pragma unroll
        for (int r = 0; r < kMaxRows; ++r) {
          if (r < nrows) {
            const int n = ty + nty * r;
            if (n < N) {
              const float2 ar = Asb[n * (kMB + 1) + mm], ai = Asb[(N + n) * (kMB + 1) + mm];
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                // ar * zr - ai * zi
                const float p1 = ar.x * z[i].x;
                const float q1 = fmaf(ar.x, z[i].x, -p1);
                const float p2 = -ai.x * z[i].z;
                const float q2 = fmaf(-ai.x, z[i].z, -p2);
                const float lo = q1 + q2 + fmaf(ar.x, z[i].y, ar.y * z[i].x) - fmaf(ai.x, z[i].w, ai.y * z[i].z);
                dd_add(accs[r][i], accc[r][i], p1);
                dd_add(accs[r][i], accc[r][i], p2);
                accc[r][i] += lo;
              }
            }
          }
        }
      }
      __syncthreads();
    }
  }
  if (e_mine < e_end) {
    const int o = cout_dir[e_mine];
#pragma unroll
    for (int r = 0; r < kMaxRows; ++r) {
      const int n = ty + nty * r;
      if (r < nrows && n < N) {
        double* dst = eb + (((size_t)iz * nO + o) * N + n) * 4;
#pragma unroll
        for (int i = 0; i < 4; ++i) atomicAdd(dst + i, (double)accs[r][i] + (double)accc[r][i]);
      }
    }
  }
}

// ------------------------------------------------------------------ DELO
// One thread per ray (Omega, nu): I_k = (Id + b K'_k)^-1 [(e Id - a K'_{k-1}) I_{k-1}
//   + a S_{k-1} + b S_k], S = eps/eta1, K' = K/eta1 - Id.  Optional: out = x - I.
template <typename T, typename A>
__device__ __forceinline__ void kprime(const T* t, A K[4][4]) {
  K[0][0] = 0; K[1][1] = 0; K[2][2] = 0; K[3][3] = 0;
  K[0][1] = K[1][0] = t[0];
  K[0][2] = K[2][0] = t[1];
  K[0][3] = K[3][0] = t[2];
  K[1][2] = t[3]; K[2][1] = -t[3];
  K[1][3] = t[4]; K[3][1] = -t[4];
  K[2][3] = t[5]; K[3][2] = -t[5];
}

// Per-point inputs of one step of the formal solution.
template <typename T, typename A>
struct DeloPoint {
  T t[10];          // K'/eta1 (6), 1/eta1, exp(-dtau), alpha, beta
  A e[4];           // emissivity
  A xs[4];          // x of y = x - Lambda eps (zero if unused)
  double ps[3];     // DELOPAR source weights
};

template <typename T, typename A>
__device__ __forceinline__ void delo_load(DeloPoint<T, A>& d, const A* __restrict__ eps, const T* __restrict__ kt,
                                          const double* __restrict__ par, const A* __restrict__ x_sub, size_t pt) {
  for (int i = 0; i < 10; ++i) d.t[i] = kt[pt * 10 + i];
  for (int s = 0; s < 4; ++s) d.e[s] = eps[pt * 4 + s];
  for (int s = 0; s < 4; ++s) d.xs[s] = x_sub ? x_sub[pt * 4 + s] : (A)0;
  if (par)
    for (int i = 0; i < 3; ++i) d.ps[i] = par[pt * 3 + i];
}

// LU factors of M = Id + b K'_k of a point (no pivoting: M is the identity plus
// b times the antisymmetric-off-diagonal K', as in the step's original form):
// strictly lower multipliers l, strictly upper entries u and the reciprocals
// of the pivots.  M depends on the tables only, so a sweep factors the next
// point while the current one is solved, and only the substitutions, which
// carry the intensity, stay on the serial chain from step to step.
template <typename A>
struct DeloFact {
  A l10, l20, l30, l21, l31, l32;
  A u01, u02, u03, u12, u13, u23;
  A i0, i1, i2, i3;
};

template <typename T, typename A>
__device__ __forceinline__ void delo_factor(const DeloPoint<T, A>& d, DeloFact<A>& F) {
  A K[4][4];
  kprime(d.t, K);
  const A be = d.t[9];
  A M[4][4];
  for (int i = 0; i < 4; ++i)
    for (int j = 0; j < 4; ++j) M[i][j] = (i == j ? (A)1 : (A)0) + be * K[i][j];
  A l[4][4], piv[4];
  for (int c0 = 0; c0 < 4; ++c0) {
    piv[c0] = (A)1 / M[c0][c0];
    for (int r = c0 + 1; r < 4; ++r) {
      const A f = M[r][c0] * piv[c0];
      l[r][c0] = f;
      for (int cc = c0; cc < 4; ++cc) M[r][cc] -= f * M[c0][cc];
    }
  }
  F.l10 = l[1][0]; F.l20 = l[2][0]; F.l30 = l[3][0]; F.l21 = l[2][1]; F.l31 = l[3][1]; F.l32 = l[3][2];
  F.u01 = M[0][1]; F.u02 = M[0][2]; F.u03 = M[0][3]; F.u12 = M[1][2]; F.u13 = M[1][3]; F.u23 = M[2][3];
  F.i0 = piv[0]; F.i1 = piv[1]; F.i2 = piv[2]; F.i3 = piv[3];
}

// One step of the formal solution (Sect. 3) at the p-th point of a ray: DELO-
// linear, or DELOPAR when `par` (the parabolic source weights psi_M, psi_O,
// psi_P of the step arriving at the point; the source vector parabolic through
// the upwind, current and downwind points, the K'I term linear with DELO-
// linear's a, b; psi = (a, b, 0) at the last point) is set; `nxt` is the next
// point (read only under DELOPAR, p + 1 < nz); F the factors of cur's
// Id + b K'.  I, Sp, Kp carry the upwind intensity, source and K' from step
// to step.
template <typename T, typename A>
__device__ __forceinline__ void delo_step(const DeloPoint<T, A>& cur, const DeloFact<A>& F,
                                          const DeloPoint<T, A>& nxt, bool par, bool has_next, int p, bool up,
                                          int boundary, double WT0, A I[4], A Sp[4], A Kp[4][4]) {
  const T* t = cur.t;
  A Kk[4][4];
  kprime(t, Kk);
  const A ie = t[6];
  A S[4];
  for (int s = 0; s < 4; ++s) S[s] = cur.e[s] * ie;
  if (p == 0) {
    I[0] = (boundary && up) ? (A)WT0 : (A)0;
    I[1] = I[2] = I[3] = (A)0;
  } else {
    // Optically thick step (e = exp(-dtau) <= 1/2): solve for D = I_k - S_k,
    //   (Id + b K'_k) D = e (I_{k-1} - S_k) + a (S_{k-1} - S_k) - a K'_{k-1} I_{k-1} - b K'_k S_k,
    // which reproduces a constant unpolarised source exactly whatever the
    // rounding of the stored weights (b = 1 - e - a enters only the dichroic
    // terms).  Thin step: the standard form for I_k, free of the
    // cancellation I_{k-1} - S_k when I << S.
    const A e = t[7], al = t[8], be = t[9];
    const bool thick = e <= (A)0.5;
    // source weights: DELO-linear (a, b, 0) or DELOPAR's parabolic ones, with the
    // downwind source S_P; psi_M + psi_O + psi_P = 1 - e in both
    A pM = al, pO = be, pP = (A)0;
    A SP[4] = {0, 0, 0, 0};
    if (par) {
      pM = (A)cur.ps[0];
      pO = (A)cur.ps[1];
      pP = (A)cur.ps[2];
      if (has_next) {
        const A ie2 = nxt.t[6];
        for (int s = 0; s < 4; ++s) SP[s] = nxt.e[s] * ie2;
      }
    }
    A rhs[4];
    for (int i = 0; i < 4; ++i) {
      A v = thick ? e * (I[i] - S[i]) + pM * (Sp[i] - S[i]) + pP * (SP[i] - S[i])
                  : e * I[i] + pM * Sp[i] + pO * S[i] + pP * SP[i];
      for (int j = 0; j < 4; ++j) v -= al * Kp[i][j] * I[j] + (thick ? be * Kk[i][j] * S[j] : (A)0);
      rhs[i] = v;
    }
    // forward substitution with the unit lower factor, back substitution with the upper one
    const A y0 = rhs[0];
    const A y1 = rhs[1] - F.l10 * y0;
    const A y2 = rhs[2] - F.l20 * y0 - F.l21 * y1;
    const A y3 = rhs[3] - F.l30 * y0 - F.l31 * y1 - F.l32 * y2;
    A D[4];
    D[3] = y3 * F.i3;
    D[2] = (y2 - F.u23 * D[3]) * F.i2;
    D[1] = (y1 - F.u12 * D[2] - F.u13 * D[3]) * F.i1;
    D[0] = (y0 - F.u01 * D[1] - F.u02 * D[2] - F.u03 * D[3]) * F.i0;
    for (int i = 0; i < 4; ++i) I[i] = thick ? S[i] + D[i] : D[i];
  }
  for (int i = 0; i < 4; ++i) {
    Sp[i] = S[i];
    for (int j = 0; j < 4; ++j) Kp[i][j] = Kk[i][j];
  }
}

// Formal solution along every ray, one thread per ray (Omega, nu); the sweep is
// sequential in height, so the inputs of the next two points are loaded while
// a point is solved.  Used where the staged sweep below does not apply (odd
// frequency counts, lines of sight, the FP64 residual path).
template <typename T, typename A>
__global__ void delo_kernel(const A* __restrict__ eps, const T* __restrict__ kt, const double* __restrict__ par,
                            const double* __restrict__ mu, const A* __restrict__ x_sub, A* __restrict__ out, int nz,
                            int nO, int N, int boundary, double WT0) {
  const int ray = blockIdx.x * blockDim.x + threadIdx.x;
  if (ray >= nO * N) return;
  const int o = ray / N, n = ray - o * N;
  const bool up = mu[o] > 0.0;
  auto point = [&](int p) { return ((size_t)(up ? p : nz - 1 - p) * nO + o) * N + n; };
  A I[4] = {0, 0, 0, 0};
  A Sp[4] = {0, 0, 0, 0};
  A Kp[4][4];
  DeloPoint<T, A> cur, nx1, nx2;
  DeloFact<A> fc, fn;
  delo_load(cur, eps, kt, par, x_sub, point(0));
  delo_factor(cur, fc);
  if (nz > 1) delo_load(nx1, eps, kt, par, x_sub, point(1));
  for (int p = 0; p < nz; ++p) {
    const size_t pt = point(p);
    if (p + 2 < nz) delo_load(nx2, eps, kt, par, x_sub, point(p + 2));
    if (p + 1 < nz) delo_factor(nx1, fn);          // off the serial chain of this step
    delo_step(cur, fc, nx1, par != nullptr, p + 1 < nz, p, up, boundary, WT0, I, Sp, Kp);
    for (int s = 0; s < 4; ++s) out[pt * 4 + s] = x_sub ? cur.xs[s] - I[s] : I[s];
    cur = nx1;
    nx1 = nx2;
    fc = fn;
  }
}

// ---- staged sweep: one CTA per (direction, chunk of kDR frequencies).  Warp 0
// lane 0 streams each height's slices of the inputs (K'/eta1 and DELO weights,
// emissivity, the x of y = x - Lambda eps, DELOPAR weights: contiguous runs of
// kDR points) with bulk asynchronous copies into a ring of kDStages heights;
// the kDR consumer threads (one per ray) take their point from shared memory.
// Needs an even frequency count (16-byte aligned slices).  Every wait is
// bounded: on expiry the CTA stops, its copies are drained, and the
// error flag is raised (PRD_E_TIMEOUT through prd_device_status).
constexpr int kDR = 128;                       // rays per CTA
constexpr int kDStages = 8;                    // heights in flight per CTA
constexpr long long kDSpin = 1ll << 24;

__device__ __forceinline__ uint32_t dsm_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool dbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred P;\n\tmbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\tselp.b32 %0, 1, 0, P;\n\t}\n"
      : "=r"(ok)
      : "r"(dsm_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool dbar_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag) {
  for (long long i = 0; i < kDSpin; ++i) {
    if (dbar_try(b, parity)) return true;
    if (*abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}

template <typename T, typename A>
struct DeloStage {
  // byte offsets of the slices inside one stage (each a multiple of 16)
  static constexpr int kKT = 0;
  static constexpr int kEps = kKT + kDR * 10 * (int)sizeof(T);
  static constexpr int kXs = kEps + kDR * 4 * (int)sizeof(A);
  static constexpr int kPar = kXs + kDR * 4 * (int)sizeof(A);
  static constexpr int kBytes = kPar + kDR * 3 * 8;
};

template <typename T, typename A>
__global__ void __launch_bounds__(32 + kDR) delo_staged_kernel(const A* __restrict__ eps, const T* __restrict__ kt,
                                                               const double* __restrict__ par,
                                                               const double* __restrict__ mu,
                                                               const A* __restrict__ x_sub, A* __restrict__ out,
                                                               int nz, int nO, int N, int boundary, double WT0,
                                                               int* err) {
  using L = DeloStage<T, A>;
  extern __shared__ __align__(128) unsigned char dsm[];
  uint64_t* full = (uint64_t*)(dsm + kDStages * L::kBytes);
  uint64_t* empty = full + kDStages;
  volatile int* abort_flag = (volatile int*)(empty + kDStages);
  const int o = blockIdx.y, n0 = blockIdx.x * kDR;
  const int R = min(kDR, N - n0);                // rays of this CTA (even)
  const bool up = mu[o] > 0.0;
  if (threadIdx.x == 0) {
    for (int d = 0; d < kDStages; ++d) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(dsm_u32(&full[d])), "r"(1));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(dsm_u32(&empty[d])), "r"(kDR));
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  auto row = [&](int p) { return ((size_t)(up ? p : nz - 1 - p) * nO + o) * N + n0; };
  int filled = 0;                                // heights thread 0 has issued copies for
  if (threadIdx.x < 32) {
    if (threadIdx.x == 0) {
      const uint32_t bkt = (uint32_t)R * 10 * sizeof(T), bv = (uint32_t)R * 4 * sizeof(A), bp = (uint32_t)R * 24;
      const uint32_t bytes = bkt + bv + (x_sub ? bv : 0u) + (par ? bp : 0u);
      int& p = filled;
      for (; p < nz; ++p) {
        const int d = p % kDStages;
        if (p >= kDStages && !dbar_wait(&empty[d], ((p / kDStages) - 1) & 1, abort_flag)) break;
        unsigned char* st = dsm + d * L::kBytes;
        const size_t r0 = row(p);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(dsm_u32(&full[d])), "r"(bytes)
                     : "memory");
        auto copy = [&](unsigned char* dst, const void* src, uint32_t nb) {
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                  dsm_u32(dst)),
              "l"((uint64_t)src), "r"(nb), "r"(dsm_u32(&full[d]))
              : "memory");
        };
        copy(st + L::kKT, kt + r0 * 10, bkt);
        copy(st + L::kEps, eps + r0 * 4, bv);
        if (x_sub) copy(st + L::kXs, x_sub + r0 * 4, bv);
        if (par) copy(st + L::kPar, par + r0 * 3, bp);
      }
    }
  } else {
    const int r = threadIdx.x - 32;
    const bool live = r < R;
    A I[4] = {0, 0, 0, 0};
    A Sp[4] = {0, 0, 0, 0};
    A Kp[4][4];
    DeloPoint<T, A> cur, nxt;
    // take point p of this ray from its stage, then release the stage
    auto take = [&](int p, DeloPoint<T, A>& dp) -> bool {
      const int d = p % kDStages;
      if (!dbar_wait(&full[d], (p / kDStages) & 1, abort_flag)) return false;
      const unsigned char* st = dsm + d * L::kBytes;
      if (live) {
        const T* tk = (const T*)(st + L::kKT) + r * 10;
        for (int i = 0; i < 10; ++i) dp.t[i] = tk[i];
        const A* ev = (const A*)(st + L::kEps) + r * 4;
        for (int s = 0; s < 4; ++s) dp.e[s] = ev[s];
        const A* xv = (const A*)(st + L::kXs) + r * 4;
        for (int s = 0; s < 4; ++s) dp.xs[s] = x_sub ? xv[s] : (A)0;
        if (par) {
          const double* pv = (const double*)(st + L::kPar) + r * 3;
          for (int i = 0; i < 3; ++i) dp.ps[i] = pv[i];
        }
      }
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(dsm_u32(&empty[d])) : "memory");
      return true;
    };
    DeloFact<A> fc, fn;
    bool ok = take(0, cur);
    if (ok && live) delo_factor(cur, fc);
    for (int p = 0; p < nz && ok; ++p) {
      if (p + 1 < nz) ok = take(p + 1, nxt);
      if (!ok) break;
      if (live) {
        if (p + 1 < nz) delo_factor(nxt, fn);      // off the serial chain of this step
        delo_step(cur, fc, nxt, par != nullptr, p + 1 < nz, p, up, boundary, WT0, I, Sp, Kp);
        A* dst = out + (row(p) + r) * 4;
        for (int s = 0; s < 4; ++s) dst[s] = x_sub ? cur.xs[s] - I[s] : I[s];
      }
      cur = nxt;
      fc = fn;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    // a wait gave up: copies that nobody has waited for may be in flight, also those of a producer
    // that had already issued its last
    ring_drain(filled, kDStages, [&](int d, uint32_t parity) {
      for (long long i = 0; i < kDSpin && !dbar_try(&full[d], parity); ++i) {
      }
    });
    if (err) atomicExch(err, 1);
  }
}

template <typename T, typename A>
static int launch_delo(Ctx* c, const A* eps, const T* kt, const double* par, const double* mu, const A* x_sub, A* out,
                       int boundary, bool allow_staged) {
  const int nz = c->nz, nO = c->nO, N = c->nnu;
  if (allow_staged && c->staged_sweep && N % 2 == 0 && c->tc_err.p) {
    using L = DeloStage<T, A>;
    const int smem = kDStages * L::kBytes + 2 * kDStages * 8 + 16;
    delo_staged_kernel<T, A><<<dim3(ceil_div(N, kDR), nO), 32 + kDR, smem, c->stream>>>(
        eps, kt, par, mu, x_sub, out, nz, nO, N, boundary, c->WT[0], (int*)c->tc_err.p);
  } else {
    delo_kernel<T, A><<<ceil_div(nO * N, 128), 128, 0, c->stream>>>(eps, kt, par, mu, x_sub, out, nz, nO, N, boundary,
                                                                    c->WT[0]);
  }
  PRD_CUDA_TRY(c, cudaPeekAtLastError());
  return PRD_OK;
}

// f = (1 - eps) W_T eta_I / [Sigma (W_T, 0, 0, 0)]_I with the line's eta_I (App. E),
// written as (1 - eps) W_T rho / (kt6 num) with rho = eta_line / eta_total (FP64)
// and kt6 the stored 1/eta_total of the formal solver's tables: the source
// f num kt6 then holds the photon budget exactly whatever the rounding of kt6
// (an FP32 1/eta against an FP64 eta would break it at 1e-7, which the
// scattering amplifies by ~1/eps).
template <typename T, typename A>
__global__ void normalise_kernel(const A* __restrict__ num, const T* __restrict__ kt, const double* __restrict__ rho,
                                 const double* __restrict__ fac, double* __restrict__ f, int nz, int nO, int N) {
  const long long pt = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (pt >= (long long)nz * nO * N) return;
  const int iz = (int)(pt / ((long long)nO * N));
  f[pt] = fac[iz] * rho[pt] / ((double)kt[pt * 10 + 6] * (double)num[pt * 4]);
}

// Coherent continuum scattering in the observer frame (App. A):
//   eps[z][o][n][i] += sigma_c[z][n] sum_{o', j} PW[o][o'][i][j] x[z][o'][n][j]
// PW = w_o' P(o, o') (dipole phase matrix); nOut output directions (the grid,
// or one line of sight), the input x on the grid's nO directions.
template <typename A>
__global__ void continuum_kernel(const A* __restrict__ x, const double* __restrict__ pw,
                                 const double* __restrict__ sig, A* __restrict__ eps, int nz, int nOut, int nO, int N) {
  const long long pt = (long long)blockIdx.x * blockDim.x + threadIdx.x;   // (z, o, n), n fastest
  if (pt >= (long long)nz * nOut * N) return;
  const int n = (int)(pt % N);
  const int o = (int)((pt / N) % nOut);
  const int iz = (int)(pt / ((long long)N * nOut));
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int op = 0; op < nO; ++op) {
    const A* xv = x + (((size_t)iz * nO + op) * N + n) * 4;
    const double* P = pw + ((size_t)o * nO + op) * 16;
    const double x0 = xv[0], x1 = xv[1], x2 = xv[2], x3 = xv[3];
    for (int i = 0; i < 4; ++i) acc[i] += P[i * 4] * x0 + P[i * 4 + 1] * x1 + P[i * 4 + 2] * x2 + P[i * 4 + 3] * x3;
  }
  const double sc = sig[(size_t)iz * N + n];
  A* e = eps + pt * 4;
  for (int i = 0; i < 4; ++i) e[i] = (A)((double)e[i] + sc * acc[i]);
}

template <typename T>
__global__ void fill_planck_kernel(T* __restrict__ x, const double* __restrict__ WT, int nz, int nO, int N) {
  const long long pt = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (pt >= (long long)nz * nO * N) return;
  const int iz = (int)(pt / ((long long)nO * N));
  x[pt * 4] = (T)WT[iz];
  x[pt * 4 + 1] = x[pt * 4 + 2] = x[pt * 4 + 3] = (T)0;
}

// ------------------------------------------------------------------ launchers
int apply_prepare(Ctx* c) {
  int rc;
  if ((rc = allow_smem(c, spline_kernel<float, 1>)) || (rc = allow_smem(c, spline_kernel<float, 4>)) ||
      (rc = allow_smem(c, spline_kernel<double, 1>)) || (rc = allow_smem(c, spline_kernel<double, 4>)) ||
      (rc = allow_smem(c, r2_simt_kernel<float, float>)) || (rc = allow_smem(c, r2_simt_kernel<float, double>)) ||
      (rc = allow_smem(c, r2_simt_kernel<double, double>)) || (rc = allow_smem(c, r2_dd_kernel)) ||
      (rc = allow_smem(c, delo_staged_kernel<float, float>)) || (rc = allow_smem(c, delo_staged_kernel<double, double>)))
    return rc;
  return PRD_OK;
}

template <typename T, typename A>
static int sigma_T(Ctx* c, const A* x, A* eps, bool normalised, A* eb_ext = nullptr, A* Ic_ext = nullptr,
                   double* J_ext = nullptr, bool t64 = false) {
  const int nz = c->nz, nO = c->nO, N = c->nnu;
  const SigmaTables tb = sigma_tables(c, t64);
  const long long npt = (long long)nz * nO * N;
  A* Ic = Ic_ext ? Ic_ext : (A*)c->scratch2.p;
  A* eb = eb_ext ? eb_ext : (A*)c->scratch3.p;
  cudaEvent_t e0;
  // S1
  stage_begin(c, ST_S1, &e0);
  launch_spline<A>(c, x, (const int*)c->iin.p, (const double*)c->tin.p, nullptr, Ic, nO);
  stage_end(c, ST_S1, e0);
  // S5 (initialises eps_bar)
  stage_begin(c, ST_S5, &e0);
  const int nuv = c->nu_st * c->nu_st;
  double* J = J_ext ? J_ext : (double*)c->r3J.p;
  PRD_CUDA_TRY(c, cudaMemsetAsync(J, 0, (size_t)nz * nuv * 2 * sizeof(double), c->stream));
  launch_r3_J<T, A>(c, Ic, J, nO, tb);
  launch_r3_out<T, A>(c, (const double*)J, (const T*)tb.r3out, eb, nO, tb);
  stage_end(c, ST_S5, e0);
  // S3 + S4
  stage_begin(c, ST_S3, &e0);
  const int nchunk = (c->max_cout + kCW - 1) / kCW;
  // CUDA-core contractions in FP64: with few work items their tiles are split between CTAs (the
  // outputs are added up with atomics either way), up to about four CTAs per SM: 80 items of 4 tiles, 21 rows, FP64
  // 292 -> 110 us; 96 items of 20 tiles, 26 rows, double-float 1120 -> 690 us
  const int ts = std::is_same<A, double>::value
                     ? std::max(1, std::min(c->ntile(), 4 * c->nsm / (nchunk * c->ncls * nz))) : 1;
  bool s3_done = false;   // the tensor-core or double-float contraction ran
  int zc = nz;            // heights of a launch of S3 + S4 and S6
  if constexpr (std::is_same<T, float>::value && std::is_same<A, float>::value) {
    if (c->use_tc && c->tc_ready && !t64) {
      zc = c->tc_zc;
      s3_done = true;       // below, with S6
    }
  }
  if constexpr (std::is_same<T, double>::value && std::is_same<A, double>::value) {
    if (t64) {
      const size_t smem = sizeof(float4) * (size_t)kMB * kCW * 4 + sizeof(float2) * (size_t)2 * N * (kMB + 1);
      r2_dd_kernel<<<dim3(nchunk * ts, c->ncls, nz), 256, smem, c->stream>>>(
          (const double*)tb.tiles, (const double*)tb.Y, Ic, (const int*)c->cls_dev.p, eb, c->ncls, c->ntile(), nO, N,
          c->npairs, tb.ld, ts);
      s3_done = true;
    }
  }
  if (!s3_done) {
    const size_t smem = sizeof(A) * (size_t)kMB * 2 * kCW * 4 + sizeof(T) * (size_t)2 * N * (kMB + 1);
    r2_simt_kernel<T, A><<<dim3(nchunk * ts, c->ncls, nz), 256, smem, c->stream>>>(
        (const unsigned char*)tb.tiles, (const T*)tb.Y, Ic, (const int*)c->cls_dev.p, eb, c->ncls, c->ntile(),
        nO, N, c->npairs, tb.ld, tb.fmt, ts);
  }
  for (int z0 = 0; z0 < nz; z0 += zc) {
    const int n = std::min(zc, nz - z0);
    RowAdds add;            // what the tensor cores contribute to eps_bar
    if constexpr (std::is_same<T, float>::value && std::is_same<A, float>::value) {
      if (c->use_tc && c->tc_ready && !t64) {
        if (z0 > 0) stage_begin(c, ST_S3, &e0);
        int rc = r2_tc_launch(c, Ic, z0, n);
        if (rc) return rc;
        add = r2_tc_adds(c, n);
      }
    }
    const bool last = z0 + n == nz;
    stage_end(c, ST_S3, e0, last);
    // S6
    stage_begin(c, ST_S6, &e0);
    launch_spline<A>(c, eb, (const int*)c->ibk.p, (const double*)c->tbk.p, normalised ? (const double*)c->f.p : nullptr,
                     eps, nO, add, z0, n);
    if (!last) stage_end(c, ST_S6, e0, false);
  }
  // continuum scattering (App. A) joins the normalised emissivity; the
  // Kirchhoff factor is computed from the line alone (normalised = false)
  if (normalised && c->has_cont())
    continuum_kernel<A><<<ceil_div(npt, 256), 256, 0, c->stream>>>(x, (const double*)c->cont_pw.p,
                                                                 (const double*)c->cont_sig.p, eps, nz, nO, nO, N);
  stage_end(c, ST_S6, e0);
  PRD_CUDA_TRY(c, cudaPeekAtLastError());
  return PRD_OK;
}

int apply_sigma(Ctx* c, const void* x, void* eps, bool normalised) {
  if (c->prec == PRD_FP64) return sigma_T<double, double>(c, (const double*)x, (double*)eps, normalised);
  return sigma_T<float, float>(c, (const float*)x, (float*)eps, normalised);
}

int apply_lambda(Ctx* c, const void* eps, void* out, const void* sub_from, bool boundary) {
  const double* dmu = (const double*)c->dmu.p;
  cudaEvent_t e0;
  stage_begin(c, ST_S7, &e0);
  int rc;
  if (c->prec == PRD_FP64)
    rc = launch_delo<double, double>(c, (const double*)eps, (const double*)c->kt.p, (const double*)c->par_active(), dmu,
                                     (const double*)sub_from, (double*)out, boundary ? 1 : 0, true);
  else
    rc = launch_delo<float, float>(c, (const float*)eps, (const float*)c->kt.p, (const double*)c->par_active(), dmu,
                                   (const float*)sub_from, (float*)out, boundary ? 1 : 0, true);
  stage_end(c, ST_S7, e0);
  return rc;
}

// Kirchhoff factor f = (1-eps) W_T eta_I / [Sigma (W_T,0,0,0)]_I (App. E).  In
// FP32 mode the unnormalised Sigma is applied to the Planck field in FP64, with
// the tables the refinement residuals use, so that f corrects the photon budget
// of exactly the operator whose solution is returned (the FP32 apply that
// drives the inner iterations differs from it only at FP32 rounding level).
int compute_normalisation(Ctx* c) {
  const int nz = c->nz, nO = c->nO, N = c->nnu;
  const long long npt = (long long)nz * nO * N;
  DBuf wt, fac, xin, num, eb, Ic;
  std::vector<double> f(nz);
  for (int iz = 0; iz < nz; ++iz) f[iz] = (1.0 - c->eps[iz]) * c->WT[iz];
  int rc;
  const size_t vb64 = nvec(c) * 8;
  auto cleanup = [&]() { dfree(wt); dfree(fac); dfree(xin); dfree(num); dfree(eb); dfree(Ic); };
  if ((rc = upload(c, wt, c->WT.data(), nz * 8)) || (rc = upload(c, fac, f.data(), nz * 8)) ||
      (rc = dalloc(c, xin, vb64)) || (rc = dalloc(c, num, vb64)) || (rc = dalloc(c, eb, vb64)) ||
      (rc = dalloc(c, Ic, vb64))) {
    cleanup();
    return rc;
  }
  if (c->prec == PRD_FP64) {
    fill_planck_kernel<double><<<ceil_div(npt, 256), 256, 0, c->stream>>>((double*)xin.p, (const double*)wt.p, nz, nO, N);
    rc = sigma_T<double, double>(c, (const double*)xin.p, (double*)num.p, false);
    if (!rc)
      normalise_kernel<double, double><<<ceil_div(npt, 256), 256, 0, c->stream>>>(
          (const double*)num.p, (const double*)c->kt.p, (const double*)c->eta_line.p, (const double*)fac.p,
          (double*)c->f.p, nz, nO, N);
  } else {
    fill_planck_kernel<double><<<ceil_div(npt, 256), 256, 0, c->stream>>>((double*)xin.p, (const double*)wt.p, nz, nO, N);
    rc = c->has64 ? sigma_T<double, double>(c, (const double*)xin.p, (double*)num.p, false, (double*)eb.p,
                                            (double*)Ic.p, nullptr, true)
                  : sigma_T<float, double>(c, (const double*)xin.p, (double*)num.p, false, (double*)eb.p,
                                           (double*)Ic.p);
    if (!rc)
      normalise_kernel<double, double><<<ceil_div(npt, 256), 256, 0, c->stream>>>(
          (const double*)num.p, (const double*)c->kt64.p, (const double*)c->eta_line.p, (const double*)fac.p,
          (double*)c->f.p, nz, nO, N);
  }
  cudaError_t e = cudaStreamSynchronize(c->stream);
  cleanup();
  if (rc) return rc;
  if (e != cudaSuccess) return fail(c, PRD_E_CUDA, std::string("normalisation: ") + cudaGetErrorString(e));
  return PRD_OK;
}

int apply_operator(Ctx* c, const void* x, void* y) {
  int rc = apply_sigma(c, x, c->gm_t.p, true);
  if (rc) return rc;
  return apply_lambda(c, c->gm_t.p, y, x, false);
}

int rhs(Ctx* c, void* b) { return apply_lambda(c, c->epsth.p, b, nullptr, true); }

// FP32 mode only: y = (Id - Lambda Sigma) x with FP64 vectors, FP64 arithmetic
// and the FP64 copy of the Sigma tables when it was kept (else the FP32 tables):
// the residuals of the refinement, which fix the accuracy of the solution.
int apply_operator_acc(Ctx* c, const double* x, double* y, double* ws /* 3 x nvec doubles */) {
  const size_t nv = nvec(c);
  double* eps = ws;
  int rc = c->has64 ? sigma_T<double, double>(c, x, eps, true, ws + nv, ws + 2 * nv, nullptr, true)
                     : sigma_T<float, double>(c, x, eps, true, ws + nv, ws + 2 * nv);
  if (rc) return rc;
  delo_kernel<double, double><<<ceil_div(c->nO * c->nnu, 128), 128, 0, c->stream>>>(
      eps, (const double*)c->kt64.p, (const double*)c->par_active(), (const double*)c->dmu.p, x, y, c->nz, c->nO,
      c->nnu, 0, c->WT[0]);
  PRD_CUDA_TRY(c, cudaPeekAtLastError());
  return PRD_OK;
}

__global__ void add_kernel(double* __restrict__ a, const double* __restrict__ b, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    a[i] += b[i];
}

// eps = eps_th + Sigma x in FP64 arithmetic on the FP64 tables (the residual
// path of the refinement in FP32 mode): the emissivity whose formal solution,
// with the boundary term, minus x is the residual b - A x.  ws: 2 N-vectors.
int emissivity_acc(Ctx* c, const double* x, double* eps, double* ws) {
  const size_t nv = nvec(c);
  int rc;
  if (c->prec == PRD_FP64) rc = sigma_T<double, double>(c, x, eps, true);
  else if (c->has64) rc = sigma_T<double, double>(c, x, eps, true, ws, ws + nv, nullptr, true);
  else rc = sigma_T<float, double>(c, x, eps, true, ws, ws + nv);
  if (rc) return rc;
  add_kernel<<<c->grid_ew(), 256, 0, c->stream>>>(eps, (const double*)(c->prec == PRD_FP64 ? c->epsth.p : c->epsth64.p),
                                                  nv);
  PRD_CUDA_TRY(c, cudaPeekAtLastError());
  return PRD_OK;
}

int rhs_acc(Ctx* c, double* b) {
  delo_kernel<double, double><<<ceil_div(c->nO * c->nnu, 128), 128, 0, c->stream>>>(
      (const double*)c->epsth64.p, (const double*)c->kt64.p, (const double*)c->par_active(), (const double*)c->dmu.p,
      nullptr, b, c->nz, c->nO, c->nnu, 1, c->WT[0]);
  cudaError_t e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return fail(c, PRD_E_CUDA, std::string("rhs_acc: ") + cudaGetErrorString(e));
  return PRD_OK;
}

// ------------------------------------------------------------------ S11
// Emergent Stokes vectors along extra lines of sight (Sect. 6.2): for each
// LOS the comoving emissivity eps_bar(z, LOS, .) is built from the solution's
// comoving field with new tiles for the angles Theta(LOS, Omega'), normalised
// with f computed from the same rows on the Planck field, moved to the
// observer frame, and one DELO sweep from the bottom boundary gives I at z_max.
template <typename T>
__global__ void planck_comoving_kernel(T* __restrict__ Ic, const double* __restrict__ WT, int nz, int nO, int N) {
  const long long pt = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (pt >= (long long)nz * nO * N) return;
  const int iz = (int)(pt / ((long long)nO * N));
  Ic[pt * 4] = (T)WT[iz];
  Ic[pt * 4 + 1] = Ic[pt * 4 + 2] = Ic[pt * 4 + 3] = (T)0;
}

// eps(z, n) = (eps_sc with f) + eps_th;  f = (1-eps) W_T eta_I / num_I, formed
// as in normalise_kernel from rho = eta_line / eta_total and the stored 1/eta_total
template <typename T, typename A>
__global__ void los_combine_kernel(const A* __restrict__ es, const A* __restrict__ ew, const T* __restrict__ kt,
                                   const double* __restrict__ rho, const T* __restrict__ eth,
                                   const double* __restrict__ fac, A* __restrict__ out, int nz, int N) {
  const int pt = blockIdx.x * blockDim.x + threadIdx.x;
  if (pt >= nz * N) return;
  const int iz = pt / N;
  const double f = fac[iz] * rho[pt] / ((double)kt[pt * 10 + 6] * (double)ew[pt * 4]);
  out[pt * 4] = (A)((double)es[pt * 4] * f + (double)eth[pt * 4]);
  for (int s = 1; s < 4; ++s) out[pt * 4 + s] = es[pt * 4 + s] + (A)eth[pt * 4 + s];
}

template <typename S, typename D>
__global__ void cast_kernel(const S* __restrict__ in, D* __restrict__ out, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = (D)in[i];
}

// R_II along one line of sight: es_bar[z][n][i] += sum over the incident directions o' (each
// its own scattering angle) and tiles of Re(T[n][m] Z[m][i]), Z = Y I~, in FP64, and the same
// for the Planck field (W_T, 0, 0, 0), which is flat in frequency: only the row sums of T and
// Y_00 enter, into the intensity of ew_bar.  A thread takes a tile row n, a CTA the tiles
// [tg * y, tg * (y + 1)) of one direction and height (grid.z = heights z0 ..): both fields share
// one read of the tile, and small problems get a CTA per tile.  FP64-bound (six operations a
// tile element); the generic contraction, a launch per height and field of one CTA per
// direction, took 6.6 ms a height at 16 directions x 41 frequencies.
template <typename T>
__global__ void los_r2_kernel(const T* __restrict__ tiles, const T* __restrict__ Y, const double* __restrict__ Ic,
                              const double* __restrict__ WT, double* __restrict__ es, double* __restrict__ ew, int z0,
                              int ncls, int nO, int nti, int N, int ld, int tiled, int tg) {
  extern __shared__ __align__(16) unsigned char lsm[];
  double* Z = reinterpret_cast<double*>(lsm);              // [m][zr(4) | zi(4)]
  const int op = blockIdx.x, zl = blockIdx.z, iz = z0 + zl, n = threadIdx.x;
  const int c = ncls == 1 ? 0 : op;                        // angle-averaged: one class for all directions
  const double4_16a* I = reinterpret_cast<const double4_16a*>(Ic) + ((size_t)iz * nO + op) * N;
  double acc[4] = {0, 0, 0, 0}, accw = 0.0;
  const double W = WT[iz];
  for (int ti = blockIdx.y * tg; ti < min(nti, (int)(blockIdx.y + 1) * tg); ++ti) {
    const T* y = Y + (((size_t)iz * nO + op) * nti + ti) * 32;
    __syncthreads();
    for (int m = threadIdx.x; m < N; m += blockDim.x) {
      const double4_16a v = I[m];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const T* yi = y + i * 8;
        Z[m * 8 + i] = (double)yi[0] * v.x + (double)yi[2] * v.y + (double)yi[4] * v.z + (double)yi[6] * v.w;
        Z[m * 8 + 4 + i] = (double)yi[1] * v.x + (double)yi[3] * v.y + (double)yi[5] * v.z + (double)yi[7] * v.w;
      }
    }
    __syncthreads();
    if (n < N) {
      const T* t = tiles + (((size_t)zl * ncls + c) * nti + ti) * N * ld;
      double sr = 0.0, si = 0.0;
#pragma unroll 4
      for (int m = 0; m < N; ++m) {
        const double ar = (double)t[tile_off(n, m, N, ld, tiled != 0)], ai = (double)t[tile_off(n, N + m, N, ld, tiled != 0)];
        const double* z = Z + m * 8;
        sr += ar;
        si += ai;
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] += ar * z[i] - ai * z[4 + i];
      }
      accw += W * ((double)y[0] * sr - (double)y[1] * si);
    }
  }
  if (n < N) {
    double* e = es + ((size_t)iz * N + n) * 4;
#pragma unroll
    for (int i = 0; i < 4; ++i) atomicAdd(e + i, acc[i]);
    atomicAdd(ew + ((size_t)iz * N + n) * 4, accw);
  }
}

// T: precision of the stored tables and of x / out; A: precision of the fields
// along the line of sight (double in FP32 mode, like the FP64-accumulated
// residual path, so the emergent spectrum carries no FP32 cancellation).

template <typename T, typename A>
static int emergent_T(Ctx* c, const T* x, int nlos, const double* mus, const double* chis, T* out) {
  const int nz = c->nz, nO = c->nO, N = c->nnu, nti = c->ntile(), nuv = c->nu_st * c->nu_st;
  const long long npt = (long long)nz * nO * N;
  const int ncl = c->mode == PRD_MODE_AA ? 1 : nO;               // scattering angles of a line of sight
  const size_t tz = (size_t)ncl * nti * N * c->ld() * sizeof(T);   // tiles of one height
  DBuf Icx, Icw, Jx, Jw, tiles, Yd, rout, ktd, ethd, kidx, ttd, es_bar, ew_bar, es, ew, eps, lam, fac, dmu, wtd,
      xa, pard, etald, cpwd;
  int rc, zb = 1;
  LosTiles* lt = los_tiles_create(c, ncl, &zb, &rc);
  if (!lt) return rc;
  auto cleanup = [&]() {
    DBuf* bs[] = {&Icx, &Icw, &Jx, &Jw, &tiles, &Yd, &rout, &ktd, &ethd, &kidx, &ttd, &es_bar, &ew_bar, &es, &ew,
                  &eps, &lam, &fac, &dmu, &wtd, &xa, &pard, &etald, &cpwd};
    for (DBuf* b : bs) dfree(*b);
    los_tiles_destroy(lt);
  };
  const size_t vb = nvec(c) * sizeof(A), lb = (size_t)nz * N * 4 * sizeof(A);
  std::vector<double> facv(nz), wt(c->WT);
  for (int iz = 0; iz < nz; ++iz) facv[iz] = (1.0 - c->eps[iz]) * c->WT[iz];
  if ((rc = dalloc(c, Icx, vb)) || (rc = dalloc(c, Icw, vb)) || (rc = dalloc(c, Jx, (size_t)nz * nuv * 16)) ||
      (rc = dalloc(c, Jw, (size_t)nz * nuv * 16)) || (rc = dalloc(c, tiles, tz * zb)) || (rc = dalloc(c, es_bar, lb)) ||
      (rc = dalloc(c, ew_bar, lb)) || (rc = dalloc(c, es, lb)) || (rc = dalloc(c, ew, lb)) ||
      (rc = dalloc(c, eps, lb)) || (rc = dalloc(c, lam, lb)) || (rc = upload(c, fac, facv.data(), nz * 8)) ||
      (rc = dalloc(c, xa, vb)) || (rc = upload(c, wtd, wt.data(), nz * 8))) {
    cleanup();
    return rc;
  }
  // comoving fields of the solution and of the Planck function, and their R_III moments
  cast_kernel<T, A><<<ceil_div(npt * 4, 256), 256, 0, c->stream>>>(x, (A*)xa.p, npt * 4);
  launch_spline<A>(c, (const A*)xa.p, (const int*)c->iin.p, (const double*)c->tin.p, nullptr, (A*)Icx.p, nO);
  planck_comoving_kernel<A><<<ceil_div(npt, 256), 256, 0, c->stream>>>((A*)Icw.p, (const double*)wtd.p, nz, nO, N);
  PRD_CUDA_TRY(c, cudaMemsetAsync(Jx.p, 0, Jx.bytes, c->stream));
  PRD_CUDA_TRY(c, cudaMemsetAsync(Jw.p, 0, Jw.bytes, c->stream));
  const SigmaTables tb = sigma_tables(c, false);
  launch_r3_J<T, A>(c, (const A*)Icx.p, (double*)Jx.p, nO, tb);
  launch_r3_J<T, A>(c, (const A*)Icw.p, (double*)Jw.p, nO, tb);
  PRD_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  for (int l = 0; l < nlos && !rc; ++l) {
    LosTables L;
    los_tables(c, mus[l], chis[l], L);
    auto up = [&](DBuf& b, const std::vector<double>& v) {
      std::vector<T> h(v.begin(), v.end());
      return upload(c, b, h.data(), h.size() * sizeof(T));
    };
    if ((rc = up(Yd, L.Y)) || (rc = up(rout, L.rout)) || (rc = up(ktd, L.kt)) || (rc = up(ethd, L.epsth)) ||
        (rc = upload(c, pard, L.par.data(), L.par.size() * 8)) ||
        (rc = upload(c, etald, L.eta_line.data(), L.eta_line.size() * 8)) ||
        (rc = upload(c, cpwd, L.cont_pw.data(), L.cont_pw.size() * 8)) ||
        (rc = upload(c, kidx, L.kidx.data(), L.kidx.size() * 4)) || (rc = upload(c, ttd, L.tt.data(), L.tt.size() * 8)) ||
        (rc = upload(c, dmu, &mus[l], 8)))
      break;
    // R_III parts initialise the comoving rows
    launch_r3_out<T, A>(c, (const double*)Jx.p, (const T*)rout.p, (A*)es_bar.p, 1, tb);
    launch_r3_out<T, A>(c, (const double*)Jw.p, (const T*)rout.p, (A*)ew_bar.p, 1, tb);
    // R_II: tiles of the heights for the LOS classes, zb heights at a time, then the contraction
    if (ncl > 1 && (rc = los_tiles_angles(c, lt, L.theta))) break;
    const int tg = nO * nz >= 4 * c->nsm ? nti : 1;      // enough CTAs for the SMs with all tiles in one
    for (int z0 = 0; z0 < nz && !rc; z0 += zb) {
      const int n = std::min(zb, nz - z0);
      if ((rc = los_tiles_gen(c, lt, z0, n, tiles.p))) break;
      los_r2_kernel<T><<<dim3(nO, (nti + tg - 1) / tg, n), (N + 31) / 32 * 32, (size_t)N * 64, c->stream>>>(
          (const T*)tiles.p, (const T*)Yd.p, (const double*)Icx.p, (const double*)wtd.p, (double*)es_bar.p,
          (double*)ew_bar.p, z0, ncl, nO, nti, N, c->ld(), c->tiled(), tg);
    }
    if (rc) break;
    PRD_CUDA_TRY(c, cudaPeekAtLastError());
    // observer frame, normalisation, thermal part, formal solution along the LOS
    launch_spline<A>(c, (const A*)es_bar.p, (const int*)kidx.p, (const double*)ttd.p, nullptr, (A*)es.p, 1);
    launch_spline<A>(c, (const A*)ew_bar.p, (const int*)kidx.p, (const double*)ttd.p, nullptr, (A*)ew.p, 1);
    los_combine_kernel<T, A><<<ceil_div(nz * N, 128), 128, 0, c->stream>>>((const A*)es.p, (const A*)ew.p,
                                                                          (const T*)ktd.p, (const double*)etald.p,
                                                                          (const T*)ethd.p,
                                                                          (const double*)fac.p, (A*)eps.p, nz, N);
    if (c->has_cont())
      continuum_kernel<A><<<ceil_div(nz * N, 128), 128, 0, c->stream>>>((const A*)xa.p, (const double*)cpwd.p,
                                                                       (const double*)c->cont_sig.p, (A*)eps.p, nz,
                                                                       1, nO, N);
    delo_kernel<T, A><<<ceil_div(N, 128), 128, 0, c->stream>>>((const A*)eps.p, (const T*)ktd.p,
                                                             c->formal ? (const double*)pard.p : nullptr,
                                                             (const double*)dmu.p, nullptr, (A*)lam.p, nz, 1, N, 1,
                                                             c->WT[0]);
    cast_kernel<A, T><<<ceil_div(N * 4, 128), 128, 0, c->stream>>>((const A*)lam.p + (size_t)(nz - 1) * N * 4,
                                                                  out + (size_t)l * N * 4, (long long)N * 4);
    PRD_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  }
  cleanup();
  return rc;
}

int emergent(Ctx* c, const void* x, int nlos, const double* mu, const double* chi, void* out) {
  if (c->prec == PRD_FP64) return emergent_T<double, double>(c, (const double*)x, nlos, mu, chi, (double*)out);
  return emergent_T<float, double>(c, (const float*)x, nlos, mu, chi, (float*)out);
}

// ------------------------------------------------------------------ static scratch
// Scratch of prd_apply_sigma_noalloc: one file-scope device array, present on
// every GPU that loads the library until the process exits.
constexpr size_t kStaticScratchBytes = (size_t)64 << 20;   // 64 MiB
static __device__ __align__(256) unsigned char g_sigma_scratch[kStaticScratchBytes];

// Device address of the static scratch in the current CUDA context.  The
// host-side symbol is only a stand-in and must not be passed to a kernel.  The
// address is looked up on every call (cudaGetSymbolAddress allocates nothing):
// a cached address would dangle after the host framework resets the device or
// re-creates its primary context, which reloads the library's device code.
static int static_scratch(Ctx* c, void** out) {
  void* p = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&p, g_sigma_scratch);
  if (e != cudaSuccess || !p)
    return fail(c, PRD_E_CUDA, std::string("cudaGetSymbolAddress(static scratch): ") + cudaGetErrorString(e));
  *out = p;
  return PRD_OK;
}

template <typename T>
static int sigma_static_T(Ctx* c, const T* x, T* eps) {
  const size_t nv = nvec(c);
  const size_t nuv = (size_t)c->nu_st * c->nu_st;
  const size_t jbytes = ((size_t)c->nz * nuv * 2 * sizeof(double) + 255) / 256 * 256;
  const size_t vb = (nv * sizeof(T) + 255) / 256 * 256;
  // the limit of the documented interface: three vectors and the R_III moments
  if (jbytes + 3 * vb > kStaticScratchBytes)
    return fail(c, PRD_E_ARG, "problem needs " + std::to_string((jbytes + 3 * vb) >> 20) +
                                  " MiB of scratch; prd_apply_sigma_noalloc supports at most 64 MiB");
  void* base = nullptr;
  int rc = static_scratch(c, &base);
  if (rc) return rc;
  unsigned char* b = (unsigned char*)base;
  double* J = (double*)b;
  T* Ic = (T*)(b + jbytes);
  T* eb = (T*)(b + jbytes + vb);
  return sigma_T<T, T>(c, x, eps, true, eb, Ic, J);
}

}  // namespace prd

extern "C" int prd_apply_sigma_noalloc(prd_ctx* ctx, const void* x_dev, void* eps_dev) {
  if (!ctx) return PRD_E_ARG;
  prd::Ctx* c = &ctx->c;
  cudaSetDevice(c->device);
  if (!c->ready) return prd::fail(c, PRD_E_STATE, "call prd_setup first");
  if (!x_dev || !eps_dev || x_dev == eps_dev) return prd::fail(c, PRD_E_ARG, "x_dev/eps_dev NULL or aliased");
  if (!prd::point_aligned(c, x_dev) || !prd::point_aligned(c, eps_dev))
    return prd::fail(c, PRD_E_ARG, "x_dev/eps_dev do not start on a whole Stokes point (4 elements)");
  if (c->prec == PRD_FP64) return prd::sigma_static_T<double>(c, (const double*)x_dev, (double*)eps_dev);
  return prd::sigma_static_T<float>(c, (const float*)x_dev, (float*)eps_dev);
}
