// Setup kernels: redistribution tiles of the R_II-AD kernel against the
// natural-spline basis (Eq. G, F after it; App. C rule i for Theta = 0; the
// Theta = pi limit kernel), R_III incident weights (Eq. RIIIQKKp) and the
// angle-averaged tiles (Eq. R_AA).
//
// A tile row n of class c and triple t = (k, kl, kl') is
//     T[n][m] = int F(Theta_c, u' + s_in, u_n + s_out) phi_m(u') du',
// s_in = s_{k kl}, s_out = s_{k kl'}, phi_m the cardinal natural cubic
// spline on the height's reduced-frequency grid continued by its end values.
// On grid interval j the spline is (1-t) y_j + t y_{j+1}
// + h_j^2/6 [((1-t)^3-(1-t)) M_j + (t^3-t) M_{j+1}], M = Q y; so a row is
// P_y + P_M Q with P_y, P_M the four moments of F on each interval.
//
// The quadrature marches Gauss-Legendre panels (8 nodes) through every interval,
// whose width is at most a quarter of the Gaussian width 2 sin(Theta/2) and
// shrinks geometrically towards the centre of the W factor (v = 0), and
// accumulates the moments in FP64.
//
// What bounds it: FP64 arithmetic (2 lanes a clock and SM), nearly all of it W and
// the exponential at the nodes; a warp instruction costs the same with one lane
// active as with 32.  So
//   - a warp takes one row and its lanes take panels, 32 at a time, whatever
//     intervals they belong to (with a lane per interval the few intervals that
//     hold most panels kept one or two lanes busy).  A lane finds its panel by
//     counting the interval's panels in FP32 pairs, which costs nothing beside
//     one node; sums of a panel's lanes go to their interval by a segmented
//     shuffle reduction, in a fixed order;
//   - a polynomial with real coefficients at a complex point takes two FMAs a term
//     (Knuth's scheme, TAOCP 4.6.4) instead of four, W beyond |z| = 8 is its
//     asymptotic series, and divisions by per-row constants are products;
//   - P_M Q is a tridiagonal solve per row (Q = T^-1 D, T symmetric), N steps
//     instead of N^2 products, the rows of a CTA side by side in one warp;
//   - an angle-averaged row has a CTA, its warps sharing the angles, and the
//     preconditioner's rows of all heights are one launch.
// Measured, setup of 4 heights x 16 directions x 60 frequencies with a first apply: 978 -> 29 ms
// (the preconditioner's rows 203 ms a height before); three lines of sight of 4 x 16 x 41
// points: 496 -> 22 ms.
#include <algorithm>
#include <cstdio>
#include <cuda_bf16.h>
#include "prd_internal.h"
#include "device_common.cuh"

namespace prd {

__constant__ WeidemanConst c_wc;
__constant__ double c_gl8x[8];
__constant__ double c_gl8w[8];

enum RowKind { ROW_R2 = 0, ROW_R3 = 1 };

// 1/d for d in the FP32 range: Newton's iteration from an FP32 reciprocal
__device__ __forceinline__ double newton_rcp(double d) {
  double r = (double)(1.0f / (float)d);
  r = fma(r, fma(-d, r, 1.0), r);
  return fma(r, fma(-d, r, 1.0), r);
}

// w(x + i y), y >= 0.  |z| <= 8: Weideman's rational expansion in Z = (L+iz)/(L-iz),
//   w = 2 p(Z)/(L - i z)^2 + 1/(sqrt(pi)(L - i z)),  p(Z) = sum_k a_k Z^k;
// beyond, the asymptotic series w ~ i/(sqrt(pi) z) sum_k (2k-1)!! / (2 z^2)^k
// (17 terms: the first one left out is below 1e-17), whose real part keeps its
// relative accuracy for small y.  Both sums by Knuth's scheme for real coefficients:
// b_k = a_k + 2 Re(Z) b_{k+1} - |Z|^2 b_{k+2}.
__device__ __forceinline__ Cx<double> faddeeva(double x, double y) {
  const double isp = 0.56418958354775628695;              // 1/sqrt(pi)
  const double q = x * x + y * y;
  if (q > 64.0) {
    const double inv = newton_rcp(q);
    const double zr = x * inv, zi = -y * inv;             // 1/z
    const double tr = zr * zr - zi * zi, ti = 2.0 * zr * zi, r = 2.0 * tr, s = inv * inv;
    constexpr double c[17] = {1.0, 0.5, 0.75, 1.875, 6.5625, 29.53125, 162.421875, 1055.7421875, 7918.06640625,
                              67303.564453125, 639383.8623046875, 6713530.55419921875, 77205601.373291015625,
                              965070017.1661376953125, 13028445231.74285888671875, 188912455860.271453857421875,
                              2928143065834.2075347900390625};
    double b1 = c[16], b2 = 0.0;
#pragma unroll
    for (int k = 15; k >= 1; --k) {
      const double b = fma(r, b1, fma(-s, b2, c[k]));
      b2 = b1;
      b1 = b;
    }
    const double Sr = fma(tr, b1, fma(-s, b2, c[0])), Si = ti * b1;
    return {-isp * (zr * Si + zi * Sr), isp * (zr * Sr - zi * Si)};
  }
  const double L = c_wc.L64;
  // L - i z = (L + y) - i x ;  L + i z = (L - y) + i x
  const double dr = L + y, di = -x, nr = L - y;
  const double inv = newton_rcp(dr * dr + di * di);
  const double Zr = (nr * dr + x * di) * inv, Zi = (x * dr - nr * di) * inv;
  const double r = 2.0 * Zr, s = Zr * Zr + Zi * Zi;
  double b1 = c_wc.a64[35], b2 = 0.0;
#pragma unroll
  for (int k = 34; k >= 1; --k) {
    const double b = fma(r, b1, fma(-s, b2, c_wc.a64[k]));
    b2 = b1;
    b1 = b;
  }
  const double pr = fma(Zr, b1, fma(-s, b2, c_wc.a64[0])), pi = Zi * b1;
  const double ir = dr * inv, ii = -di * inv;             // 1/(L - i z)
  const double i2r = ir * ir - ii * ii, i2i = 2.0 * ir * ii;
  return {2.0 * (pr * i2r - pi * i2i) + isp * ir, 2.0 * (pr * i2i + pi * i2r) + isp * ii};
}

// The kernel of one row as a function of the incident node u'.
//   R_II: F(Theta, u' + s_in, x), x = u_n + s_out (Eq. G), times wscale;
//   R_III: the incident bracket W(u' + s_in) + W(u' + s_out)^* of Eq. RIIIQKKp.
struct RowKernel {
  double x, s_in, s_out, a;
  double inv_g, inv_2c, y, scale;   // 1/(2 sin), 1/(2 cos), a/cos of Theta/2, wscale/sin(Theta)
  bool back;                        // Theta = pi
};

template <int KIND>
__device__ __forceinline__ Cx<double> row_eval(const RowKernel& k, double up) {
  if (KIND == ROW_R3) {
    const Cx<double> w1 = faddeeva(up + k.s_in, k.a), w2 = faddeeva(up + k.s_out, k.a);
    return {w1.re + w2.re, w1.im - w2.im};
  }
  const double xp = up + k.s_in;
  if (k.back) {
    const double v = 0.5 * (k.x + xp), d = k.x - xp;
    const double g = k.scale * exp(-0.25 * d * d) / (2.0 * 1.7724538509055160 * (v * v + k.a * k.a));
    return {g * k.a, g * v};
  }
  const double d = (k.x - xp) * k.inv_g;
  const double g = exp(-d * d) * k.scale;
  const Cx<double> w = faddeeva((k.x + xp) * k.inv_2c, k.y);
  return {g * w.re, g * w.im};
}

// An unevaluated pair of floats: positions within an interval, to ~2^-45
struct FF { float h, l; };
__device__ __forceinline__ FF ff(double v) {
  const float h = (float)v;
  return {h, (float)(v - (double)h)};
}
__device__ __forceinline__ float ff_diff(FF a, FF b) { return (a.h - b.h) + (a.l - b.l); }
__device__ __forceinline__ FF ff_add(FF a, float w) {
  const float s = a.h + w, bb = s - a.h;
  const float e = (a.h - (s - bb)) + (w - bb) + a.l;
  const float h = s + e;
  return {h, e - (h - s)};
}

// The panels of one interval [x0, x1], positions as offsets from x0.
struct Marcher {
  FF end, c1, c2;      // x1, and the centres to refine towards: uV (R_II) or -s_in, -s_out (R_III)
  float hV, hG;
  template <int KIND>
  __device__ __forceinline__ float width(FF pos, float rem) const {
    if (KIND == ROW_R2) {
      const float gap = ff_diff(c1, pos), q = 0.25f * hV;
      float w = fminf(hG, fmaxf(q, 0.5f * fabsf(gap)));
      // never wider than the Gaussian limit, and a panel ends at the W centre
      if (gap > 0.f && gap < rem) w = gap > q ? fminf(w, fmaxf(0.5f * gap, q)) : fminf(w, gap);
      return w;
    }
    // R_III profiles: smooth on scale 1 around their centres
    const float g1 = ff_diff(c1, pos), g2 = ff_diff(c2, pos);
    float w = fmaxf(0.25f, 0.25f * fminf(fabsf(g1), fabsf(g2)));
    if (g1 > 0.f && g1 < w) w = fmaxf(g1, 0.05f);
    if (g2 > 0.f && g2 < w) w = fmaxf(g2, 0.05f);
    return w;
  }
};
constexpr int kMaxPanels = 4096;         // panels of one interval

template <int KIND>
__device__ __forceinline__ int count_panels(const Marcher& m) {
  FF pos = {0.f, 0.f};
  int n = 0;
  for (; n < kMaxPanels; ++n) {
    const float rem = ff_diff(m.end, pos);
    if (!(rem > 0.f)) break;
    const float w = m.width<KIND>(pos, rem);
    if (!(w > 0.f)) break;
    if (w >= rem) return n + 1;
    pos = ff_add(pos, w);
  }
  return n;
}

__device__ __forceinline__ int find_interval(const double* u, int N, double x) {
  // largest j with u[j] <= x, clamped to [0, N-2]; -1 if x < u[0]; N-1 if x >= u[N-1]
  if (x < u[0]) return -1;
  if (x >= u[N - 1]) return N - 1;
  int lo = 0, hi = N - 1;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (u[mid] <= x) lo = mid; else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ double shfl_down_d(double v, int d) { return __shfl_down_sync(0xffffffffu, v, d); }

// Moments of one row (P_y in acc[0..2N), P_M in acc[2N..4N), Re then Im) over the
// support of R_II or the grid span of R_III, added to acc by one warp.  off: N + 2 ints.
template <int KIND>
__device__ void row_moments(double theta, double a, double s_in, double s_out, double un, const double* u, int N,
                            double* acc, int* off, double wscale) {
  const int lane = threadIdx.x & 31;
  double* PyR = acc;
  double* PyI = acc + N;
  double* PmR = acc + 2 * N;
  double* PmI = acc + 3 * N;
  if (KIND == ROW_R2 && theta == 0.0) {
    if (lane == 0) {
      // App. C rule i: sqrt(pi) W(a, x) delta(u' - (x - s_in))
      const double x = un + s_out, p = x - s_in;
      const Cx<double> w = faddeeva(x, a);
      const double cr = 1.7724538509055160 * w.re * wscale, ci = 1.7724538509055160 * w.im * wscale;
      const int j = find_interval(u, N, p);
      if (j < 0) { PyR[0] += cr; PyI[0] += ci; }
      else if (j >= N - 1) { PyR[N - 1] += cr; PyI[N - 1] += ci; }
      else {
        const double h = u[j + 1] - u[j], t = (p - u[j]) / h, omt = 1.0 - t, k6 = h * h / 6.0;
        PyR[j] += cr * omt; PyI[j] += ci * omt;
        PyR[j + 1] += cr * t; PyI[j + 1] += ci * t;
        PmR[j] += cr * k6 * (omt * omt * omt - omt); PmI[j] += ci * k6 * (omt * omt * omt - omt);
        PmR[j + 1] += cr * k6 * (t * t * t - t); PmI[j + 1] += ci * k6 * (t * t * t - t);
      }
    }
    __syncwarp();
    return;
  }
  RowKernel rk{un + s_out, s_in, s_out, a, 0.0, 0.0, 0.0, wscale, false};
  double L, R, uV = 0.0;
  float hV = 1.f, hG = 1.f;
  if (KIND == ROW_R2) {
    rk.back = theta >= 3.14159265358979;
    const double s2 = rk.back ? 1.0 : sin(0.5 * theta), c2 = rk.back ? 0.0 : cos(0.5 * theta);
    if (!rk.back) {
      rk.inv_g = 1.0 / (2.0 * s2);
      rk.inv_2c = 1.0 / (2.0 * c2);
      rk.y = a / c2;
      rk.scale = wscale / sin(theta);
    }
    const double g = 2.0 * s2, uG = rk.x - s_in;
    L = uG - 6.5 * g;
    R = uG + 6.5 * g;
    uV = -rk.x - s_in;
    hV = (float)(2.0 * fmax(c2, a));
    hG = (float)(0.25 * g);
  } else {
    L = u[0];
    R = u[N - 1];
  }
  // regions: left extension (-1), intervals 0..N-2, right extension (N-1)
  const int jlo = find_interval(u, N, L), jhi = find_interval(u, N, R), nj = jhi - jlo + 1;
  auto ends = [&](int j, double& x0, double& x1) {
    x0 = j < 0 ? L : fmax(L, u[j]);
    x1 = j >= N - 1 ? R : fmin(R, u[j + 1]);
  };
  auto marcher = [&](double x0, double x1) {
    Marcher m;
    m.end = ff(x1 - x0);
    m.c1 = ff(KIND == ROW_R2 ? uV - x0 : -s_in - x0);
    m.c2 = ff(KIND == ROW_R2 ? 0.0 : -s_out - x0);
    m.hV = hV;
    m.hG = hG;
    return m;
  };
  // panels per interval and their running sum
  int total = 0;
  for (int b = 0; b < nj; b += 32) {
    int cnt = 0;
    if (b + lane < nj) {
      double x0, x1;
      ends(jlo + b + lane, x0, x1);
      if (x1 > x0) cnt = count_panels<KIND>(marcher(x0, x1));
    }
    int inc = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += v;
    }
    if (b + lane < nj) off[b + lane] = total + inc - cnt;
    total += __shfl_sync(0xffffffffu, inc, 31);
  }
  if (lane == 0) off[nj] = total;
  __syncwarp();
  for (int p0 = 0; p0 < total; p0 += 32) {
    const int p = p0 + lane;
    int j = -2 - lane;                                   // no panel: a key of its own
    double Ar = 0, Ai = 0, Br = 0, Bi = 0, Cr = 0, Ci = 0, Dr = 0, Di = 0;
    if (p < total) {
      int lo = 0, hi = nj;                               // largest interval with off <= p
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= p) lo = mid; else hi = mid;
      }
      j = jlo + lo;
      double x0, x1;
      ends(j, x0, x1);
      const Marcher m = marcher(x0, x1);
      FF pos = {0.f, 0.f};
      for (int q = p - off[lo]; q > 0; --q) pos = ff_add(pos, m.width<KIND>(pos, ff_diff(m.end, pos)));
      const float rem = ff_diff(m.end, pos), w = m.width<KIND>(pos, rem);
      const double xl = x0 + ((double)pos.h + (double)pos.l);
      double xr = x1;
      if (w < rem) {
        const FF e = ff_add(pos, w);
        xr = x0 + ((double)e.h + (double)e.l);
      }
      const bool ext = j < 0 || j >= N - 1;
      // a constant continuation has its whole weight on the end node (t = 0)
      const double uj = ext ? 0.0 : u[j], hj = ext ? 0.0 : u[j + 1] - u[j], ih = ext ? 0.0 : 1.0 / hj, k6 = hj * hj / 6.0;
      const double half = 0.5 * (xr - xl), mid = 0.5 * (xr + xl);
#pragma unroll 1
      for (int g = 0; g < 8; ++g) {
        const double up = fma(half, c_gl8x[g], mid), wq = half * c_gl8w[g];
        const Cx<double> f = row_eval<KIND>(rk, up);
        const double fr = f.re * wq, fi = f.im * wq;
        const double t = (up - uj) * ih, omt = 1.0 - t;
        const double cC = k6 * (omt * omt * omt - omt), cD = k6 * (t * t * t - t);
        Ar += fr * omt; Ai += fi * omt;
        Br += fr * t; Bi += fi * t;
        Cr += fr * cC; Ci += fi * cC;
        Dr += fr * cD; Di += fi * cD;
      }
      if (j < 0) {                                       // left of the grid: node 0 is the right node of "interval" -1
        Br = Ar; Bi = Ai;
        Ar = Ai = 0.0;
      }
    }
    // sum over the lanes of one interval into its first lane
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int jn = __shfl_down_sync(0xffffffffu, j, d);
      const bool same = lane + d < 32 && jn == j;
      double v;
      v = shfl_down_d(Ar, d); if (same) Ar += v;
      v = shfl_down_d(Ai, d); if (same) Ai += v;
      v = shfl_down_d(Br, d); if (same) Br += v;
      v = shfl_down_d(Bi, d); if (same) Bi += v;
      v = shfl_down_d(Cr, d); if (same) Cr += v;
      v = shfl_down_d(Ci, d); if (same) Ci += v;
      v = shfl_down_d(Dr, d); if (same) Dr += v;
      v = shfl_down_d(Di, d); if (same) Di += v;
    }
    const int jp = __shfl_up_sync(0xffffffffu, j, 1);
    const bool lead = p < total && (lane == 0 || jp != j);
    // left nodes, then right nodes: each address once in either pass
    if (lead && j >= 0) { PyR[j] += Ar; PyI[j] += Ai; PmR[j] += Cr; PmI[j] += Ci; }
    __syncwarp();
    if (lead && j < N - 1) { PyR[j + 1] += Br; PyI[j + 1] += Bi; PmR[j + 1] += Dr; PmI[j + 1] += Di; }
    __syncwarp();
  }
}

// P_M -> T^-1 P_M on the interior nodes of the natural spline (its end values are
// constants), by one lane per (row, Re or Im): v points at its N moments, tab at the
// height's spline tables.
__device__ __forceinline__ void fold_solve(double* v, const double* tab, int N) {
  v[0] = v[N - 1] = 0.0;
  const double *idn = tab + kSpIden * N, *cg = tab + kSpCg * N, *cp = tab + kSpCp * N;
  double prev = 0.0;
#pragma unroll 4
  for (int i = 1; i < N - 1; ++i) {
    prev = v[i] * idn[i - 1] - cg[i - 1] * prev;
    v[i] = prev;
  }
  double next = 0.0;
#pragma unroll 4
  for (int i = N - 2; i >= 1; --i) {
    next = v[i] - cp[i - 1] * next;
    v[i] = next;
  }
}
// node m of the folded row: P_y + D^T (T^-1 P_M)
__device__ __forceinline__ double fold_node(const double* Py, const double* w, const double* tab, int N, int m) {
  const double* s = tab + kSp6h * N;
  const double sl = m > 0 ? s[m - 1] : 0.0, sr = m < N - 1 ? s[m] : 0.0;
  double v = Py[m] - (sl + sr) * w[m];
  if (m > 0) v += sl * w[m - 1];
  if (m < N - 1) v += sr * w[m + 1];
  return v;
}

struct TileParams {
  const double* u;        // [nz][N]
  const double* sp;       // [nz][kSpTabs][N] spline tables
  const double* a;        // [nz]
  const double* shift;    // [nz][nu][nl]
  const int* trip;        // [ntrip][3] (k, kl, kl')
  const double* theta;    // [ncls] (AA: unused)
  const double* aa_th;    // AA Theta nodes
  const double* aa_w;     // AA weights (1/2 sin(Theta) dTheta)
  int n_aa;
  int N, nu, nl, ntrip, ncls, z0;
};
struct TileRow {
  int n, c, iz;
  double s_in, s_out;
};
__device__ __forceinline__ TileRow tile_row(const TileParams& p, long long row) {
  // row -> (z - z0, c, t, n)
  TileRow r;
  r.n = (int)(row % p.N);
  long long q = row / p.N;
  const int t = (int)(q % p.ntrip);
  q /= p.ntrip;
  r.c = (int)(q % p.ncls);
  r.iz = p.z0 + (int)(q / p.ncls);
  const int k = p.trip[3 * t], kl = p.trip[3 * t + 1], klp = p.trip[3 * t + 2];
  r.s_in = p.shift[((size_t)r.iz * p.nu + k) * p.nl + kl];
  r.s_out = p.shift[((size_t)r.iz * p.nu + k) * p.nl + klp];
  return r;
}

constexpr int kRowsPerBlock = 8;     // rows (warps) of a CTA
static size_t tile_smem(int N) { return (size_t)kRowsPerBlock * (4 * N * sizeof(double) + (N + 2 + (N & 1)) * sizeof(int)); }

// One row per warp.
__global__ void __launch_bounds__(32 * kRowsPerBlock) tile_kernel(TileParams p, double* tiles, long long nrows) {
  extern __shared__ double sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, N = p.N;
  double* acc = sm + (size_t)warp * 4 * N;
  int* off = reinterpret_cast<int*>(sm + (size_t)kRowsPerBlock * 4 * N) + (size_t)warp * (N + 2 + (N & 1));
  const long long row0 = (long long)blockIdx.x * kRowsPerBlock, row = row0 + warp;
  const bool live = row < nrows;
  const TileRow r = tile_row(p, live ? row : row0);
  const double* tab = p.sp + (size_t)r.iz * kSpTabs * N;
  if (live) {
    for (int i = lane; i < 4 * N; i += 32) acc[i] = 0.0;
    __syncwarp();
    const double* u = p.u + (size_t)r.iz * N;
    row_moments<ROW_R2>(p.theta[r.c], p.a[r.iz], r.s_in, r.s_out, u[r.n], u, N, acc, off, 1.0);
  }
  __syncthreads();
  if (threadIdx.x < 2 * kRowsPerBlock && row0 + (threadIdx.x >> 1) < nrows)
    fold_solve(sm + (size_t)(threadIdx.x >> 1) * 4 * N + (2 + (threadIdx.x & 1)) * N,
               p.sp + (size_t)tile_row(p, row0 + (threadIdx.x >> 1)).iz * kSpTabs * N, N);
  __syncthreads();
  if (live) {
    double* out = tiles + (size_t)row * 2 * N;
    for (int i = lane; i < 2 * N; i += 32) {
      const int im = i >= N, m = i - im * N;
      out[i] = fold_node(acc + im * N, acc + (2 + im) * N, tab, N, m);
    }
  }
}

// One angle-averaged row per CTA: its warps take the Theta nodes in turn.
__global__ void __launch_bounds__(32 * kRowsPerBlock) tile_aa_kernel(TileParams p, double* tiles, long long nrows) {
  extern __shared__ double sm[];
  const int warp = threadIdx.x >> 5, N = p.N;
  double* acc = sm + (size_t)warp * 4 * N;
  int* off = reinterpret_cast<int*>(sm + (size_t)kRowsPerBlock * 4 * N) + (size_t)warp * (N + 2 + (N & 1));
  for (int i = threadIdx.x; i < kRowsPerBlock * 4 * N; i += blockDim.x) sm[i] = 0.0;
  __syncthreads();
  const TileRow r = tile_row(p, blockIdx.x);
  const double* u = p.u + (size_t)r.iz * N;
  for (int g = warp; g < p.n_aa; g += kRowsPerBlock)
    row_moments<ROW_R2>(p.aa_th[g], p.a[r.iz], r.s_in, r.s_out, u[r.n], u, N, acc, off, p.aa_w[g]);
  __syncthreads();
  for (int i = threadIdx.x; i < 4 * N; i += blockDim.x) {
    double v = sm[i];
#pragma unroll
    for (int w = 1; w < kRowsPerBlock; ++w) v += sm[(size_t)w * 4 * N + i];
    sm[i] = v;
  }
  __syncthreads();
  const double* tab = p.sp + (size_t)r.iz * kSpTabs * N;
  if (threadIdx.x < 2) fold_solve(sm + (2 + threadIdx.x) * N, tab, N);
  __syncthreads();
  double* out = tiles + (size_t)blockIdx.x * 2 * N;
  for (int i = threadIdx.x; i < 2 * N; i += blockDim.x) {
    const int im = i >= N, m = i - im * N;
    out[i] = fold_node(sm + im * N, sm + (2 + im) * N, tab, N, m);
  }
}

struct R3Params {
  const double* u;
  const double* sp;
  const double* a;
  const double* shift;
  int N, nu, nl;
};

// R_III incident weights r[z][q][m], q = (ku, kv, kl):
// int_{u_1}^{u_N} [W(a, u'+s_{kv kl}) + W(a, u'+s_{ku kl})^*] phi_m(u') du', one row per warp,
// to an FP32 and an FP64 table (either may be NULL).
__global__ void __launch_bounds__(32 * kRowsPerBlock) r3_kernel(R3Params p, float* out32, double* out64, int nz) {
  extern __shared__ double sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int N = p.N, nq = p.nu * p.nu * p.nl, nrows = nz * nq;
  double* acc = sm + (size_t)warp * 4 * N;
  int* off = reinterpret_cast<int*>(sm + (size_t)kRowsPerBlock * 4 * N) + (size_t)warp * (N + 2 + (N & 1));
  const int row0 = blockIdx.x * kRowsPerBlock, row = row0 + warp;
  const bool live = row < nrows;
  const int q = live ? row % nq : 0, iz = live ? row / nq : 0;
  if (live) {
    const int kl = q % p.nl, kv = (q / p.nl) % p.nu, ku = q / (p.nl * p.nu);
    for (int i = lane; i < 4 * N; i += 32) acc[i] = 0.0;
    __syncwarp();
    const double s1 = p.shift[((size_t)iz * p.nu + kv) * p.nl + kl];
    const double s2 = p.shift[((size_t)iz * p.nu + ku) * p.nl + kl];
    row_moments<ROW_R3>(0.0, p.a[iz], s1, s2, 0.0, p.u + (size_t)iz * N, N, acc, off, 1.0);
  }
  __syncthreads();
  if (threadIdx.x < 2 * kRowsPerBlock && row0 + (int)(threadIdx.x >> 1) < nrows)
    fold_solve(sm + (size_t)(threadIdx.x >> 1) * 4 * N + (2 + (threadIdx.x & 1)) * N,
               p.sp + (size_t)((row0 + (threadIdx.x >> 1)) / nq) * kSpTabs * N, N);
  __syncthreads();
  if (live)
    for (int i = lane; i < 2 * N; i += 32) {
      const int im = i >= N, m = i - im * N;
      const double v = fold_node(acc + im * N, acc + (2 + im) * N, p.sp + (size_t)iz * kSpTabs * N, N, m);
      if (out32) out32[(size_t)row * 2 * N + i] = (float)v;
      if (out64) out64[(size_t)row * 2 * N + i] = v;
    }
}

// Group-mean / deviation split of the FP64 tiles of one height:
//   tiles[c][g][.]        = mean over the triples t of group g of G_t
//   tiles[c][ngrp + t][.] = G_t - mean of its group
// so that the large dispersion parts that cancel between Zeeman components
// of one J level are summed once, in FP64, before rounding to the storage type.
// One CTA per (row n, class, height); formats of the stored element (n, k):
//   TILE_PLAIN  T, rows of ld
//   TILE_F32    FP32 in the K-step layout of tile_off
//   TILE_BF16   bf16 planes (BF16x3), TILE_BF16HI the hi plane alone (BF16x2)
constexpr int kSplitThreads = 128;

template <typename T>
__global__ void __launch_bounds__(kSplitThreads) group_split_kernel(const double* __restrict__ src, T* __restrict__ dst,
                                                                    const int* __restrict__ grp, int ncls, int ntrip,
                                                                    int ngrp, int N, int ld, int fmt) {
  const int n = blockIdx.x, c = blockIdx.y, z = blockIdx.z, nti = ngrp + ntrip;
  const size_t rowlen = (size_t)2 * N * N;             // one FP64 scratch tile: N rows of 2N
  src += ((size_t)z * ncls + c) * ntrip * rowlen + (size_t)n * 2 * N;
  const size_t tsz = (size_t)N * ld;                   // elements of one stored tile
  const size_t t0 = ((size_t)z * ncls + c) * nti;
  auto means = [&](int k, double (&mean)[2]) {
    int cnt[2] = {0, 0};
    mean[0] = mean[1] = 0.0;
    for (int t = 0; t < ntrip; ++t) {
      const int g = grp[t];
      mean[g] += src[t * rowlen + k];
      cnt[g] += 1;
    }
    for (int g = 0; g < ngrp; ++g) mean[g] = cnt[g] ? mean[g] / cnt[g] : 0.0;
  };
  auto store = [&](int ti, int k, double v) {
    if (fmt <= TILE_F32) {
      dst[(t0 + ti) * tsz + tile_off(n, k, N, ld, fmt == TILE_F32)] = (T)v;
    } else if (fmt == TILE_BF16) {
      __nv_bfloat16* t = reinterpret_cast<__nv_bfloat16*>(dst) + (t0 + ti) * tsz * 2;
      const float w = (float)v;
      const __nv_bfloat16 hi = __float2bfloat16_rn(w);
      t[tile_off_split(n, k, N, ld, false)] = hi;
      t[tile_off_split(n, k, N, ld, true)] = __float2bfloat16_rn(w - __bfloat162float(hi));
    } else {
      reinterpret_cast<__nv_bfloat16*>(dst)[(t0 + ti) * tsz + tile_off_hi(n, k, N, ld)] = __float2bfloat16_rn((float)v);
    }
  };
  for (int k = threadIdx.x; k < 2 * N; k += kSplitThreads) {
    double mean[2];
    means(k, mean);
    for (int g = 0; g < ngrp; ++g) store(g, k, mean[g]);
    for (int t = 0; t < ntrip; ++t) store(ngrp + t, k, src[t * rowlen + k] - mean[grp[t]]);
  }
}

// -------------------------------------------------------------- launchers
static int upload_consts(Ctx* c) {
  WeidemanConst wc;
  double a64[36], L64;
  weideman_coeffs(kWeidemanN64, a64, &L64);
  for (int i = 0; i < 36; ++i) wc.a64[i] = a64[i];
  wc.L64 = L64;
  PRD_CUDA_TRY(c, cudaMemcpyToSymbol(c_wc, &wc, sizeof(wc)));
  // 8-point Gauss-Legendre on [-1, 1]
  const double x8[8] = {-0.9602898564975363, -0.7966664774136267, -0.5255324099163290, -0.1834346424956498,
                        0.1834346424956498, 0.5255324099163290, 0.7966664774136267, 0.9602898564975363};
  const double w8[8] = {0.1012285362903763, 0.2223810344533745, 0.3137066458778873, 0.3626837833783620,
                        0.3626837833783620, 0.3137066458778873, 0.2223810344533745, 0.1012285362903763};
  PRD_CUDA_TRY(c, cudaMemcpyToSymbol(c_gl8x, x8, sizeof(x8)));
  PRD_CUDA_TRY(c, cudaMemcpyToSymbol(c_gl8w, w8, sizeof(w8)));
  return PRD_OK;
}

// Device inputs of the tile kernels, uploaded once and shared by their launches.
struct TileGen {
  DBuf u, a, shift, trip, theta, aa_th, aa_w, scr, grp;
  TileParams p{};
  bool aa = false;
  ~TileGen() {
    for (DBuf* b : {&u, &a, &shift, &trip, &theta, &aa_th, &aa_w, &scr, &grp}) dfree(*b);
  }
  int init(Ctx* c, const std::vector<double>& sh, int nu, int nl, const std::vector<int>& tr,
           const std::vector<double>& th, const std::vector<double>& ath, const std::vector<double>& aw) {
    int rc = upload_consts(c);
    if (rc) return rc;
    aa = !ath.empty();
    const std::vector<double> one(1, 0.0);
    const std::vector<double>&t1 = aa ? ath : one, &w1 = aa ? aw : one;
    if ((rc = upload(c, u, c->u.data(), c->u.size() * 8)) || (rc = upload(c, a, c->a.data(), c->nz * 8)) ||
        (rc = upload(c, shift, sh.data(), sh.size() * 8)) || (rc = upload(c, trip, tr.data(), tr.size() * 4)) ||
        (rc = upload(c, theta, th.data(), th.size() * 8)) || (rc = upload(c, aa_th, t1.data(), t1.size() * 8)) ||
        (rc = upload(c, aa_w, w1.data(), w1.size() * 8)))
      return rc;
    p = TileParams{(const double*)u.p, (const double*)c->sp.p, (const double*)a.p, (const double*)shift.p,
                   (const int*)trip.p, (const double*)theta.p, (const double*)aa_th.p, (const double*)aa_w.p,
                   aa ? (int)ath.size() : 0, c->nnu, nu, nl, (int)tr.size() / 3, aa ? 1 : (int)th.size(), 0};
    PRD_CUDA_TRY(c, cudaFuncSetAttribute(tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
    PRD_CUDA_TRY(c, cudaFuncSetAttribute(tile_aa_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
    PRD_CUDA_TRY(c, cudaFuncSetAttribute(r3_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
    return PRD_OK;
  }
  // FP64 rows [z][class][triple][n][2N] of the heights z0 .. z0 + n - 1
  int rows(Ctx* c, int z0, int n, double* out) {
    p.z0 = z0;
    const long long nrows = (long long)n * p.ncls * p.ntrip * p.N;
    const size_t smem = tile_smem(p.N);
    if (aa)
      tile_aa_kernel<<<(unsigned)nrows, 32 * kRowsPerBlock, smem, c->stream>>>(p, out, nrows);
    else
      tile_kernel<<<ceil_div(nrows, kRowsPerBlock), 32 * kRowsPerBlock, smem, c->stream>>>(p, out, nrows);
    PRD_CUDA_TRY(c, cudaPeekAtLastError());
    return PRD_OK;
  }
  // Stored tiles (group means, then deviations) of the heights z0 .. z0 + n - 1 from their rows in scr
  template <typename T>
  int split(Ctx* c, int n, T* dst, int ld, int fmt) {
    group_split_kernel<T><<<dim3(p.N, p.ncls, n), kSplitThreads, 0, c->stream>>>(
        (const double*)scr.p, dst, (const int*)grp.p, p.ncls, p.ntrip, c->ngrp, p.N, ld, fmt);
    PRD_CUDA_TRY(c, cudaPeekAtLastError());
    return PRD_OK;
  }
};

// Heights whose FP64 rows share one launch: as many as fit in 256 MB of scratch (small
// problems fill the chip with all heights at once), at least one.
static int heights_per_launch(const Ctx* c, int ncls, int nz) {
  const size_t per = (size_t)ncls * c->ntrip * c->nnu * 2 * c->nnu * 8;
  return (int)std::max<size_t>(1, std::min<size_t>(nz, ((size_t)256 << 20) / per));
}

static std::vector<int> triples(const Ctx* c) {
  std::vector<int> t;
  for (int i = 0; i < c->ntrip; ++i) t.insert(t.end(), {c->trip_k[i], c->trip_l[i], c->trip_lp[i]});
  return t;
}

int launch_tiles(Ctx* c) {
  const int nz = c->nz, N = c->nnu, zb = heights_per_launch(c, c->ncls, nz);
  TileGen g;
  const bool aa = c->mode == PRD_MODE_AA;
  int rc = g.init(c, c->shift, c->nu_st, c->nl_st, triples(c), c->theta, aa ? c->aa_theta : std::vector<double>(),
                  c->aa_w);
  if (rc || (rc = dalloc(c, g.scr, (size_t)zb * g.p.ncls * c->ntrip * N * 2 * N * 8)) ||
      (rc = upload(c, g.grp, c->trip_grp.data(), c->trip_grp.size() * 4)))
    return rc;
  const size_t ztile = (size_t)c->ncls * c->ntile() * N * c->ld();
  for (int z0 = 0; z0 < nz && !rc; z0 += zb) {
    const int n = std::min(zb, nz - z0);
    // W in FP64 in both modes: the per-triple tiles are differenced against
    // their group mean, so their errors must be far below the storage epsilon
    if ((rc = g.rows(c, z0, n, (double*)g.scr.p))) break;
    if (c->prec == PRD_FP64) {
      rc = g.split<double>(c, n, (double*)c->tiles.p + z0 * ztile, c->ld(), TILE_PLAIN);
    } else {
      rc = g.split<float>(c, n, (float*)((char*)c->tiles.p + z0 * ztile * c->tile_esz()), c->ld(), c->tile_fmt());
      if (!rc && c->has64)
        rc = g.split<double>(c, n, (double*)c->tiles64.p + (size_t)z0 * c->ncls * c->ntile() * N * c->ld64(), c->ld64(),
                             TILE_PLAIN);
    }
  }
  if (!rc) {
    R3Params q{(const double*)g.u.p, (const double*)c->sp.p, (const double*)g.a.p, (const double*)g.shift.p, N,
               c->nu_st, c->nl_st};
    const int nq = c->nu_st * c->nu_st * c->nl_st;
    const bool f64 = c->prec == PRD_FP64;
    r3_kernel<<<ceil_div((long long)nz * nq, kRowsPerBlock), 32 * kRowsPerBlock, tile_smem(N), c->stream>>>(
        q, f64 ? nullptr : (float*)c->r3w.p,
        f64 ? (double*)c->r3w.p : (c->has64 ? (double*)c->r3w64.p : nullptr), nz);
  }
  const cudaError_t e = cudaStreamSynchronize(c->stream);
  if (rc) return rc;
  if (e != cudaSuccess) return fail(c, PRD_E_CUDA, std::string("tile generation: ") + cudaGetErrorString(e));
  return PRD_OK;
}

// Tiles of a list of scattering angles per height (one class per entry), stored like the main
// tiles [class][group means, deviations][n][2N], for heights_per_launch heights at a time.
struct LosTiles {
  TileGen g;
};
LosTiles* los_tiles_create(Ctx* c, int ncl, int* zb, int* rc) {
  LosTiles* t = new LosTiles;
  *zb = heights_per_launch(c, ncl, c->nz);
  const bool aa = c->mode == PRD_MODE_AA;
  if ((*rc = t->g.init(c, c->shift, c->nu_st, c->nl_st, triples(c), std::vector<double>(ncl, 0.0),
                       aa ? c->aa_theta : std::vector<double>(), c->aa_w)) ||
      (*rc = dalloc(c, t->g.scr, (size_t)*zb * ncl * c->ntrip * c->nnu * 2 * c->nnu * 8)) ||
      (*rc = upload(c, t->g.grp, c->trip_grp.data(), c->trip_grp.size() * 4))) {
    delete t;
    return nullptr;
  }
  return t;
}
void los_tiles_destroy(LosTiles* t) { delete t; }
// angles of the next line of sight
int los_tiles_angles(Ctx* c, LosTiles* t, const std::vector<double>& thetas) {
  PRD_CUDA_TRY(c, cudaMemcpyAsync(t->g.theta.p, thetas.data(), thetas.size() * 8, cudaMemcpyHostToDevice, c->stream));
  PRD_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return PRD_OK;
}
// tiles of the heights z0 .. z0 + n - 1 in the context's plain or tiled element layout
int los_tiles_gen(Ctx* c, LosTiles* t, int z0, int n, void* out) {
  int rc = t->g.rows(c, z0, n, (double*)t->g.scr.p);
  if (rc) return rc;
  return c->prec == PRD_FP64 ? t->g.split<double>(c, n, (double*)out, c->ld(), TILE_PLAIN)
                             : t->g.split<float>(c, n, (float*)out, c->ld(), TILE_F32);
}

// Angle-averaged tiles and R_III incident weights of the unmagnetised J-level
// components (shifts shift_g[z][g]) for the preconditioner, returned in FP64.
int launch_pc_tiles(Ctx* c, const std::vector<double>& shift_g, std::vector<double>& aa_tiles,
                    std::vector<double>& r3g) {
  const int nz = c->nz, N = c->nnu, ng = c->ngrp;
  std::vector<double> x, w, th, tw;
  gauss_legendre(kAAThetaNodes, x, w);
  for (int h = 0; h < 2; ++h) {
    const double lo = h * 0.5 * kPi, hi = lo + 0.5 * kPi;
    for (int i = 0; i < kAAThetaNodes; ++i) {
      const double t = 0.5 * (hi - lo) * x[i] + 0.5 * (hi + lo);
      th.push_back(t);
      tw.push_back(0.5 * 0.5 * (hi - lo) * w[i] * std::sin(t));
    }
  }
  std::vector<int> trip;
  for (int g = 0; g < ng; ++g) trip.insert(trip.end(), {g, 0, 0});
  TileGen g;
  DBuf out, out3;
  const size_t n2 = (size_t)nz * ng * N * 2 * N, n3 = (size_t)nz * ng * ng * 2 * N;
  int rc = g.init(c, shift_g, ng, 1, trip, std::vector<double>(1, 0.0), th, tw);
  if (!rc && !(rc = dalloc(c, out, n2 * 8)) && !(rc = dalloc(c, out3, n3 * 8)) && !(rc = g.rows(c, 0, nz, (double*)out.p))) {
    R3Params q{(const double*)g.u.p, (const double*)c->sp.p, (const double*)g.a.p, (const double*)g.shift.p, N, ng, 1};
    r3_kernel<<<ceil_div((long long)nz * ng * ng, kRowsPerBlock), 32 * kRowsPerBlock, tile_smem(N), c->stream>>>(
        q, nullptr, (double*)out3.p, nz);
  }
  cudaError_t e = cudaStreamSynchronize(c->stream);
  if (!rc && e == cudaSuccess) {
    aa_tiles.resize(n2);
    r3g.resize(n3);
    e = cudaMemcpy(aa_tiles.data(), out.p, n2 * 8, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(r3g.data(), out3.p, n3 * 8, cudaMemcpyDeviceToHost);
  }
  dfree(out);
  dfree(out3);
  if (rc) return rc;
  if (e != cudaSuccess) return fail(c, PRD_E_CUDA, std::string("preconditioner tiles: ") + cudaGetErrorString(e));
  return PRD_OK;
}

}  // namespace prd
