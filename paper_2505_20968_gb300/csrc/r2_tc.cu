// S3+S4 R_II contraction on the 5th-generation tensor cores (tcgen05, sm_103a).
//
// For a height z, a scattering-angle class c and up to 32 output entries (an output
// direction with at most two incident directions of the class) a CTA computes
//     eps_bar(o, i)[n] += sum_t sum_{o', j} Re( Y_{t,ij}(o, o') sum_k T_t[n][k] I~_j(o', k) )
// tile by tile: the tensor cores contract the stored tile with the raw incident field,
//     W[n][(o', j)] = sum_k A[n][k] I~[(o', j)][k]      (once for the Re, once for the Im half),
// and the CUDA cores apply Y from TMEM: a thread owns the tile rows n, so the outputs
// stay in its registers over all tiles of the class, and Y is uniform over a warp.
//
// Why this order: I~ does not depend on the tile, so its operand is built (split,
// swizzled) once per CTA and stays in shared memory, and a K step is nothing but one tile
// step landing and its products.  Folding Y in first, B = Y I~, needs a new operand
// for every K step; its 16 builder warps (256 FMAs, a split and two handshakes a step)
// held the kernel at 2000 clocks a step of 16 columns and 200 rows, against the 630 in
// which HBM delivers it.
//
// Here the tiles are stored as bf16 planes (PRD_FP32_BF16X3: hi and lo, PRD_FP32_BF16X2: hi alone), the
// operands of the products as they land; r2_tc32.cu has the same contraction for FP32 tiles.
// v = hi + lo, and a product is hi hi + hi lo + lo hi (2^-15 of it left out) in FP32.
//
// The entries' contributions go to a buffer of their own and are added per output, in a fixed
// order, where the frame change back reads its rows: the sums of repeated applies agree to the
// bit (added with atomics they differed by the order the classes finished in, which far-wing
// optical depths amplify a thousandfold; R_III's moments are still FP64 atomics, whose order moves
// their last bits), and 20 us of atomics an apply (8 heights) go.
//
// Roles (640 threads): warp 0 streams the tile into a ring of K step pairs with two bulk
// asynchronous copies a step (the planes are stored pre-swizzled, step by step) and owns the
// TMEM allocation; warp 1 issues tcgen05.mma; warps 4-19 stage I~ and Y and apply Y.  TMEM:
// [half][row block of 128][128 columns (o', j)], so the products of one half run
// while Y is applied to the other.  Every mbarrier wait is bounded; on expiry the CTA
// records an error flag, drains what it issued and returns.
//
// What shaped it, in turn (contraction of Mg II 8 heights x 64 directions x 200 frequencies, both
// planes in FP16): the products' order above 2795 -> 1515 us; products issued by an elected lane of a
// uniform warp 1200; K steps in pairs and 16 Y warps of 8 entries each instead of 8 of 16 1100; bare
// poll loops in the products' warp 967.  HBM alone takes 722, the copies without products
// 804, the products without copies or Y about 800; the rest is their overlap, the operand's build
// (7 us a CTA) and a last wave.
// Measured (operator apply, BF16x3, Mg II 4 x 64 x 163; before: the operand formed per K step by builder
// warps): 1316 -> 580 us.
#include <algorithm>
#include <cstdio>
#include <vector>
#include "device_common.cuh"
#include "r2_tc.cuh"

namespace prd {

namespace tc {

// warps 0, 1: copies, products (2, 3 fill their warpgroup); then the Y warps
constexpr int kThreads = 128 + kEpi;
// registers a thread: launched with 96, the first warpgroup gives up what the Y warps'
// accumulators need (128 * 32 + 512 * 112 = 640 * 96)
constexpr int kRegsFew = 32, kRegsMany = 112;
__host__ __device__ constexpr int plane_bytes(int N) { return (N <= 64 ? 128 : rows16(N)) * 32; }
__host__ __device__ constexpr int step_bytes(int N, bool hi) { return plane_bytes(N) * (hi ? 1 : 2); }
// Shared memory of one CTA: the tile ring, the resident I~ operand (two planes), two Y
// buffers, the auxiliary tables, 1 KB to align the base.  The second row block of a
// tile plane reads past its rows (into what follows: rows nobody uses), so the
// operand stands behind the ring.
__host__ __device__ constexpr int smem_bytes(int N, int st, bool hi) {
  return st * kSteps * step_bytes(N, hi) + rows16(N) / kKC * 2 * kPlane + 2 * tiles_per_pass(N) * kYBytes + kAuxBytes + 1024;
}

// NB: row blocks of 128 (N <= 128: 1, else 2).  G: tiles per pass (1, or 2 or 4 where N is
// small).  HI: the tiles hold the hi plane alone (BF16x2: products hi hi + hi lo(I~)).
template <int NB, int G, bool HI>
__global__ void __launch_bounds__(kThreads, 1) r2_tc_kernel(Params p) {
  extern __shared__ __align__(1024) unsigned char smraw[];
  // 1024-byte aligned base, derived by offset so that the compiler keeps the
  // shared address space on every pointer below (plain LDS/STS, no generic access)
  unsigned char* sm = smraw + ((1024u - (smem_u32(smraw) & 1023u)) & 1023u);
  const int N = p.N, nst = p.nst;
  const int SA = step_bytes(N, HI);              // one K step of the tile
  const int PA = plane_bytes(N);                 // one plane of it (of the pass's G tiles)
  const int KCH = p.ld / kKC, KH = KCH >> 1;     // K steps per tile and per half
  unsigned char* Iop = sm + nst * kSteps * SA;   // [K step][hi | lo][128 rows][32 bytes]
  float* Ys = (float*)(Iop + KH * 2 * kPlane);   // [buffer][tile of the pass][entry][pair][kYS]
  int* rec = (int*)((unsigned char*)Ys + 2 * G * kYBytes);
  uint64_t* full = (uint64_t*)(((uintptr_t)(rec + kRec) + 7) & ~(uintptr_t)7);
  uint64_t* empty = full + kStagesMax;
  uint64_t* accfull = empty + kStagesMax;        // [half] products of the half complete
  uint64_t* accfree = accfull + 2;               // [half] Y applied
  uint64_t* iready = accfree + 2;
  uint64_t* done = iready + 1;
  uint32_t* tmem_slot = (uint32_t*)(done + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  // work item (z, record) and part of its tiles
  const int past = max((int)blockIdx.x - p.split0, 0);
  const int item = min((int)blockIdx.x, p.split0) + past / p.zs;
  const int nparts = item >= p.split0 ? p.zs : 1, part = item >= p.split0 ? past % p.zs : 0;
  const int zl = item / p.nwork, iz = p.z0 + zl;
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;   // uniform
  const int et = threadIdx.x - 128;              // index among the Y threads
  constexpr uint32_t tm_cols = NB * 256u;
  const int t0 = p.ntile * part / nparts, t1 = p.ntile * (part + 1) / nparts;

  for (int i = threadIdx.x; i < kRec; i += kThreads) rec[i] = p.work[(size_t)(item - zl * p.nwork) * kRec + i];
  if (threadIdx.x == 0) {
    for (int s = 0; s < nst; ++s) {
      mbar_init(&full[s], 1);        // armed by the producer with the bytes of the tile copy
      mbar_init(&empty[s], 1);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(&accfull[h], 1);
      mbar_init(&accfree[h], kEpiWarps);   // one arrival a warp
    }
    mbar_init(iready, kEpiWarps);
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(tm_cols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  const int c = rec[0], E = rec[1], ns = rec[2];
  const int* vinfo = rec + 4;
  const int* vpair = rec + 36;
  const int* sdir = rec + 100;
  const int passes = (t1 - t0 + G - 1) / G, iters = passes * KH;   // stages of kSteps = 2 steps
  int filled = 0;                                // stages warp 0 has filled

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsFew));
    if (warp == 0) {
      // ---------------- producer: the warp waits for a free stage and arms its barrier with the
      // bytes of the copies, then each lane issues its one (plane, step, tile of the pass), up
      // to nst stages ahead of the products
      const uint64_t pol_t = policy_evict_first();
      const uint32_t pbytes = (uint32_t)N * 32;     // one plane of a step
      const size_t sbytes = (size_t)pbytes * (HI ? 1 : 2);
      const int pl = lane & 1, c2 = (lane >> 1) & 1, g = lane >> 2;
      const unsigned char* src = p.tiles + (((size_t)iz * p.ncls + c) * p.ntile + t0 + g) * KCH * sbytes + c2 * sbytes + pl * pbytes;
      unsigned char* dst = sm + c2 * SA + pl * PA + g * (4096 / G);
      int j = 0, left = t1 - t0;                     // stage of the pass; tiles left
      filled = ring_produce(
          iters, nst, [&](int s, uint32_t par) { return mbar_wait_warp(&empty[s], par, abort_flag, p.spin); },
          [&](int s) {
            // rows n >= N of the stage (and the places of a last pass's missing tiles) keep stale
            // data: they only reach accumulator rows that nobody reads
            const int g1 = min(G, left);
            if (lane == 0) mbar_expect_tx(&full[s], (uint32_t)(kSteps * sbytes) * g1);
            __syncwarp();
            if (g < g1 && (!HI || pl == 0)) bulk_load(dst + s * kSteps * SA, src, pbytes, &full[s], pol_t);
            src += kSteps * sbytes;
            if (++j == KH) {
              j = 0;
              left -= G;
              src += (size_t)(G - 1) * KCH * sbytes;
            }
          });
      __syncwarp();
    } else if (warp == 1) {
      // ---------------- products: the warp runs uniformly (waits by all lanes, descriptors in
      // uniform registers) and an elected lane issues; a loop of one lane issued a product
      // every 160 clocks, three times what it takes to execute
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(rows16(4 * ns) >> 3) << 17) | ((128u >> 4) << 24);
      const uint64_t a0 = sdesc32(sm), b0 = sdesc32(Iop);    // the address field counts 16 bytes
      // A stage's waits are kept to a bare poll loop, without a vote on their outcome or a look
      // at the abort flag (either cost 100 to 200 clocks a stage in this warp of few
      // registers).  A lane whose wait gives up raises the flag and polls no more (lim = 0).
      // The products, their commits and with them a stage's return to the producer are the
      // elected lane's, which leaves them out from then on: no stage goes back whose copies
      // may be in flight.  The flag ends the loop at the next pass.
      int lim = p.spin;
      auto wait = [&](uint64_t* b, uint32_t par) {
        bool r = false;
        for (int i = 0; i < lim && !r; ++i) r = mbar_try(b, par);
        if (!r) {
          *abort_flag = 1;
          lim = 0;
        }
        __syncwarp();
      };
      {
        // I~ takes microseconds to build: plain polls, so that a short poll limit expires here
        bool r = false;
        for (int i = 0; i < lim && !r; ++i) r = mbar_test(iready, 0);
        if (!r) {
          *abort_flag = 1;
          lim = 0;
        }
        __syncwarp();
      }
      RingPos pos;
      bool issued = false;
      for (int t = 0; t < passes; ++t) {
        if (__any_sync(0xffffffffu, *abort_flag != 0)) break;
        int h = 0, kc = 0;                           // half and K step within it
        for (int j = 0; j < KH; ++j) {
          ring_take(
              pos, nst, lim,
              [&](int s, uint32_t par, int& limit) {
                wait(&full[s], par);
                // a half's accumulators are free once Y has been applied to the pass before
                if (t > 0 && kc == 0) wait(&accfree[h], (t - 1) & 1);
                if (t > 0 && kc + 1 == KH && h == 0) wait(&accfree[1], (t - 1) & 1);
                return limit > 0;
              },
              [&](int s, bool landed) {
                // orders the products behind the Y warps' reads of the accumulators
                if (kc == 0 || kc + 1 == KH) asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t as = a0 + (uint64_t)((uint32_t)(s * kSteps * SA) >> 4);
                if (elect_one() && landed) {
                  int h2 = h, k2 = kc;
#pragma unroll
                  for (int u = 0; u < kSteps; ++u) {
                    const uint64_t ah = as + (uint64_t)((uint32_t)(u * SA) >> 4), al = ah + (uint64_t)((uint32_t)PA >> 4);
                    const uint64_t bh = b0 + (uint64_t)((uint32_t)(k2 * 2 * kPlane) >> 4), bl = bh + (kPlane >> 4);
#pragma unroll
                    for (int b = 0; b < NB; ++b) {
                      const uint32_t d = tmem + (uint32_t)(h2 * NB + b) * 128u;
                      mma_bf16(d, ah + b * 256, bh, idesc, k2 > 0 ? 1u : 0u);
                      mma_bf16(d, ah + b * 256, bl, idesc, 1u);
                      if constexpr (!HI) mma_bf16(d, al + b * 256, bh, idesc, 1u);
                    }
                    if (++k2 == KH) {
                      mma_commit(&accfull[h2]);
                      k2 = 0;
                      ++h2;
                    }
                  }
                  mma_commit(&empty[s]);
                }
              });
          kc += kSteps;
          if (kc >= KH) { kc -= KH; ++h; }
          issued = true;
        }
      }
      // every product issued completes before TMEM is released
      __syncwarp();
      if (issued) {
        if (elect_one()) mma_commit(done);
        for (int i = 0; i < kSpin && !mbar_try(done, 0); ++i) {
        }
      }
    }
  } else {
    // ---------------- Y warps
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsMany));
    const int q = warp & 3;                        // TMEM lane quarter of this warp
    const int og = (warp - 4) >> 2;                // entries of this warp: 4 i + og
    // Y of a tile: thread (pair slot, i) moves the 8 coefficients of output Stokes i
    // (tiles of the pass are shared out between the two halves of the threads)
    constexpr int GY = (G + 1) / 2;
    const int yp = (et & 255) >> 2, yi = et & 3;   // pair slot 2 entry + pair, Stokes i
    const int yg = et >> 8;                        // tiles yg, yg + 2 of the pass
    const int ypair = (yp >> 1) < E && yg < G ? vpair[yp] : -1;
    const float4* ysrc = reinterpret_cast<const float4*>(p.Y + (((size_t)iz * p.npairs + max(ypair, 0)) * p.ntile + t0) * 32 + yi * 8);
    float4 ya[GY], yb[GY];
    auto load_y = [&](int t) {                     // Y of pass t's tiles
#pragma unroll
      for (int k = 0; k < GY; ++k) {
        const int ti = t * G + yg + 2 * k;
        if (ypair >= 0 && ti < t1 - t0) { ya[k] = ysrc[ti * 8]; yb[k] = ysrc[ti * 8 + 1]; }
      }
    };
#pragma unroll
    for (int k = 0; k < GY; ++k) ya[k] = yb[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    load_y(0);
    build_operand<2>(Iop, p.Ic, sdir, warp - 4, ns, iz, p.nO, N, KH);
    __syncwarp();
    if (lane == 0) mbar_arrive(iready);
    bool ok = true;

    // tile of the pass and row of this lane
    const int gt = q * G / 4, n0 = (q % (4 / G)) * 32 + lane;
    const bool live0 = (q % (4 / G)) * 32 < N, live1 = NB > 1 && 128 + q * 32 < N;
    float acc[kEV][NB][4];
#pragma unroll
    for (int i = 0; i < kEV; ++i)
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[i][b][k] = 0.f;
    const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
    for (int t = 0; t < passes; ++t) {
      float* Yb = Ys + (t & 1) * (G * kYBytes / 4);
#pragma unroll
      for (int k = 0; k < GY; ++k) {
        const int g = yg + 2 * k;
        if (g >= G) break;
        float* d = Yb + g * (kYBytes / 4) + yp * kYS + yi;             // [half][j][i]
        d[0] = ya[k].x; d[4] = ya[k].z; d[8] = yb[k].x; d[12] = yb[k].z;
        d[16] = -ya[k].y; d[20] = -ya[k].w; d[24] = -yb[k].y; d[28] = -yb[k].w;
      }
      ok = epi_all(ok);
      if (!ok) break;
      if (t + 1 < passes) load_y(t + 1);
      for (int h = 0; h < 2 && ok; ++h) {
        ok = mbar_wait_warp(&accfull[h], t & 1, abort_flag, p.spin);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (live0 && (G == 1 || t * G + gt < t1 - t0)) {
          const uint32_t ta = tq + (uint32_t)(h * NB) * 128u;
          const float* Yh = Yb + gt * (kYBytes / 4) + h * 16;
#pragma unroll
          for (int i = 0; i < kEV; ++i) {
            const int v = 4 * i + og;
            if (v >= E) break;
            const int info = vinfo[v], np = info >> 16;
            const uint32_t ca = ta + (uint32_t)(info & 255) * 4u, cb = ta + (uint32_t)((info >> 8) & 255) * 4u;
            float w[2 * NB][4];                    // [pair, row block]
#pragma unroll
            for (int b = 0; b < NB; ++b) tmem_ld4(w[b], ca + b * 128u);
            if (np > 1) {
#pragma unroll
              for (int b = 0; b < NB; ++b) tmem_ld4(w[NB + b], cb + b * 128u);
            }
            tmem_wait<2 * NB>(w);
#pragma unroll
            for (int pr = 0; pr < 2; ++pr) {
              if (pr < np) {
                const float4* y4 = reinterpret_cast<const float4*>(Yh + (2 * v + pr) * kYS);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  const float4 y = y4[j];
#pragma unroll
                  for (int b = 0; b < NB; ++b) {
                    const float x = w[pr * NB + b][j];
                    acc[i][b][0] += y.x * x;
                    acc[i][b][1] += y.y * x;
                    acc[i][b][2] += y.z * x;
                    acc[i][b][3] += y.w * x;
                  }
                }
              }
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&accfree[h]);
      }
    }
    if (ok) {
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const int n = b * 128 + n0;
        if (n >= N || (b > 0 && !live1)) continue;
#pragma unroll
        for (int i = 0; i < kEV; ++i) {
          const int v = 4 * i + og;
          if (v < E) {
            float4* dst = part == 0 ? p.ent + add_off(gt, zl * p.nent + rec[3] + v, p.nz * p.nent, N, 0, n)
                                    : p.tail + (part - 1) * (size_t)G * p.nsplit * kMaxE * N +
                                          add_off(gt, (item - p.split0) * kMaxE + v, p.nsplit * kMaxE, N, 0, n);
            *dst = make_float4(acc[i][b][0], acc[i][b][1], acc[i][b][2], acc[i][b][3]);
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) atomicExch(p.err, 1);
  if (warp == 0) {
    // a wait gave up: copies that nobody has waited for may be in flight (with every wait met
    // all stages have been used)
    if (*abort_flag)
      ring_drain(filled, nst, [&](int s, uint32_t par) {
        for (int i = 0; i < kSpin && !mbar_try(&full[s], par); ++i) {
        }
      });
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tm_cols));
  }
}

}  // namespace tc

// The kernel of a context's tiles (bf16 planes) for N rows.
using R2Kernel = void (*)(tc::Params);
template <int NB, int G>
static R2Kernel r2_tc_pick(bool hi) {
  return hi ? tc::r2_tc_kernel<NB, G, true> : tc::r2_tc_kernel<NB, G, false>;
}
static R2Kernel r2_tc_pick(const Ctx* c) {
  switch (tc::tiles_per_pass(c->nnu)) {
    case 4: return r2_tc_pick<1, 4>(c->hi_only);
    case 2: return r2_tc_pick<1, 2>(c->hi_only);
    default: return c->nnu <= 128 ? r2_tc_pick<1, 1>(c->hi_only) : r2_tc_pick<2, 1>(c->hi_only);
  }
}

// Tile stages for N rows: the most (<= kStagesMax) whose shared memory fits.
static int r2_tc_stages(const Ctx* c) {
  if (!c->split_tiles) return r2_f32_stages(c->nnu);
  for (int st = tc::kStagesMax; st >= 2; --st)
    if (tc::smem_bytes(c->nnu, st, c->hi_only) <= kMaxSmem) return st;
  return 0;
}
// Rows from which a pass takes several tiles, and how many
static void r2_tc_packed(const Ctx* c, int* n0, int* G) {
  *n0 = !c->split_tiles && c->nnu > 128 ? 128 : 0;
  *G = tc::tiles_per_pass(c->nnu - *n0);
}

// Every item takes about as long, one CTA per SM: whole waves of a launch's items run as they are, and
// the tiles of the rest, the n items from split0 on, are split between zs CTAs each, on the SMs of a
// last wave (at least 4 tiles, or two passes, a CTA).  On 152 SMs, contraction of Mg II 8 heights (768
// items) 1000 -> 954 us, H I 4 heights x 96 directions 812 -> 779, angle-averaged 512 items 309 -> 272
// (three FP16 products).
struct R2Split {
  int split0, n, zs;
};
static R2Split r2_tc_split(const Ctx* c, int nz) {
  const int items = c->tc_nwork * nz, rest = items % c->nsm;
  const int zs = rest ? std::min(c->ntile() / std::max(4, 2 * tc::tiles_per_pass(c->nnu)), c->nsm / rest) : 1;
  return {items - rest, rest, std::max(1, zs)};
}
constexpr size_t kEntBytes = (size_t)1 << 30;

// Work records of the contraction: every class's outputs cut into entries of at most two
// incident directions each (an output with more, as all are in angle-averaged mode,
// takes several entries, which add up in eps_bar) and the entries packed into records of
// at most 32 entries and 32 incident directions.  Where entries are many they are
// taken by blocks of 32 incident directions, so that a record's entries share them.
// entry_out: the output direction of every entry.
static void r2_tc_records(const Ctx* c, std::vector<int>& out, std::vector<int>& entry_out) {
  using namespace tc;
  struct Entry { int o, p[2], n; };
  out.clear();
  for (int k = 0; k < c->ncls; ++k) {
    std::vector<Entry> es;
    bool many = false;
    for (int e = c->cout_ptr[k]; e < c->cout_ptr[k + 1]; ++e) {
      many = many || c->pair_ptr[e + 1] - c->pair_ptr[e] > 2;
      for (int p = c->pair_ptr[e]; p < c->pair_ptr[e + 1]; p += 2) {
        Entry x{c->cout_dir[e], {p, -1}, 1};
        if (p + 1 < c->pair_ptr[e + 1]) { x.p[1] = p + 1; x.n = 2; }
        es.push_back(x);
      }
    }
    if (many)
      std::stable_sort(es.begin(), es.end(), [&](const Entry& a, const Entry& b) {
        return c->pair_in[a.p[0]] / kMaxIn < c->pair_in[b.p[0]] / kMaxIn;
      });
    std::vector<int> slots;
    int rec = -1;
    for (const Entry& x : es) {
      std::vector<int> add;
      for (int i = 0; i < x.n; ++i) {
        const int d = c->pair_in[x.p[i]];
        if (std::find(slots.begin(), slots.end(), d) == slots.end() && std::find(add.begin(), add.end(), d) == add.end())
          add.push_back(d);
      }
      if (rec < 0 || out[rec + 1] == kMaxE || (int)(slots.size() + add.size()) > kMaxIn) {
        rec = (int)out.size();
        out.resize(out.size() + kRec, 0);
        out[rec] = k;
        out[rec + 3] = (int)entry_out.size();
        slots.clear();
        add.clear();
        for (int i = 0; i < x.n; ++i) {
          const int d = c->pair_in[x.p[i]];
          if (std::find(add.begin(), add.end(), d) == add.end()) add.push_back(d);
        }
      }
      for (int d : add) {
        out[rec + 100 + (int)slots.size()] = d;
        slots.push_back(d);
      }
      out[rec + 2] = (int)slots.size();
      const int v = out[rec + 1]++;
      int sl[2] = {0, 0};
      for (int i = 0; i < x.n; ++i)
        sl[i] = (int)(std::find(slots.begin(), slots.end(), c->pair_in[x.p[i]]) - slots.begin());
      entry_out.push_back(x.o);
      out[rec + 4 + v] = sl[0] | (sl[1] << 8) | (x.n << 16);
      out[rec + 36 + 2 * v] = x.p[0];
      out[rec + 36 + 2 * v + 1] = x.n > 1 ? x.p[1] : -1;
    }
  }
}

// Work list and error flag of the tensor-core contraction.
int r2_tc_prepare(Ctx* c) {
  // the device error flag of the bounded waits (contraction and staged sweep), all precisions
  if (!c->tc_err.p) {
    int rc = dalloc(c, c->tc_err, sizeof(int));
    if (rc) return rc;
    PRD_CUDA_TRY(c, cudaMemset(c->tc_err.p, 0, sizeof(int)));
  }
  if (c->prec != PRD_FP32 || c->lambda_only) return PRD_OK;   // no contraction
  if (!c->tiled() || c->nnu > 224 || r2_tc_stages(c) < 2)
    return fail(c, PRD_E_ARG, "tensor-core contraction needs FP32 tiles and N small enough for two tile stages "
                              "beside the resident I~ (N <= 224)");
  std::vector<int> work, eo;
  r2_tc_records(c, work, eo);
  c->tc_nwork = (int)work.size() / tc::kRec;
  c->tc_nent = (int)eo.size();
  // entries of each output direction, in order: [nO + 1] starts, then (entry, record * kMaxE + its place)
  std::vector<int> lists(c->nO + 1, 0), place(eo.size());
  for (int r = 0; r < c->tc_nwork; ++r)
    for (int v = 0; v < work[(size_t)r * tc::kRec + 1]; ++v) place[work[(size_t)r * tc::kRec + 3] + v] = r * tc::kMaxE + v;
  for (int o : eo) ++lists[o + 1];
  for (int o = 0; o < c->nO; ++o) lists[o + 1] += lists[o];
  std::vector<int> at(lists.begin(), lists.end() - 1);
  const int l0 = c->nO + 1 + (c->nO + 1) % 2;          // pairs start 8-byte aligned
  lists.resize(l0 + 2 * eo.size());
  for (int e = 0; e < c->tc_nent; ++e) {
    int* l = &lists[l0 + 2 * at[eo[e]]++];
    l[0] = e;
    l[1] = place[e];
  }
  // The contributions wait in tc_ent for the frame change back, at most kEntBytes of them or one height's
  // (with all directions as partners an entry count grows as their square), so that they stay a
  // small part of a context; more heights take several launches (of the contraction and the frame
  // change back, whose last waves then cost: at 256 MiB, 32 of 70 heights of the full Mg II problem a
  // launch, the frame change took 0.69 ms instead of 0.47).
  int n0, G;
  r2_tc_packed(c, &n0, &G);
  const size_t rows = c->nnu + (size_t)(G - 1) * (c->nnu - n0);   // stored per entry (RowAdds)
  const size_t per = c->tc_nent * rows * sizeof(float4);
  c->tc_zc = (int)std::max<size_t>(1, std::min<size_t>(c->nz, kEntBytes / per));
  size_t tail = 16;
  for (int n : {c->tc_zc, c->nz % c->tc_zc}) {
    const R2Split s = r2_tc_split(c, n);
    tail = std::max(tail, (size_t)(s.zs - 1) * s.n * tc::kMaxE * rows * sizeof(float4));
  }
  int rc;
  if ((rc = upload(c, c->tc_work, work.data(), work.size() * sizeof(int))) ||
      (rc = upload(c, c->tc_lists, lists.data(), lists.size() * sizeof(int))) ||
      (rc = dalloc(c, c->tc_ent, c->tc_zc * per)) ||
      (rc = dalloc(c, c->tc_tail, tail)))
    return rc;
  if (c->split_tiles) PRD_CUDA_TRY(c, cudaFuncSetAttribute(r2_tc_pick(c), cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
  else if ((rc = r2_f32_prepare(c))) return rc;
  PRD_CUDA_TRY(c, cudaMemset(c->tc_err.p, 0, sizeof(int)));
  c->tc_ready = true;
  return PRD_OK;
}

RowAdds r2_tc_adds(const Ctx* c, int n) {
  const int* lists = (const int*)c->tc_lists.p;
  const R2Split s = r2_tc_split(c, n);
  RowAdds a{(const float4*)c->tc_ent.p, (const float4*)c->tc_tail.p, lists, reinterpret_cast<const int2*>(lists + c->nO + 1 + (c->nO + 1) % 2),
            c->tc_nent, 1, 0, s.zs, s.split0, c->tc_nwork, s.n};
  r2_tc_packed(c, &a.n0, &a.G);
  return a;
}

int r2_tc_launch(Ctx* c, const float* Ic, int z0, int n) {
  // the deepest ring that fits, or the caller's (autotuned) depth if smaller
  const int nmax = r2_tc_stages(c);
  const int nst = c->tc_stages >= 2 ? std::min(c->tc_stages, nmax) : nmax;
  const R2Split s = r2_tc_split(c, n);
  const int grid = s.split0 + s.n * s.zs;
  tc::Params p{(const unsigned char*)c->tiles.p, (const float*)c->Y.p, Ic, (const int*)c->tc_work.p, (float4*)c->tc_ent.p,
               (float4*)c->tc_tail.p, (int*)c->tc_err.p, c->ncls, c->ntile(), c->nO, c->nnu, c->npairs, c->ld(), c->tc_nent,
               n, c->tc_nwork, z0, s.split0, s.n, s.zs, nst, 0,
               c->tc_spin > 0 ? (int)std::min<long long>(c->tc_spin, INT32_MAX) : tc::kSpin};
  if (c->split_tiles) r2_tc_pick(c)<<<grid, tc::kThreads, tc::smem_bytes(c->nnu, nst, c->hi_only), c->stream>>>(p);
  else r2_f32_launch(c, p, grid);
  PRD_CUDA_TRY(c, cudaPeekAtLastError());
  return PRD_OK;
}

int r2_tc_check_error(Ctx* c) {
  int h = 0;
  PRD_CUDA_TRY(c, cudaMemcpy(&h, c->tc_err.p, sizeof(int), cudaMemcpyDeviceToHost));
  if (h) {
    cudaMemset(c->tc_err.p, 0, sizeof(int));
    return fail(c, PRD_E_TIMEOUT, "tensor-core contraction: a bounded wait expired");
  }
  return PRD_OK;
}

}  // namespace prd
