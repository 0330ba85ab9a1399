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
// Operands are pairs of 16-bit planes, v = hi + lo, and a product is hi hi + hi lo + lo hi in
// FP32: FP16 planes scaled by powers of two (one per tile row, one per incident direction
// and Stokes parameter, from their largest element; undone exactly in FP32), which hold an
// FP32 value to 2^-24 of itself down to 2^-17 of the row's largest element and to 2^-40
// of that below, leaving <= 3 * 2^-24 a product.  TF32 products left 3 * 2^-22 at half the
// rate.  BF16 contexts use bf16 planes, unscaled.
//
// Roles (320 threads): warp 0 streams the tile into a ring of K steps with two bulk
// asynchronous copies each (the planes are stored pre-swizzled, step by step) and owns the
// TMEM allocation; warp 1 issues tcgen05.mma; warps 2-9 stage I~ and Y and apply Y.  TMEM:
// [half][row block of 128][128 columns (o', j)], so the products of one half run
// while Y is applied to the other.  Every mbarrier wait is bounded; on expiry the CTA
// records an error flag, drains what it issued and returns.
//
// Measured (operator apply, FP32): Mg II 8 heights x 64 directions x 200 frequencies
// 2952 -> 1693 us, H I 4 x 96 x 150 2680 -> 1423 us, H I angle-averaged 8 x 64 x 91
// 12480 -> 690 us, Mg II 10 x 16 x 27 201 -> 161 us; BF16x3, Mg II 4 x 64 x 163, 1313 -> 918 us.
#include <algorithm>
#include <cstdio>
#include <vector>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include "prd_internal.h"
#include "device_common.cuh"

namespace prd {

namespace tc {

constexpr int kStagesMax = 8;                 // tile ring depth: 2..8, the most that fit beside the rest
constexpr int kKC = 16;                       // columns of a K step (32-byte rows per plane)
constexpr int kMaxE = 32;                     // output entries per CTA
constexpr int kMaxIn = 32;                    // incident directions per CTA (128 operand rows)
constexpr int kPlane = 4 * kMaxIn * 32;       // bytes of one K step of one I~ plane
constexpr int kEpiWarps = 8;
constexpr int kEpi = 32 * kEpiWarps;          // threads of the Y warps
constexpr int kThreads = 64 + kEpi;
constexpr int kYS = 36;                       // floats of a staged pair: Re [j][i], -Im [j][i], 4 of padding (banks)
constexpr int kYBytes = 2 * kMaxE * kYS * 4;  // one tile's Y (two buffers)
constexpr int kRec = 4 + 32 + 32 + 64 + 32;   // ints of a work record
constexpr int kAuxBytes = 2048;               // work record, column scales, barriers, TMEM slot, abort flag
__host__ __device__ constexpr int rows16(int N) { return (N + 15) / 16 * 16; }
__host__ __device__ constexpr int stage_bytes(int N, bool hi) { return rows16(N) * (hi ? 32 : 64); }
// Shared memory of one CTA: the tile ring, the resident I~ operand (two planes), two Y
// buffers, the auxiliary tables, 1 KB to align the base.  The second row block of a
// tile plane reads past its rows (into what follows: rows nobody uses), so the
// operand stands behind the ring.
__host__ __device__ constexpr int smem_bytes(int N, int st, bool hi) {
  return st * stage_bytes(N, hi) + rows16(N) / kKC * 2 * kPlane + 2 * kYBytes + kAuxBytes + 1024;
}
constexpr long long kSpin = 1ll << 24;        // bounded waits (default limit of the pipeline waits; drains)

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred P;\n\tmbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\tselp.b32 %0, 1, 0, P;\n\t}\n"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded pipeline wait of at most `limit` polls; returns false (and raises the
// CTA abort flag) on expiry or when another role has aborted
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag, long long limit) {
  for (long long i = 0; i < limit; ++i) {
    if (mbar_try(b, parity)) return true;
    if (*abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}

// bulk asynchronous copy global -> shared (16-byte aligned ends, size a multiple
// of 16) with an L2 eviction-priority policy
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
      ::"r"(smem_u32(dst)), "l"((uint64_t)src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
      : "memory");
}
// the tiles are streamed once per apply: first out of L2, so that I~ and Y stay resident
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
// 16-bit operands (kind::f16, both of one type), FP32 accumulation, K = 16 per instruction
__device__ __forceinline__ void mma_f16(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
      ::"r"(dtmem), "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
// shared-memory matrix descriptor: K-major, 32-byte swizzle (rows of 16 values),
// 8-row groups 256 B apart
__device__ __forceinline__ uint64_t sdesc32(const void* p) {
  const uint64_t addr = (smem_u32(p) & 0x3FFFF) >> 4;
  const uint64_t lbo = 1;            // unused for swizzled K-major
  const uint64_t sbo = 256 >> 4;
  return addr | (lbo << 16) | (sbo << 32) | (1ull << 46) | (6ull << 61);
}
// byte offset of the 4 values of k-group g (k = 4g .. 4g + 3, g < 4) of `row` in a
// K-major 32-byte-swizzled operand: the 16-byte half (g >> 1) is exchanged with
// the other in rows whose bit 2 is set
__device__ __forceinline__ uint32_t swz32(int row, int g) {
  return (uint32_t)row * 32u + (uint32_t)(((g >> 1) ^ ((row >> 2) & 1)) * 16) + (uint32_t)(g & 1) * 8u;
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}


// Four values split into planes of the operand type: hi = rn(v), lo = rn(v - hi).
template <bool BF>
__device__ __forceinline__ void split4(float4 v, uint2& hi, uint2& lo) {
  if constexpr (BF) {
    const __nv_bfloat162 h0 = __floats2bfloat162_rn(v.x, v.y), h1 = __floats2bfloat162_rn(v.z, v.w);
    const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
    const __nv_bfloat162 l0 = __floats2bfloat162_rn(v.x - f0.x, v.y - f0.y);
    const __nv_bfloat162 l1 = __floats2bfloat162_rn(v.z - f1.x, v.w - f1.y);
    hi = {*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1)};
    lo = {*reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1)};
  } else {
    const __half2 h0 = __floats2half2_rn(v.x, v.y), h1 = __floats2half2_rn(v.z, v.w);
    const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
    const __half2 l0 = __floats2half2_rn(v.x - f0.x, v.y - f0.y), l1 = __floats2half2_rn(v.z - f1.x, v.w - f1.y);
    hi = {*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1)};
    lo = {*reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1)};
  }
}

struct Params {
  const unsigned char* tiles;   // [z][class][tile] pre-swizzled K steps of [plane][N][16]
  const float* tsc;     // [z][class][N] power-of-two scale to undo per tile row (NULL: none)
  const float* Y;       // [z][pair][ntile][16][2]
  const float* Ic;      // [z][o][N][4]
  const int* work;      // [item][kRec]: class, entries, incident directions, -, output direction of each entry,
                        // its slots (a | b << 8 | pairs << 16), its pairs' indices, direction of each slot
  float* eb;            // [z][o][N][4]
  int* err;
  int ncls, ntile, nO, N, npairs, ld;
  int nst;              // tile stages
  long long spin;       // poll limit of the pipeline waits (the drains keep kSpin)
};

// barrier over the Y warps only (named barrier 1), returning whether v holds on all of
// them (keeps their loop exits uniform, so none waits at the barrier for one that left)
__device__ __forceinline__ bool epi_all(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbar.red.and.pred q, 1, %2, p;\n\tselp.b32 %0, 1, 0, q;\n\t}\n"
      : "=r"(r)
      : "r"((uint32_t)v), "n"(kEpi)
      : "memory");
  return r != 0;
}

// four TMEM columns of the warp's 32 lanes; the values are there after tmem_wait
__device__ __forceinline__ void tmem_ld4(float (&w)[4], uint32_t addr) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=f"(w[0]), "=f"(w[1]), "=f"(w[2]), "=f"(w[3])
               : "r"(addr));
}
template <int K>
__device__ __forceinline__ void tmem_wait(float (&w)[K][4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
  // the values pass through here, so that no use of them moves above the wait
#pragma unroll
  for (int k = 0; k < K; ++k) asm volatile("" : "+f"(w[k][0]), "+f"(w[k][1]), "+f"(w[k][2]), "+f"(w[k][3]));
}

// NB: row blocks of 128 (N <= 128: 1, else 2).  BF: bf16 planes, else scaled FP16.  HI: the
// tiles hold the hi plane alone (BF16x2: products hi hi + hi lo(I~)).  CONV: FP16 tiles
// contracted with bf16 products (PRD_OPT_CONTRACTION): warp 1 re-splits each landed step
// in place before its products.
template <int NB, bool BF, bool HI, bool CONV>
__global__ void __launch_bounds__(kThreads, 1) r2_tc_kernel(Params p) {
  extern __shared__ __align__(1024) unsigned char smraw[];
  // 1024-byte aligned base, derived by offset so that the compiler keeps the
  // shared address space on every pointer below (plain LDS/STS, no generic access)
  unsigned char* sm = smraw + ((1024u - (smem_u32(smraw) & 1023u)) & 1023u);
  const int N = p.N, nst = p.nst;
  const int SA = stage_bytes(N, HI);             // one K step of the tile
  const int PA = rows16(N) * 32;                 // one plane of it
  const int KCH = p.ld / kKC, KH = KCH >> 1;     // K steps per tile and per half
  unsigned char* Iop = sm + nst * SA;            // [K step][hi | lo][128 rows][32 bytes]
  float* Ys = (float*)(Iop + KH * 2 * kPlane);   // [buffer][entry][pair][kYS]
  int* rec = (int*)((unsigned char*)Ys + 2 * kYBytes);
  float* colinv = (float*)(rec + kRec);          // scale to undo per operand row (o', j)
  uint64_t* full = (uint64_t*)(((uintptr_t)(colinv + 4 * kMaxIn) + 7) & ~(uintptr_t)7);
  uint64_t* empty = full + kStagesMax;
  uint64_t* accfull = empty + kStagesMax;        // [half] products of the half complete
  uint64_t* accfree = accfull + 2;               // [half] Y applied
  uint64_t* iready = accfree + 2;
  uint64_t* done = iready + 1;
  uint32_t* tmem_slot = (uint32_t*)(done + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);

  const int iz = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int et = threadIdx.x - 64;               // index among the Y threads
  constexpr uint32_t tm_cols = NB * 256u;
  // tiles of this CTA (grid.z splits them where there are too few work items)
  const int t0 = p.ntile * (int)blockIdx.z / (int)gridDim.z, t1 = p.ntile * ((int)blockIdx.z + 1) / (int)gridDim.z;

  for (int i = threadIdx.x; i < kRec; i += kThreads) rec[i] = p.work[(size_t)blockIdx.x * kRec + i];
  if (threadIdx.x == 0) {
    for (int s = 0; s < nst; ++s) {
      mbar_init(&full[s], 1);        // armed by the producer with the bytes of the tile copy
      mbar_init(&empty[s], 1);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(&accfull[h], 1);
      mbar_init(&accfree[h], kEpi);
    }
    mbar_init(iready, kEpi);
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
  const int* vdir = rec + 4;
  const int* vinfo = rec + 36;
  const int* vpair = rec + 68;
  const int* sdir = rec + 132;
  const int iters = (t1 - t0) * KCH;

  if (warp == 0) {
    // ---------------- producer: lane 0 waits for a free stage, arms its barrier with the
    // bytes of the step and copies the planes, up to nst steps ahead of the products
    if (lane == 0) {
      int it = 0;
      const uint64_t pol_t = policy_evict_first();
      const uint32_t pbytes = (uint32_t)N * 32;   // one plane of a step
      const size_t sbytes = (size_t)pbytes * (HI ? 1 : 2);
      const unsigned char* src = p.tiles + (((size_t)iz * p.ncls + c) * p.ntile + t0) * KCH * sbytes;
      int s = 0, ps = 0;                          // it % nst and (it / nst) & 1
      for (; it < iters; ++it, src += sbytes, s = (s + 1 == nst) ? (ps ^= 1, 0) : s + 1) {
        if (it >= nst && !mbar_wait(&empty[s], ps ^ 1, abort_flag, p.spin)) break;
        // rows n >= N of the stage keep stale data: they only reach accumulator rows
        // that nobody reads
        mbar_expect_tx(&full[s], (uint32_t)sbytes);
        bulk_load(sm + s * SA, src, pbytes, &full[s], pol_t);
        if constexpr (!HI) bulk_load(sm + s * SA + PA, src + pbytes, pbytes, &full[s], pol_t);
      }
      if (*abort_flag) {
        // drain copies that were issued and may not have been consumed
        for (int j = max(0, it - nst); j < it; ++j)
          for (long long i = 0; i < kSpin && !mbar_try(&full[j % nst], (j / nst) & 1); ++i) {
          }
      }
    }
  } else if (warp == 1) {
    // ---------------- products.  CONV: the whole warp re-splits a step first, so every lane
    // takes part in the waits; otherwise lane 0 alone.
    if (CONV || lane == 0) {
      const uint32_t ty = BF ? 1u : 0u;
      const uint32_t idesc = (1u << 4) | (ty << 7) | (ty << 10) | ((uint32_t)(rows16(4 * ns) >> 3) << 17) | ((128u >> 4) << 24);
      auto wait = [&](uint64_t* b, uint32_t par) {
        const bool r = mbar_wait(b, par, abort_flag, p.spin);
        return CONV ? (bool)__all_sync(0xffffffffu, r) : r;
      };
      bool ok = wait(iready, 0);
      int s = 0, ps = 0;
      bool issued = false;
      for (int t = 0; t < t1 - t0 && ok; ++t)
        for (int h = 0; h < 2 && ok; ++h) {
          if (t > 0) ok = wait(&accfree[h], (t - 1) & 1);
          for (int kc = 0; kc < KH && ok; ++kc) {
            ok = wait(&full[s], ps);
            if (!ok) break;
            unsigned char* A = sm + s * SA;
            if constexpr (CONV) {
              for (int i = lane; i < PA / 16; i += 32) {
                uint4 h4 = reinterpret_cast<uint4*>(A)[i], l4 = reinterpret_cast<uint4*>(A + PA)[i];
                uint32_t* hp = &h4.x;
                uint32_t* lp = &l4.x;
#pragma unroll
                for (int q = 0; q < 4; q += 2) {
                  const float2 a = __half22float2(*reinterpret_cast<__half2*>(hp + q)), b = __half22float2(*reinterpret_cast<__half2*>(lp + q));
                  const float2 e = __half22float2(*reinterpret_cast<__half2*>(hp + q + 1)), f = __half22float2(*reinterpret_cast<__half2*>(lp + q + 1));
                  uint2 hi, lo;
                  split4<true>(make_float4(a.x + b.x, a.y + b.y, e.x + f.x, e.y + f.y), hi, lo);
                  hp[q] = hi.x; hp[q + 1] = hi.y;
                  lp[q] = lo.x; lp[q + 1] = lo.y;
                }
                reinterpret_cast<uint4*>(A)[i] = h4;
                reinterpret_cast<uint4*>(A + PA)[i] = l4;
              }
              asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
              __syncwarp();
            }
            if (lane == 0) {
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              const uint64_t bh = sdesc32(Iop + kc * 2 * kPlane), bl = sdesc32(Iop + kc * 2 * kPlane + kPlane);
#pragma unroll
              for (int b = 0; b < NB; ++b) {
                const uint32_t d = tmem + (uint32_t)(h * NB + b) * 128u;
                const uint64_t ah = sdesc32(A + b * 4096);
                mma_f16(d, ah, bh, idesc, kc > 0 ? 1u : 0u);
                mma_f16(d, ah, bl, idesc, 1u);
                if constexpr (!HI) mma_f16(d, sdesc32(A + PA + b * 4096), bh, idesc, 1u);
              }
              mma_commit(&empty[s]);
              if (kc == KH - 1) mma_commit(&accfull[h]);
              issued = true;
            }
            s = (s + 1 == nst) ? (ps ^= 1, 0) : s + 1;
          }
        }
      // every product issued completes before TMEM is released
      if (lane == 0 && issued) {
        mma_commit(done);
        for (long long i = 0; i < kSpin && !mbar_try(done, 0); ++i) {
        }
      }
    }
  } else {
    // ---------------- Y warps
    const int q = warp & 3;                        // TMEM lane quarter of this warp
    const int og = (warp - 2) >> 2;                // entries of this warp: 2 i + og
    // Y of a tile: thread (pair slot, i) moves the 8 coefficients of output Stokes i
    const int yp = et >> 2, yi = et & 3;           // pair slot 2 entry + pair, Stokes i
    const int ypair = (yp >> 1) < E ? vpair[yp] : -1;
    const float4* ysrc = reinterpret_cast<const float4*>(p.Y + (((size_t)iz * p.npairs + max(ypair, 0)) * p.ntile + t0) * 32 + yi * 8);
    float4 ya = make_float4(0.f, 0.f, 0.f, 0.f), yb = ya;
    if (ypair >= 0) { ya = ysrc[0]; yb = ysrc[1]; }
    // I~ operand: a warp per incident direction; the scale of each of its 4 rows brings
    // the largest element to [2^13, 2^14)
    for (int sl = warp - 2; sl < ns; sl += kEpiWarps) {
      const float4* src = reinterpret_cast<const float4*>(p.Ic) + ((size_t)iz * p.nO + sdir[sl]) * N;
      float sc[4] = {1.f, 1.f, 1.f, 1.f};
      if constexpr (!BF) {
        float m[4] = {0.f, 0.f, 0.f, 0.f};
        for (int k = lane; k < N; k += 32) {
          const float4 v = src[k];
          m[0] = fmaxf(m[0], fabsf(v.x)); m[1] = fmaxf(m[1], fabsf(v.y));
          m[2] = fmaxf(m[2], fabsf(v.z)); m[3] = fmaxf(m[3], fabsf(v.w));
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
          for (int x = 16; x > 0; x >>= 1) m[j] = fmaxf(m[j], __shfl_xor_sync(0xffffffffu, m[j], x));
          // 2^(13 - exponent), kept where it and its inverse are normal FP32 numbers
          const int ex = (int)(__float_as_uint(m[j]) >> 23);          // biased exponent
          const int e = (ex == 255 || m[j] == 0.f) ? 127 : min(253, max(1, 127 + 13 + 127 - ex));
          sc[j] = __uint_as_float((uint32_t)e << 23);
          if (lane == j) colinv[sl * 4 + j] = __uint_as_float((uint32_t)(254 - e) << 23);
        }
      } else if (lane < 4) {
        colinv[sl * 4 + lane] = 1.f;
      }
      for (int g = lane; g < KH * 4; g += 32) {
        float4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = 4 * g + k < N ? src[4 * g + k] : make_float4(0.f, 0.f, 0.f, 0.f);
        unsigned char* dst = Iop + (g >> 2) * 2 * kPlane;
        const float4 r[4] = {make_float4(v[0].x, v[1].x, v[2].x, v[3].x), make_float4(v[0].y, v[1].y, v[2].y, v[3].y),
                             make_float4(v[0].z, v[1].z, v[2].z, v[3].z), make_float4(v[0].w, v[1].w, v[2].w, v[3].w)};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          uint2 hi, lo;
          split4<BF>(make_float4(r[j].x * sc[j], r[j].y * sc[j], r[j].z * sc[j], r[j].w * sc[j]), hi, lo);
          const uint32_t o = swz32(sl * 4 + j, g & 3);
          *(uint2*)(dst + o) = hi;
          *(uint2*)(dst + kPlane + o) = lo;
        }
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive(iready);
    bool ok = epi_all(true);                       // colinv is complete

    float ci[4] = {1.f, 1.f, 1.f, 1.f};            // column scales of this thread's Y
    if (ypair >= 0) {
      const int info = vinfo[yp >> 1], sl = (yp & 1) ? (info >> 8) & 255 : info & 255;
#pragma unroll
      for (int j = 0; j < 4; ++j) ci[j] = colinv[sl * 4 + j];
    }
    const bool live0 = q * 32 < N, live1 = NB > 1 && 128 + q * 32 < N;
    float acc[16][NB][4];
#pragma unroll
    for (int i = 0; i < 16; ++i)
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[i][b][k] = 0.f;
    const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
    for (int t = 0; t < t1 - t0; ++t) {
      float* Yb = Ys + (t & 1) * (kYBytes / 4);
      {
        float* d = Yb + yp * kYS + yi;             // [half][j][i]
        d[0] = ya.x * ci[0]; d[4] = ya.z * ci[1]; d[8] = yb.x * ci[2]; d[12] = yb.z * ci[3];
        d[16] = -ya.y * ci[0]; d[20] = -ya.w * ci[1]; d[24] = -yb.y * ci[2]; d[28] = -yb.w * ci[3];
      }
      ok = epi_all(ok);
      if (!ok) break;
      if (ypair >= 0 && t + 1 < t1 - t0) { ya = ysrc[(t + 1) * 8]; yb = ysrc[(t + 1) * 8 + 1]; }
      for (int h = 0; h < 2 && ok; ++h) {
        ok = __all_sync(0xffffffffu, mbar_wait(&accfull[h], t & 1, abort_flag, p.spin));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (live0) {
          const uint32_t ta = tq + (uint32_t)(h * NB) * 128u;
          const float* Yh = Yb + h * 16;
          // entry i + 1's columns are read while Y is applied to entry i's
          float w[2][2 * NB][4];                   // [buffer][pair, row block]
          auto load = [&](int i) {
            const int v = 2 * i + og;
            if (v >= E) return;
            const int info = vinfo[v];
            float(&x)[2 * NB][4] = w[i & 1];
            tmem_ld4(x[0], ta + (uint32_t)(info & 255) * 4u);
            if (NB > 1) tmem_ld4(x[NB - 1], ta + 128u + (uint32_t)(info & 255) * 4u);
            if ((info >> 16) > 1) {
              const uint32_t cb = (uint32_t)((info >> 8) & 255) * 4u;
              tmem_ld4(x[NB], ta + cb);
              if (NB > 1) tmem_ld4(x[2 * NB - 1], ta + 128u + cb);
            }
          };
          load(0);
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int v = 2 * i + og;
            if (v >= E) break;
            tmem_wait<2 * NB>(w[i & 1]);
            if (i + 1 < 16) load(i + 1);
            const int np = vinfo[v] >> 16;
#pragma unroll
            for (int pr = 0; pr < 2; ++pr) {
              if (pr < np) {
                const float4* y4 = reinterpret_cast<const float4*>(Yh + (2 * v + pr) * kYS);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  const float4 y = y4[j];
#pragma unroll
                  for (int b = 0; b < NB; ++b) {
                    if (b > 0 && !live1) continue;
                    const float x = w[i & 1][pr * NB + b][j];
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
        mbar_arrive(&accfree[h]);
      }
    }
    if (ok) {
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const int n = b * 128 + q * 32 + lane;
        if (n >= N) continue;
        const float sc = p.tsc ? p.tsc[((size_t)iz * p.ncls + c) * N + n] : 1.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int v = 2 * i + og;
          if (v < E) {
            float* dst = p.eb + (((size_t)iz * p.nO + vdir[v]) * N + n) * 4;
            asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst), "f"(acc[i][b][0] * sc),
                         "f"(acc[i][b][1] * sc), "f"(acc[i][b][2] * sc), "f"(acc[i][b][3] * sc)
                         : "memory");
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*abort_flag && threadIdx.x == 0) atomicExch(p.err, 1);
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tm_cols));
  }
}

}  // namespace tc

// Tile stages for N rows: the most (<= kStagesMax) whose shared memory fits.
static int r2_tc_stages(int N, bool hi) {
  for (int st = tc::kStagesMax; st >= 2; --st)
    if (tc::smem_bytes(N, st, hi) <= kMaxSmem) return st;
  return 0;
}

template <int NB>
static int r2_tc_attr(Ctx* c) {
  for (auto k : {tc::r2_tc_kernel<NB, false, false, false>, tc::r2_tc_kernel<NB, true, false, false>,
                 tc::r2_tc_kernel<NB, true, true, false>, tc::r2_tc_kernel<NB, true, false, true>})
    PRD_CUDA_TRY(c, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
  return PRD_OK;
}

// Work records of the contraction: every class's outputs cut into entries of at most two
// incident directions each (an output with more, as all are in angle-averaged mode,
// takes several entries, which add up in eps_bar) and the entries packed into records of
// at most 32 entries and 32 incident directions.  Where entries are many they are
// taken by blocks of 32 incident directions, so that a record's entries share them.
void r2_tc_records(const Ctx* c, std::vector<int>& out) {
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
        slots.clear();
        add.clear();
        for (int i = 0; i < x.n; ++i) {
          const int d = c->pair_in[x.p[i]];
          if (std::find(add.begin(), add.end(), d) == add.end()) add.push_back(d);
        }
      }
      for (int d : add) {
        out[rec + 132 + (int)slots.size()] = d;
        slots.push_back(d);
      }
      out[rec + 2] = (int)slots.size();
      const int v = out[rec + 1]++;
      int sl[2] = {0, 0};
      for (int i = 0; i < x.n; ++i)
        sl[i] = (int)(std::find(slots.begin(), slots.end(), c->pair_in[x.p[i]]) - slots.begin());
      out[rec + 4 + v] = x.o;
      out[rec + 36 + v] = sl[0] | (sl[1] << 8) | (x.n << 16);
      out[rec + 68 + 2 * v] = x.p[0];
      out[rec + 68 + 2 * v + 1] = x.n > 1 ? x.p[1] : -1;
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
  if (c->prec != PRD_FP32) return PRD_OK;
  if (!c->tiled() || c->nnu > 224 || r2_tc_stages(c->nnu, c->hi_only) < 2)
    return fail(c, PRD_E_ARG, "tensor-core contraction needs FP32 tiles and N small enough for two tile stages "
                              "beside the resident I~ (N <= 224)");
  std::vector<int> work;
  r2_tc_records(c, work);
  c->tc_nwork = (int)work.size() / tc::kRec;
  dfree(c->tc_work);
  int rc = dalloc(c, c->tc_work, work.size() * sizeof(int));
  if (rc || (rc = r2_tc_attr<1>(c)) || (rc = r2_tc_attr<2>(c))) return rc;
  PRD_CUDA_TRY(c, cudaMemcpy(c->tc_work.p, work.data(), work.size() * sizeof(int), cudaMemcpyHostToDevice));
  PRD_CUDA_TRY(c, cudaMemset(c->tc_err.p, 0, sizeof(int)));
  c->tc_ready = true;
  return PRD_OK;
}

int r2_tc_launch(Ctx* c, const float* Ic, float* eb) {
  // the deepest ring that fits, or the caller's (autotuned) depth if smaller
  const int nmax = r2_tc_stages(c->nnu, c->hi_only);
  const int nst = c->tc_stages >= 2 ? std::min(c->tc_stages, nmax) : nmax;
  tc::Params p{(const unsigned char*)c->tiles.p, (const float*)c->tile_scale.p, (const float*)c->Y.p, Ic,
               (const int*)c->tc_work.p, eb, (int*)c->tc_err.p, c->ncls, c->ntile(), c->nO, c->nnu, c->npairs,
               c->ld(), nst, c->tc_spin > 0 ? c->tc_spin : tc::kSpin};
  const int smem = tc::smem_bytes(c->nnu, nst, c->hi_only);
  // fewer CTAs than SMs: split the tiles of a work item (at least 4 tiles each)
  const int items = c->tc_nwork * c->nz;
  const int zs = std::max(1, std::min(c->ntile() / 4, c->nsm / std::max(1, items)));
  auto go = [&](auto k1, auto k2) -> int {
    const dim3 g(c->tc_nwork, c->nz, zs);
    if (c->nnu <= 128) k1<<<g, tc::kThreads, smem, c->stream>>>(p);
    else k2<<<g, tc::kThreads, smem, c->stream>>>(p);
    PRD_CUDA_TRY(c, cudaPeekAtLastError());
    return PRD_OK;
  };
  if (c->hi_only) return go(tc::r2_tc_kernel<1, true, true, false>, tc::r2_tc_kernel<2, true, true, false>);
  if (c->split_tiles) return go(tc::r2_tc_kernel<1, true, false, false>, tc::r2_tc_kernel<2, true, false, false>);
  if (c->tc_bf16) return go(tc::r2_tc_kernel<1, true, false, true>, tc::r2_tc_kernel<2, true, false, true>);
  return go(tc::r2_tc_kernel<1, false, false, false>, tc::r2_tc_kernel<2, false, false, false>);
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
