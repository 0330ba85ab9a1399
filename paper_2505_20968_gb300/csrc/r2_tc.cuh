// What the two tensor-core contraction kernels share (r2_tc.cu: tiles stored as bf16 planes;
// r2_tc32.cu: FP32 tiles): work records, barriers, operand layouts and products.
#pragma once
#include <cuda_bf16.h>
#include "prd_internal.h"
#include "ring.h"

namespace prd {

namespace tc {

constexpr int kStagesMax = 8;                 // tile ring depth: 2..8, the most that fit beside the rest
constexpr int kKC = 16;                       // columns of a K step
constexpr int kSteps = 2;                     // K steps per stage: a stage's waits and commits cost the
                                              // issuing warp some 300 clocks, a product 64
constexpr int kMaxE = 32;                     // output entries per CTA
constexpr int kMaxIn = 32;                    // incident directions per CTA (128 operand rows)
constexpr int kPlane = 4 * kMaxIn * 32;       // bytes of one K step of one I~ plane
constexpr int kEpiWarps = 16;
constexpr int kEV = kMaxE / (kEpiWarps / 4);   // entries of a Y warp (4 warps share a lane quarter)
constexpr int kEpi = 32 * kEpiWarps;          // threads of the Y warps
constexpr int kYS = 36;                       // floats of a staged pair: Re [j][i], -Im [j][i], 4 of padding (banks)
constexpr int kYBytes = 2 * kMaxE * kYS * 4;  // one tile's Y
constexpr int kRec = 4 + 32 + 64 + 32;        // ints of a work record
constexpr int kAuxBytes = 2048;               // work record, barriers, TMEM slot, abort flag
__host__ __device__ constexpr int rows16(int N) { return (N + 15) / 16 * 16; }
// Tiles per pass: up to 64 (32) rows, two (four) tiles share the 128 accumulator rows, each
// with its own lane quarters and Y, so a small tile does not leave most of a product
// and of the Y warps idle.
__host__ __device__ constexpr int tiles_per_pass(int rows) { return rows <= 32 ? 4 : (rows <= 64 ? 2 : 1); }
constexpr int kSpin = 1 << 24;                // bounded waits (default limit of the pipeline waits; drains)

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
// the same without the suspension of try_wait
__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred P;\n\tmbarrier.test_wait.parity.shared::cta.b64 P, [%1], %2;\n\tselp.b32 %0, 1, 0, P;\n\t}\n"
      : "=r"(ok)
      : "r"(smem_u32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded pipeline wait of at most `limit` polls; returns false (and raises the
// CTA abort flag) on expiry or when another role has aborted, which it looks at
// between bursts of polls
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag, int limit) {
  bool r = mbar_try(b, parity);
  for (int n = 1; !r && n < limit && !*abort_flag;) {
    const int m = min(n + 64, limit);
    for (; n < m && !r; ++n) r = mbar_try(b, parity);
  }
  if (!r) *abort_flag = 1;
  return r;
}
// the same by a converged warp
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* b, uint32_t parity, volatile int* abort_flag, int limit) {
  const bool r = mbar_wait(b, parity, abort_flag, limit);
  return __all_sync(0xffffffffu, r);
}
// the same after a look ahead: a look at a barrier takes some 150 clocks, which a role that has other
// work spends on it (ok: that mbar_test)
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* b, uint32_t parity, volatile int* abort_flag, int limit, bool ok) {
  return __all_sync(0xffffffffu, ok) || mbar_wait_warp(b, parity, abort_flag, limit);
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
// bf16 operands, FP32 accumulation, K = 16 per instruction
__device__ __forceinline__ void mma_bf16(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
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


// The next bf16 plane of two values, rounded to nearest, which keep the remainders: after three,
// nothing is left of an FP32 value (8 + 8 + 8 significant bits; |remainder| <= 2^-8 of the value
// after one plane, 2^-17 after two).
// The remainder is a mixed-precision fma, v - 1 hi, which takes the plane's halves as they are: unpacked
// by shifts and masks first, three of five instructions sat in the half-rate integer pipe (165
// clocks of a scheduler for 16 values of 32 lanes and three planes, 101 this way).
__device__ __forceinline__ uint32_t split2(float& a, float& b) {
  uint32_t h;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(b), "f"(a));
  asm("{\n\t.reg .b16 l, u, m;\n\tmov.b32 {l, u}, %2;\n\tmov.b16 m, 0xBF80;\n\t"
      "fma.rn.f32.bf16 %0, l, m, %0;\n\tfma.rn.f32.bf16 %1, u, m, %1;\n\t}"
      : "+f"(a), "+f"(b)
      : "r"(h));
  return h;
}

// one lane of a converged warp (the same one every time)
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}\n" : "=r"(r));
  return r != 0;
}

struct Params {
  const unsigned char* tiles;   // [z][class][tile] pre-swizzled K steps of FP32 [N][16] or bf16 [plane][N][16]
  const float* Y;       // [z][pair][ntile][16][2]
  const float* Ic;      // [z][o][N][4]
  const int* work;      // [item][kRec]: class, entries, incident directions, first entry, then of each entry its
                        // slots (a | b << 8 | pairs << 16) and its pairs' indices, and the direction of each slot
  float4* ent;          // contributions of the entries (RowAdds)
  float4* tail;         // those of the further parts of split items
  int* err;
  int ncls, ntile, nO, N, npairs, ld, nent, nz, nwork;   // nz: heights of this launch
  int z0;               // first height: the items count from it
  int split0, nsplit, zs;   // the nsplit work items from split0 on have their tiles split between zs CTAs
  int nst;              // tile stages
  int ring;             // bytes of the tile ring (FP32 tiles)
  int spin;             // poll limit of the pipeline waits (the drains keep kSpin)
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
  asm volatile("tcgen05.wait::ld.sync.aligned;");
  // the values pass through here, so that no use of them moves above the wait
#pragma unroll
  for (int k = 0; k < K; ++k) asm volatile("" : "+f"(w[k][0]), "+f"(w[k][1]), "+f"(w[k][2]), "+f"(w[k][3]));
}

// The resident I~ operand, by a warp: K step by K step IP planes of 128 rows (incident direction,
// Stokes parameter) of 32 bytes under the 32-byte swizzle.  A warp takes every kEpiWarps-th
// incident direction from sl on, a lane four frequencies of its four rows.
template <int IP>
__device__ __forceinline__ void build_operand(unsigned char* Iop, const float* Ic, const int* sdir, int sl, int ns, int iz,
                                              int nO, int N, int KH) {
  for (; sl < ns; sl += kEpiWarps) {
    const float4* src = reinterpret_cast<const float4*>(Ic) + ((size_t)iz * nO + sdir[sl]) * N;
    for (int g = threadIdx.x & 31; g < KH * 4; g += 32) {
      float4 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = 4 * g + k < N ? src[4 * g + k] : make_float4(0.f, 0.f, 0.f, 0.f);
      unsigned char* dst = Iop + (g >> 2) * IP * kPlane;
      float4 r[4] = {make_float4(v[0].x, v[1].x, v[2].x, v[3].x), make_float4(v[0].y, v[1].y, v[2].y, v[3].y),
                     make_float4(v[0].z, v[1].z, v[2].z, v[3].z), make_float4(v[0].w, v[1].w, v[2].w, v[3].w)};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t o = swz32(sl * 4 + j, g & 3);
#pragma unroll
        for (int k = 0; k < IP; ++k) *(uint2*)(dst + k * kPlane + o) = make_uint2(split2(r[j].x, r[j].y), split2(r[j].z, r[j].w));
      }
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

}  // namespace tc

// FP32 tiles (r2_tc32.cu)
int r2_f32_stages(int N);
int r2_f32_prepare(Ctx* c);
void r2_f32_launch(Ctx* c, tc::Params p, int grid);

}  // namespace prd
