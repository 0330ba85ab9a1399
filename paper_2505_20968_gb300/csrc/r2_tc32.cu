// S3+S4 R_II contraction of FP32 tiles on the tensor cores: the same order and work records as
// r2_tc.cu (tile times the raw incident field, W[n][(o', j)] = sum_k A[n][k] I~[(o', j)][k], then Y
// from TMEM), with products that keep FP32's accuracy at any exponent.
//
// An FP32 value is three bf16 planes, hi + mid + lo, exactly; of the nine products of two values the
// six with at most two steps down (hi hi, hi mid, hi lo, mid hi, mid mid, lo hi) are taken, and
// what is left out is 2^-24 of the product.  (Scaled FP16 pairs take three products, but hold a
// value to 2^-38 of its row's largest only.)  PRD_OPT_CONTRACTION = BF16X3 keeps hi and mid of both
// and three products, as contexts of bf16 planes do.
//
// What bounds it: the tensor pipe (64 clocks a product of 128 x 128 x 16) and shared memory,
// which at 128 bytes a clock can feed both operands of one such product in just that time; beside
// them the schedulers, which the split and Y share with the warp that issues the products (ncu, 4
// heights of the problem below: tensor pipe 65 %, issue slots 56 %, HBM 45 % of the measured rate).
// So the tile goes through registers into TMEM, the one place that a product can take its first
// operand from without shared memory: four warps, a thread a row, read a landed FP32 step, split it
// and store its planes as packed columns, and only I~ is read from shared memory.  TMEM
// holds the accumulators of one block of 128 rows (Re and Im half, 128 columns each: Y is applied
// to one while the other is formed) and two slots of planes, so a CTA takes all its tiles
// for the rows 0 .. 127 and then for the rest; rows beyond 128 are packed like small tiles, two or
// four tiles a pass where they are at most 64 or 32.
//
// What shaped it (contraction of Mg II 8 heights x 64 directions x 200 frequencies): planes written back
// to shared memory for the products, 2350 us; through TMEM, 1570 with eight split warps in one step
// each; remainders by mixed-precision fma and barriers looked at ahead 1530; hand-overs of four K
// steps 1505; four split warps of two steps each (fewer instructions beside the products' warp)
// 1455; the look ahead in the middle of a turn 1420.  The products alone take 1140 to 1250 here
// (a loop without other warps: 970), split, Y and copies without them 1270.
// Without gain: fetching the tiles into L2 ahead (the ring is shallow, three stages, at 200
// frequencies), Y's columns read an entry ahead, eight Y warps of 16 entries, a split group for each
// slot, registers moved to the Y warps (setmaxnreg).
// Measured, contraction (before: scaled FP16 pairs, three products; before that: three TF32 products of
// an operand formed per K step): that problem 2795, 954, now 1420 us; H I 4 x 96 x 150 779 -> 816; H I
// angle-averaged 8 x 64 x 91 272 -> 379; Mg II 10 x 16 x 27 24 -> 29.
//
// Roles (704 threads): warp 0 streams the tile into a ring of K step pairs (bulk copies) and owns the
// TMEM allocation; warp 1 issues tcgen05.mma; warps 2-5 split; warps 6-21 stage I~ and Y and apply
// Y.  Every mbarrier wait is bounded; on expiry the CTA records an error flag, drains what it issued
// and returns.
#include <algorithm>
#include "device_common.cuh"
#include "r2_tc.cuh"

namespace prd {

namespace tc {

constexpr int kSplit0 = 2, kSplitWarps = 4;   // warps that split (a lane quarter each)
constexpr int kY0 = kSplit0 + kSplitWarps;    // first Y warp
constexpr int kThreads32 = 32 * kY0 + kEpi;
// Planes in TMEM: two slots of two stages (four K steps) each.  A look at a barrier takes 150 clocks and an
// arrival 100, so the hand-over is per slot.
constexpr int kSlots = 2, kTurn = 2 * kSteps;
// Bytes of a landed K step of a row block, and stages that a ring of `ring` bytes takes: where
// the second block has a single tile a pass, its steps lie closer and more of them are in flight
__host__ __device__ constexpr int step32(int N, int blk) {
  return blk && N - 128 > 64 ? rows16(N - 128) * 64 : 128 * 64;
}
__host__ __device__ constexpr int stages32(int N, int blk, int ring) {
  return ring / (kSteps * step32(N, blk)) < kStagesMax ? ring / (kSteps * step32(N, blk)) : kStagesMax;
}
// Y buffers: two, so that the next pass's Y is staged beside the one in use, where there is room
// (N <= 128); a barrier more a pass otherwise
__host__ __device__ constexpr int y_bufs(int N) { return N <= 128 ? 2 : 1; }
// tiles per pass: of the first 128 rows, of the rest, and the larger of the two
__host__ __device__ constexpr int tpp(int N, int blk) { return tiles_per_pass(blk ? N - 128 : (N < 128 ? N : 128)); }
__host__ __device__ constexpr int tpp_max(int N) { return N > 128 ? tpp(N, 1) : tpp(N, 0); }
// Shared memory of one CTA but for the tile ring: the resident I~ operand, the Y buffers, the
// auxiliary tables, 1 KB to align the base.
__host__ __device__ constexpr int smem32(int N, int ip) {
  return rows16(N) / kKC * ip * kPlane + y_bufs(N) * tpp_max(N) * kYBytes + kAuxBytes + 1024;
}
// (The split reads 128 rows of every step; those past a closer step, N > 192, lie in the next ones or, behind the
// ring, in the operand: read, and of no effect.)

__device__ __forceinline__ void mma_commit_if(uint64_t* bar, bool yes) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %1, 0;\n\t"
      "@p tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}\n" ::"r"(smem_u32(bar)),
      "r"((uint32_t)yes)
      : "memory");
}
// first operand in TMEM
__device__ __forceinline__ void mma_bf16_t(uint32_t dtmem, uint32_t atmem, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n"
      ::"r"(dtmem), "r"(atmem), "l"(b), "r"(idesc), "r"(acc));
}
// eight TMEM columns of the warp's 32 lanes
__device__ __forceinline__ void tmem_st8(uint32_t addr, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(addr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}

// IP: planes of an operand (3: six products, 2: three)
template <int IP>
__global__ void __launch_bounds__(kThreads32, 1) r2_f32_kernel(Params p) {
  extern __shared__ __align__(1024) unsigned char smraw[];
  // 1024-byte aligned base, derived by offset so that the compiler keeps the
  // shared address space on every pointer below (plain LDS/STS, no generic access)
  unsigned char* sm = smraw + ((1024u - (smem_u32(smraw) & 1023u)) & 1023u);
  const int N = p.N;
  const int KCH = p.ld / kKC, KH = KCH >> 1;     // K steps per tile and per half
  unsigned char* Iop = sm + p.ring;              // [K step][plane][128 rows][32 bytes]
  float* Ys = (float*)(Iop + KH * IP * kPlane);  // [buffer][tile of the pass][entry][pair][kYS]
  const int YB = y_bufs(N);
  int* rec = (int*)((unsigned char*)Ys + YB * tpp_max(N) * kYBytes);
  uint64_t* full = (uint64_t*)(((uintptr_t)(rec + kRec) + 7) & ~(uintptr_t)7);
  uint64_t* empty = full + 2 * kStagesMax;       // both [row block][stage]
  uint64_t* aready = empty + 2 * kStagesMax;     // [slot] planes written
  uint64_t* afree = aready + kSlots;             // [slot] products that read them complete
  uint64_t* accfull = afree + kSlots;            // [half] products of the half complete
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
  const int t0 = p.ntile * part / nparts, nt = p.ntile * (part + 1) / nparts - t0;   // this part's tiles

  for (int i = threadIdx.x; i < kRec; i += kThreads32) rec[i] = p.work[(size_t)(item - zl * p.nwork) * kRec + i];
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2 * kStagesMax; ++s) {
      mbar_init(&full[s], 1);              // armed by the producer with the bytes of the copies
      mbar_init(&empty[s], kSplitWarps);
    }
    for (int s = 0; s < kSlots; ++s) {
      mbar_init(&aready[s], kSplitWarps);
      mbar_init(&afree[s], 1);
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
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot, atmem = tmem + 256;
  constexpr uint32_t kACols = 8 * IP, kSlotCols = kTurn * kACols;   // TMEM columns of a step's planes, of a slot
  const int c = rec[0], E = rec[1], ns = rec[2];
  const int* vinfo = rec + 4;
  const int* vpair = rec + 36;
  const int* sdir = rec + 100;
  // passes over the tiles, of both row blocks, and their stages of kSteps = 2 steps
  const int nblk = N > 128 ? 2 : 1;
  auto blk_passes = [&](int blk) { return (nt + tpp(N, blk) - 1) / tpp(N, blk); };
  const int passes = blk_passes(0) + (nblk > 1 ? blk_passes(1) : 0);
  int filled[2] = {0, 0};                        // stages warp 0 has filled, by row block

  if (warp == 0) {
    // ---------------- producer: the warp waits for a free stage and arms its barrier with the
    // bytes of the copies, then each lane issues its one (step, tile of the pass), up to nst
    // stages ahead of the split
    const uint64_t pol_t = policy_evict_first();
    const size_t step = (size_t)N * 64;
    const int c2 = lane & 1, g = lane >> 1;
    bool ok = true;
    for (int blk = 0; blk < nblk && ok; ++blk) {
      const int G = tpp(N, blk), n = stages32(N, blk, p.ring), iters = blk_passes(blk) * KH, S = step32(N, blk);
      const uint32_t bytes = (uint32_t)min(N - blk * 128, 128) * 64;   // one copy
      const unsigned char* src = p.tiles + (((size_t)iz * p.ncls + c) * p.ntile + t0 + g) * KCH * step + c2 * step + blk * (128 * 64);
      unsigned char* dst = sm + c2 * S + g * (8192 / G);
      int j = 0, left = nt;                          // stage of the pass, tiles left
      auto wait_empty = [&](int s, uint32_t par) { return mbar_wait_warp(&empty[blk * kStagesMax + s], par, abort_flag, p.spin); };
      const int done_ = ring_produce(iters, n, wait_empty, [&](int s) {
        // the stage's other rows (and the places of a last pass's missing tiles) keep stale
        // data: they only reach accumulator rows that nobody reads
        uint64_t* f = &full[blk * kStagesMax + s];
        const int g1 = min(G, left);
        if (lane == 0) mbar_expect_tx(f, kSteps * bytes * g1);
        __syncwarp();
        if (g < g1) bulk_load(dst + s * kSteps * S, src, bytes, f, pol_t);
        src += kSteps * step;
        if (++j == KH) {
          j = 0;
          left -= G;
          src += (size_t)(G - 1) * KCH * step;
        }
      });
      if (blk == 0) filled[0] = done_; else filled[1] = done_;
      // the next block's stages lie elsewhere in the ring: all of this one's are back first
      ok = done_ == iters && (blk + 1 == nblk || ring_close(iters, n, wait_empty));
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- products: the warp runs uniformly (waits by all lanes, descriptors in
    // uniform registers) and an elected lane issues; a loop of one lane issued a product
    // every 160 clocks, three times what it takes to execute
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(rows16(4 * ns) >> 3) << 17) | ((128u >> 4) << 24);
    const uint64_t b0 = sdesc32(Iop);              // the address field counts 16 bytes
    const uint32_t b0lo = (uint32_t)b0, b0hi = (uint32_t)(b0 >> 32);
    // Everything here is uniform, the outcome of a wait by a vote, so that descriptors stay in
    // uniform registers: moved there for every product they cost 80 clocks of it.  A wait that
    // gives up raises the flag, and nothing is waited for, issued or committed any more, so no
    // slot goes back.  (The flag is looked at once a pass: a look costs 100 clocks.)
    bool live = true;
    auto wait = [&](uint64_t* b, uint32_t par) {
      if (!live) return;
      bool r = false;
      for (int i = 0; i < p.spin && !r; ++i) r = __all_sync(0xffffffffu, mbar_try(b, par));
      if (!r) *abort_flag = 1;
      live = r;
    };
    {
      // I~ takes microseconds to build: plain polls, so that a short poll limit expires here
      bool r = false;
      for (int i = 0; i < p.spin && !r; ++i) r = __all_sync(0xffffffffu, mbar_test(iready, 0));
      if (!r) *abort_flag = 1;
      live = r;
    }
    // A slot (four K steps) a turn, whose barrier is looked at in the middle of the turn before (at its
    // start the slot is still being filled, and the wait cost 2 % more).  What may come in
    // the middle of a turn, the end of a half and the next one's wait for its accumulators, costs
    // no branch between the products: the commit is predicated, the wait taken at the turn's start
    // (branches a step cost 100 clocks a stage).  Halves of less than a turn (and a last turn of one
    // stage) take it step by step: their accumulators may be freed by a commit of the same turn.
    const int iters = passes * KH;
    int t = 0, h = 0, kc = 0;                      // pass, half, K step within it
    int sl = 0;
    uint32_t ph = 0;
    bool ahead = false;
    auto products = [&](int v, int hv, int k) {    // step v of the turn: step k of half hv
      const uint32_t d = tmem + (uint32_t)hv * 128u, ah = atmem + (uint32_t)sl * kSlotCols + v * kACols, am = ah + 8, al = ah + 16;
      const uint32_t o = b0lo + (uint32_t)k * (IP * kPlane >> 4);
      const uint64_t bh = (uint64_t)b0hi << 32 | o, bm = (uint64_t)b0hi << 32 | (o + (kPlane >> 4)),
                     bl = (uint64_t)b0hi << 32 | (o + 2 * (kPlane >> 4));
      mma_bf16_t(d, ah, bh, idesc, k > 0 ? 1u : 0u);
      mma_bf16_t(d, ah, bm, idesc, 1u);
      mma_bf16_t(d, am, bh, idesc, 1u);
      if constexpr (IP == 3) {
        mma_bf16_t(d, ah, bl, idesc, 1u);
        mma_bf16_t(d, am, bm, idesc, 1u);
        mma_bf16_t(d, al, bh, idesc, 1u);
      }
      mma_commit_if(&accfull[hv], k + 1 == KH);
    };
    for (int it = 0; it < iters && live; it += 2) {
      const int cnt = min(2, iters - it);
      if (!__all_sync(0xffffffffu, ahead)) wait(&aready[sl], ph);
      ahead = false;
      if (cnt == 2 && KH >= kTurn) {
        // a half's accumulators are free once Y has been applied to the pass before
        const bool starts = kc == 0, next = kc + kTurn > KH;
        if (starts && t > 0) wait(&accfree[h], (t - 1) & 1);
        if (next && t + h > 0) wait(&accfree[h ^ 1], (t + h - 1) & 1);
        // orders the products behind the planes' stores and the Y warps' reads
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int v = 0; v < kTurn; ++v) {
          const bool wrap = kc + v >= KH;
          if (live && elect_one()) products(v, wrap ? h ^ 1 : h, wrap ? kc + v - KH : kc + v);
          if (v == 1) ahead = it + 2 < iters && mbar_test(&aready[sl ^ 1], ph ^ sl);
        }
        kc += kTurn;
        if (kc >= KH) {
          kc -= KH;
          if ((h ^= 1) == 0) {
            ++t;
            if (__any_sync(0xffffffffu, *abort_flag != 0)) live = false;
          }
        }
      } else {
        for (int v = 0; v < cnt * kSteps; ++v) {
          if (kc == 0 && t > 0) wait(&accfree[h], (t - 1) & 1);
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (live && elect_one()) products(v, h, kc);
          if (++kc == KH) {
            kc = 0;
            if ((h ^= 1) == 0) {
              ++t;
              if (__any_sync(0xffffffffu, *abort_flag != 0)) live = false;
            }
          }
        }
      }
      if (live && elect_one()) mma_commit(&afree[sl]);
      ph ^= sl;
      sl ^= 1;
    }
    // every product issued completes before TMEM is released
    __syncwarp();
    if (elect_one()) mma_commit(done);
    for (int i = 0; i < kSpin && !mbar_try(done, 0); ++i) {
    }
  } else if (warp < kY0) {
    // ---------------- split: thread = row of the block.  A landed row of 64 bytes lies under the
    // 64-byte swizzle; its planes go to 8 columns each (two neighbouring k a column) of a slot.
    const int q = warp & 3, row = q * 32 + lane;   // TMEM lane quarter of this warp
    const uint32_t at = atmem + ((uint32_t)(q * 32) << 16);
    const int iters0 = blk_passes(0) * KH, iters = passes * KH;
    RingPos pos, slot;                             // stage to take, slot to fill
    int lim = p.spin, blk = 0, n = stages32(N, 0, p.ring), S = step32(N, 0);
    bool ahead_full = mbar_test(&full[0], 0), ahead_free = true;   // looks at the next stage and slot
    for (int it = 0; it < iters && lim > 0; ++it) {
      ring_take(
          pos, n, lim,
          [&](int s, uint32_t par, int& limit) {
            return mbar_wait_warp(&full[blk * kStagesMax + s], par, abort_flag, limit, ahead_full);
          },
          [&](int s, bool landed) {
            // a slot's first stage: the products that read the slot before are complete
            if (landed && (it & 1) == 0) landed = mbar_wait_warp(&afree[slot.s], slot.ph ^ 1, abort_flag, lim, ahead_free);
            if (!landed) {
              lim = 0;                             // the same on all lanes
              return;
            }
            const int own = blk * kStagesMax;
            float v[kSteps][16];
#pragma unroll
            for (int u = 0; u < kSteps; ++u) {
              const float4* a = reinterpret_cast<const float4*>(sm + (s * kSteps + u) * S + row * 64);
#pragma unroll
              for (int k = 0; k < 4; ++k) *reinterpret_cast<float4*>(&v[u][4 * k]) = a[k ^ ((row >> 1) & 3)];
            }
            RingPos next = pos;
            next.next(n);
            if (it + 1 == iters0) {                // on to the second row block's stages
              next = RingPos();
              pos = RingPos{n - 1, 1};             // from which ring_take steps to the same
              blk = 1;
              n = stages32(N, 1, p.ring);
              S = step32(N, 1);
            }
            ahead_full = mbar_test(&full[blk * kStagesMax + next.s], next.ph);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int k = 0; k < IP; ++k) {
#pragma unroll
              for (int u = 0; u < kSteps; ++u) {
                uint32_t w[8];
#pragma unroll
                for (int m = 0; m < 8; ++m) w[m] = split2(v[u][2 * m], v[u][2 * m + 1]);
                tmem_st8(at + (uint32_t)slot.s * kSlotCols + ((it & 1) * kSteps + u) * kACols + k * 8, w);
              }
              if (k == 0) {                        // the stage has been read
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[own + s]);
              }
            }
            if ((it & 1) || it + 1 == iters) {     // the slot is full
              asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
              asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
              __syncwarp();
              if (lane == 0) mbar_arrive(&aready[slot.s]);
              slot.next(kSlots);
              ahead_free = it + 1 < 2 * kSlots || mbar_test(&afree[slot.s], slot.ph ^ 1);
            }
          });
    }
  } else {
    // ---------------- Y warps
    const int et = threadIdx.x - 32 * kY0;         // index among the Y threads
    const int q = warp & 3;                        // TMEM lane quarter of this warp
    const int og = (warp - kY0) >> 2;              // entries of this warp: 4 i + og
    // Y of a tile: thread (pair slot, i) moves the 8 coefficients of output Stokes i
    // (tiles of the pass are shared out between the two halves of the threads)
    const int yp = (et & 255) >> 2, yi = et & 3;   // pair slot 2 entry + pair, Stokes i
    const int yg = et >> 8;                        // tiles yg, yg + 2 of the pass
    const int ypair = (yp >> 1) < E ? vpair[yp] : -1;
    const float4* ysrc = reinterpret_cast<const float4*>(p.Y + (((size_t)iz * p.npairs + max(ypair, 0)) * p.ntile + t0) * 32 + yi * 8);
    build_operand<IP>(Iop, p.Ic, sdir, warp - kY0, ns, iz, p.nO, N, KH);
    __syncwarp();
    if (lane == 0) mbar_arrive(iready);
    bool ok = true;
    const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
    int use = 0;                                   // pass, over both row blocks
    for (int blk = 0; blk < nblk; ++blk) {
      if (blk > 0 && !(ok = epi_all(ok))) break;   // all warps go on, or none
      const int G = tpp(N, blk), r0 = blk * 128, rows = min(N - r0, 128), np_ = (nt + G - 1) / G;
      // tile of the pass and row of this lane
      const int gt = q * G / 4, nl = (q % (4 / G)) * 32 + lane;
      const bool live = (q % (4 / G)) * 32 < rows;
      float4 ya[2], yb[2];
      auto load_y = [&](int t) {                   // Y of pass t's tiles
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int g = yg + 2 * k, ti = t * G + g;
          ya[k] = yb[k] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (ypair >= 0 && g < G && ti < nt) { ya[k] = ysrc[ti * 8]; yb[k] = ysrc[ti * 8 + 1]; }
        }
      };
      load_y(0);
      float acc[kEV][4];
#pragma unroll
      for (int i = 0; i < kEV; ++i)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[i][k] = 0.f;
      for (int t = 0; t < np_; ++t, ++use) {
        float* Yb = Ys + (YB == 2 ? use & 1 : 0) * (tpp_max(N) * kYBytes / 4);
        if (YB == 1) ok = epi_all(ok);             // every warp has used the Y of the pass before
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int g = yg + 2 * k;
          if (g >= G) break;
          float* d = Yb + g * (kYBytes / 4) + yp * kYS + yi;           // [half][j][i]
          d[0] = ya[k].x; d[4] = ya[k].z; d[8] = yb[k].x; d[12] = yb[k].z;
          d[16] = -ya[k].y; d[20] = -ya[k].w; d[24] = -yb[k].y; d[28] = -yb[k].w;
        }
        ok = epi_all(ok);
        if (!ok) break;
        if (t + 1 < np_) load_y(t + 1);
        for (int h = 0; h < 2 && ok; ++h) {
          ok = mbar_wait_warp(&accfull[h], use & 1, abort_flag, p.spin);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (live && t * G + gt < nt) {
            const uint32_t ta = tq + (uint32_t)h * 128u;
            const float* Yh = Yb + gt * (kYBytes / 4) + h * 16;
#pragma unroll
            for (int i = 0; i < kEV; ++i) {
              const int v = 4 * i + og;
              if (v >= E) break;
              const int info = vinfo[v], np = info >> 16;
              float w[2][4];                       // [pair]
              tmem_ld4(w[0], ta + (uint32_t)(info & 255) * 4u);
              if (np > 1) tmem_ld4(w[1], ta + (uint32_t)((info >> 8) & 255) * 4u);
              tmem_wait<2>(w);
#pragma unroll
              for (int pr = 0; pr < 2; ++pr) {
                if (pr < np) {
                  const float4* y4 = reinterpret_cast<const float4*>(Yh + (2 * v + pr) * kYS);
#pragma unroll
                  for (int j = 0; j < 4; ++j) {
                    const float4 y = y4[j];
                    const float x = w[pr][j];
                    acc[i][0] += y.x * x;
                    acc[i][1] += y.y * x;
                    acc[i][2] += y.z * x;
                    acc[i][3] += y.w * x;
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
      if (ok && nl < rows) {
        const int n = r0 + nl, n0 = N > 128 ? 128 : 0, GX = tpp_max(N);
#pragma unroll
        for (int i = 0; i < kEV; ++i) {
          const int v = 4 * i + og;
          if (v < E) {
            float4* dst = part == 0 ? p.ent + add_off(gt, zl * p.nent + rec[3] + v, p.nz * p.nent, N, n0, n)
                                    : p.tail + (part - 1) * (size_t)p.nsplit * kMaxE * (N + (GX - 1) * (N - n0)) +
                                          add_off(gt, (item - p.split0) * kMaxE + v, p.nsplit * kMaxE, N, n0, n);
            *dst = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
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
      for (int blk = 0; blk < nblk; ++blk)
        ring_drain(filled[blk], stages32(N, blk, p.ring), [&](int s, uint32_t par) {
          for (int i = 0; i < kSpin && !mbar_try(&full[blk * kStagesMax + s], par); ++i) {
          }
        });
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  }
}

}  // namespace tc

int r2_f32_stages(int N) { return tc::stages32(N, 0, kMaxSmem - tc::smem32(N, 3)); }

using R2Kernel32 = void (*)(tc::Params);
static R2Kernel32 r2_f32_pick(int ip) { return ip == 2 ? tc::r2_f32_kernel<2> : tc::r2_f32_kernel<3>; }

int r2_f32_prepare(Ctx* c) {
  for (int ip = 2; ip <= 3; ++ip)
    PRD_CUDA_TRY(c, cudaFuncSetAttribute(r2_f32_pick(ip), cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem));
  return PRD_OK;
}

void r2_f32_launch(Ctx* c, tc::Params p, int grid) {
  const int ip = c->tc_bf16 ? 2 : 3, rest = tc::smem32(p.N, ip);
  // the caller's depth, or all there is for the ring (both row blocks' stages, up to kStagesMax)
  const int most = tc::kStagesMax * tc::kSteps * 128 * 64;
  p.ring = c->tc_stages >= 2 ? p.nst * tc::kSteps * 128 * 64 : std::min(most, (kMaxSmem - rest) / 1024 * 1024);
  r2_f32_pick(ip)<<<grid, tc::kThreads32, p.ring + rest, c->stream>>>(p);
}

}  // namespace prd
