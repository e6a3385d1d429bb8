// GEMM of prompts on pairs of CTAs (sm_100a, tcgen05 cta_group::2): Y[T][N] = X[T][K] W^T for the two 4-bit block formats and for
// fp16 matrices; fp16 operands (4-bit: w = rn16(scale * code), one rounding), fp32 accumulation.
//
// The weights are the A operand (M = 256 features, 128 per CTA), the tokens are the instruction's N (multiples of 16 up to 256, chosen from T; fp16
// weights also tiles of 512 tokens, two instructions).
// 4-bit weights are expanded into tensor memory: a thread of the sixteen dequantization warps turns 32-weight blocks of one
// feature (its lane) into sixteen columns each; nothing is stored to shared memory, no swizzle, no proxy fence.  (With the
// weights as a shared-memory operand a 64-k step of 256 features took about 1700 cycles, whatever the number of tokens, for the
// chain wait - store - fence - arrive that every warp went through in every step.)  fp16 weights go to shared memory by TMA.
//
// Unit of work: 128 k of a tile.  4-bit: codes and scales of a unit stream through a ring in shared memory by TMA (rows whose
// scales are not 16-byte aligned: 4-byte asynchronous copies), activations through another (each CTA loads half of the
// tokens), the expanded weights through `stages` slots of 64 tensor-memory columns.  fp16: one ring of 64-k steps, activations and
// weights together.  The leader's MMA warp issues for both CTAs.  Eight epilogue warps move the accumulator through shared memory
// to 16-byte stores (optionally + residual, or SwiGLU of 64 gate and 64 up features per CTA).  Two accumulators take turns where
// tensor memory has room (fp16 weights; tiles of at most 128 tokens), so that the epilogue of one runs under the MMAs of the next.
// The tensor core truncates what it adds to an accumulator, so long chains drift: where units_at_once says so, a stretch is
// added up in parts, rounding, in words of the scratch that belong to the thread that reads them back (two parts of a split tile: in an
// accumulator each, where there are two).
//
// Work division: the (feature tile, token tile) tiles go to the pairs (one CTA per SM, persistent) in waves of neighbours, which
// read the same weights and tokens from L2 at the same time (contiguous ranges of tiles per pair instead: 2048 tokens, fp16 gate
// and up 447 us against 346, 4096 x 14336 254 against 196).  The units of the tiles that are left for the last wave form one line
// of work that is cut into equal contiguous ranges.  A tile that falls into several of them is summed through fp32 partials in
// the scratch: every contributor leaves its part there, 32 tokens at a time; the last one to do so for these tokens adds the parts in
// ascending k order (so the result does not depend on who that is) and writes them.  Nobody waits for anybody.
//
// What bounds it: 4-bit, up to about 128 tokens, the MMA warp's chain among the expanding warps of its scheduler; a wait that is not known
// to be over when it begins costs 200 cycles: that is why the barriers are tested ahead and why activations come two units at a time.  A
// unit takes 0.32 to 0.39 us, of which the MMAs of 80 tokens are 0.16 and the expansion alone would be 0.16 (HBM 0.21).  The roles branch on a
// warp number that the compiler knows to be the same for the warp, and nothing in the MMA warp's loop looks as if lanes could differ: else
// every operand of every MMA is moved to a uniform register by itself, and eight MMAs and two commits take 180 cycles to issue where they
// take 80 (430 among the expanding warps; a unit 0.42 to 0.48 us; 77 tokens MXFP4, 28672 x 4096 31.5 -> 27.7 us, 512 tokens Q4, 4096 x 14336
// 59.2 -> 54.9).  fp16 there the weights' way from memory; with tiles for all pairs the MMAs and the power limit; with few tiles the launch
// (5 us and more: entry, the pair's meeting, first loads, output) and the sum of split tiles.  72 registers a thread are all that 896 threads
// leave: the compiler spills 96 to 104 bytes, in the epilogue's sums.
// Back to back on new weights, single-CTA kernel (with reduction, residual and SwiGLU launches) -> pairs:
//   77 tokens MXFP4: 28672 x 4096 with SwiGLU 66 -> 32 us, 4096 x 14336 41 -> 24
//   512 tokens Q4: gate and up 143 -> 91 us, 4096 x 14336 78 -> 60;  2048 tokens: gate and up 462 -> 328 to 351 (1372 TFLOP/s)
//   2048 tokens fp16: q, k, v 152 -> 78 us, o 66 -> 59, gate and up 451 -> 346 (1390 TFLOP/s)
//
// Roles per CTA: warp 0 = activation loads (fp16: and weights), warp 1 = tensor-memory allocation and (leader) MMA issue, warps 2, 3
// = code and scale loads, warps 4..11 = epilogue, warps 12..27 = dequantization: four groups of four.  Every mbarrier wait is
// bounded; on expiry the CTA raises the status word, skips the rest, and every thread still reaches the closing cluster barrier.
#include <cuda.h>

#include <cmath>

#include "gemm_tiles.cuh"

namespace ats {

namespace {

constexpr int kFeat = 128;                 // features per CTA
constexpr int kUnitK = 128;                // k per unit of work: 64 bytes of codes per row
constexpr int kMaxCodes = 12, kMaxX = 12;  // ring depths at most
constexpr int kCodeBytes = kFeat * 64;     // 8 KB
constexpr int kScaleBytes = kFeat * 16;    // per row: the eight scales of the 256-k line (or, unaligned, six halves)
constexpr int kStagePitch = 272;           // bytes per token of the output staging: 128 halves + 16
constexpr int kW16Bytes = kFeat * 128;     // fp16 weights of a 64-k step: 16 KB
constexpr int kW16StageTok = 64;           // tokens staged at a time with fp16 weights (the ring has the rest of shared memory)
enum { kFmtQ4 = 0, kFmtMx = 1, kFmtW16 = 2 };
constexpr int kPairThreads = 28 * 32;
constexpr int kMaxA = 4;                   // weight stages in tensor memory at most
constexpr int kMaxParts = 4;               // contributors of a split tile at most
constexpr uint32_t kColA = 256;            // tensor-memory columns: accumulator 0..255, weight stages from 256 on
constexpr uint32_t kClearPeer = 0xFEFFFFFFu;

struct PairParams : TileWork {  // (workers: pairs; units: 128 k)
  int ksteps;             // 64-k steps per tile
  int stages, codes, xs;  // depths of the rings: weights in tensor memory, codes (a multiple of it), activations
  int xu;             // units of activations that a place in their ring holds
  int sc16;           // scale rows are 16-byte aligned
  __half* y;          // (SwiGLU: may be null)
  int ldy;
  const __half* res;  // optional: y2 = rn16(res + y)
  __half* y2;
  int ldact;
  float* partial;     // slots of 2 * 128 features x slot_tok tokens
  int slot_tok;
  int slots2;         // a pair may leave a part of two tiles (ranges not cut at equal fractions of a tile)
  float* own;         // a further slot per pair: sums of a stretch in several parts
  int stage_tok;      // tokens that the staging holds: a multiple of 64, or all
  int max_units;      // units that one accumulator adds up at most
  int* counters;      // [2 * pairs], zero between launches
  int* status;
  unsigned long long grp_stride;
};

__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void pair_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void pair_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void pair_sync() {
  pair_arrive();
  pair_wait();
}
// arrival on the leader's copy of a barrier (from either CTA)
__device__ __forceinline__ void arrive_leader(uint64_t* own) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(smem_u32(own)));
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(a) : "memory");
}
__device__ __forceinline__ void tma_pair_2d(uint32_t one, uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* own_bar) {
  asm volatile(
      "{\n.reg .pred q;\nsetp.ne.b32 q, %5, 0;\n@q cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3}], [%4];\n}" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(smem_u32(own_bar) & kClearPeer), "r"(one)
      : "memory");
}
__device__ __forceinline__ void tma_pair_3d(uint32_t one, uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* own_bar) {
  asm volatile(
      "{\n.reg .pred q;\nsetp.ne.b32 q, %6, 0;\n@q cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4}], [%5];\n}" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(0), "r"(smem_u32(own_bar) & kClearPeer), "r"(one)
      : "memory");
}
__device__ __forceinline__ void umma_ts_pair(uint32_t one, uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.b32 p, %4, 0;\nsetp.ne.b32 q, %5, 0;\n@q tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(
          d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(one)
      : "memory");
}
__device__ __forceinline__ void umma_ss_pair(uint32_t one, uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.b32 p, %4, 0;\nsetp.ne.b32 q, %5, 0;\n@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(
          d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(one)
      : "memory");
}
// arrives on the same barrier of both CTAs when the pair's MMAs issued so far are done
__device__ __forceinline__ void umma_commit_both(uint32_t one, uint64_t* bar) {
  asm volatile(
      "{\n.reg .pred q;\n.reg .b16 m;\nmov.b16 m, 3;\nsetp.ne.b32 q, %1, 0;\n@q "
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], m;\n}" ::"r"(smem_u32(bar)),
      "r"(one)
      : "memory");
}
__device__ __forceinline__ void cp_async4z(uint32_t dst, const void* src, bool live) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(live ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
template <int N>
struct Int {
  static constexpr int value = N;
};
struct PairMaps {
  CUtensorMap codes[3], scales[3];  // of the segments (scales: where their rows are 16-byte aligned)
};
// Units that go into an accumulator before it is handed over: a stretch in equal parts of p.max_units at most.
__device__ __forceinline__ int seg_units(const PairParams& p, int n) {
  return n <= p.max_units ? n : (n + (n - 1) / p.max_units) / ((n + p.max_units - 1) / p.max_units);
}

template <int FMT>
__global__ void __launch_bounds__(kPairThreads, 1) gemm_pair_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ PairMaps wmap,
                                                                const __grid_constant__ PairParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t afull[kMaxA], aempty[kMaxA], xfull[kMaxX], xempty[kMaxX], cfull[kMaxCodes], cempty[kMaxCodes], acc_full[2], d_empty[2];
  __shared__ uint32_t tmem_s;
  __shared__ int last_s[2][4], n_blocks_s;
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // (the same for the warp, and known to be)
  const uint32_t rank = cta_rank();
  const int pair = blockIdx.x >> 1;
  const int S = p.stages, NC = p.codes, NX = p.xs;
  const int xbytes = p.nt / 2 * 128;                 // this CTA's activation bytes of a 64-k step
  uint8_t* x_s = smem;                               // [NX][2 xu][nt / 2 rows][128 bytes], swizzled
  const int step_bytes = xbytes + kW16Bytes;         // (fp16 weights: [NX] of a step's activations and weights, nothing else)
  uint8_t* code_s = x_s + (size_t)NX * (FMT == kFmtW16 ? step_bytes : p.xu * 2 * xbytes);   // [NC][128 rows][64 bytes], 16-byte pieces swizzled by row pair
  uint8_t* scale_s = code_s + (size_t)NC * kCodeBytes;
  uint8_t* out_s = scale_s + (size_t)NC * kScaleBytes;  // [nt][kStagePitch]
  // two accumulators that take turns: of 128 columns beside the weights, of 256 where those are not in tensor memory; a tile of 512
  // tokens (fp16 weights) is all 512 columns
  const bool wide = FMT == kFmtW16 && p.nt > 256;
  const bool two = FMT == kFmtW16 ? !wide : p.nt <= 128;
  constexpr uint32_t kAcc = FMT == kFmtW16 ? 256 : 128;
  const int sc_pitch = p.sc16 ? 16 : 12;

  if (warp == 4 && lane == 0) {
    prefetch_map(&xmap);
    for (int i = 0; i < p.n_seg; ++i) {
      prefetch_map(&wmap.codes[i]);
      if (p.sc16) prefetch_map(&wmap.scales[i]);
    }
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&afull[s], 8);      // (leader) four dequantization warps of each CTA
      mbar_init(&aempty[s], 1);
    }
    for (int s = 0; s < NX; ++s) {
      mbar_init(&xfull[s], 1);      // (leader) expect_tx
      mbar_init(&xempty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&acc_full[s], 1);
      mbar_init(&d_empty[s], 16);   // (leader) eight epilogue warps of each CTA
    }
    mbar_fence_init();
  }
  if (warp == 2 && lane == 0) {     // (the loaders' own barriers: they start before the CTAs have met)
    for (int s = 0; s < NC; ++s) {
      mbar_init(&cfull[s], p.sc16 ? 2 : 1 + 64);
      mbar_init(&cempty[s], 4);     // the warps of the stage's group
    }
    mbar_fence_init();
  }
  // The weights do not depend on the preceding kernel; the activations (and the grouped form's row offsets) do.  What the
  // epilogue touches is ordered behind the activation loads.  Whoever has something to wait for or to request does so between its arrival
  // and its wait for the other CTA (with the first requests ahead of the arrival the CTAs met 1.5 us later, and the activations were
  // requested another 2 us after that).
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_s)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  if (FMT != kFmtW16 && (warp == 2 || warp == 3)) asm volatile("bar.sync 2, 64;" ::: "memory");  // the loaders' barriers are initialised
  tc_fence_before();
  __syncwarp();
  pair_arrive();
  if ((warp == 0 && FMT != kFmtW16) || p.grp_off) asm volatile("griddepcontrol.wait;" ::: "memory");
  // Grouped form: every CTA lists the blocks of rows for itself from the experts' offsets.
  uint32_t* const blocks = reinterpret_cast<uint32_t*>(smem + p.list_at);
  int n_whole = p.n_whole;
  if (p.grp_off) {
    if (warp == 4) {
      const int n = list_blocks(p, blocks, lane);
      if (lane == 31) n_blocks_s = n;
    }
    __syncthreads();
    n_whole = n_blocks_s * p.ft_per;
  }
  // ---- code loads (warp 2) and scale loads (warp 3; both where the scales' rows are not 16-byte aligned).  Weights depend on nothing:
  // the first units are requested before the CTAs of the pair meet, the rest by the loaders' own branch below.
  bool ok = true;
  Stretch st;
  Walk ld_walk(p, pair, n_whole);
  int ld_n = 0, ld_u = 0, ld_end = 0, ld_cs = 0;   // units requested; next and last unit of the current stretch; ring place
  int ld_first = 0, ld_e = 0, ld_sa = 0, ld_sb = 0;
  uint32_t ld_par = 1;
  auto load_units = [&](int upto) {
    const uint32_t one = elect_one();
    const int half_k = p.K / 2, nblk = p.K / 32;
    while (ld_n < upto) {
      if (ld_u == ld_end) {
        if (!uniform(ld_walk.next(st))) return;
        const Tile tl = tile_of(p, st.tile, blocks);
        ld_u = uniform(st.u0);
        ld_end = uniform(st.u1);
        ld_e = uniform(tl.expert);
        ld_sa = p.act ? 0 : uniform(tl.sg);
        ld_sb = p.act ? 1 : ld_sa;
        ld_first = uniform(p.act ? tl.row0 + (int)rank * 64 : tl.row0 + (int)rank * kFeat);
      }
      if (ld_n >= NC) {
        ok = wait_warp(&cempty[ld_cs], ld_par);
        if (!ok) return;
      }
      uint64_t* bar = &cfull[ld_cs];
      const uint32_t sdst = smem_u32(scale_s) + (uint32_t)(ld_cs * kScaleBytes);
      const int second = p.act ? ld_first : ld_first + 64;
      // (two warps: one alone needed 770 cycles per unit for its four loads, as long as the unit takes at 16 tokens; 18944 x 14336
      // 59.8 -> 56.7 us)
      if (warp == 2) {  // rows beyond the matrix and k beyond its end read as zeros
        const uint32_t dst = smem_u32(code_s) + (uint32_t)(ld_cs * kCodeBytes);
        expect_tx_one(one, bar, (uint32_t)kCodeBytes);
        tma_3d_one(one, dst, &wmap.codes[ld_sa], ld_u * 64, ld_first, ld_e, bar);
        tma_3d_one(one, dst + kCodeBytes / 2, &wmap.codes[ld_sb], ld_u * 64, second, ld_e, bar);
      } else if (p.sc16) {  // (a line of eight scales serves two units: 16 bytes are the least that a copy takes)
        expect_tx_one(one, bar, (uint32_t)kScaleBytes);
        tma_3d_one(one, sdst, &wmap.scales[ld_sa], (ld_u >> 1) * 8, ld_first, ld_e, bar);
        tma_3d_one(one, sdst + kScaleBytes / 2, &wmap.scales[ld_sb], (ld_u >> 1) * 8, second, ld_e, bar);
      }
      if (!p.sc16) {
        // six halves of each row from the 4-byte boundary at or below the unit's first scale; the reader skips the odd one.
        // Words that begin beyond the matrix's scales are not read.
        const int l = (warp - 2) * 32 + lane, rows = p.seg[ld_sa].n_rows;
        const size_t hi = (size_t)rows * nblk * 2;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int gr = (j ? second : ld_first) + l;
          const bool live = gr < rows;
          const uint8_t* sc = p.seg[j ? ld_sb : ld_sa].base + (unsigned long long)ld_e * p.grp_stride + (size_t)rows * half_k;
          const size_t lo = (((size_t)(live ? gr : 0) * nblk + ld_u * 4) * 2) & ~(size_t)3;
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const bool in = live && lo + 4 * q < hi;
            cp_async4z(sdst + (uint32_t)((l + 64 * j) * 12 + 4 * q), sc + (in ? lo + 4 * q : 0), in);
          }
        }
        cp_async_arrive(bar);
      }
      ++ld_n;
      ++ld_u;
      if (++ld_cs == NC) ld_cs = 0, ld_par ^= 1u;
    }
  };
  if (FMT != kFmtW16 && (warp == 2 || warp == 3)) load_units(min(4, NC));
  __syncwarp();
  pair_wait();
  tc_fence_after();
  const uint32_t tmem = tmem_s;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // 72 registers a thread at launch; the epilogue's sums need more: 56 + 4 x 64 + 2 x 96 = 7 x 72
  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    if (warp == 0) {
      // ------------------------------------------------------------ activations
      const uint32_t one = elect_one();
      Walk mine(p, pair, n_whole);
      const uint32_t x0 = smem_u32(x_s);
      int s = 0, n = 0;
      uint32_t par = 1;
      while (uniform(ok && mine.next(st))) {
        const Tile tl = tile_of(p, st.tile, blocks);
        const int u0 = uniform(st.u0), u1 = uniform(st.u1);
        const int row = uniform(tl.rowoff + tl.t0 + (int)rank * (p.nt / 2));
        if constexpr (FMT == kFmtW16) {
          const int sa = p.act ? 0 : uniform(tl.sg), sb = p.act ? 1 : sa;
          const int wa = uniform(tl.row0 + (int)rank * (p.act ? 64 : kFeat)), wb = p.act ? wa : wa + 64;
          const int k1 = min(2 * u1, p.ksteps);
          auto weights = [&](int ks, int place) {
            const uint32_t dw = x0 + (uint32_t)(place * step_bytes + xbytes);
            if (rank == 0) expect_tx_one(one, &xfull[place], (uint32_t)(2 * step_bytes));
            tma_pair_3d(one, dw, &wmap.codes[sa], ks * 64, wa, &xfull[place]);
            tma_pair_3d(one, dw + kW16Bytes / 2, &wmap.codes[sb], ks * 64, wb, &xfull[place]);
          };
          // The weights of the first steps do not wait for the preceding kernel, their activations do (18944 x 1024, 32 tokens 11.9 -> 10.6 us).
          const int ahead = n == 0 ? min(NX, k1 - 2 * u0) : 0;
          if (n == 0) {
            for (int i = 0; i < ahead; ++i) weights(2 * u0 + i, i);
            asm volatile("griddepcontrol.wait;" ::: "memory");
          }
          for (int ks = 2 * u0; ks < k1; ++ks) {
            if (n >= NX && !wait_warp(&xempty[s], par)) {
              ok = false;
              break;
            }
            ++n;
            if (ks - 2 * u0 >= ahead) weights(ks, s);
            const uint32_t dst = x0 + (uint32_t)(s * step_bytes);
            // (wide: tokens 128 rank .. of each half of the tile, so that either half is one operand of the pair)
            tma_pair_2d(one, dst, &xmap, ks * 64, wide ? row - (int)rank * 128 : row, &xfull[s]);
            if (wide) tma_pair_2d(one, dst + (uint32_t)(xbytes / 2), &xmap, ks * 64, row - (int)rank * 128 + 256, &xfull[s]);
            if (++s == NX) s = 0, par ^= 1u;
          }
          continue;
        }
        auto load = [&](auto units_of_a_place) {
          constexpr int XU = decltype(units_of_a_place)::value;
          for (int u = u0; u < u1; u += XU) {
            if (n >= NX && !wait_warp(&xempty[s], par)) {
              ok = false;
              break;
            }
            ++n;
            const int n_ks = min(2 * min(u + XU, u1), p.ksteps) - 2 * u;
            const uint32_t dst = x0 + (uint32_t)(s * XU * 2 * xbytes);
            if (rank == 0) expect_tx_one(one, &xfull[s], (uint32_t)(n_ks * 2 * xbytes));
#pragma unroll
            for (int j = 0; j < 2 * XU; ++j)
              if (j < n_ks) tma_pair_2d(one, dst + (uint32_t)(j * xbytes), &xmap, u * 128 + j * 64, row, &xfull[s]);
            if (++s == NX) s = 0, par ^= 1u;
          }
        };
        if (p.xu == 2) load(Int<2>{});
        else load(Int<1>{});
      }
    } else if (warp == 1) {
      // ------------------------------------------------------------ MMA issue (leader)
      // (the units of a place as a constant: with one of them to a place the loop has nothing to count.  18944 x 6144 over 160 tokens 37.4 -> 36.7
      // us, over 132 35.4 -> 34.6)
      auto issue = [&](auto units_of_a_place) {
        constexpr int XU = decltype(units_of_a_place)::value;
        const uint32_t one = elect_one();
        const uint32_t idesc = umma_idesc_f16(2 * kFeat, wide ? 256 : p.nt);
        const uint64_t xd = umma_desc_sw128(smem_u32(x_s));
        Walk mine(p, pair, n_whole);
        int s = 0, sx = 0, xi = 0, seg = 0;  // places in the rings, unit of the activations' place, accumulator segments so far
        uint32_t par = 0, parx = 0;
        bool ready = false, readyx = false;
        while (uniform(mine.next(st))) {
          const int u0 = uniform(st.u0), u1 = uniform(st.u1);
          int left = 0;  // units until the accumulator is handed over
          uint32_t d = 0, accumulate = 0;
          const int part = seg_units(p, u1 - u0);
          for (int u = u0; u < u1; ++u) {
            if (left == 0) {
              left = min(part, u1 - u);
              accumulate = 0;
              const int b = two ? seg & 1 : 0, use = two ? seg >> 1 : seg;
              d = kAcc * b;
              if (use > 0 && !wait_warp(&d_empty[b], (use - 1) & 1)) return false;
            }
            if constexpr (FMT == kFmtW16) {
              for (int ks = 2 * u; ks < min(2 * u + 2, p.ksteps); ++ks) {
                if (!__all_sync(0xffffffffu, readyx) && !wait_warp(&xfull[sx], parx)) return false;
                tc_fence_after();
                const int sxn = sx + 1 == NX ? 0 : sx + 1;
                const uint32_t parxn = sx + 1 == NX ? parx ^ 1u : parx;
                readyx = peek(&xfull[sxn], parxn);
                const uint64_t bd = xd + (uint64_t)((uint32_t)sx * (uint32_t)(step_bytes >> 4)), ad = bd + (uint64_t)(xbytes >> 4);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                  umma_ss_pair(one, d, ad + (uint64_t)(2 * kk), bd + (uint64_t)(2 * kk), idesc, kk > 0 ? 1u : accumulate);
                if (wide) {
#pragma unroll
                  for (int kk = 0; kk < 4; ++kk)
                    umma_ss_pair(one, d + 256u, ad + (uint64_t)(2 * kk), bd + (uint64_t)((xbytes >> 5) + 2 * kk), idesc, kk > 0 ? 1u : accumulate);
                }
                accumulate = 1;
                umma_commit_both(one, &xempty[sx]);
                sx = sxn, parx = parxn;
              }
              if (--left == 0) {
                umma_commit_both(one, &acc_full[two ? seg & 1 : 0]);
                ++seg;
              }
              continue;
            }
            if (!__all_sync(0xffffffffu, ready) && !wait_warp(&afull[s], par)) return false;
            if (xi == 0 && !__all_sync(0xffffffffu, readyx) && !wait_warp(&xfull[sx], parx)) return false;
            tc_fence_after();
            const int sn = s + 1 == S ? 0 : s + 1, sxn = sx + 1 == NX ? 0 : sx + 1;
            const uint32_t parn = s + 1 == S ? par ^ 1u : par, parxn = sx + 1 == NX ? parx ^ 1u : parx;
            const bool xlast = xi + 1 == XU || u + 1 == u1;  // the place in the activations' ring is done with
            ready = peek(&afull[sn], parn);
            if (xlast) readyx = peek(&xfull[sxn], parxn);
            const uint64_t bd = xd + (uint64_t)((uint32_t)(sx * XU + xi) * 2u * (uint32_t)(xbytes >> 4));
            const uint32_t at = kColA + 64u * s;  // (all 512 columns are this CTA's: the allocation starts at 0)
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) umma_ts_pair(one, d, at + 8u * kk, bd + (uint64_t)(2 * kk), idesc, kk > 0 ? 1u : accumulate);
            if (2 * u + 1 < p.ksteps) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                umma_ts_pair(one, d, at + 32u + 8u * kk, bd + (uint64_t)((uint32_t)(xbytes >> 4) + 2 * kk), idesc, 1);
            }
            accumulate = 1;
            umma_commit_both(one, &aempty[s]);
            if (xlast) umma_commit_both(one, &xempty[sx]);
            if (--left == 0) {
              umma_commit_both(one, &acc_full[two ? seg & 1 : 0]);
              ++seg;
            }
            s = sn, par = parn;
            xi = xlast ? 0 : xi + 1;
            if (xlast) sx = sxn, parx = parxn;
          }
        }
        return true;
      };
      if (rank == 0) {
        if (FMT != kFmtW16 && p.xu == 2) ok = issue(Int<2>{});
        else ok = issue(Int<1>{});
      }
    } else {
      // ------------------------------------------------------------ code and scale loaders, continued
      if (FMT != kFmtW16) load_units(0x7fffffff);
      asm volatile("cp.async.wait_all;" ::: "memory");
    }
  } else if (warp >= 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    // ------------------------------------------------------------ dequantization: thread = (feature, one 32-k block of a step)
    // Four groups of four warps, one for each weight stage, so that four of these chains of latencies (barrier, shared memory,
    // arithmetic, tensor-memory store, barrier) run side by side.  A group takes every S-th unit; the code ring's depth is a
    // multiple of S, so every barrier belongs to one group (a phase's parity says which one it is only to a waiter that has
    // seen the one before).
    const int quarter = warp & 3, grp = (warp - 12) >> 2;
    const int row = quarter * 32 + lane;
    const int nblk = p.K / 32;
    const uint32_t a_col = tmem + ((uint32_t)(quarter * 32) << 16) + kColA + 64u * grp;
    const uint32_t code_row = smem_u32(code_s) + (uint32_t)(row * 64), scale_row = smem_u32(scale_s) + (uint32_t)(row * sc_pitch);
    const uint32_t swz = (uint32_t)((row >> 1) & 3) << 4;
    Walk mine(p, pair, n_whole);
    int skip = grp;               // units until this group's next
    int cs = grp;                 // its place in the code ring
    uint32_t cpar = 0, apar = 1;  // (the first wait for an empty stage passes at once)
    while (FMT != kFmtW16 && ok && grp < S && mine.next(st)) {
      int odd = 0;
      if (!p.sc16) {  // units start at even offsets: the row decides
        const Tile tl = tile_of(p, st.tile, blocks);
        odd = ((p.act ? tl.row0 + (int)rank * 64 + (row & 63) : tl.row0 + (int)rank * kFeat + row) & nblk) & 1;
      }
      int u = st.u0 + skip;
      for (; u < st.u1; u += S) {
        if (!wait_warp(&cfull[cs], cpar)) {
          ok = false;
          break;
        }
        const bool free_seen = peek(&aempty[grp], apar);
        const uint32_t cr = code_row + (uint32_t)(cs * kCodeBytes), sr = scale_row + (uint32_t)(cs * kScaleBytes);
        uint2 sw;  // four scales
        if (p.sc16) {
          sw = lds64(sr + (uint32_t)(u & 1) * 8);
        } else {
          const uint32_t w0 = lds32(sr), w1 = lds32(sr + 4), w2 = lds32(sr + 8);
          sw = odd ? make_uint2(__byte_perm(w0, w1, 0x5432), __byte_perm(w1, w2, 0x5432)) : make_uint2(w0, w1);
          const int left = nblk - u * 4;  // blocks that exist; what follows belongs to the next row
          if (left < 4) sw.y &= left < 3 ? 0u : 0x0000FFFFu;
          if (left < 2) sw.x &= 0x0000FFFFu;
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t o[32];
          const uint32_t pairs = c ? sw.y : sw.x;
#pragma unroll
          for (int b = 0; b < 2; ++b) {
            const uint4 q = lds128(cr + (((uint32_t)(2 * c + b) << 4) ^ swz));
            const __half2 sc = as_h2(__byte_perm(pairs, 0, b ? 0x3232 : 0x1010));
            expand_word<FMT == kFmtMx>(q.x, sc, o + 16 * b);
            expand_word<FMT == kFmtMx>(q.y, sc, o + 16 * b + 4);
            expand_word<FMT == kFmtMx>(q.z, sc, o + 16 * b + 8);
            expand_word<FMT == kFmtMx>(q.w, sc, o + 16 * b + 12);
          }
          if (c == 0) {
            if (!__all_sync(0xffffffffu, free_seen) && !wait_warp(&aempty[grp], apar)) {
              ok = false;
              break;
            }
            tc_fence_after();
          }
          tmem_st_x32(a_col + 32u * c, o);
        }
        if (!ok) break;
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          arrive_leader(&afull[grp]);
          mbar_arrive(&cempty[cs]);
        }
        apar ^= 1u;
        cs += S;
        if (cs >= NC) cs -= NC, cpar ^= 1u;
      }
      skip = u - st.u1;
    }
  } else {
    // ------------------------------------------------------------ epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 96;");
    const int quarter = warp & 3;
    const int half = (warp - 4) >> 2;        // two warps per quarter: even and odd runs of 32 tokens
    const int tid = threadIdx.x - 128;       // 0..255
    const int feat = quarter * 32 + lane;    // this thread's feature of the CTA's 128
    const uint32_t d_col = tmem + ((uint32_t)(quarter * 32) << 16), out_u = smem_u32(out_s);
    auto epi_sync = [] { asm volatile("bar.sync 1, 256;" ::: "memory"); };
    auto epi_all = [](bool v) {
      uint32_t r;
      asm volatile("{\n.reg .pred a, b;\nsetp.ne.u32 a, %1, 0;\nbarrier.cta.red.and.pred b, 1, 256, a;\nselp.u32 %0, 1, 0, b;\n}"
                   : "=r"(r)
                   : "r"((uint32_t)v)
                   : "memory");
      return r != 0;
    };
    Walk mine(p, pair, n_whole);
    int seg = 0;
    while (ok && mine.next(st)) {
      const Tile tl = tile_of(p, st.tile, blocks);
      const int ntok = min(p.nt, tl.T - tl.t0);
      // ---- all parts but the last of the stretch: added up in this thread's own words of the scratch
      const int n = st.u1 - st.u0, part = seg_units(p, n), n_part = part == n ? 1 : (n + part - 1) / part;
      // (two parts of a split tile meet in tensor memory, one in each accumulator, without a way through the scratch: 6144 x 4096 over 77 tokens
      // 17.8 -> 16.3 us, 4096 x 4096 16.2 -> 14.5; a whole tile's first part makes room for the next tile instead)
      const bool meet = two && n_part == 2 && n < p.units;
      uint32_t col = 0, col0 = 0;
      float* own = p.own + (size_t)blockIdx.x * kFeat * p.slot_tok + feat;
      auto add_own = [&](float* v, int c0, auto n_tok) {  // (all loads before the first addition)
        constexpr int NT = decltype(n_tok)::value;
        float w[NT];
#pragma unroll
        for (int i = 0; i < NT; ++i) w[i] = c0 + i < ntok ? __ldcg(own + (size_t)(c0 + i) * kFeat) : 0.f;
#pragma unroll
        for (int i = 0; i < NT; ++i) v[i] += w[i];
      };
      for (int g = 0; g < n_part; ++g, ++seg) {
        const int b = two ? seg & 1 : 0, use = two ? seg >> 1 : seg;
        if (meet && g == 0) {
          col0 = d_col + kAcc * b;
          continue;
        }
        bool got = true;  // (one warp polls, the others sleep at the barrier: polls take issue slots from the expansion)
        if (warp == 4) got = wait_warp(&acc_full[b], use & 1);
        ok = epi_all(got);
        if (!ok) break;
        tc_fence_after();
        col = d_col + kAcc * b;
        if (g + 1 == n_part) break;
        // (16 tokens at a time: the registers of 32 sums and their 32 words are not there, and what is spilled is fetched one after the other
        // while the MMAs wait for the accumulator.  5376 x 7680 over 438 tokens, three parts: 41.7 -> 41.2 us)
#pragma unroll 1
        for (int c = 32 * half; c < ntok; c += c & 16 ? 48 : 16) {
          float v[16];
          tmem_ld_x16(col + c, reinterpret_cast<uint32_t*>(v));
          tmem_ld_wait_x16(reinterpret_cast<uint32_t*>(v));
          if (g) add_own(v, c, Int<16>{});
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (c + i < ntok) __stcg(own + (size_t)(c + i) * kFeat, v[i]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_leader(&d_empty[b]);
      }
      if (!ok) break;
      const int last_b = two ? seg & 1 : 0;
      ++seg;
      auto stage = [&](const float* v, auto n_tok, int row) {  // this thread's feature of n_tok tokens
        const uint32_t o = out_u + (uint32_t)(row * kStagePitch + 2 * feat);
#pragma unroll
        for (int i = 0; i < decltype(n_tok)::value; ++i) sts16(o + (uint32_t)(i * kStagePitch), __float2half_rn(v[i]));
      };
      // The staged tokens h0 .. h1-1 (rows row0 ..) to memory, by N threads.
      auto write_out = [&](auto n_thr, int id, int h0, int h1, int row0) {
        constexpr int N = decltype(n_thr)::value;
        const uint32_t rows = out_u + (uint32_t)(row0 * kStagePitch);
        const size_t trow = (size_t)tl.rowoff + tl.t0;
        if (p.act) {
          const int F = p.seg[0].n_rows, f0 = tl.row0 + (int)rank * 64;
          const int c = (id & 7) * 8;
          const int live = F - f0 - c;  // F is a multiple of 8: a run of eight is live or not
          if (live > 0) {
#pragma unroll 2
            for (int t = h0 + (id >> 3); t < h1; t += N / 8) {
              const uint4 g4 = lds128(rows + (uint32_t)((t - h0) * kStagePitch + c * 2));
              const uint4 u4 = lds128(rows + (uint32_t)((t - h0) * kStagePitch + 128 + c * 2));
              const uint32_t gw[4] = {g4.x, g4.y, g4.z, g4.w}, uw[4] = {u4.x, u4.y, u4.z, u4.w};
              uint32_t a[4];
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const float2 g = __half22float2(as_h2(gw[q])), u = __half22float2(as_h2(uw[q]));
                a[q] = as_u32(__floats2half2_rn(silu_times(g.x, u.x), silu_times(g.y, u.y)));
              }
              *reinterpret_cast<uint4*>(p.act + (trow + t) * p.ldact + f0 + c) = make_uint4(a[0], a[1], a[2], a[3]);
              if (p.y) {
                *reinterpret_cast<uint4*>(p.y + (trow + t) * p.ldy + f0 + c) = g4;
                *reinterpret_cast<uint4*>(p.y + (trow + t) * p.ldy + F + f0 + c) = u4;
              }
            }
          }
          return;
        }
        const int r0 = tl.row0 + (int)rank * kFeat;
        const int live = min(kFeat, p.seg[tl.sg].n_rows - r0);
        const int colbase = p.seg[tl.sg].col0 + r0;
        const bool vec = (p.ldy % 8 == 0) && (colbase % 8 == 0) &&
                         (((reinterpret_cast<uintptr_t>(p.y) | reinterpret_cast<uintptr_t>(p.res) | reinterpret_cast<uintptr_t>(p.y2)) & 15) == 0);
        const int c = (id & 15) * 8;
        if (vec && c + 8 <= live) {
          for (int tb = h0 + (id >> 4); tb < h1; tb += N / 4) {
            // four tokens at a time, their residuals requested before anything is stored
            uint4 r4[4];
            if (p.res) {
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (tb + N / 16 * q < h1) r4[q] = __ldg(reinterpret_cast<const uint4*>(p.res + (trow + tb + N / 16 * q) * p.ldy + colbase + c));
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int t = tb + N / 16 * q;
              if (t >= h1) break;
              const uint4 o4 = lds128(rows + (uint32_t)((t - h0) * kStagePitch + c * 2));
              const size_t off = (trow + t) * p.ldy + colbase + c;
              *reinterpret_cast<uint4*>(p.y + off) = o4;
              if (p.res) {
                const uint32_t ow[4] = {o4.x, o4.y, o4.z, o4.w}, rw[4] = {r4[q].x, r4[q].y, r4[q].z, r4[q].w};
                uint32_t z[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const float2 a = __half22float2(as_h2(ow[e])), b = __half22float2(as_h2(rw[e]));
                  z[e] = as_u32(__floats2half2_rn(b.x + a.x, b.y + a.y));
                }
                *reinterpret_cast<uint4*>(p.y2 + off) = make_uint4(z[0], z[1], z[2], z[3]);
              }
            }
          }
        } else if (c < live) {
          for (int t = h0 + (id >> 4); t < h1; t += N / 16) {
            const __half* o = reinterpret_cast<const __half*>(out_s + (size_t)(row0 + t - h0) * kStagePitch) + c;
            const size_t off = (trow + t) * p.ldy + colbase + c;
            for (int q = 0; q < min(8, live - c); ++q) {
              p.y[off + q] = o[q];
              if (p.res) p.y2[off + q] = __float2half_rn(__half2float(p.res[off + q]) + __half2float(o[q]));
            }
          }
        }
      };
      if (st.u0 == 0 && st.u1 == p.units) {  // a whole tile, as many tokens at a time as the staging holds
        for (int h0 = 0; h0 < ntok; h0 += p.stage_tok) {
          const int h1 = min(h0 + p.stage_tok, ntok);
#pragma unroll 1
          for (int c0 = h0 + 32 * half; c0 < h1; c0 += 64) {
            float v[32];
            tmem_ld_x32(col + c0, reinterpret_cast<uint32_t*>(v));
            tmem_ld_wait_x32(reinterpret_cast<uint32_t*>(v));
            if (n_part > 1) add_own(v, c0, Int<32>{});
            stage(v, Int<32>{}, c0 - h0);
          }
          if (h1 == ntok) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_leader(&d_empty[last_b]);  // the accumulator may be overwritten
          }
          epi_sync();
          write_out(Int<256>{}, tid, h0, h1, 0);
          epi_sync();  // the staging may be filled again
        }
        continue;
      }
      // ---- A split tile.  Its contributors are the pairs whose ranges meet it: pair q holds units n q / P .. n (q + 1) / P - 1, so unit u
      // lies with q = ((u + 1) P - 1) / n.  Each leaves its part in the scratch, 32 tokens at a time, and counts itself in for these
      // tokens; the last one to do so adds their parts up in ascending k order and writes them.  The contributors, which finish at
      // about the same time, begin with different tokens, so that each is the last for some of them (4-bit, 4096 x 14336 in four parts: 77
      // tokens 28.6 -> 25.1 us, 256 tokens in two parts 46.9 -> 40.2, against one contributor that sums the whole tile).  The warps of even
      // and odd runs of tokens go their own ways.
      const unsigned n_units = (unsigned)(p.n_ft * p.n_tt - p.n_whole) * p.units, lo = (unsigned)(st.tile - p.n_whole) * p.units;
      const int first = (int)(((lo + 1) * p.split_workers - 1) / n_units);
      const int n_con = (int)(((lo + p.units) * p.split_workers - 1) / n_units) - first + 1;
      auto part_of = [&](int q) {  // this CTA's half of what pair q leaves of the tile
        // (the first contributor begins the tile, the others come upon it at the start of their range)
        return p.partial + ((size_t)(p.slots2 && q == first ? p.split_workers + q : q) * 2 + rank) * kFeat * p.slot_tok + feat;
      };
      auto half_sync = [&] { asm volatile("bar.sync %0, 128;" ::"r"(3 + half) : "memory"); };
      unsigned* cnt = reinterpret_cast<unsigned*>(p.counters) + 2 * first + rank;  // four bits for every 32 tokens
      const int n_run = ((ntok + 31) / 32 - half + 1) / 2;  // runs of this half
      const int turn = (pair - first) * n_run / n_con;
      {
        float* dst = part_of(pair);
        uint32_t prev = 0;
        int mine_j = -1;
#pragma unroll 1
        for (int i = 0; i < n_run; ++i) {
          const int j = turn + i < n_run ? turn + i : turn + i - n_run, c0 = 64 * j + 32 * half;
          float v[32];
          tmem_ld_x32(col + c0, reinterpret_cast<uint32_t*>(v));
          tmem_ld_wait_x32(reinterpret_cast<uint32_t*>(v));
          if (meet) {
#pragma unroll
            for (int h = 0; h < 32; h += 16) {
              float w[16];
              tmem_ld_x16(col0 + c0 + h, reinterpret_cast<uint32_t*>(w));
              tmem_ld_wait_x16(reinterpret_cast<uint32_t*>(w));
#pragma unroll
              for (int t = 0; t < 16; ++t) v[h + t] += w[t];
            }
          } else if (n_part > 1) {
            add_own(v, c0, Int<32>{});
          }
#pragma unroll
          for (int t = 0; t < 32; ++t)
            if (c0 + t < ntok) __stcg(dst + (size_t)(c0 + t) * kFeat, v[t]);
          half_sync();  // the run's words are written: one thread releases them (another warp's each time: nobody waits for the count)
          if (quarter == i && lane == 0) {
            mine_j = j;
            asm volatile("atom.add.release.gpu.global.u32 %0, [%1], %2;" : "=r"(prev) : "l"(cnt), "r"(1u << (4 * (2 * j + half))) : "memory");
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_leader(&d_empty[last_b]);  // the accumulator may be overwritten
        if (lane == 0 && meet) arrive_leader(&d_empty[last_b ^ 1]);
        if (mine_j >= 0) {
          const int at = 4 * (2 * mine_j + half);
          const bool last = ((prev >> at) & 15u) == (uint32_t)(n_con - 1);
          asm volatile("fence.acq_rel.gpu;" ::: "memory");
          if (last) atomicSub(cnt, (uint32_t)n_con << at);  // ready for the next launch
          last_s[half][mine_j] = last;
        }
        half_sync();
      }
#pragma unroll 1
      for (int j = 0; j < n_run; ++j) {
        if (!last_s[half][j]) continue;
        const int c0 = 64 * j + 32 * half, c1 = min(c0 + 32, ntok), row = 32 * half;
#pragma unroll 1
        for (int h = c0; h < c1; h += 16) {
          float v[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = 0.f;
#pragma unroll 1
          for (int q = 0; q < n_con; q += 2) {  // two parts' words on their way at a time
            const float *s0 = part_of(first + q) + (size_t)h * kFeat, *s1 = part_of(first + min(q + 1, n_con - 1)) + (size_t)h * kFeat;
            float w0[16], w1[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              w0[i] = h + i < ntok ? __ldcg(s0 + i * kFeat) : 0.f;
              w1[i] = h + i < ntok && q + 1 < n_con ? __ldcg(s1 + i * kFeat) : 0.f;
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = (v[i] + w0[i]) + w1[i];
          }
          stage(v, Int<16>{}, row + h - c0);
        }
        half_sync();
        write_out(Int<128>{}, tid & 127, c0, c1, row);
        half_sync();  // the staging may be filled again
      }
      epi_sync();
    }
  }
  __syncwarp();
  if (!ok && lane == 0) raise_status(p.status, 3);
  __syncwarp();
  // nobody leaves or frees tensor memory while the partner may still read or signal it
  tc_fence_before();
  pair_sync();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// ------------------------------------------------------------------------------------------------- host side
// Units that one accumulator adds up at most.  The tensor core truncates each sum, and what a chain drops grows with its
// length: of the fp16 results 0.5 % differ from the exact sum's rounding after 1024 k, 1.7 % after 4096, 5 % after 14336.  So no
// chain is longer (by more than part of a unit) than the single-CTA kernel's for the same product (fp16: for each matrix by itself, as that
// kernel takes them), except that 1536 k are allowed where plan_of says so (`longer`), and fp16 matrices of enough large tiles (112 CTAs of 256 features x 256
// tokens) are added up in one.
int units_at_once(const int* rows, int n_seg, int T, int K, bool w16, bool longer) {
  int chain = K;
  for (int i = 0; w16 && i < n_seg; ++i)
    if (T < 384 || (rows[i] + 255) / 256 * ((T + 511) / 512) < 56) chain = std::min(chain, gemm_chain(rows + i, 1, T, K));
  if (!w16) chain = gemm_chain(rows, n_seg, T, K);
  return ((longer ? std::max(1536, chain) : chain) + kUnitK - 1) / kUnitK;
}
// Feature tiles of a segment (fused SwiGLU: a tile is 128 gate and 128 up rows, all counted with the gate).
int feature_tiles(const int* rows, int seg, bool act) {
  return act ? (seg ? 0 : (rows[0] + kFeat - 1) / kFeat) : (rows[seg] + 2 * kFeat - 1) / (2 * kFeat);
}

// Time in us of the ways to divide the work (see the kernel's comment).  A unit costs its MMAs, the expansion of its weights
// or their way from memory, whichever is longest; a tile its epilogue; a stretch that is added up in several parts their way out and
// back, less where the MMAs go on meanwhile in the other accumulator; a split tile the parts' way through L2.  The figures are fitted
// to launches back to back on new weights: the 4-bit formats' to 330, 14 shapes of 6 to 66 MB, 12 to 1000 tokens, in the ways that come
// within a third of the best (6 % rms off; many waves run 8 % slower, at the power limit; later 8 products whose contributors have several parts,
// 6144 x 4096 over 160 tokens among them, taken at 21.4 us for 24.2, where the single-CTA kernel needs 22.5), fp16's to about 400 with the sums
// of split tiles as they were when one contributor made them (10 %).  pairs = 0: the scratch holds none.
GemmPairPlan pair_plan(const int* rows, int n_seg, bool act, int T, int K, bool w16, bool longer, int max_pairs, uint64_t scratch_bytes) {
  GemmPairPlan best{};
  best.us = 1e300;
  int n_ft = 0;
  for (int i = 0; i < n_seg; ++i) n_ft += feature_tiles(rows, i, act);
  const int units = (K + kUnitK - 1) / kUnitK, max_units = units_at_once(rows, n_seg, T, K, w16, longer);
  double weights_mb = 0;
  for (int i = 0; i < n_seg; ++i) weights_mb += 2e-6 * rows[i] * K;
  int last = 0;
  for (int most : {512, 256, 192, 128}) {
    const int n_tt = (T + most - 1) / most;
    if (most == 512 ? !w16 || T <= 256 || n_ft * n_tt > max_pairs : n_tt == last) continue;
    last = most == 512 ? 0 : n_tt;
    const int nt = most == 512 ? 512 : ((T + n_tt - 1) / n_tt + 15) / 16 * 16;
    const uint64_t slot = 2ull * kFeat * std::min(nt, T) * 4;
    // (fp16 tiles of 512 tokens: the weights serve two operands, but nothing runs under the epilogue and the ring is four steps deep.  Where
    // they make one wave they are the faster ones: 4096 x 14336 over 2048 tokens 204 -> 186 us, 14336 x 4096 over 512 67 -> 55; in several
    // waves they are not: 28672 x 4096 over 3000 tokens 527 -> 649.  fp16 weights that several token tiles share come out of L2 for all but
    // one)
    const double unit = w16 ? std::max(n_tt > 1 ? 0.55 : 0.729, nt == 512 ? 1.55 : 0.40 + 0.00165 * nt) : std::max(0.416, 0.155 + 0.0020 * nt) * (n_ft * n_tt >= 4 * max_pairs ? 1.08 : 1.0);
    const double launch = w16 ? 5.0 : 4.9, tile = w16 ? (nt == 512 ? 6.0 : 0.0) : 0.0077 * nt;
    const double flush = w16 ? 1.1 : std::max(0.3, 0.0284 * nt - 1.56);
    const int tok = std::min(nt, T), batches = tok <= 16 ? 1 : (tok + 63) / 64 * 2;  // (16 tokens a batch and warp, two warps side by side)
    // (slots: of a split tile.  Its contributors' parts come back from the scratch in the way of the sum, where they do not meet in tensor
    // memory; those that do cost less than `flush`, which is not counted on: near the line the single-CTA kernel keeps what it had)
    auto stretch = [&](double len, int slots) {
      const double parts = std::ceil(len / max_units);
      const bool back = slots == 1 && parts > 1 && !w16 && (parts > 2 || nt > 128);
      return len * unit + (parts - 1) * flush + (back ? 0.012 * std::max(0, nt - 24) : 0.0) + tile;
    };
    auto sum = [&](double con) { return w16 ? 1.0 + batches * (con > 2 ? 2.7 : 1.6) : 2.2 + 0.0284 * tok + 0.1 * con; };
    // whole tiles in waves of one per pair; the rest, `rem`, whole in a wave of its own or divided over n pairs, `len` units each
    const int tiles = n_ft * n_tt, waves = tiles / max_pairs, rem = tiles % max_pairs;
    auto take = [&](double us, double len, int n, int slots) {
      const bool parts = std::max(len, waves || !slots ? (double)units : 0.0) > max_units;
      const int pairs = waves ? max_pairs : slots ? n : rem;
      const uint64_t need = ((uint64_t)n * slots + (parts ? pairs : 0)) * slot;
      if (need > scratch_bytes || (nt == 512 && need)) return;  // (tiles of 512 tokens: whole ones in one part)
      us += launch + waves * stretch(units, 0);
      if (w16) us = std::max(us, weights_mb / 4.5);
      if (us >= best.us) return;
      best = GemmPairPlan{nt, n_tt, pairs, slots ? tiles - rem : tiles, n, slots == 2, parts, max_units, us, need};
    };
    take(rem ? stretch(units, 0) : 0.0, units, 0, 0);
    for (int s = 2; s <= kMaxParts && s <= units && rem && rem * s <= max_pairs; ++s)
      if (units % s == 0 || units > 4 * s) take(stretch((units + s - 1) / s, 1) + sum(s), (units + s - 1) / s, rem * s, 1);
    const double per = (double)rem * units / max_pairs;
    if (per >= 1 && units <= per * (kMaxParts - 2))  // (a tile meets at most units / per + 2 ranges)
      take(stretch(std::ceil(per), 2) + sum(std::ceil(units / per) + 1) + (w16 ? 3.1 : 6.2), std::ceil(per), max_pairs, 2);
  }
  return best;
}

int pairs_of_device(int sm_count) { return std::min(sm_count / 2, kAttnMaxCounters / 2); }

// 16-byte rows of y: others the single-CTA kernel stores by the element, so that it is no match for the pairs.
bool rows_aligned(const GemmParams& g) { return g.ldy % 8 == 0 && (reinterpret_cast<uintptr_t>(g.y) & 15) == 0; }

// Time of the product on the single-CTA kernel, which takes fp16 matrices one by one and has SwiGLU as a launch of its own beside it.
double single_cta_us(const GemmParams& g) {
  int rows[3] = {0, 0, 0};
  double us = 0;
  for (int i = 0; i < g.n_seg; ++i) rows[i] = g.seg[i].n_rows;
  for (int i = 0; g.w16 && i < g.n_seg; ++i) us += gemm_us(rows + i, 1, g.T, g.K, true);
  if (!g.w16) us = gemm_us(rows, g.n_seg, g.T, g.K, false);
  if (g.act) us += 2.0 + 6e-6 / 4 * g.T * rows[0];
  return us;
}

// The plan of a launch depends on its shapes, and on the scratch in one point only: the best plan where the scratch holds it, else
// the best one that the scratch of the single-CTA kernel's plan holds, which every caller has (there may be none).
// `single`: time of the single-CTA kernel.  Chains of 1536 k are for products that the pairs take in clearly less: where both kernels are
// about equally fast, the one that drops more has nothing to offer.  The more contributors a tile has, the fewer the tiles and the shorter
// the single-CTA kernel's own chains (6144 x 4096, 77 tokens: three contributors would sum 1408 k in one accumulator against its 704).
GemmPairPlan plan_of(const GemmParams& g, int sm_count, double single) {
  int rows[3] = {0, 0, 0}, n = 0, n_ft = 0;
  for (int i = 0; i < g.n_seg; ++i) n += rows[i] = g.seg[i].n_rows;
  for (int i = 0; i < g.n_seg; ++i) n_ft += feature_tiles(rows, i, g.act != nullptr);
  auto plan = [&](bool longer, uint64_t bytes) {
    return pair_plan(rows, g.n_seg, g.act != nullptr, g.T, g.K, g.w16, longer, pairs_of_device(sm_count), bytes);
  };
  GemmPairPlan best = plan(true, ~0ull);
  const int split = n_ft * best.n_tt - best.n_whole;  // tiles that several pairs share
  const double most = best.split_pairs == 0 ? 0.96 : best.split_pairs <= 2 * split ? 0.93 : 0.75;
  const bool longer = !rows_aligned(g) || best.us <= most * single;
  if (!longer) best = plan(false, ~0ull);
  const uint64_t have = g.scratch ? g.scratch_bytes : 0;
  return best.scratch <= have ? best : plan(longer, std::min(have, gemm_scratch_bytes(g.T, n, g.K)));
}

}  // namespace

bool gemm_pair_eligible(const GemmParams& g, int sm_count, GemmPairPlan* plan) {
  if ((g.w16 && g.grp_off) || g.n_seg < 1 || g.n_seg > 3 || !g.counters || g.K % (g.w16 ? 8 : 32) || g.K > (1 << 24) || g.ldx % 8) return false;
  if (reinterpret_cast<uintptr_t>(g.x) & 15) return false;
  if ((g.res != nullptr) != (g.y2 != nullptr)) return false;
  for (int i = 0; i < g.n_seg; ++i) {
    if (reinterpret_cast<uintptr_t>(g.seg[i].base) & 15) return false;
    if (g.grp_tab[i]) return false;
  }
  if (g.act && (g.n_seg != 2 || g.seg[0].n_rows != g.seg[1].n_rows || g.seg[0].n_rows % 8 || g.ldact % 8 || g.ldy % 8 || g.res ||
                ((reinterpret_cast<uintptr_t>(g.act) | reinterpret_cast<uintptr_t>(g.y)) & 15)))
    return false;
  if (g.grp_off) return (g.n_seg == 1 || g.act) && g.grp_stride % 16 == 0 && !g.res;
  // The pairs win where there are tiles for most of them (4-bit 4096 x 4096: 128 tokens 15.7 us against 18.2, 512 tokens 23.5 against 27.7);
  // where tiles have to be split the single-CTA kernel, with smaller tiles, eight splits and the sum as a launch of its own, can be the
  // faster one (4-bit 4096 x 14336, 256 tokens: 40.3 against 38.7; fp16: 43 against 41.5).  It takes fp16 matrices one by
  // one, SwiGLU is a launch of its own beside it, and rows of y that are not 16-byte aligned it stores by the element (3333 x 9984, 300
  // tokens: 53 against 85).
  double single = single_cta_us(g);
  const GemmPairPlan pl = *plan = plan_of(g, sm_count, single);
  if (!rows_aligned(g)) return pl.pairs > 0;
  if (g.w16 && pl.n_whole > pl.pairs) single *= 1.06;  // (the fit is that far off there: 14336 x 4096 over 700 tokens 83 us on the pairs, 97)
  return pl.pairs > 0 && pl.us <= single;
}

int gemm_pair_chain(const GemmParams& g, const GemmPairPlan& pl) {
  int rows[3] = {0, 0, 0}, n_ft = 0;
  for (int i = 0; i < g.n_seg; ++i) rows[i] = g.seg[i].n_rows;
  for (int i = 0; i < g.n_seg; ++i) n_ft += feature_tiles(rows, i, g.act != nullptr);
  const int units = (g.K + kUnitK - 1) / kUnitK, split = n_ft * pl.n_tt - pl.n_whole;
  auto chain = [&](int n) { return !pl.own || n <= pl.max_units ? n : (n + (n - 1) / pl.max_units) / ((n + pl.max_units - 1) / pl.max_units); };
  int most = pl.n_whole ? chain(units) : 1;
  if (split) most = std::max(most, chain(std::min(units, (int)(((long long)split * units + pl.split_pairs - 1) / pl.split_pairs))));
  return std::min(g.K, most * kUnitK);
}

GemmOther gemm_other(const GemmParams& g, int sm_count, bool pairs) {
  GemmParams all = g;
  all.scratch = reinterpret_cast<void*>(16);
  all.scratch_bytes = ~0ull;
  int rows[3] = {0, 0, 0};
  for (int i = 0; i < g.n_seg; ++i) rows[i] = g.seg[i].n_rows;
  GemmPairPlan pl{};
  if (!pairs || !gemm_pair_eligible(all, sm_count, &pl)) return GemmOther{single_cta_us(g), gemm_chain(rows, g.n_seg, g.T, g.K)};
  return GemmOther{pl.us, gemm_pair_chain(g, pl)};
}

cudaError_t launch_gemm_pair(const GemmParams& g, const GemmPairPlan& pl, int sm_count, cudaStream_t st, uint64_t* n_launch, std::string* err) {
  TensorMapEncodeFn enc = tensor_map_encode();
  if (!enc) {
    if (err) *err = "cuTensorMapEncodeTiled is not available from the driver";
    return cudaErrorNotSupported;
  }
  PairParams p{};
  p.n_seg = g.n_seg;
  int rows[3] = {0, 0, 0}, n_ft = 0, col = 0;
  for (int i = 0; i < g.n_seg; ++i) {
    rows[i] = g.seg[i].n_rows;
    p.seg[i] = TileSeg{g.seg[i].base, rows[i], n_ft, col};
    n_ft += feature_tiles(rows, i, g.act != nullptr);
    col += g.seg[i].n_rows;
  }
  p.K = g.K;
  p.T = g.T;
  p.units = (g.K + kUnitK - 1) / kUnitK;
  p.ksteps = (g.K + 63) / 64;
  p.tile_rows = g.act ? kFeat : 2 * kFeat;
  const int max_pairs = pairs_of_device(sm_count);
  p.max_units = p.units;
  int max_blocks = 0;  // of an expert's rows, at most
  if (g.grp_off) {
    if (g.n_groups <= 0 || g.n_groups > 1024 || g.T <= 0 || g.T >= 1 << 22) return cudaErrorInvalidValue;
    // The rows of an expert are known on the device only: blocks as high as an expert's rows are expected to be at most where the pairs
    // spread evenly (mean + 3 standard deviations), in equal parts of at most 256.  An expert with more takes more blocks, each of which
    // reads and expands its weights; low blocks, whose rows cost next to nothing, get 5 deviations (300 tokens, all through the same four
    // of 64 experts: 32 -> 48 rows, 98.7 -> 84 us for the layer; 40 through the same eight: 16 -> 32 rows, 118.6 -> 98.6.  Blocks of 64 or 96
    // rows whatever the mean cost evenly spread ones 1 to 6 %, and so does a height that the device chooses: the loops then count in registers).
    const double mean = (double)g.T / g.n_groups;
    auto height = [&](double rows) {
      const int parts = (int)std::ceil(rows / 256);
      return std::min(256, ((int)std::ceil(rows / parts) + 15) / 16 * 16);
    };
    p.nt = std::max(height(mean + 3 * std::sqrt(mean)), std::min(64, height(mean + 5 * std::sqrt(mean))));
    p.n_groups = g.n_groups;
    max_blocks = std::min(g.n_groups, g.T) + g.T / p.nt;
    p.ft_per = n_ft;
    p.n_tt = 1;
    p.workers = (int)std::min<long long>((long long)n_ft * max_blocks, max_pairs);
  } else {
    if (!pl.pairs) return cudaErrorInvalidValue;
    p.nt = pl.nt;
    p.n_tt = pl.n_tt;
    p.n_ft = n_ft;
    p.workers = pl.pairs;
    p.n_whole = pl.n_whole;
    p.split_workers = pl.split_pairs;
    p.slots2 = pl.slots2;
    if (pl.own) p.max_units = pl.max_units;
  }
  p.sc16 = !g.w16 && g.K % 256 == 0;
  p.y = g.y;
  p.ldy = g.ldy;
  p.res = g.res;
  p.y2 = g.y2;
  p.act = g.act;
  p.ldact = g.ldact;
  p.partial = (float*)g.scratch;
  p.slot_tok = std::min(p.nt, g.T);
  p.own = p.partial + (size_t)(p.split_workers * (p.slots2 ? 2 : 1)) * 2 * kFeat * p.slot_tok;
  p.counters = g.counters;
  p.status = g.status;
  p.grp_off = g.grp_off;
  p.grp_stride = g.grp_stride;
  CUtensorMap xmap;
  const cuuint64_t dims[2] = {(cuuint64_t)g.K, (cuuint64_t)g.T}, strides[1] = {(cuuint64_t)g.ldx * 2};
  const cuuint32_t box[2] = {64, (cuuint32_t)(p.nt > 256 ? p.nt / 4 : p.nt / 2)}, es[2] = {1, 1};
  if (enc(&xmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(g.x), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
          CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
    if (err) *err = "cuTensorMapEncodeTiled failed for the activation tile";
    return cudaErrorInvalidValue;
  }
  PairMaps maps;
  for (int i = 0; i < 3; ++i) {
    if (i >= g.n_seg) {
      maps.codes[i] = maps.codes[0];
      maps.scales[i] = maps.scales[0];
      continue;
    }
    const GemvSeg& sg = g.seg[i];
    const cuuint64_t row = g.w16 ? (cuuint64_t)g.K * 2 : (cuuint64_t)g.K / 2, groups = g.grp_off ? (cuuint64_t)g.n_groups : 1;
    const cuuint64_t wd[3] = {g.w16 ? (cuuint64_t)g.K : row, (cuuint64_t)sg.n_rows, groups};
    const cuuint64_t ws[2] = {row, g.grp_off ? (cuuint64_t)g.grp_stride : row * sg.n_rows};
    const cuuint32_t wb[3] = {64, 64, 1}, we[3] = {1, 1, 1};
    if (enc(&maps.codes[i], g.w16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t*>(sg.base), wd, ws, wb, we,
            CU_TENSOR_MAP_INTERLEAVE_NONE, g.w16 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
            g.w16 ? CU_TENSOR_MAP_L2_PROMOTION_L2_256B : CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
      if (err) *err = "cuTensorMapEncodeTiled failed for the weights";
      return cudaErrorInvalidValue;
    }
    maps.scales[i] = maps.codes[i];
    if (p.sc16) {  // scales: [n_rows][K / 32] halves behind the codes, eight at a time
      const cuuint64_t sd[3] = {(cuuint64_t)g.K / 32, wd[1], wd[2]}, ss[2] = {(cuuint64_t)g.K / 16, ws[1]};
      const cuuint32_t sb[3] = {8, 64, 1};
      if (enc(&maps.scales[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<uint8_t*>(sg.base) + (size_t)sg.n_rows * (g.K / 2), sd, ss, sb, we,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) !=
          CUDA_SUCCESS) {
        if (err) *err = "cuTensorMapEncodeTiled failed for the scales";
        return cudaErrorInvalidValue;
      }
    }
  }
  constexpr size_t kMost = 227 * 1024 - 1024;
  size_t smem;
  if (g.w16) {  // a ring of steps, as deep as a staging of 64 tokens leaves room for
    p.stage_tok = kW16StageTok;
    const size_t fixed = 1024 + (size_t)kW16StageTok * kStagePitch, step = (size_t)p.nt * 64 + kW16Bytes;
    p.xs = (int)std::min<size_t>(kMaxX, (kMost - fixed) / step);
    smem = fixed + p.xs * step;
  } else {  // three activation stages and a code ring twice as deep as the weight stages, then more activations
    p.stage_tok = (p.nt + 31) / 32 * 32;
    p.xu = p.nt <= 128 ? 2 : 1;
    const size_t xs = (size_t)p.nt * 128 * p.xu, cs = kCodeBytes + kScaleBytes, list = g.grp_off ? (size_t)(max_blocks + 1) * sizeof(uint32_t) : 0;
    // (beside three places for 256 rows there is room for a list of 255 blocks; more of them: the staging in two halves.  8 experts, 32768 rows:
    // a list of 8 bytes a block had left two places, 829 -> 807 us for the layer)
    if (1024 + (size_t)p.stage_tok * kStagePitch + list + 3 * xs + 6 * cs > kMost) p.stage_tok = 128;
    const size_t fixed = 1024 + (size_t)p.stage_tok * kStagePitch + list;
    p.stages = fixed + 3 * xs + 8 * cs <= kMost ? 4 : 3;
    p.codes = 2 * p.stages;
    p.xs = (int)std::min<size_t>(kMaxX, (kMost - fixed - p.codes * cs) / xs);
    while (p.codes + p.stages <= kMaxCodes && fixed + p.xs * xs + (p.codes + p.stages) * cs <= kMost) p.codes += p.stages;
    smem = fixed + p.xs * xs + p.codes * cs;
    p.list_at = (int)(smem - 1024 - list);
  }
  static std::atomic<uint64_t> attr_done;
  const cudaError_t e = smem_limit_once(&attr_done, {reinterpret_cast<const void*>(gemm_pair_kernel<kFmtQ4>), reinterpret_cast<const void*>(gemm_pair_kernel<kFmtMx>),
                                                     reinterpret_cast<const void*>(gemm_pair_kernel<kFmtW16>)}, kMost);
  if (e != cudaSuccess) return e;
  ++*n_launch;
  auto run = [&](auto* kernel) { return launch_dep(kernel, dim3(2 * p.workers), dim3(kPairThreads), smem, st, g.pdl, 2, xmap, maps, p); };
  return g.w16 ? run(gemm_pair_kernel<kFmtW16>) : g.mx ? run(gemm_pair_kernel<kFmtMx>) : run(gemm_pair_kernel<kFmtQ4>);
}

}  // namespace ats
