// GEMM of few tokens to a tile (at most 128) on single CTAs (sm_100a, tcgen05): Y[T][N] = X[T][K] W^T for the two 4-bit block formats;
// fp16 operands (w = rn16(scale * code), one rounding), fp32 accumulation.
//
// As on the pairs of CTAs (kernels_gemm_pair.cu) the weights are the A operand, expanded straight into tensor memory (a thread has one
// feature, its lane), and the tokens the instruction's N.  There the one MMA warp of a pair was the bottleneck up to 128 tokens and beyond:
// every unit went through mbarriers of two CTAs, and a wait that is not over when it begins costs 200 cycles.  Here a CTA has two halves with
// an MMA warp each, and expansion meets MMA at named barriers of the CTA, so that 128 k of 128 features take 410 to 440 cycles (pairs: 630 to
// 760; the expansion alone 310 to 340, the MMAs 4 per token).  What the halves take:
//   wide    two blocks of 128 features, the same 256 k: activations are read once for both
//   SwiGLU  128 gate and the 128 up features to them: silu(g) u in the epilogue, whose threads have both accumulators of a feature
//   deep    128 features, half of the k each, the two sums added up in the epilogue: half as high tiles where there are few
// With whole tiles the sums are written as they are.  Few tiles are shared by a cluster of CTAs (2 to 6, each with a range of the k): runs of
// 16 tokens belong to its CTAs in turn, each sends what it has of the others' runs into their shared memory (st.async, counted on a barrier
// there) and adds up its own in ascending order of k.  (Through scratch memory and arrival counts the same took 4 us instead of 1: 4096 x 4096,
// 16 tokens, 9.4 us; whole tiles 9.3; in clusters 7.2.)
//
// The tensor core truncates what it adds, so chains are no longer than on the kernels that would take the product otherwise with all the scratch they
// want (gemm_other; with less the pairs have another plan, whose chains are shorter by up to a fifth for 1.6 % of products: their limit would cost these 7 % of
// their time, up to 46, for an error against 64 bits that is the same to the fifth digit, 2.0753e-4).  A half's
// steps go to up to four accumulators in turn where a CTA has one tile and tensor memory has room, or an accumulator is handed over and the
// sums so far wait in the scratch.
//
// What bounds it: up to 64 tokens HBM where every SM has a CTA (6.3 TB/s of weights; an SM's share of the rate is 396 cycles for 128 k of 128 features,
// the expansion stays just under it), with 128 the MMAs at the power limit (1.3 to
// 1.4 PFLOP/s); products of few tiles launch, first loads and output (2.5 to 4 us) and the exchange.  Back to back on new weights, before (pairs or
// gemm_q4_kernel) -> now, us:
//   1024 x 1024, 16 tokens Q4       5.8 -> 3.3      4096 x 4096, 16 / 77 / 512 tokens MXFP4   10.8 / 13.9 / 21.5 -> 7.2 / 10.6 / 17.5
//   14336 x 4096, 16 / 128 Q4       17.0 / 20.7 -> 11.3 / 15.3      4096 x 14336, 16 / 77 / 512 Q4   17.8 / 21.2 / 55.7 -> 14.2 / 18.0 / 50
//   2880 x 2880, 16 / 300 Q4        10.2 / 17.9 -> 6.9 / 11.7       13600 x 4000, 16 / 77 MXFP4               21.7 / 24.8 -> 13.0 / 14.4
//   28672 x 4096, 16 / 77 MXFP4     24.8 / 26.9 -> 17.4 / 20.3      2048 x 5632, 16 / 300 MXFP4   10.3 / 23.9 -> 7.0 / 15
//
// Roles per CTA: warp 0 = activation loads, warps 1 and 2 = MMA issue (and tensor-memory allocation), warp 3 = code and scale loads, warps 4..11 =
// epilogue, warps 12..27 = expansion: four groups of four, each with a slot of 64 tensor-memory columns (128 k).  Every mbarrier wait is
// bounded; on expiry the CTA raises the status word, goes on meeting at its named barriers without work, and every thread reaches the end.
#include <cuda.h>

#include <cmath>
#include <type_traits>

#include "gemm_tiles.cuh"

namespace ats {

namespace {

constexpr int kRows = 128;                  // features that one MMA takes: tensor memory's lanes
constexpr int kUnitK = 256;                 // k per unit of work: 128 bytes of codes and one 16-byte line of scales per row
constexpr int kCodeBytes = kRows * 128;     // of 128 rows: 16 KB
constexpr int kScaleBytes = kRows * 16;     // 2 KB
// K no multiple of 256: a warp fetches the scales of its 32 rows for 128 k itself, three words of each from the 4-byte boundary at or below the
// first, three steps ahead.  (From one warp, five words of each row for a unit: 0.93 us a unit where this takes 0.44; as a flag instead of a kernel of
// its own it cost the other products 0.4 us of instruction fetch.)
constexpr int kFeed = 4, kFeedBytes = 32 * 12;
constexpr int kMaxCodes = 8, kMaxX = 12;    // ring depths at most
constexpr int kStagePitch = 272;            // bytes per token of the output staging: 128 halves + 16
constexpr int kStageTok = 16;               // tokens staged at a time
constexpr int kStageBytes = 2 * 2 * kStageTok * kStagePitch;  // two sets of epilogue warps, two buffers each
constexpr int kFewThreads = 28 * 32;
constexpr int kMaxTok = 128;                // tokens of a tile at most
constexpr int kMaxParts = 6;                // CTAs of a cluster that share a tile at most
constexpr int kPartBytes = kRows * kStageTok * 4;  // fp32 sums of 16 tokens and 128 features: 8 KB
constexpr uint32_t kColA = 256;             // tensor-memory columns: accumulators 0..255, expanded weights from 256 on
enum { kWide, kSwiglu, kDeep };             // what the two halves of a CTA take, see above
// What becomes of a CTA's sums.  (Kernels of their own: a launch runs every line of the epilogue for the first time, and what it does not need
// cost 0.3 to 0.7 us, 14336 x 1024 over 16 tokens 5.1 -> 5.8.)
enum {
  kPlain,   // written as they are
  kShared,  // added up from several accumulators, and from the CTAs of a cluster that share a tile
  kHanded   // added up in parts, in words of the scratch
};

struct FewParams : TileWork {  // (workers: CTAs; units: 256 k)
  int codes, xs;      // depths of the rings
  unsigned long long grp_stride;
  __half* y;          // (SwiGLU: may be null)
  int ldy;
  const __half* res;  // optional: y2 = rn16(res + y)
  __half* y2;
  int ldact;
  int turns;          // accumulators of a half (1, 2, 4) that take its steps in turn; more than one: a CTA has a single tile
  int max_units;      // units that an accumulator adds up before it is handed over; the sums so far wait in ...
  float* own;         // ... words of the scratch that belong to the thread that reads them back: nt x 128 per CTA (and half)
  int parts;          // CTAs of a cluster, which divide the units of their tile among them (1: a CTA has tiles of its own)
  int* status;
};
struct FewMaps {
  CUtensorMap codes[3], scales[3];  // of the segments
  CUtensorMap x[kMaxTok / 16];      // activations, in boxes of 16, 32, .. tokens (those that occur)
};
// A CTA's stretches, the same sequence in every role: whole tiles, or its share of the cluster's one tile.
struct FewWalk {
  int tile, step, n, u0, u1;
  __device__ __forceinline__ FewWalk(const FewParams& p, bool cluster, int rank, int n_tiles) {
    tile = blockIdx.x;
    step = p.workers;
    n = n_tiles;
    u0 = 0;
    u1 = p.units;
    if (cluster) {
      tile = blockIdx.x / p.parts;
      u0 = p.units * rank / p.parts;
      u1 = p.units * (rank + 1) / p.parts;
    }
  }
  __device__ __forceinline__ bool next(int* t) {
    if (tile >= n) return false;
    *t = tile;
    tile += step;
    return true;
  }
};
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Tokens that a tile's MMAs take: those it has, in multiples of 16.
__device__ __forceinline__ int tokens_of(const FewParams& p, const Tile& tl) { return (min(p.nt, tl.T - tl.t0) + 15) & ~15; }
// Remote shared memory: four words to another CTA of the cluster, counted on a barrier there.
__device__ __forceinline__ uint32_t remote(uint32_t saddr, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(saddr), "r"(rank));
  return a;
}
__device__ __forceinline__ void st_async4(uint32_t dst, uint32_t bar, const float* v) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%2, %3, %4, %5}, [%1];" ::"r"(dst), "r"(bar),
               "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3]))
               : "memory");
}

// Units that go into an accumulator at a time: a stretch in equal parts of p.max_units at most.
__device__ __forceinline__ int part_units(const FewParams& p, int n) {
  return n <= p.max_units ? n : (n + (n - 1) / p.max_units) / ((n + p.max_units - 1) / p.max_units);
}

template <bool MX, int MODE, int SUMS, bool LINES>
__global__ void __launch_bounds__(kFewThreads, 1) gemm_few_kernel(const __grid_constant__ FewMaps maps, const __grid_constant__ FewParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint64_t aempty[4], xfull[kMaxX], xempty[kMaxX], cfull[kMaxCodes], cempty[kMaxCodes], acc_full[2][2], d_empty[2][2];
  __shared__ uint32_t tmem_s;
  __shared__ uint64_t recv_full[2];
  __shared__ int n_blocks_s;
  constexpr bool kJoined = MODE != kWide;             // both halves' accumulators meet in the epilogue
  constexpr int kSubs = MODE == kDeep ? 1 : 2;        // 128-row blocks of weights in a unit
  constexpr uint32_t kPlaceBytes = kSubs * kCodeBytes;
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // (the same for the warp, and known to be)
  const bool cluster = SUMS == kShared && p.parts > 1;
  const int rank = cluster ? (int)cluster_rank() : 0;
  const int NC = p.codes, NX = p.xs;
  const uint32_t xbytes = (uint32_t)p.nt * 256;       // a place for activations of 128 k: two chunks of 64, rows of 128 bytes, swizzled
  uint8_t* x_s = smem;
  uint8_t* code_s = x_s + (size_t)NX * xbytes;
  uint8_t* scale_s = code_s + (size_t)NC * kPlaceBytes;
  uint8_t* out_s = scale_s + (LINES ? NC * kSubs * kScaleBytes : 16 * kFeed * kFeedBytes);  // (LINES: K is a multiple of 256)
  uint8_t* recv_s = out_s + kStageBytes;              // sums from the other CTAs of the cluster
  // Several accumulators per half where tensor memory has room: two that take tiles in turn, or the steps of a CTA's one tile (shorter
  // chains).  Accumulator i of half s lies at s * pitch + i * 2 * pitch.
  const bool two = p.nt <= 64 && (SUMS != kShared || p.turns == 1);
  const uint32_t pitch = two ? 64u : SUMS == kShared ? 128u / p.turns : 128u;

  if (threadIdx.x == 0) {
    for (int s = 0; s < 4; ++s) mbar_init(&aempty[s], 1);
    for (int s = 0; s < NX; ++s) {
      mbar_init(&xfull[s], 1);
      mbar_init(&xempty[s], MODE == kDeep ? 1 : 2);
    }
    for (int s = 0; s < 4; ++s) {
      mbar_init(&acc_full[s >> 1][s & 1], 1);
      mbar_init(&d_empty[s >> 1][s & 1], kJoined ? 8 : 4);
    }
    if (SUMS == kShared)
      for (int s = 0; s < 2; ++s) mbar_init(&recv_full[s], 1);
    prefetch_map(&maps.x[p.nt / 16 - 1]);
    mbar_fence_init();
  }
  if (warp == 3 && lane == 0) {  // (the loader's own barriers: it starts before the others are ready)
    for (int i = 0; i < p.n_seg; ++i) {
      prefetch_map(&maps.codes[i]);
      if (LINES) prefetch_map(&maps.scales[i]);
    }
    for (int s = 0; s < NC; ++s) {
      mbar_init(&cfull[s], 1);
      mbar_init(&cempty[s], MODE == kDeep ? 8 : 16);
    }
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_s, 512);
  __syncwarp();
  // The weights do not depend on the preceding kernel; the activations (and the grouped form's row offsets) do.  What the
  // epilogue touches is ordered behind the activation loads.
  if (cluster) cluster_arrive();  // (behind this CTA's barriers)
  if (p.grp_off) asm volatile("griddepcontrol.wait;" ::: "memory");
  uint32_t* const blocks = reinterpret_cast<uint32_t*>(smem + p.list_at);
  int n_tiles = p.n_whole;
  if (p.grp_off) {
    if (warp == 4) {
      const int n = list_blocks(p, blocks, lane);
      if (lane == 31) n_blocks_s = n;
    }
    __syncthreads();
    n_tiles = n_blocks_s * p.ft_per;
  }
  bool ok = true;
  int tile;
  auto total_units = [&] {
    FewWalk mine(p, cluster, rank, n_tiles);
    int n = 0;
    while (mine.next(&tile)) n += mine.u1 - mine.u0;
    return n;
  };
  FewWalk ld_walk(p, cluster, rank, n_tiles);
  int ld_u = 0, ld_end = 0, ld_cs = 0;  // next unit and end of the current stretch; ring place
  int ld_first = 0, ld_e = 0, ld_sa = 0, ld_sb = 0;
  uint32_t ld_par = 0;
  auto load_units = [&](int most, bool used) {  // used: the places have held units before
    const uint32_t one = elect_one();
    for (int n = 0; n < most; ++n) {
      if (ld_u == ld_end) {
        if (!uniform(ld_walk.next(&tile))) return;
        const Tile tl = tile_of(p, tile, blocks);
        ld_u = uniform(ld_walk.u0);
        ld_end = uniform(ld_walk.u1);
        ld_e = uniform(tl.expert);
        ld_sa = MODE == kSwiglu ? 0 : uniform(tl.sg);
        ld_sb = MODE == kSwiglu ? 1 : ld_sa;
        ld_first = uniform(tl.row0);
      }
      if (used && !wait_warp(&cempty[ld_cs], ld_par)) {
        ok = false;
        return;
      }
      uint64_t* bar = &cfull[ld_cs];
      const uint32_t dst = smem_u32(code_s) + (uint32_t)ld_cs * kPlaceBytes, sdst = smem_u32(scale_s) + (uint32_t)(ld_cs * kSubs * kScaleBytes);
      const int second = MODE == kSwiglu ? ld_first : ld_first + kRows;
      expect_tx_one(one, bar, kPlaceBytes + (LINES ? (uint32_t)(kSubs * kScaleBytes) : 0u));
      // rows beyond the matrix and k beyond its end read as zeros
      tma_3d_one(one, dst, &maps.codes[ld_sa], ld_u * 128, ld_first, ld_e, bar);
      if (kSubs == 2) tma_3d_one(one, dst + kCodeBytes, &maps.codes[ld_sb], ld_u * 128, second, ld_e, bar);
      if (LINES) tma_3d_one(one, sdst, &maps.scales[ld_sa], ld_u * 8, ld_first, ld_e, bar);
      if (LINES && kSubs == 2) tma_3d_one(one, sdst + kScaleBytes, &maps.scales[ld_sb], ld_u * 8, second, ld_e, bar);
      ++ld_u;
      if (++ld_cs == NC) {
        ld_cs = 0;
        if (used) ld_par ^= 1u;
      }
    }
  };
  if (warp == 3) load_units(NC, false);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_s;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // 72 registers a thread at launch; the epilogue's sums need more: 56 + 4 x 64 + 2 x 96 = 7 x 72
  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    if (warp == 0) {
      // ------------------------------------------------------------ activations: 128 k at a time
      asm volatile("griddepcontrol.wait;" ::: "memory");
      const uint32_t one = elect_one();
      FewWalk mine(p, cluster, rank, n_tiles);
      const uint32_t x0 = smem_u32(x_s);
      int s = 0;
      uint32_t par = 1;
      while (uniform(ok && mine.next(&tile))) {
        const Tile tl = tile_of(p, tile, blocks);
        const int i1 = 2 * uniform(mine.u1), row = uniform(tl.rowoff + tl.t0), box = uniform(tokens_of(p, tl) / 16);
        for (int i = 2 * uniform(mine.u0); i < i1; ++i) {
          if (!wait_warp(&xempty[s], par)) {  // (the first wait for an empty place passes at once)
            ok = false;
            break;
          }
          expect_tx_one(one, &xfull[s], (uint32_t)box * 4096u);
          if (LINES) {  // (both chunks in one box)
            tma_3d_one(one, x0 + (uint32_t)s * xbytes, &maps.x[box - 1], 0, row, 2 * i, &xfull[s]);
          } else {
            tma_3d_one(one, x0 + (uint32_t)s * xbytes, &maps.x[box - 1], 128 * i, row, 0, &xfull[s]);
            tma_3d_one(one, x0 + (uint32_t)s * xbytes + (uint32_t)box * 2048u, &maps.x[box - 1], 128 * i + 64, row, 0, &xfull[s]);
          }
          if (++s == NX) s = 0, par ^= 1u;
        }
      }
    } else if (warp < 3) {
      // ------------------------------------------------------------ MMA issue: one warp for each half
      // It meets the four warps that expanded its weights at a barrier of the CTA (on an mbarrier a wait that is not known to be
      // over when it begins costs 200 cycles).  Nothing in the loop may look as if lanes could differ: operands are then moved to
      // uniform registers one by one, and eight MMAs and two commits take 600 cycles to issue instead of 80.
      const int sub = warp - 1;
      int m = 0;  // steps of 128 k so far; slots take turns
      auto meet = [&] { asm volatile("bar.sync %0, 160;" ::"r"(1 + 2 * sub + (m++ & 1)) : "memory"); };
      auto issue = [&] {
        const uint32_t one = elect_one();
        const uint64_t xd = umma_desc_sw128(smem_u32(x_s));
        FewWalk mine(p, cluster, rank, n_tiles);
        int sx = MODE == kDeep ? sub : 0, seg = 0;
        uint32_t parx = 0;
        bool readyx = false;
        while (uniform(mine.next(&tile))) {
          const int tokens = uniform(tokens_of(p, tile_of(p, tile, blocks)));
          const uint32_t idesc = umma_idesc_f16(kRows, tokens), chunk = (uint32_t)tokens * 8;  // (16-byte pieces of a chunk)
          int left = uniform(mine.u1 - mine.u0) * (MODE == kDeep ? 1 : 2);
          const int most = SUMS == kHanded ? uniform(part_units(p, mine.u1 - mine.u0)) * (MODE == kDeep ? 1 : 2) : left;
          const uint32_t last_turn = SUMS == kShared ? (uint32_t)p.turns - 1 : 0;
          for (; left > 0; left -= most) {
            const int steps = min(most, left);
            const int b = two ? seg & 1 : 0, use = two ? seg >> 1 : seg;
            const uint32_t d = pitch * (2 * b + sub);
            ++seg;
            if (use > 0 && !wait_warp(&d_empty[sub][b], (use - 1) & 1)) return false;
              uint32_t accumulate = 0;
            for (int i = 0; i < steps; ++i) {
              const int slot = 2 * sub + (m & 1);
              const uint32_t da = SUMS == kShared ? d + 2u * pitch * ((uint32_t)i & last_turn) : d;
              meet();
              if (!__all_sync(0xffffffffu, readyx) && !wait_warp(&xfull[sx], parx)) return false;
              tc_fence_after();
              int sxn = sx + (MODE == kDeep ? 2 : 1);
              uint32_t parxn = parx;
              if (sxn >= NX) sxn -= NX, parxn ^= 1u;
              readyx = peek(&xfull[sxn], parxn);
              const uint64_t bd = xd + (uint64_t)((uint32_t)sx * (xbytes >> 4));
              const uint32_t at = kColA + 64u * slot;  // (all 512 columns are this CTA's: the allocation starts at 0)
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) umma_ts(one, da, at + 8u * kk, bd + (uint64_t)(2 * kk), idesc, kk > 0 ? 1u : accumulate);
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) umma_ts(one, da, at + 32u + 8u * kk, bd + (uint64_t)(chunk + 2 * kk), idesc, 1);
              umma_commit_to(one, &aempty[slot]);
              umma_commit_to(one, &xempty[sx]);
              accumulate = SUMS != kShared || (uint32_t)i >= last_turn;
              sx = sxn, parx = parxn;
            }
            umma_commit_to(one, &acc_full[sub][b]);
          }
        }
        return true;
      };
      ok = issue();
      if (!ok) {  // whoever gives up goes on meeting the others at the barriers
        const int steps = total_units() * (MODE == kDeep ? 1 : 2);
        while (m < steps) meet();
      }
    } else {
      load_units(0x7fffffff, true);
    }
  } else if (warp >= 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    // ------------------------------------------------------------ expansion: thread = feature; a group of four warps per slot of 128 k
    const int quarter = warp & 3, slot = (warp - 12) >> 2, sub = slot >> 1, h = slot & 1;
    const int row = quarter * 32 + lane;
    const int kh = MODE == kDeep ? sub : h;  // which 128 k of a unit
    const uint32_t a_col = tmem + ((uint32_t)(quarter * 32) << 16) + kColA + 64u * slot;
    const uint32_t code_row = smem_u32(code_s) + (uint32_t)((MODE == kDeep ? 0 : sub * kCodeBytes) + row * 128);
    const uint32_t scale_row = LINES ? smem_u32(scale_s) + (uint32_t)((MODE == kDeep ? 0 : sub * kScaleBytes) + row * 16 + kh * 8)
                                     : smem_u32(scale_s) + (uint32_t)((warp - 12) * kFeed * kFeedBytes);
    const int nblk = p.K / 32;
    const uint32_t swz = (uint32_t)(row & 7) << 4;
    constexpr int kStep = MODE == kDeep ? 2 : 1;  // (deep: the groups of a half take turns)
    int m = 0;  // units of this group so far
    auto expand = [&] {
      FewWalk mine(p, cluster, rank, n_tiles);
      int skip = MODE == kDeep ? h : 0, cs = skip;
      // scales, three steps ahead: tile, next unit and its end, this lane's three words (row, word) = (l / 3, l % 3), l = lane + 32 j
      FewWalk fd(p, cluster, rank, n_tiles);
      const uint8_t* fd_base = nullptr;
      uint32_t fd_at[3] = {0, 0, 0}, fd_hi = 0, fd_place = 0;
      int fd_u = skip, fd_end = 0;
      auto feed = [&] {
        while (fd_u >= fd_end) {
          int t;
          if (!fd.next(&t)) {
            fd_u = fd_end;
            break;
          }
          const Tile tl = tile_of(p, t, blocks);
          const TileSeg& sg = p.seg[MODE == kSwiglu ? sub : tl.sg];
          fd_u = fd.u0 + fd_u - fd_end;
          fd_end = fd.u1;
          fd_base = sg.base + (unsigned long long)tl.expert * p.grp_stride + (size_t)sg.n_rows * (p.K / 2);
          fd_hi = (uint32_t)sg.n_rows * nblk * 2;
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            const int l = lane + 32 * j, r = tl.row0 + (MODE == kWide ? sub * kRows : 0) + quarter * 32 + l / 3;
            fd_at[j] = r < sg.n_rows ? (((uint32_t)r * nblk * 2) & ~3u) + kh * 8 + l % 3 * 4 : 0x80000000u;  // (at most 2 GB of scales, see the plan)
          }
        }
        if (fd_u < fd_end) {
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            const uint32_t lo = fd_at[j] + (uint32_t)fd_u * 16;
            const bool in = lo < fd_hi;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(scale_row + fd_place * kFeedBytes + (uint32_t)(lane + 32 * j) * 4),
                         "l"(fd_base + (in ? lo : 0)), "r"(in ? 4 : 0)
                         : "memory");
          }
          fd_u += kStep;
        }
        fd_place = (fd_place + 1) & (kFeed - 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
      };
      if (!LINES) {
        feed();
        feed();
        feed();
      }
      uint32_t cpar = 0, apar = 1;  // (the first wait for an empty slot passes at once)
      while (mine.next(&tile)) {
        int u = mine.u0 + skip, odd = 0;
        if (!LINES) {  // units begin at even scales: the row decides
          const Tile tl = tile_of(p, tile, blocks);
          odd = ((tl.row0 + (MODE == kWide ? sub * kRows : 0) + row) & nblk) & 1;
        }
        for (; u < mine.u1; u += kStep) {
          if (!wait_warp(&cfull[cs], cpar)) return false;
          const bool free_seen = peek(&aempty[slot], apar);
          const uint32_t cr = code_row + (uint32_t)cs * kPlaceBytes;
          uint2 sw;  // four scales
          if (LINES) {
            sw = lds64(scale_row + (uint32_t)(cs * kSubs * kScaleBytes));
          } else {
            asm volatile("cp.async.wait_group 2;" ::: "memory");
            __syncwarp();
            const uint32_t sr = scale_row + (uint32_t)((m & (kFeed - 1)) * kFeedBytes + lane * 12);
            const uint32_t w0 = lds32(sr), w1 = lds32(sr + 4), w2 = lds32(sr + 8);
            sw = odd ? make_uint2(__byte_perm(w0, w1, 0x5432), __byte_perm(w1, w2, 0x5432)) : make_uint2(w0, w1);
            const int left = nblk - (u * 8 + kh * 4);  // blocks that exist; what follows belongs to the next row
            if (left < 4) sw.y &= left < 3 ? 0u : 0x0000FFFFu;
            if (left < 2) sw.x &= left < 1 ? 0u : 0x0000FFFFu;
            feed();  // (into the place that was read one step ago)
          }
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            uint32_t o[32];
            const uint32_t pairs = c ? sw.y : sw.x;
#pragma unroll
            for (int b = 0; b < 2; ++b) {
              const uint4 q = lds128(cr + (((uint32_t)(4 * kh + 2 * c + b) << 4) ^ swz));
              const __half2 sc = as_h2(__byte_perm(pairs, 0, b ? 0x3232 : 0x1010));
              expand_word<MX>(q.x, sc, o + 16 * b);
              expand_word<MX>(q.y, sc, o + 16 * b + 4);
              expand_word<MX>(q.z, sc, o + 16 * b + 8);
              expand_word<MX>(q.w, sc, o + 16 * b + 12);
            }
            if (c == 0) {
              // (the limit is above all that the MMA warp may wait for: nobody comes to the barrier below a second time before it did)
              if (!__all_sync(0xffffffffu, free_seen) && !__all_sync(0xffffffffu, mbar_wait_suspending(&aempty[slot], apar, 8 * kWaitLimitCycles)))
                return false;
              tc_fence_after();
            }
            tmem_st_x32(a_col + 32u * c, o);
          }
          tmem_st_wait();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&cempty[cs]);
          asm volatile("bar.arrive %0, 160;" ::"r"(1 + slot) : "memory");
          ++m;
          apar ^= 1u;
          cs += kStep;
          if (cs >= NC) cs -= NC, cpar ^= 1u;
        }
        skip = u - mine.u1;
      }
      return true;
    };
    ok = expand();
    if (!LINES) asm volatile("cp.async.wait_all;" ::: "memory");
    if (!ok) {  // whoever gives up goes on meeting the MMA warp, and does not come to the barrier before that has been there
      const int total = MODE == kDeep ? (total_units() - h + 1) / 2 : total_units();
      for (; m < total; ++m) asm volatile("bar.sync %0, 160;" ::"r"(1 + slot) : "memory");
    }
  } else {
    // ------------------------------------------------------------ epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 96;");
    if (cluster) cluster_wait();  // (the other CTAs' barriers are initialised)
    // Two sets of four warps.  Wide: a set for each half's 128 features.  Else a thread has both accumulators of its feature and the
    // sets take turns: whole tiles 16 tokens at a time, split ones 32.
    const int quarter = warp & 3, set = (warp - 4) >> 2, tid = (threadIdx.x - 128) & 127;
    const int feat = quarter * 32 + lane;
    const uint32_t d_col = tmem + ((uint32_t)(quarter * 32) << 16);
    const uint32_t out_u = smem_u32(out_s) + (uint32_t)(set * 2 * kStageTok * kStagePitch);
    auto set_sync = [&] { asm volatile("bar.sync %0, 128;" ::"r"(5 + set) : "memory"); };
    auto set_all = [&](bool v) {
      uint32_t r;
      asm volatile("{\n.reg .pred a, b;\nsetp.ne.u32 a, %1, 0;\nbarrier.cta.red.and.pred b, %2, 128, a;\nselp.u32 %0, 1, 0, b;\n}"
                   : "=r"(r)
                   : "r"((uint32_t)v), "r"(5 + set)
                   : "memory");
      return r != 0;
    };
    constexpr int kPlanes = MODE == kSwiglu ? 2 : 1;  // values per feature and token that a thread has: gate, up
    FewWalk mine(p, cluster, rank, n_tiles);
    int seg = 0, buf = 0;
    while (mine.next(&tile)) {
      const Tile tl = tile_of(p, tile, blocks);
      const int ntok = min(p.nt, tl.T - tl.t0);
      int b = 0;
      auto wait_sums = [&] {
        b = two ? seg & 1 : 0;
        const int use = two ? seg >> 1 : seg;
        ++seg;
        bool got = true;  // (one warp polls, the others sleep at the barrier: polls take issue slots from the expansion)
        if (quarter == 0) {
          if (kJoined) got = wait_warp(&acc_full[0][b], use & 1) && wait_warp(&acc_full[1][b], use & 1);
          else got = wait_warp(&acc_full[set][b], use & 1);
        }
        got = set_all(got);
        tc_fence_after();
        return got;
      };
      auto add16 = [&](uint32_t col, float* v) {
        float w[16];
        tmem_ld_x16(col, reinterpret_cast<uint32_t*>(w));
        tmem_ld_wait_x16(reinterpret_cast<uint32_t*>(w));
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] += w[i];
      };
      // 16 tokens' sums of this thread's feature (SwiGLU: gate, then up)
      auto sums = [&](int c0, float* v) {
        const uint32_t col0 = d_col + pitch * (2 * b), col1 = col0 + pitch;
        const uint32_t a = (MODE == kWide && set ? col1 : col0) + c0;
        tmem_ld_x16(a, reinterpret_cast<uint32_t*>(v));
        if (MODE == kSwiglu) tmem_ld_x16(col1 + c0, reinterpret_cast<uint32_t*>(v + 16));
        tmem_ld_wait_x16(reinterpret_cast<uint32_t*>(v));
        if (MODE == kSwiglu) tmem_ld_wait_x16(reinterpret_cast<uint32_t*>(v + 16));
        if (MODE == kDeep) add16(col1 + c0, v);
#pragma unroll 1
        for (int i = 1; SUMS == kShared && i < p.turns; ++i) {
          const uint32_t t = 2u * pitch * (uint32_t)i;
          add16(a + t, v);
          if (MODE == kSwiglu) add16(col1 + c0 + t, v + 16);
          if (MODE == kDeep) add16(col1 + c0 + t, v);
        }
      };
      auto release = [&] {  // the accumulators may be overwritten
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (kJoined) mbar_arrive(&d_empty[0][b]), mbar_arrive(&d_empty[1][b]);
          else mbar_arrive(&d_empty[set][b]);
        }
      };
      // Tokens c0 .. c0+15 of the tile (those below ntok) through shared memory to 16-byte stores.
      const size_t trow = (size_t)tl.rowoff + tl.t0;
      const int r0 = MODE == kWide ? tl.row0 + set * kRows : tl.row0;
      const int live = min(kRows, p.seg[tl.sg].n_rows - r0);
      const int colbase = p.seg[tl.sg].col0 + r0;
      const int c = (tid & 15) * 8, tq = tid >> 4;
      const bool vec = MODE == kSwiglu || ((p.ldy % 8 == 0) && (colbase % 8 == 0) &&
                       (((reinterpret_cast<uintptr_t>(p.y) | reinterpret_cast<uintptr_t>(p.res) | reinterpret_cast<uintptr_t>(p.y2)) & 15) == 0));
      auto emit = [&](const float* v, int c0) {
        const int n = min(kStageTok, ntok - c0);
        if (MODE == kSwiglu) {
          const uint32_t o = out_u + 2 * feat;
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            sts16(o + (uint32_t)(i * kStagePitch), __float2half_rn(v[i]));
            sts16(o + (uint32_t)((kStageTok + i) * kStagePitch), __float2half_rn(v[16 + i]));
          }
          set_sync();
          const int F = p.seg[0].n_rows;
          if (c < live) {  // F is a multiple of 8: a run of eight is live or not
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const int t = tq + 8 * q;
              if (t >= n) break;
              const uint4 g4 = lds128(out_u + (uint32_t)(t * kStagePitch + c * 2));
              const uint4 u4 = lds128(out_u + (uint32_t)((kStageTok + t) * kStagePitch + c * 2));
              const uint32_t gw[4] = {g4.x, g4.y, g4.z, g4.w}, uw[4] = {u4.x, u4.y, u4.z, u4.w};
              uint32_t a[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const float2 g = __half22float2(as_h2(gw[e])), u = __half22float2(as_h2(uw[e]));
                a[e] = as_u32(__floats2half2_rn(silu_times(g.x, u.x), silu_times(g.y, u.y)));
              }
              const size_t tr = trow + c0 + t;
              *reinterpret_cast<uint4*>(p.act + tr * p.ldact + r0 + c) = make_uint4(a[0], a[1], a[2], a[3]);
              if (p.y) {
                *reinterpret_cast<uint4*>(p.y + tr * p.ldy + r0 + c) = g4;
                *reinterpret_cast<uint4*>(p.y + tr * p.ldy + F + r0 + c) = u4;
              }
            }
          }
          set_sync();  // the staging may be filled again
          return;
        }
        const bool mine8 = vec && c + 8 <= live;
        uint4 r4[2];
        if (p.res && mine8) {
#pragma unroll
          for (int q = 0; q < 2; ++q)
            if (tq + 8 * q < n) r4[q] = __ldg(reinterpret_cast<const uint4*>(p.res + (trow + c0 + tq + 8 * q) * p.ldy + colbase + c));
        }
        const uint32_t rows = out_u + (uint32_t)(buf * kStageTok * kStagePitch);
#pragma unroll
        for (int i = 0; i < 16; ++i) sts16(rows + (uint32_t)(i * kStagePitch + 2 * feat), __float2half_rn(v[i]));
        set_sync();  // (whoever fills this buffer again has passed the other one's barrier, behind these reads)
        buf ^= 1;
        if (mine8) {
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int t = tq + 8 * q;
            if (t >= n) break;
            const uint4 o4 = lds128(rows + (uint32_t)(t * kStagePitch + c * 2));
            const size_t off = (trow + c0 + t) * p.ldy + colbase + c;
            *reinterpret_cast<uint4*>(p.y + off) = o4;
            if (p.res) {
              const uint32_t ow[4] = {o4.x, o4.y, o4.z, o4.w}, rw[4] = {r4[q].x, r4[q].y, r4[q].z, r4[q].w};
              uint32_t z[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const float2 a = __half22float2(as_h2(ow[e])), r = __half22float2(as_h2(rw[e]));
                z[e] = as_u32(__floats2half2_rn(r.x + a.x, r.y + a.y));
              }
              *reinterpret_cast<uint4*>(p.y2 + off) = make_uint4(z[0], z[1], z[2], z[3]);
            }
          }
        } else if (c < live) {
          for (int t = tq; t < n; t += 8) {
            const size_t off = (trow + c0 + t) * p.ldy + colbase + c;
            for (int q = 0; q < min(8, live - c); ++q) {
              const uint32_t a = rows + (uint32_t)(t * kStagePitch + (c + q) * 2);
              uint16_t hv;
              asm volatile("ld.shared.u16 %0, [%1];" : "=h"(hv) : "r"(a));
              const __half o = __ushort_as_half(hv);
              p.y[off + q] = o;
              if (p.res) p.y2[off + q] = __float2half_rn(__half2float(p.res[off + q]) + __half2float(o));
            }
          }
        }
      };
      // ---- all parts but the last: added up in this thread's own words
      float* const own = p.own + ((size_t)blockIdx.x * (MODE == kDeep ? 1 : 2) + (MODE == kWide ? set : 0)) * kRows * p.nt + feat;
      auto add_own = [&](int c0, float* v) {  // (all loads before the first addition)
        float w[16 * kPlanes];
#pragma unroll
        for (int g = 0; g < kPlanes; ++g)
#pragma unroll
          for (int i = 0; i < 16; ++i) w[16 * g + i] = __ldcg(own + (size_t)(g * p.nt + c0 + i) * kRows);
#pragma unroll
        for (int i = 0; i < 16 * kPlanes; ++i) v[i] += w[i];
      };
      const int c_first = kJoined ? kStageTok * set : 0, c_step = kJoined ? 2 * kStageTok : kStageTok;
      int n_part = 1;
      if (SUMS == kHanded) {
        const int n_units = mine.u1 - mine.u0, part = part_units(p, n_units);
        n_part = (n_units + part - 1) / part;
#pragma unroll 1
        for (int q = 0; q + 1 < n_part && ok; ++q) {
          ok = wait_sums();
#pragma unroll 1
          for (int c0 = c_first; c0 < ntok && ok; c0 += c_step) {
            float v[16 * kPlanes];
            sums(c0, v);
            if (q) add_own(c0, v);
#pragma unroll
            for (int g = 0; g < kPlanes; ++g)
#pragma unroll
              for (int i = 0; i < 16; ++i) __stcg(own + (size_t)(g * p.nt + c0 + i) * kRows, v[16 * g + i]);
          }
          release();
        }
      }
      if (ok) ok = wait_sums();
      if (!ok) break;
      if (SUMS != kShared) {
        if (c_first >= ntok) release();
#pragma unroll 1
        for (int c0 = c_first; c0 < ntok; c0 += c_step) {
          float v[16 * kPlanes];
          sums(c0, v);
          if (c0 + c_step >= ntok) release();
          if (SUMS == kHanded && n_part > 1) add_own(c0, v);
          emit(v, c0);
        }
        continue;
      }
      // ---- The cluster's CTAs have a part of the sums each.  Runs of 16 tokens belong to them in turn: a CTA sends what it has of
      // the others' runs into their shared memory, 64 bytes to a thread, and adds up its own in ascending order of k.
      // (16-byte pieces are swizzled, so that eight lanes' pieces lie in different banks.)
      const uint32_t swz = (uint32_t)((lane >> 1) & 3);
      const uint32_t mine_at = (uint32_t)(feat * 64), recv_u = smem_u32(recv_s), bar_u = smem_u32(&recv_full[set]);
      // what CTA q leaves of run r: place of the run among the owner's, then of q among the others
      const int own_runs = ((ntok + kStageTok - 1) / kStageTok + p.parts - 1) / p.parts;  // of one CTA at most
      auto slot_of = [&](int r, int owner, int q) {
        return (uint32_t)((((r / p.parts) + (MODE == kWide ? set * own_runs : 0)) * (p.parts - 1) + (q < owner ? q : q - 1)) * kPlanes * kPartBytes);
      };
      int expect = 0;
      for (int r = c_first / kStageTok; r * kStageTok < ntok; r += c_step / kStageTok) expect += r % p.parts == rank;
      if (tid == 0 && expect) mbar_expect_tx(&recv_full[set], (uint32_t)(expect * (p.parts - 1) * kPlanes * kPartBytes));
#pragma unroll 1
      for (int c0 = c_first; c0 < ntok; c0 += c_step) {
        const int r = c0 / kStageTok, owner = r % p.parts;
        if (owner == rank) continue;
        float v[16 * kPlanes];
        sums(c0, v);
        const uint32_t dst = remote(recv_u + slot_of(r, owner, rank) + mine_at, owner), bar = remote(bar_u, owner);
#pragma unroll
        for (int g = 0; g < kPlanes; ++g)
#pragma unroll
          for (int i = 0; i < 4; ++i) st_async4(dst + g * kPartBytes + 16u * (i ^ swz), bar, v + 16 * g + 4 * i);
      }
      if (expect) {
        bool here = true;
        if (quarter == 0) here = wait_warp(&recv_full[set], 0);
        ok = set_all(here);
        if (!ok) break;
      }
#pragma unroll 1
      for (int c0 = c_first; c0 < ntok; c0 += c_step) {
        const int r = c0 / kStageTok;
        if (r % p.parts != rank) continue;
        float v[16 * kPlanes];
#pragma unroll
        for (int i = 0; i < 16 * kPlanes; ++i) v[i] = 0.f;
#pragma unroll 1
        for (int q = 0; q < p.parts; ++q) {
          if (q == rank) {
            float w[16 * kPlanes];
            sums(c0, w);
#pragma unroll
            for (int i = 0; i < 16 * kPlanes; ++i) v[i] += w[i];
            continue;
          }
          const uint32_t src = recv_u + slot_of(r, rank, q) + mine_at;
#pragma unroll
          for (int g = 0; g < kPlanes; ++g)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const uint4 w = lds128(src + g * kPartBytes + 16u * (i ^ swz));
              float* o = v + 16 * g + 4 * i;
              o[0] += __uint_as_float(w.x), o[1] += __uint_as_float(w.y), o[2] += __uint_as_float(w.z), o[3] += __uint_as_float(w.w);
            }
        }
        emit(v, c0);
      }
    }
  }
  __syncwarp();
  if (!ok && lane == 0) raise_status(p.status, 3);
  __syncwarp();
  tc_fence_before();
  if (cluster) {  // nobody leaves while another CTA may send to it
    if (warp < 4 || warp >= 12) cluster_wait();
    cluster_arrive();
    cluster_wait();
  } else {
    __syncthreads();
  }
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}


// ------------------------------------------------------------------------------------------------- host side
int feature_tiles(const GemmParams& g, int mode, int seg) {
  if (mode == kSwiglu) return seg ? 0 : (g.seg[0].n_rows + kRows - 1) / kRows;
  const int rows = mode == kDeep ? kRows : 2 * kRows;
  return (g.seg[seg].n_rows + rows - 1) / rows;
}

template <int N>
using Const = std::integral_constant<int, N>;

// Depths of the rings, and the shared memory of a CTA (0: it does not fit).  The places for codes (HBM: three units at least on their way) and
// activations (L2: three halves of a unit).  With `deep` both are even: a place belongs to one group, or half, so that a phase's parity tells
// its waiter which one it is.
constexpr size_t kMostSmem = 227 * 1024 - 1024;
struct FewRings {
  int codes, xs;
  size_t smem;
};
FewRings rings_of(int mode, int nt, int parts, bool lines, size_t list) {
  const size_t own_runs = ((nt + kStageTok - 1) / kStageTok + parts - 1) / parts;
  const size_t fixed = 1024 + kStageBytes + own_runs * (parts - 1) * (mode == kDeep ? 1 : 2) * kPartBytes + list + (lines ? 0 : 16 * kFeed * kFeedBytes);
  const size_t xb = (size_t)nt * 256, cb = (size_t)(mode == kDeep ? 1 : 2) * (kCodeBytes + (lines ? kScaleBytes : 0));
  const int step = mode == kDeep ? 2 : 1;
  auto fits = [&](int codes, int xs) { return fixed + xs * xb + codes * cb <= kMostSmem; };
  FewRings r{mode == kDeep ? 4 : 3, mode == kDeep ? 4 : 3, 0};
  if (!fits(r.codes, r.xs)) r.codes = 2;
  if (!fits(r.codes, r.xs)) return r;
  for (bool more = true; more;) {
    more = false;
    if (r.xs < 2 * r.codes && r.xs + step <= kMaxX && fits(r.codes, r.xs + step)) r.xs += step, more = true;
    if (r.codes + step <= kMaxCodes && fits(r.codes + step, r.xs)) r.codes += step, more = true;
  }
  r.smem = fixed + r.xs * xb + r.codes * cb;
  return r;
}

// Time in us of one way to divide the work: launch and first loads, waves of units (expansion or MMAs, whichever is longer, and what the CTAs take
// from each other in the L2 cache), accumulators in turn, the cluster's exchange, sums that are handed over.  Fitted to 2939 launches back to
// back on new weights (21 products, 12 to 640 tokens; 5 % rms within 1.15 times the best way; the way chosen is 1.3 % slower than the best one);
// long launches run at the power limit.  `active`: the part of the SMs that have a CTA.
double few_us(const GemmParams& g, int rows, int mode, int nt, int n_tt, double active, int waves, int units, int parts, int turns, int handed) {
  const bool deep = mode == kDeep;
  const double e = (deep ? 0.407 : 0.933) * (g.mx ? 1.0 : 1.056), m = (deep ? 0.0042 : 0.0093) * nt;
  const double unit = std::pow(e * e * e * e + m * m * m * m, 0.25) + (deep ? 0.00063 : 0.0) * nt * active;
  const double us = 0.78 + 3.15 * active + 0.0157 * nt + waves * units * unit + (parts > 1 || turns > 1 || handed ? 0.72 : 0.0) + 0.22 * (turns - 1) +
                    (parts > 1 ? 0.02 * nt + 0.44 * parts : 0.0) + waves * handed * (nt <= 64 ? 0.23 : 0.48 + 0.0147 * nt);
  return std::max(us, 1.0 + 2e-6 / 1286 * nt * n_tt * rows * g.K);
}

// The fastest way whose chains are no longer than `limit` k (at least one unit).
GemmFewPlan plan_of(const GemmParams& g, int sm_count, int limit) {
  GemmFewPlan best{};
  best.us = 1e300;
  const int units = (g.K + kUnitK - 1) / kUnitK;
  limit = std::max(limit, kUnitK);
  int n = 0;
  for (int i = 0; i < g.n_seg; ++i) n += g.seg[i].n_rows;
  // (what every caller has, so that a plan is a function of the shapes)
  const uint64_t scratch = g.scratch ? std::min(g.scratch_bytes, gemm_scratch_bytes(g.T, n, g.K)) : 0;
  for (int mode : {kWide, kSwiglu, kDeep}) {
    if ((mode == kSwiglu) != (g.act != nullptr)) continue;
    int n_ft = 0, last = 0;
    for (int i = 0; i < g.n_seg; ++i) n_ft += feature_tiles(g, mode, i);
    for (int most : {128, 112, 96, 80, 64, 48, 32, 16}) {
      const int n_tt = (g.T + most - 1) / most, nt = ((g.T + n_tt - 1) / n_tt + 15) / 16 * 16;
      if (n_tt == last || (long long)n_ft * n_tt > 16ll * sm_count) continue;
      last = n_tt;
      const int tiles = n_ft * n_tt;
      for (int parts = 1; parts <= std::min(kMaxParts, units); ++parts) {
        // (clusters of more than two do not fill the machine: 33 of four, 26 of five, 22 of six at a time of 148 SMs)
        if (parts > 1 && tiles > (parts == 2 ? sm_count / 2 : (sm_count - 20) / parts)) break;
        const FewRings r = rings_of(mode, nt, parts, g.K % kUnitK == 0, 0);
        if (!r.smem || r.codes < (mode == kDeep ? 4 : 2)) continue;
        const int active = std::min(tiles * parts, sm_count), waves = (tiles * parts + sm_count - 1) / sm_count;
        const int per = (units + parts - 1) / parts, steps = mode == kDeep ? per : 2 * per;
        int turns = 1;
        while (turns < 4 && 2 * turns * nt <= 128 && waves == 1 && 2 * turns <= (mode == kDeep ? units / parts : 2 * (units / parts)) &&
               (steps + turns - 1) / turns * 128 > limit)
          turns *= 2;
        int max_units = per;
        uint64_t own = 0;
        if ((steps + turns - 1) / turns * 128 > limit) {
          if (parts > 1) continue;
          turns = 1;
          max_units = limit / (mode == kDeep ? 128 : 256);
          own = (uint64_t)std::min(tiles, sm_count) * (mode == kDeep ? 1 : 2) * kRows * nt * 4;
          if (own > scratch) continue;
        }
        const int handed = (per + max_units - 1) / max_units - 1;
        const double us = few_us(g, n, mode, nt, n_tt, (double)active / sm_count, waves, per, parts, turns, handed);
        if (us < best.us) best = GemmFewPlan{mode, nt, n_tt, parts, turns, max_units, us};
      }
    }
  }
  return best;
}

}  // namespace

int gemm_few_chain(const GemmParams& g, const GemmFewPlan& pl) {
  const int units = (g.K + kUnitK - 1) / kUnitK, per = (units + pl.parts - 1) / pl.parts, steps = pl.mode == kDeep ? 1 : 2;  // (of 128 k, a unit)
  int n = per;
  if (n > pl.max_units) n = (n + (n - 1) / pl.max_units) / ((n + pl.max_units - 1) / pl.max_units);
  return std::min(g.K, (n * steps + pl.turns - 1) / pl.turns * 128);
}

bool gemm_few_eligible(const GemmParams& g, int sm_count, bool pairs, GemmFewPlan* plan) {
  if (g.w16 || g.n_seg < 1 || g.n_seg > 3 || g.K % 32 || g.K > (1 << 24) || g.ldx % 8) return false;
  if (reinterpret_cast<uintptr_t>(g.x) & 15) return false;
  if ((g.res != nullptr) != (g.y2 != nullptr)) return false;
  for (int i = 0; i < g.n_seg; ++i) {
    if (reinterpret_cast<uintptr_t>(g.seg[i].base) & 15) return false;
    if (g.grp_tab[i] || (long long)g.seg[i].n_rows * (g.K / 16) >= 1ll << 31) return false;
  }
  if (g.act && (g.n_seg != 2 || g.seg[0].n_rows != g.seg[1].n_rows || g.seg[0].n_rows % 8 || g.ldact % 8 || g.ldy % 8 || g.res ||
                ((reinterpret_cast<uintptr_t>(g.act) | reinterpret_cast<uintptr_t>(g.y)) & 15)))
    return false;
  // (grouped: up to 80 rows to an expert.  512 tokens through 8 of 128 experts, 32 rows, 187 -> 140 us for the layer; 300 through 4 of 16, 75 rows,
  // 94 -> 88; 1500 through 4 of 64, 94 rows, 218 -> 217; 2048 through 8 of 128, 128 rows, 346 -> 366)
  if (g.grp_off) return g.n_groups > 0 && g.T <= 80 * g.n_groups && (g.n_seg == 1 || g.act) && g.grp_stride % 16 == 0 && !g.res;
  // (against the best of all ways and kernels the choice loses 1.5 %: both models are off by about 5 %)
  const GemmOther other = gemm_other(g, sm_count, pairs);
  const GemmFewPlan pl = *plan = plan_of(g, sm_count, other.chain);
  return pl.parts && pl.us <= 0.96 * other.us;
}

cudaError_t launch_gemm_few(const GemmParams& g, const GemmFewPlan& pl, int sm_count, cudaStream_t st, uint64_t* n_launch, std::string* err) {
  TensorMapEncodeFn enc = tensor_map_encode();
  if (!enc) {
    if (err) *err = "cuTensorMapEncodeTiled is not available from the driver";
    return cudaErrorNotSupported;
  }
  const int mode = g.grp_off ? (g.act ? kSwiglu : kWide) : pl.mode;
  FewParams p{};
  p.n_seg = g.n_seg;
  int n_ft = 0, col = 0;
  for (int i = 0; i < g.n_seg; ++i) {
    p.seg[i] = TileSeg{g.seg[i].base, g.seg[i].n_rows, n_ft, col};
    n_ft += feature_tiles(g, mode, i);
    col += g.seg[i].n_rows;
  }
  p.K = g.K;
  p.T = g.T;
  p.units = (g.K + kUnitK - 1) / kUnitK;
  const bool lines = g.K % kUnitK == 0;
  p.grp_stride = g.grp_stride;
  p.tile_rows = mode == kWide ? 2 * kRows : kRows;
  p.n_ft = n_ft;
  int max_blocks = 0;  // of an expert's rows, at most
  if (g.grp_off) {
    if (g.n_groups <= 0 || g.n_groups > 1024 || g.T <= 0 || g.T >= 1 << 22) return cudaErrorInvalidValue;
    const double mean = (double)g.T / g.n_groups;
    auto height = [&](double rows) {
      const int parts = (int)std::ceil(rows / kMaxTok);
      return std::min(kMaxTok, ((int)std::ceil(rows / parts) + 15) / 16 * 16);
    };
    p.nt = std::max(height(mean + 3 * std::sqrt(mean)), std::min(64, height(mean + 5 * std::sqrt(mean))));
    p.n_groups = g.n_groups;
    max_blocks = std::min(g.n_groups, g.T) + g.T / p.nt;
    p.ft_per = n_ft;
    p.n_tt = 1;
    p.workers = (int)std::min<long long>((long long)n_ft * max_blocks, sm_count);
  } else {
    p.nt = pl.nt;
    p.n_tt = pl.n_tt;
    p.n_whole = n_ft * pl.n_tt;
    p.workers = std::min(p.n_whole, sm_count / pl.parts);
  }
  p.y = g.y;
  p.ldy = g.ldy;
  p.res = g.res;
  p.y2 = g.y2;
  p.act = g.act;
  p.ldact = g.ldact;
  p.parts = g.grp_off ? 1 : pl.parts;
  p.turns = g.grp_off ? 1 : pl.turns;
  p.max_units = g.grp_off ? p.units : pl.max_units;
  p.own = (float*)g.scratch;
  p.status = g.status;
  p.grp_off = g.grp_off;
  FewMaps maps{};
  // activations as [64 k][tokens][chunks of 64 k]; boxes as high as tiles may be (grouped: any height)
  // (K no multiple of 256: as [k][tokens], so that k beyond its end read as zeros, in boxes of 64 k)
  const cuuint64_t xd[3] = {lines ? 64 : (cuuint64_t)g.K, (cuuint64_t)g.T, lines ? (cuuint64_t)g.K / 64 : 1}, xs[2] = {(cuuint64_t)g.ldx * 2, 128};
  const cuuint32_t one[3] = {1, 1, 1};
  const int last = ((g.T - (p.n_tt - 1) * p.nt) + 15) / 16;
  for (int h = 1; h <= p.nt / 16; ++h) {
    if (!g.grp_off && h != p.nt / 16 && h != last) continue;
    const cuuint32_t xb[3] = {64, (cuuint32_t)(16 * h), lines ? 2u : 1u};
    if (enc(&maps.x[h - 1], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<__half*>(g.x), xd, xs, xb, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
      if (err) *err = "cuTensorMapEncodeTiled failed for the activation tile";
      return cudaErrorInvalidValue;
    }
  }
  for (int i = 0; i < 3; ++i) {
    if (i >= g.n_seg) {
      maps.codes[i] = maps.codes[0];
      maps.scales[i] = maps.scales[0];
      continue;
    }
    const GemvSeg& sg = g.seg[i];
    const cuuint64_t row = (cuuint64_t)g.K / 2, groups = g.grp_off ? (cuuint64_t)g.n_groups : 1, slice = g.grp_off ? (cuuint64_t)g.grp_stride : row * sg.n_rows;
    const cuuint64_t wd[3] = {row, (cuuint64_t)sg.n_rows, groups}, ws[2] = {row, slice};
    const cuuint32_t wb[3] = {128, kRows, 1};
    // scales: [n_rows][K / 32] halves behind the codes, eight at a time
    const cuuint64_t sd[3] = {(cuuint64_t)g.K / 32, wd[1], groups}, ss[2] = {(cuuint64_t)g.K / 16, slice};
    const cuuint32_t sb[3] = {8, kRows, 1};
    maps.scales[i] = maps.codes[0];
    if (enc(&maps.codes[i], CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t*>(sg.base), wd, ws, wb, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS ||
        (lines && enc(&maps.scales[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, const_cast<uint8_t*>(sg.base) + (size_t)sg.n_rows * (g.K / 2), sd, ss, sb, one,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)) {
      if (err) *err = "cuTensorMapEncodeTiled failed for the weights";
      return cudaErrorInvalidValue;
    }
  }
  const size_t list = g.grp_off ? (size_t)(max_blocks + 1) * sizeof(uint32_t) : 0;
  const FewRings rings = rings_of(mode, p.nt, p.parts, lines, list);
  if (!rings.smem) return cudaErrorInvalidValue;
  p.codes = rings.codes;
  p.xs = rings.xs;
  p.list_at = (int)(rings.smem - 1024 - list);
  const size_t smem = rings.smem;
  ++*n_launch;
  const int how = p.parts > 1 || p.turns > 1 ? kShared : p.max_units < p.units ? kHanded : kPlain;
  auto run = [&](auto mode_of, auto how_of) {
    constexpr int kMode = decltype(mode_of)::value, kHow = decltype(how_of)::value;
    auto kernel = g.mx ? lines ? gemm_few_kernel<true, kMode, kHow, true> : gemm_few_kernel<true, kMode, kHow, false>
                       : lines ? gemm_few_kernel<false, kMode, kHow, true> : gemm_few_kernel<false, kMode, kHow, false>;
    static std::atomic<uint64_t> attr_done[4];
    const cudaError_t e = smem_limit_once(&attr_done[(g.mx ? 2 : 0) + lines], {reinterpret_cast<const void*>(kernel)}, kMostSmem);
    if (e != cudaSuccess) return e;
    return launch_dep(kernel, dim3(p.workers * p.parts), dim3(kFewThreads), smem, st, g.pdl, p.parts, maps, p);
  };
  auto with = [&](auto mode_of) {
    return how == kPlain ? run(mode_of, Const<kPlain>{}) : how == kShared ? run(mode_of, Const<kShared>{}) : run(mode_of, Const<kHanded>{});
  };
  return mode == kWide ? with(Const<kWide>{}) : mode == kSwiglu ? with(Const<kSwiglu>{}) : with(Const<kDeep>{});
}

}  // namespace ats
