// What the prompt GEMMs with persistent workers share (kernels_gemm_pair.cu: a worker is a pair of CTAs; kernels_gemm_few.cu: a CTA):
// the division of the tiles among the workers, the list of the experts' blocks of rows, the expansion of 4-bit codes, and
// warp-wide forms of loads, barriers and tests.
#pragma once
#include "ats_internal.h"
#include "sm100_umma.cuh"

namespace ats {
namespace {

struct TileSeg {
  const uint8_t* base;
  int n_rows;
  int tile0;  // first feature tile of the segment
  int col0;   // first output column of the segment
};
struct TileWork {
  TileSeg seg[3];
  int n_seg;
  int K, T;
  int n_ft, n_tt;     // feature tiles, token tiles
  int tile_rows;      // features of a tile (SwiGLU: gate features)
  int nt;             // tokens per tile
  int units;          // per tile
  int workers;
  int n_whole;        // tiles that a worker has to itself; the units of the others are divided over ...
  int split_workers;  // ... this many workers
  __half* act;        // SwiGLU of segments 0 (gate) and 1 (up)
  const int* grp_off; // grouped form: row offsets per expert
  int ft_per, n_groups, list_at;  // ... feature tiles per expert, experts, place of the list of blocks in shared memory
};

// One stretch of a worker's work: units u0 .. u1-1 of a tile.
struct Stretch {
  int tile, u0, u1;
};
// Walks a worker's stretches; the same sequence in every role.
struct Walk {
  int tile, step, n_whole;  // whole tiles: worker, worker + workers, ... (neighbours in L2 run at the same time)
  int units;
  unsigned at, end;         // the worker's range of the last tiles' units, counted from tile n_whole on
  __device__ __forceinline__ Walk(const TileWork& p, int worker, int whole) {
    units = p.units;
    tile = worker;
    step = p.workers;
    n_whole = whole;
    const unsigned n = p.grp_off ? 0u : (unsigned)(p.n_ft * p.n_tt - whole) * units;  // (below 148 tiles of 128k units: K is at most 2^24)
    at = worker < p.split_workers ? n * worker / p.split_workers : 0;
    end = worker < p.split_workers ? n * (worker + 1) / p.split_workers : 0;
  }
  __device__ __forceinline__ bool next(Stretch& s) {
    if (tile < n_whole) {
      s.tile = tile;
      s.u0 = 0;
      s.u1 = units;
      tile += step;
      return true;
    }
    if (at >= end) return false;
    const int t = (int)(at / (unsigned)units);
    s.tile = n_whole + t;
    s.u0 = (int)at - t * units;
    s.u1 = min(units, s.u0 + (int)(end - at));
    at += s.u1 - s.u0;
    return true;
  }
};
// Which rows, tokens and expert a tile stands for.
struct Tile {
  int sg, row0;        // segment, first feature row of the tile within it
  int t0, T, rowoff;   // first token, tokens of the matrix (of the block of an expert's rows), its first row
  int expert;
};
// Grouped form: the experts' rows in blocks of at most nt, in shared memory: expert | first row << 10.  The blocks follow one another, so the
// next one's first row ends it (behind the last: all rows).
__device__ __forceinline__ Tile tile_of(const TileWork& p, int tile, const uint32_t* blocks) {
  Tile r;
  int ft = tile / (p.grp_off ? p.ft_per : p.n_tt);
  if (p.grp_off) {  // feature tiles of one block after another
    const uint32_t b = blocks[ft], e = blocks[ft + 1];
    ft = tile - ft * p.ft_per;
    r.expert = (int)(b & 1023u);
    r.t0 = 0;
    r.rowoff = (int)(b >> 10);
    r.T = (int)(e >> 10) - r.rowoff;
  } else {
    r.expert = 0;
    r.t0 = (tile - ft * p.n_tt) * p.nt;
    r.T = p.T;
    r.rowoff = 0;
  }
  r.sg = 0;
  if (!p.act)
    while (r.sg + 1 < p.n_seg && ft >= p.seg[r.sg + 1].tile0) ++r.sg;
  r.row0 = (ft - p.seg[r.sg].tile0) * p.tile_rows;
  return r;
}
// Lists the blocks (one warp); returns their number in lane 31.
__device__ __forceinline__ int list_blocks(const TileWork& p, uint32_t* blocks, int lane) {
  const int per = (p.n_groups + 31) / 32, e0 = min(lane * per, p.n_groups), e1 = min(e0 + per, p.n_groups);
  int n = 0, incl;
  for (int e = e0; e < e1; ++e) n += (p.grp_off[e + 1] - p.grp_off[e] + p.nt - 1) / p.nt;
  incl = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  int at = incl - n;
  for (int e = e0; e < e1; ++e) {
    const int hi = p.grp_off[e + 1];
    for (int r = p.grp_off[e]; r < hi; r += p.nt) blocks[at++] = (uint32_t)(e | r << 10);
  }
  if (lane == 31) blocks[incl] = (uint32_t)p.T << 10;
  return incl;
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) { asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory"); }
// Loads are issued like MMAs: by all lanes of a warp, in flow that is the same for the warp, with the instruction left to one.
__device__ __forceinline__ void tma_3d_one(uint32_t one, uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "{\n.reg .pred q;\nsetp.ne.b32 q, %6, 0;\n@q cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, "
      "{%2, %3, %4}], [%5];\n}" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar)), "r"(one)
      : "memory");
}
__device__ __forceinline__ void expect_tx_one(uint32_t one, uint64_t* bar, uint32_t bytes) {
  asm volatile("{\n.reg .pred q;\nsetp.ne.b32 q, %2, 0;\n@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}" ::"r"(smem_u32(bar)),
               "r"(bytes), "r"(one)
               : "memory");
}
// The value of any lane (all hold the same) as one the compiler knows to be the same for the warp.
__device__ __forceinline__ int uniform(int v) { return (int)__reduce_max_sync(0xffffffffu, (unsigned)v); }
// (32-bit shared addresses: the pointers into the aligned dynamic array would make generic accesses)
__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts16(uint32_t a, __half v) { asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"(__half_as_ushort(v)) : "memory"); }
__device__ __forceinline__ __half2 as_h2(uint32_t v) {
  __half2 h;
  *reinterpret_cast<uint32_t*>(&h) = v;
  return h;
}
__device__ __forceinline__ uint32_t as_u32(__half2 h) { return *reinterpret_cast<uint32_t*>(&h); }
// (v & mask) | or_bits in one instruction (left to itself the compiler takes eight logic operations per word, not five)
__device__ __forceinline__ uint32_t and_or(uint32_t v, uint32_t mask, uint32_t or_bits) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(v), "r"(mask), "r"(or_bits));
  return d;
}
// One code word (8 codes, internal nibble order) times the block scale -> 8 fp16 weights, k ascending.
template <bool MX>
__device__ __forceinline__ void expand_word(uint32_t w, __half2 s2, uint32_t* o) {
  if (MX) {
    // byte j of a word: codes (0, 2), (4, 6), (1, 3), (5, 7); half of the instructions of shifts and masks (77 tokens, 28672 x
    // 4096: 41.1 -> 37.2 us)
    uint32_t c[4];
    cvt_e2m1x8(w, c);
    o[0] = as_u32(__hmul2(as_h2(__byte_perm(c[0], c[2], 0x5410)), s2));
    o[1] = as_u32(__hmul2(as_h2(__byte_perm(c[0], c[2], 0x7632)), s2));
    o[2] = as_u32(__hmul2(as_h2(__byte_perm(c[1], c[3], 0x5410)), s2));
    o[3] = as_u32(__hmul2(as_h2(__byte_perm(c[1], c[3], 0x7632)), s2));
  } else {
    const uint32_t kMagic = 0x64006400u, w8 = w >> 8;
    const __half2 k1032 = as_h2(0x64086408u), k16th = as_h2(0x2C002C00u), kM72 = as_h2(0xD480D480u);
    o[0] = as_u32(__hmul2(__hsub2(as_h2(and_or(w, 0x000F000Fu, kMagic)), k1032), s2));
    o[1] = as_u32(__hmul2(__hfma2(as_h2(and_or(w, 0x00F000F0u, kMagic)), k16th, kM72), s2));
    o[2] = as_u32(__hmul2(__hsub2(as_h2(and_or(w8, 0x000F000Fu, kMagic)), k1032), s2));
    o[3] = as_u32(__hmul2(__hfma2(as_h2(and_or(w8, 0x00F000F0u, kMagic)), k16th, kM72), s2));
  }
}
// A warp waits with all its lanes; try_wait lets the hardware park it, so that the many waiting warps leave the issue slots
// and the barrier unit to those that work (polling with test_wait cost 3 to 20 %).
__device__ __forceinline__ bool wait_warp(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait_suspending(bar, parity));
}
// A test whose result is looked at later: its latency (about 200 cycles here) passes under other work.
__device__ __forceinline__ bool peek(uint64_t* bar, uint32_t parity) { return mbar_test_wait(bar, parity); }

__device__ __forceinline__ void tmem_ld_x16(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
        "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait_x16(uint32_t* v) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]),
                 "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])::"memory");
}

}  // namespace
}  // namespace ats
