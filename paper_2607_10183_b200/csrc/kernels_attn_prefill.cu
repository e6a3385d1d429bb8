// Causal grouped-query attention of a prompt chunk over the KV cache on the 5th-generation tensor cores (sm_100a).
//
// A CTA owns two tiles of 128 query rows: the same 128 tokens of two query heads that share a kv head (or, when the group
// is odd, two consecutive token blocks of one head).  Where that leaves half of the SMs idle, both are the same tokens of one head, over the even and
// the odd key blocks, and their sums meet at the end.  Key and value blocks of 128 cache rows stream through a ring in shared
// memory by TMA and serve both tiles.  Per tile and block: S = Q K^T (both operands in shared memory, 128 x 128 fp32
// accumulator in tensor memory), softmax by four warps with one query row per thread (the row lies along the thread's
// tensor-memory lane, so maximum and sum need no shuffles), P as fp16 back into tensor memory over S, O += P V with P as
// the tensor-memory operand and V as the MN-major shared-memory operand (the cache's own row layout).  The tensor core works
// on one tile while the softmax of the other runs.
//
// When a row's running maximum grows, the accumulated O has to be scaled down, a round trip through tensor memory: four warps
// of their own do that, from factors that the softmax warps leave in shared memory, while those go on with the exponentials.
//
// What bounds it: per tile and block the chain S -> softmax -> P V is serial and the two tiles only overlap each other; the
// exponentials (16 a cycle and SM: 2048 cycles for both tiles' 128 x 128 scores) are the busiest unit.  Measured with 32
// query and 8 kv heads of 128: 2048 tokens after 2048 others 127 us = 812 TFLOP/s, 512 tokens from position 0 17.3 us; the
// mma.sync kernel takes 720 and 34 us there.
//
// Roles: warp 0 = TMA producer, warp 1 = tensor-memory allocation and MMA issue, warps 4..7 / 8..11 = softmax and output of
// the first / second tile, warps 12..15 = rescaling of O.  Heavy token blocks (long contexts) are scheduled first.  Every
// mbarrier wait is bounded; on expiry the CTA raises the status word, skips the rest of its work, frees its tensor memory
// and returns.
#include "ats_internal.h"
#include "sm100_umma.cuh"

namespace ats {

namespace {

constexpr int kQRows = 128;   // query rows per tile (MMA M)
constexpr int kKeys = 128;    // cache rows per block
constexpr int kRing = 5;      // key / value blocks in flight
constexpr int kAttnThreads = 512;

struct AttnTcParams {
  __half* out;        // [T][n_q][D]
  int T, n_q, group, pos0;
  int pair_heads;     // 1: the two tiles are two heads of one token block; 0: two token blocks of one head
  int n_tb;           // token blocks (or pairs of them) in the grid
  float scale_log2;   // 1/sqrt(d) * log2(e)
  int* status;
};

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_half2(float a, float b) {
  const __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// SPLIT: the two tiles are one, tile x taking the key blocks 2 j + x.
template <int D, bool SPLIT>
__global__ void __launch_bounds__(kAttnThreads, 1)
    attn_prefill_tc_kernel(const __grid_constant__ CUtensorMap qmap, const __grid_constant__ CUtensorMap kmap,
                           const __grid_constant__ CUtensorMap vmap, const AttnTcParams p) {
  constexpr int NC = D / 64;                   // 64-element chunks of a head row (one swizzle row each)
  constexpr int kTileBytes = kQRows * D * 2;   // one query tile
  constexpr int kSlot = kKeys * D * 2;         // one key or value block
  constexpr int kChunk = 128 * 128;            // bytes of one 64-element chunk of 128 rows
  constexpr uint32_t kColO = 256;              // accumulators: S (then P) of tile x at 128 x, O at 256 + 128 x
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* q_s = smem;
  uint8_t* kv_s = smem + 2 * kTileBytes;
  __shared__ uint64_t q_full, kv_full[kRing], kv_empty[kRing], s_full[2], p_full[2], f_full[2], o_ok[2], o_done[2];
  __shared__ float factor_s[2][kQRows];  // what the row's O shrinks by
  __shared__ uint32_t tmem_s;
  __shared__ int fail_s;
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // (the same for the warp, and known to be)

  // ---- which tiles
  const int per_tb = gridDim.x / p.n_tb;                // work items of a token block: head pairs or heads
  const int tb = p.n_tb - 1 - (int)blockIdx.x / per_tb;  // the longest contexts first
  const int item = blockIdx.x % per_tb;
  const int head0 = p.pair_heads ? 2 * item : item, head1 = p.pair_heads ? head0 + 1 : head0;
  const bool same_tb = p.pair_heads || SPLIT;
  const int t0[2] = {same_tb ? tb * kQRows : tb * 2 * kQRows, same_tb ? tb * kQRows : tb * 2 * kQRows + kQRows};
  const int kvh = head0 / p.group;
  const int last_t = min(p.T, t0[1] + kQRows) - 1;      // last token either tile holds (a second tile may lie beyond T)
  const int n_kb = (p.pos0 + max(last_t, min(p.T, t0[0] + kQRows) - 1)) / kKeys + 1;
  const int nb0 = SPLIT ? (n_kb + 1) / 2 : n_kb, nb1 = SPLIT ? n_kb / 2 : n_kb;  // key blocks of each tile

  if (threadIdx.x == 0) {
    fail_s = 0;
    mbar_init(&q_full, 1);
    for (int s = 0; s < kRing; ++s) {
      mbar_init(&kv_full[s], 1);
      mbar_init(&kv_empty[s], 1);
    }
    for (int x = 0; x < 2; ++x) {
      mbar_init(&s_full[x], 1);
      mbar_init(&p_full[x], 4);
      mbar_init(&f_full[x], 4);
      mbar_init(&o_ok[x], 4);
      mbar_init(&o_done[x], 1);
    }
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_s, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_s;
  if (warp == 0) asm volatile("griddepcontrol.wait;" ::: "memory");  // everything read comes through this warp's copies
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // 128 registers a thread at launch; the softmax warps need more: 56 + 88 + 2 x 184 = 4 x 128
  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    if (warp == 0) {
      if (lane == 0) {
        mbar_expect_tx(&q_full, 2 * kTileBytes);
        for (int x = 0; x < 2; ++x)
          for (int c = 0; c < NC; ++c)
            tma_load_3d(q_s + x * kTileBytes + c * kChunk, &qmap, c * 64, x ? head1 : head0, t0[x], &q_full);
        // ring contents: K0, V0, K1, V1, ...
        for (int i = 0; i < 2 * n_kb; ++i) {
          const int s = i % kRing;
          if (i >= kRing && !mbar_wait(&kv_empty[s], ((i / kRing) - 1) & 1)) {
            fail_s = 1;
            break;
          }
          mbar_expect_tx(&kv_full[s], kSlot);
          for (int c = 0; c < NC; ++c)
            tma_load_3d(kv_s + s * kSlot + c * kChunk, (i & 1) ? &vmap : &kmap, c * 64, (i >> 1) * kKeys, kvh, &kv_full[s]);
        }
      }
    } else if (warp == 1) {
      constexpr uint32_t idesc_s = umma_idesc_f16(128, kKeys), idesc_o = umma_idesc_f16(128, D, true);
      const uint32_t one = elect_one();
      const uint64_t qd = umma_desc_sw128(smem_u32(q_s));
      const uint64_t kd = umma_desc_sw128(smem_u32(kv_s)), vd = umma_desc_sw128(smem_u32(kv_s), kChunk);
      auto issue_s = [&](int x, int slot) {
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint64_t off = (uint64_t)((kk / 4) * (kChunk >> 4) + (kk % 4) * 2);
          umma_ss(one, 128u * x, qd + (uint64_t)(x * (kTileBytes >> 4)) + off, kd + off + (uint64_t)(slot * (kSlot >> 4)), idesc_s,
                  kk > 0);
        }
        umma_commit_to(one, &s_full[x]);
      };
      auto issue_o = [&](int x, int slot, bool accumulate) {
#pragma unroll
        for (int kk = 0; kk < kKeys / 16; ++kk)
          umma_ts(one, kColO + 128u * x, 128u * x + 8u * kk, vd + (uint64_t)(slot * (kSlot >> 4) + kk * (2048 >> 4)), idesc_o,
                  accumulate || kk > 0);
      };
      bool ok = mbar_wait_all(&q_full, 0) && mbar_wait_all(&kv_full[0], 0);
      if (ok && SPLIT) {
        // every block serves one tile: K_b at position 2 b of the ring's sequence, V_b behind it
        auto full = [&](int i) { return mbar_wait_all(&kv_full[i % kRing], (i / kRing) & 1); };
        tc_fence_after();
        issue_s(0, 0);
        umma_commit_to(one, &kv_empty[0]);
        if (nb1) {
          ok = full(2);
          if (ok) {
            tc_fence_after();
            issue_s(1, 2 % kRing);
            umma_commit_to(one, &kv_empty[2 % kRing]);
          }
        }
        for (int j = 0; j < nb0 && ok; ++j) {
#pragma unroll
          for (int x = 0; x < 2 && ok; ++x) {
            if (j >= (x ? nb1 : nb0)) break;
            const int iv = 2 * (2 * j + x) + 1, ik = iv + 3;  // V of this block, K of the tile's next
            ok = full(iv) && (j == 0 || mbar_wait_all(&o_ok[x], (j - 1) & 1)) && mbar_wait_all(&p_full[x], j & 1);
            if (!ok) break;
            tc_fence_after();
            issue_o(x, iv % kRing, j > 0);
            if (j + 1 == (x ? nb1 : nb0)) umma_commit_to(one, &o_done[x]);
            umma_commit_to(one, &kv_empty[iv % kRing]);
            if (j + 1 < (x ? nb1 : nb0)) {
              ok = full(ik);
              if (!ok) break;
              issue_s(x, ik % kRing);  // behind the product that reads P out of the same columns
              umma_commit_to(one, &kv_empty[ik % kRing]);
            }
          }
        }
      } else {
        if (ok) {
          tc_fence_after();
          issue_s(0, 0);
          issue_s(1, 0);
          umma_commit_to(one, &kv_empty[0]);
        }
        for (int j = 0; j < n_kb && ok; ++j) {
          const int iv = 2 * j + 1, ik = 2 * j + 2;  // ring positions of V_j and K_{j+1}
          const int sv = iv % kRing, sk = ik % kRing;
#pragma unroll
          for (int x = 0; x < 2 && ok; ++x) {
            ok = (x || mbar_wait_all(&kv_full[sv], (iv / kRing) & 1)) && (j == 0 || mbar_wait_all(&o_ok[x], (j - 1) & 1)) &&
                 mbar_wait_all(&p_full[x], j & 1);
            if (!ok) break;
            tc_fence_after();
            issue_o(x, sv, j > 0);
            if (j + 1 == n_kb) umma_commit_to(one, &o_done[x]);
            if (x) umma_commit_to(one, &kv_empty[sv]);
            if (j + 1 < n_kb) {
              ok = x || mbar_wait_all(&kv_full[sk], (ik / kRing) & 1);
              if (!ok) break;
              issue_s(x, sk);  // behind the product that reads P out of the same columns
              if (x) umma_commit_to(one, &kv_empty[sk]);
            }
          }
        }
      }
      if (!ok && lane == 0) fail_s = 1;
    }
  } else if (warp >= 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
    const int quarter = warp & 3;
    const uint32_t t_o = tmem + ((uint32_t)(quarter * 32) << 16) + kColO;
    bool ok = true;
    for (int j = 1; j < nb0 && ok; ++j) {
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        if (j >= (x ? nb1 : nb0)) break;
        ok = mbar_wait_warp(&f_full[x], (j - 1) & 1, lane);
        if (!ok) break;
        tc_fence_after();
        const float f = factor_s[x][quarter * 32 + lane];
        if (__any_sync(0xffffffffu, f != 1.f)) {
          // the scores of this block are there, so the product that wrote O before them is complete
#pragma unroll
          for (int c = 0; c < D; c += 32) {
            uint32_t o[32];
            tmem_ld_x32(t_o + 128u * x + c, o);
            tmem_ld_wait_x32(o);
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
            tmem_st_x32(t_o + 128u * x + c, o);
          }
          tmem_st_wait();
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&o_ok[x]);
      }
    }
    if (!ok) fail_s = 1;
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 184;");
    const int x = (warp - 4) >> 2;                     // which tile
    const int quarter = warp & 3;                      // tensor-memory lanes this warp may access
    const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
    const uint32_t t_s = tmem + lanes + 128u * x, t_o = tmem + lanes + kColO + 128u * x;
    const int row = quarter * 32 + lane;
    const int t = t0[x] + row, qpos = p.pos0 + t;
    const int warp_pos = p.pos0 + t0[x] + quarter * 32;  // position of the warp's first row
    float m = 0.f;                                      // running maximum (scaled, log2)
    float2 l = make_float2(0.f, 0.f);                   // running sums (even and odd keys)
    bool ok = true;
    for (int j = 0; j < (x ? nb1 : nb0); ++j) {
      const int key0 = (SPLIT ? 2 * j + x : j) * kKeys;  // first key of the block
      ok = mbar_wait_warp(&s_full[x], j & 1, lane);
      if (!ok) break;
      tc_fence_after();
      float s[kKeys];
#pragma unroll
      for (int c = 0; c < kKeys; c += 32) tmem_ld_x32(t_s + c, reinterpret_cast<uint32_t*>(s) + c);
#pragma unroll
      for (int c = 0; c < kKeys; c += 32) tmem_ld_wait_x32(reinterpret_cast<uint32_t*>(s) + c);
      if (key0 + kKeys - 1 > warp_pos) {
#pragma unroll
        for (int i = 0; i < kKeys; ++i)
          if (key0 + i > qpos) s[i] = -INFINITY;
      }
      float mx[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
      for (int i = 4; i < kKeys; i += 8)
#pragma unroll
        for (int q = 0; q < 4; ++q) mx[q] = fmaxf(fmaxf(mx[q], s[i + q]), i + 4 + q < kKeys ? s[i + 4 + q] : s[i + q]);
      const float mb = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * p.scale_log2;
      if (j == 0) {
        m = SPLIT ? fmaxf(mb, -1e30f) : mb;  // finite: key 0 is visible to every row (split: no key of an odd block need be)
      } else {
        const float mn = fmaxf(m, mb), f = ex2(m - mn);
        m = mn;
        l.x *= f;
        l.y *= f;
        factor_s[x][row] = f;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&f_full[x]);
      }
      const float2 c2 = make_float2(p.scale_log2, p.scale_log2), m2 = make_float2(-m, -m);
#pragma unroll
      for (int c = 0; c < kKeys / 2; c += 32) {
        uint32_t pk[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          float2 e = fma_x2(make_float2(s[2 * (c + i)], s[2 * (c + i) + 1]), c2, m2);
          e.x = ex2(e.x);
          e.y = ex2(e.y);
          l = add_x2(l, e);
          pk[i] = pack_half2(e.x, e.y);
        }
        tmem_st_x32(t_s + c, pk);
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&p_full[x]);
    }
    float sum = l.x + l.y, scale0 = 1.f, scale1 = 0.f;
    if (ok && (x ? nb1 : nb0)) ok = mbar_wait_warp(&o_done[x], 0, lane);
    if (SPLIT) {
      // the odd blocks' sums go where queries and keys were (all that read them is done when both tiles are), the even tile adds them up
      float* odd_o = reinterpret_cast<float*>(kv_s);     // [D][128 rows]
      float2* odd_s = reinterpret_cast<float2*>(q_s);    // maximum and sum of a row over the odd blocks
      if (x == 1 && ok) {
        ok = mbar_wait_warp(&o_done[0], 0, lane);
        odd_s[row] = nb1 ? make_float2(m, sum) : make_float2(-1e30f, 0.f);
        if (ok && nb1) {
          tc_fence_after();
#pragma unroll
          for (int c = 0; c < D; c += 32) {
            uint32_t o[32];
            tmem_ld_x32(t_o + c, o);
            tmem_ld_wait_x32(o);
#pragma unroll
            for (int i = 0; i < 32; ++i) odd_o[(c + i) * kQRows + row] = __uint_as_float(o[i]);
          }
        }
      }
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (x == 0 && nb1) {
        const float2 od = odd_s[row];
        const float mm = fmaxf(m, od.x);
        scale0 = ex2(m - mm);
        scale1 = ex2(od.x - mm);
        sum = sum * scale0 + od.y * scale1;
      }
    }
    if (ok) {
      tc_fence_after();
      const float inv = 1.0f / sum;
      const float* odd_o = reinterpret_cast<const float*>(kv_s) + row;
      const bool merge = SPLIT && nb1;
      __half* dst = p.out + ((size_t)t * p.n_q + (x ? head1 : head0)) * D;
#pragma unroll
      for (int c = 0; c < D && !(SPLIT && x); c += 32) {
        uint32_t o[32];
        tmem_ld_x32(t_o + c, o);
        tmem_ld_wait_x32(o);
        if (merge) {
#pragma unroll
          for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * scale0 + odd_o[(c + i) * kQRows] * scale1);
        }
        if (t < p.T) {
#pragma unroll
          for (int i = 0; i < 32; i += 8) {
            uint4 v;
            v.x = pack_half2(__uint_as_float(o[i]) * inv, __uint_as_float(o[i + 1]) * inv);
            v.y = pack_half2(__uint_as_float(o[i + 2]) * inv, __uint_as_float(o[i + 3]) * inv);
            v.z = pack_half2(__uint_as_float(o[i + 4]) * inv, __uint_as_float(o[i + 5]) * inv);
            v.w = pack_half2(__uint_as_float(o[i + 6]) * inv, __uint_as_float(o[i + 7]) * inv);
            *reinterpret_cast<uint4*>(dst + c + i) = v;
          }
        }
      }
    } else {
      fail_s = 1;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (fail_s && threadIdx.x == 0) raise_status(p.status, 9);
  if (warp == 1) tmem_dealloc(tmem, 512);
}

template <int D, bool SPLIT>
cudaError_t launch_tc(const CUtensorMap& qm, const CUtensorMap& km, const CUtensorMap& vm, const AttnTcParams& p, int grid, cudaStream_t st,
                      int pdl) {
  constexpr size_t smem = (size_t)(2 * kQRows + kRing * kKeys) * D * 2 + 1024;
  static std::atomic<uint64_t> attr_done;
  const cudaError_t e = smem_limit_once(&attr_done, {reinterpret_cast<const void*>(attn_prefill_tc_kernel<D, SPLIT>)}, smem);
  if (e != cudaSuccess) return e;
  return launch_dep(attn_prefill_tc_kernel<D, SPLIT>, dim3(grid), dim3(kAttnThreads), smem, st, pdl, 1, qm, km, vm, p);
}

}  // namespace

bool attn_prefill_tc_eligible(const __half* q_rot16, const __half* kc, const __half* vc, const __half* a16, int T, int d) {
  return (d == 64 || d == 128) && T > 128 &&
         (((reinterpret_cast<uintptr_t>(q_rot16) | reinterpret_cast<uintptr_t>(kc) | reinterpret_cast<uintptr_t>(vc) |
            reinterpret_cast<uintptr_t>(a16)) & 15) == 0);
}

cudaError_t launch_attn_prefill_tc(const __half* q_rot16, const __half* kc, const __half* vc, __half* a16, int T, int n_q, int n_kv, int d,
                                   int cap, int pos0, int* status, int sm_count, cudaStream_t st, uint64_t* n_launch, int pdl) {
  // rows beyond the context (and query rows beyond T) read as zeros: the cache may hold anything there
  CUtensorMap qm, km, vm;
  const uint64_t row = (uint64_t)d * 2;
  if (!encode_map_f16_3d(&qm, q_rot16, d, n_q, T, row, row * n_q, 64, 1, kQRows) ||
      !encode_map_f16_3d(&km, kc, d, pos0 + T, n_kv, row, row * cap, 64, kKeys, 1) ||
      !encode_map_f16_3d(&vm, vc, d, pos0 + T, n_kv, row, row * cap, 64, kKeys, 1))
    return cudaErrorInvalidValue;
  AttnTcParams p{};
  p.out = a16;
  p.T = T;
  p.n_q = n_q;
  p.group = n_q / n_kv;
  p.pos0 = pos0;
  // One tile to a CTA, its key blocks in two, where all such CTAs run at once and there are blocks enough for the merge (2 us) to pay.  Layers of 4096,
  // 130 tokens after 2000: 152.9 -> 139.2 us, 300 after 1500 184.5 -> 175.1; of 2048, 1000 after 300: 143.0 -> 131.9; 700 tokens of 24 heads of 64
  // 81.3 -> 78.3.  With four blocks (400 tokens of 40 heads, 228.7) it was 2 us slower.
  const bool split = (T + kQRows - 1) / kQRows * n_q <= sm_count && (pos0 + T + kKeys - 1) / kKeys >= 6;
  p.pair_heads = p.group % 2 == 0 && !split;
  const int tokens = p.pair_heads || split ? kQRows : 2 * kQRows;
  p.n_tb = (T + tokens - 1) / tokens;
  p.scale_log2 = 1.4426950408889634f / sqrtf((float)d);
  p.status = status;
  const int grid = p.n_tb * (p.pair_heads ? n_q / 2 : n_q);
  ++*n_launch;
  if (split) return d == 128 ? launch_tc<128, true>(qm, km, vm, p, grid, st, pdl) : launch_tc<64, true>(qm, km, vm, p, grid, st, pdl);
  return d == 128 ? launch_tc<128, false>(qm, km, vm, p, grid, st, pdl) : launch_tc<64, false>(qm, km, vm, p, grid, st, pdl);
}

}  // namespace ats
