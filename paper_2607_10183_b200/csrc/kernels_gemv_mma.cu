// Few-row GEMV for the two 4-bit block formats on the warp-level tensor-core instruction (mma.sync m16n8k16, fp16
// operands, fp32 accumulation): y[m][n] = sum_k w[n][k] x[m][k] for M <= 8 rows of x.
//
// The generic GEMV decodes every weight to fp32 and spends a fused multiply-add per weight and activation row: about five
// thread instructions per weight, which is what bounds it (not HBM) for the microscaling format and for several rows.
// Here a warp owns 16 weight rows; the weights of a 16 x 16 tile are the A operand, decoded straight into fp16 pairs in
// the fragment layout (two shifts and two logic operations per pair for the microscaling format, one logic
// operation and one fp16 operation for the integer codes), the M activation rows
// are the eight columns of the B operand, and one instruction does the 16 x 16 x 8 products.  Products of fp16 values are
// exact in fp32; the two k-steps of a 32-wide block accumulate in the instruction's fp32 accumulator, the block's scale
// is applied in fp32 and blocks are summed in fp32, so weights stay exact as in the generic kernel.  The layout:
//   A (16 x 16, row):  reg0 = (row g, kk 2t..2t+1), reg1 = (row g+8, same kk), reg2 = (row g, kk 2t+8..2t+9), reg3 = (row g+8, ..)
//   B (16 x 8, col):   reg0 = (kk 2t..2t+1, column g), reg1 = (kk 2t+8..2t+9, column g)
//   C (16 x 8):        c0 c1 = (row g, columns 2t 2t+1), c2 c3 = (row g+8, columns 2t 2t+1)        g = lane / 4, t = lane % 4
// The instruction sums over its sixteen kk whatever they stand for, so the k of a 32-wide block are dealt to the two
// instructions in the order that suits the data: lane t takes k = 8t .. 8t+7 of the block, that is ONE code word per row
// (word t of the block's four) and 16 contiguous bytes of x, with the word's pairs (2j, 2j+1), j = 0..3, as
// (instruction j / 2, reg 0/1 or 2/3 by j % 2) on both operands.  All shifts of the decode are compile-time constants.
//
// A unit is 16 consecutive output rows (SwiGLU: 16 gate rows and the 16 up rows of the same outputs).  1, 2, 4 or 8 warps of
// the CTA share a unit, each on its own part of K; partial tiles meet in shared memory and are added in fixed order.
// Code loads are 4 bytes per thread, row and block (the quad's four words are the block's 16 contiguous bytes), sixteen
// blocks in flight, the first batch issued before the grid dependency resolves (weights do not depend on the preceding
// kernel).
#include "ats_internal.h"
#include "sm100_sync.cuh"

namespace ats {

namespace {

struct MmaGemvParams {
  const uint8_t* base[3];
  int n_rows[3];
  int n_seg, K, M, mode, ksplit;
  const __half* x;
  int ldx;
  float* y32;
  __half* y16;
  int ldy;
  const float* res32;
  const __half* res16;
  int ldres;
};

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The four pairs (k = 2j, 2j+1 in nibbles j and j + 4) of a code word as fp16 pairs.
//   MX = false: offset-binary integer codes u = c + 8.  (w & 0x000F000F) | 0x6400.. is the fp16 pair 1024 + u, the
//     0x00F000F0 pair is 1024 + 16 u: one subtraction or one multiply-add gives c exactly.
//   MX = true: microscaling floats: magnitude bits onto bits 11..9 of each half, sign onto bit 15: element * 2^-14.
template <bool MX>
__device__ __forceinline__ void decode_word(uint32_t w, uint32_t (&a)[4]) {
  if (MX) {
    const uint32_t kMag = 0x0E000E00u, kSgn = 0x80008000u;
    a[0] = ((w << 9) & kMag) | ((w << 12) & kSgn);
    a[1] = ((w << 5) & kMag) | ((w << 8) & kSgn);
    a[2] = ((w << 1) & kMag) | ((w << 4) & kSgn);
    a[3] = ((w >> 3) & kMag) | (w & kSgn);
  } else {
    auto h2 = [](uint32_t v) { __half2 h; *reinterpret_cast<uint32_t*>(&h) = v; return h; };
    auto u32 = [](__half2 h) { return *reinterpret_cast<uint32_t*>(&h); };
    const uint32_t kMagic = 0x64006400u, w8 = w >> 8;
    const __half2 k1032 = h2(0x64086408u), k16th = h2(0x2C002C00u), kM72 = h2(0xD480D480u);
    a[0] = u32(__hsub2(h2((w & 0x000F000Fu) | kMagic), k1032));
    a[1] = u32(__hfma2(h2((w & 0x00F000F0u) | kMagic), k16th, kM72));
    a[2] = u32(__hsub2(h2((w8 & 0x000F000Fu) | kMagic), k1032));
    a[3] = u32(__hfma2(h2((w8 & 0x00F000F0u) | kMagic), k16th, kM72));
  }
}

// N (4, 8 or 16) consecutive block scales of a row as packed fp16 pairs: one or two vector loads where the address allows,
// else scalar loads; blocks at or beyond b_hi read as zero.
template <int N>
__device__ __forceinline__ void load_scales(const __half* sp, int b0, int b_hi, bool live, uint32_t (&s)[N / 2]) {
  if (live && b0 + N <= b_hi && (reinterpret_cast<uintptr_t>(sp + b0) & (2 * N > 16 ? 15 : 2 * N - 1)) == 0) {
    if (N == 4) {
      const uint2 v = __ldg(reinterpret_cast<const uint2*>(sp + b0));
      s[0] = v.x; s[1] = v.y;
    } else {
#pragma unroll
      for (int i = 0; i < N / 8; ++i) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(sp + b0) + i);
        s[4 * i] = v.x; s[4 * i + 1] = v.y; s[4 * i + 2] = v.z; s[4 * i + 3] = v.w;
      }
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < N / 2; ++j) {
    const unsigned short a = (live && b0 + 2 * j < b_hi) ? __half_as_ushort(__ldg(sp + b0 + 2 * j)) : (unsigned short)0;
    const unsigned short b = (live && b0 + 2 * j + 1 < b_hi) ? __half_as_ushort(__ldg(sp + b0 + 2 * j + 1)) : (unsigned short)0;
    s[j] = (uint32_t)a | ((uint32_t)b << 16);
  }
}
template <int N2>
__device__ __forceinline__ float scale_of(const uint32_t (&s)[N2], int j) {
  return __half2float(__ushort_as_half((unsigned short)(s[j >> 1] >> (16 * (j & 1)))));
}

// One thread per (unit, row of the tile, activation row) adds the K parts in fixed order and writes the output.
template <bool SW, int NT>
__device__ __forceinline__ void write_units(const MmaGemvParams& p, const float (&red_s)[8][NT][16][8], int u0, int upc, int ks, int n_rows) {
  for (int e = threadIdx.x; e < upc * 16 * p.M; e += blockDim.x) {
    const int m = e % p.M, row = (e / p.M) % 16, sl = e / (16 * p.M);
    const int r = 16 * (u0 + sl) + row;
    if (r >= n_rows) continue;
    float s0 = 0.f, s1 = 0.f;
    for (int q2 = 0; q2 < ks; ++q2) {
      s0 += red_s[sl * ks + q2][0][row][m];
      if (SW) s1 += red_s[sl * ks + q2][NT - 1][row][m];
    }
    const size_t o = (size_t)m * p.ldy + r, ro = (size_t)m * p.ldres + r;
    switch (p.mode) {
      case GEMV_OUT_F32: p.y32[o] = s0; break;
      case GEMV_OUT_F16: p.y16[o] = __float2half_rn(s0); break;
      case GEMV_RES16_OUT_F32: p.y32[o] = __half2float(p.res16[ro]) + s0; break;
      case GEMV_RES32_OUT_F16: p.y16[o] = __float2half_rn(p.res32[ro] + s0); break;
      case GEMV_RES16_OUT_F16: p.y16[o] = __float2half_rn(__half2float(p.res16[ro]) + s0); break;
      case GEMV_SWIGLU_F16: p.y16[o] = __float2half_rn(s0 / (1.0f + expf(-s0)) * s1); break;
      default: break;
    }
  }
}

template <bool MX, bool SW>
__global__ void __launch_bounds__(256) gemv_mma_kernel(const MmaGemvParams p) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  bool waited = false;  // x and the residual come from the preceding kernel; the first weight loads need not wait for it
  constexpr int NT = SW ? 2 : 1;   // weight tiles per unit
  constexpr int NBK = SW ? 8 : 16;  // blocks in flight per thread and row
  __shared__ float red_s[8][NT][16][8];
  const int lane = threadIdx.x & 31, w = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // (the same for the warp, and known to be)
  const int g = lane >> 2, t = lane & 3;
  const int K = p.K, nblk = K / 32, M = p.M;
  int n_rows = p.n_rows[0];  // rows side by side (SwiGLU: outputs)
  if (!SW) n_rows += (p.n_seg > 1 ? p.n_rows[1] : 0) + (p.n_seg > 2 ? p.n_rows[2] : 0);
  // codes and scales of weight row r of tile kind nt (SwiGLU: 0 = gate, 1 = up; otherwise rows run across the segments)
  auto row_ptrs = [&](int r, int nt, const uint4*& codes, const __half*& scales) {
    const uint8_t* base = p.base[0];
    int rows = p.n_rows[0];
    if (SW) {
      if (nt) base = p.base[1];
    } else if (p.n_seg > 1 && r >= p.n_rows[0]) {
      r -= p.n_rows[0];
      base = p.base[1];
      rows = p.n_rows[1];
      if (p.n_seg > 2 && r >= p.n_rows[1]) {
        r -= p.n_rows[1];
        base = p.base[2];
        rows = p.n_rows[2];
      }
    }
    codes = reinterpret_cast<const uint4*>(base + (size_t)r * (K / 2));
    scales = reinterpret_cast<const __half*>(base + (size_t)rows * (K / 2)) + (size_t)r * nblk;
  };
  const int n_units = (n_rows + 15) / 16;
  const int ks = p.ksplit, upc = 8 / ks;
  const int part = w % ks, slot = w / ks;
  const int per = (((nblk + ks - 1) / ks) + 15) & ~15;  // blocks per part: whole batches, so that scale loads stay aligned
  const int b_lo = part * per, b_hi = min(nblk, b_lo + per);
  const uint32_t zero_word = MX ? 0u : 0x88888888u;  // eight zeros in either format
  const __half* xrow = p.x + (size_t)min(g, M - 1) * p.ldx + 8 * t;
  const bool xlive = g < M;
  for (int u0 = blockIdx.x * upc; u0 < n_units; u0 += gridDim.x * upc) {
    const int u = u0 + slot;
    float acc[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[nt][i] = 0.f;
    if (u < n_units) {
      const uint4* cp[NT][2];
      const __half* sp[NT][2];
      bool live[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = 16 * u + g + 8 * h;
        live[h] = r < n_rows;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) row_ptrs(live[h] ? r : 0, nt, cp[nt][h], sp[nt][h]);
      }
      for (int b0 = b_lo; b0 < b_hi; b0 += NBK) {
        // Lane t of a quad loads word t of every block of its two rows (the quad's four words are the block's 16 contiguous
        // bytes), NBK blocks in flight.
        uint32_t q[NBK][NT][2];
        uint32_t sc[NT][2][NBK / 2];
#pragma unroll
        for (int j = 0; j < NBK; ++j) {
          const int b = b0 + j;
#pragma unroll
          for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int h = 0; h < 2; ++h)
              q[j][nt][h] = (live[h] && b < b_hi) ? __ldg(reinterpret_cast<const uint32_t*>(cp[nt][h] + b) + t) : zero_word;
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int h = 0; h < 2; ++h) load_scales<NBK>(sp[nt][h], b0, b_hi, live[h], sc[nt][h]);
        if (!waited) {
          asm volatile("griddepcontrol.wait;" ::: "memory");
          waited = true;
        }
#pragma unroll
        for (int j = 0; j < NBK; ++j) {
          const int b = b0 + j;
          if (b >= b_hi) break;  // uniform over the warp
          // x[b * 32 + 8 t .. + 7]: the four pairs this lane's word multiplies, in instruction order
          const uint4 xv = xlive ? __ldg(reinterpret_cast<const uint4*>(xrow + b * 32)) : make_uint4(0, 0, 0, 0);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            uint32_t a0[4], a1[4];
            decode_word<MX>(q[j][nt][0], a0);
            decode_word<MX>(q[j][nt][1], a1);
            float c[4] = {0.f, 0.f, 0.f, 0.f};
            const uint32_t f0[4] = {a0[0], a1[0], a0[1], a1[1]}, f1[4] = {a0[2], a1[2], a0[3], a1[3]};
            mma16816(c, f0, xv.x, xv.y);
            mma16816(c, f1, xv.z, xv.w);
            const float s0 = scale_of(sc[nt][0], j), s1 = scale_of(sc[nt][1], j);
            acc[nt][0] = fmaf(s0, c[0], acc[nt][0]);
            acc[nt][1] = fmaf(s0, c[1], acc[nt][1]);
            acc[nt][2] = fmaf(s1, c[2], acc[nt][2]);
            acc[nt][3] = fmaf(s1, c[3], acc[nt][3]);
          }
        }
      }
    }
    if (!waited) {  // no block for this warp
      asm volatile("griddepcontrol.wait;" ::: "memory");
      waited = true;
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const float f = MX ? 16384.f : 1.f;  // the microscaling decode left a factor 2^-14 on every element
      red_s[w][nt][g][2 * t] = acc[nt][0] * f;
      red_s[w][nt][g][2 * t + 1] = acc[nt][1] * f;
      red_s[w][nt][g + 8][2 * t] = acc[nt][2] * f;
      red_s[w][nt][g + 8][2 * t + 1] = acc[nt][3] * f;
    }
    __syncthreads();
    write_units<SW, NT>(p, red_s, u0, upc, ks, n_rows);
    __syncthreads();
  }
  if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The same product for K a multiple of 256 and rows whose scales are 16-byte aligned: a warp streams its rows through a ring
// of its own in shared memory with 16-byte asynchronous copies, a stage being 256 k of 16 rows (SwiGLU: of 16 gate and
// 16 up rows), and goes from one unit to the next with the ring full.  (Loads of 4 bytes per lane into registers, as above,
// touch sixteen lines per row pair and block; the L1's tag stage and the gaps between batches set the pace.  5 rows, before
// -> now: MXFP4 14336 x 4096 22.3 -> 10.2 us, 4096 x 14336 24.7 -> 10.3, 28672 x 4096 46.0 -> 18.1; Q4 21.6 -> 12.0, 24.7 -> 12.0,
// 45.6 -> 20.8.)  Code rows have a pitch of 144 bytes in the ring: lane (g, t) reads word t of row g without bank conflicts.
// Microscaling words are unpacked by cvt_e2m1x8, whose pairs (0, 2), (4, 6), (1, 3), (5, 7) the activations follow; products,
// accumulation and the order of the sums are those of the kernel above.
constexpr int kRingPitch = 144, kRingTile = 16 * kRingPitch + 16 * 16;  // bytes of a 16-row x 256-k tile: codes, then scales
constexpr int kRingWarps = 8;
// Four stages are in flight per warp, two with gate and up; a fifth takes from the L1 what the activations need (11.3 us for 10.2).
constexpr int kRingStages = 4, kRingStagesSw = 2;

// Asynchronous copies of step k's tile: codes of rows lane / 8 + 4 q (piece lane % 8), scales of row lane (lanes 0..15).
__device__ __forceinline__ void ring_request(uint32_t dst, const uint8_t* const (&cp)[4], const uint8_t* sp, int k, int lane) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (uint32_t)(((lane >> 3) + 4 * q) * kRingPitch + (lane & 7) * 16)),
                 "l"(cp[q] + (size_t)k * 128)
                 : "memory");
  if (lane < 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (uint32_t)(16 * kRingPitch + lane * 16)), "l"(sp + (size_t)k * 16) : "memory");
}

// A stage's 256 k of NT tiles: lane (g, t) holds rows g, g + 8 of column pair t and gives the activations xv of column g.
template <bool MX, int NT>
__device__ __forceinline__ void ring_step(const uint8_t* st, int g, int t, const uint4 (&xv)[8], float (&acc)[NT][4]) {
  uint4 sc[NT][2];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int h = 0; h < 2; ++h) sc[nt][h] = *reinterpret_cast<const uint4*>(st + nt * kRingTile + 16 * kRingPitch + (g + 8 * h) * 16);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    uint4 x = xv[j];
    if (MX)
      x = make_uint4(__byte_perm(x.x, x.y, 0x5410u), __byte_perm(x.z, x.w, 0x5410u), __byte_perm(x.x, x.y, 0x7632u),
                     __byte_perm(x.z, x.w, 0x7632u));
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const uint8_t* tile = st + nt * kRingTile + j * 16 + t * 4;
      const uint32_t q0 = *reinterpret_cast<const uint32_t*>(tile + g * kRingPitch);
      const uint32_t q1 = *reinterpret_cast<const uint32_t*>(tile + (g + 8) * kRingPitch);
      uint32_t a0[4], a1[4];
      if (MX) {
        cvt_e2m1x8(q0, a0);
        cvt_e2m1x8(q1, a1);
      } else {
        decode_word<false>(q0, a0);
        decode_word<false>(q1, a1);
      }
      float c[4] = {0.f, 0.f, 0.f, 0.f};
      const uint32_t f0[4] = {a0[0], a1[0], a0[1], a1[1]}, f1[4] = {a0[2], a1[2], a0[3], a1[3]};
      mma16816(c, f0, x.x, x.y);
      mma16816(c, f1, x.z, x.w);
      const uint32_t w0[4] = {sc[nt][0].x, sc[nt][0].y, sc[nt][0].z, sc[nt][0].w}, w1[4] = {sc[nt][1].x, sc[nt][1].y, sc[nt][1].z, sc[nt][1].w};
      const float s0 = scale_of(w0, j), s1 = scale_of(w1, j);
      acc[nt][0] = fmaf(s0, c[0], acc[nt][0]);
      acc[nt][1] = fmaf(s0, c[1], acc[nt][1]);
      acc[nt][2] = fmaf(s1, c[2], acc[nt][2]);
      acc[nt][3] = fmaf(s1, c[3], acc[nt][3]);
    }
  }
}

template <bool MX, bool SW>
__global__ void __launch_bounds__(32 * kRingWarps, 2) gemv_mma_ring_kernel(const MmaGemvParams p) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int NT = SW ? 2 : 1;     // weight tiles per unit
  constexpr int S = SW ? kRingStagesSw : kRingStages;
  extern __shared__ __align__(16) uint8_t ring[];
  __shared__ __align__(16) float red_s[2][kRingWarps][NT][16][8];
  const int lane = threadIdx.x & 31, w = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // (the same for the warp, and known to be)
  const int g = lane >> 2, t = lane & 3;
  const int K = p.K, nblk = K / 32, M = p.M, n_step = K / 256;
  int n_rows = p.n_rows[0];
  if (!SW) n_rows += (p.n_seg > 1 ? p.n_rows[1] : 0) + (p.n_seg > 2 ? p.n_rows[2] : 0);
  const int n_units = (n_rows + 15) / 16;
  const int ks = p.ksplit, upc = kRingWarps / ks, part = w % ks, slot = w / ks;
  const int per = (n_step + ks - 1) / ks, k_lo = min(part * per, n_step), k_hi = min(k_lo + per, n_step);
  uint8_t* my = ring + (size_t)w * S * NT * kRingTile;
  const uint32_t my_u = (uint32_t)__cvta_generic_to_shared(my);
  // ---- requests: unit by unit, step by step, S - 1 stages ahead of their use
  int ru = blockIdx.x * upc + slot, rk = k_lo, rs = 0;
  const uint8_t* cp[NT][4];   // this lane's four 16-byte pieces of a step's codes: rows lane / 8 + 4 q, piece lane % 8
  const uint8_t* sp[NT];      // (lanes 0..15) the row's eight scales of a step
  auto row_codes = [&](int r, int nt, const uint8_t*& scales) {  // rows beyond the last: the last (their sums are not written)
    r = min(r, n_rows - 1);
    const uint8_t* base = p.base[0];
    int rows = p.n_rows[0];
    if (SW) {
      if (nt) base = p.base[1];
    } else if (p.n_seg > 1 && r >= p.n_rows[0]) {
      r -= p.n_rows[0];
      base = p.base[1];
      rows = p.n_rows[1];
      if (p.n_seg > 2 && r >= p.n_rows[1]) {
        r -= p.n_rows[1];
        base = p.base[2];
        rows = p.n_rows[2];
      }
    }
    scales = base + (size_t)rows * (K / 2) + (size_t)r * nblk * 2;
    return base + (size_t)r * (K / 2);
  };
  auto request = [&] {
    if (ru < n_units && k_lo < k_hi) {
      if (rk == k_lo) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          const uint8_t* unused;
#pragma unroll
          for (int q = 0; q < 4; ++q) cp[nt][q] = row_codes(16 * ru + (lane >> 3) + 4 * q, nt, unused) + (lane & 7) * 16;
          row_codes(16 * ru + (lane & 15), nt, sp[nt]);
        }
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) ring_request(my_u + (uint32_t)((rs * NT + nt) * kRingTile), cp[nt], sp[nt], rk, lane);
      if (++rk == k_hi) rk = k_lo, ru += gridDim.x * upc;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (++rs == S) rs = 0;
  };
#pragma unroll
  for (int i = 0; i < S - 1; ++i) request();
  asm volatile("griddepcontrol.wait;" ::: "memory");  // x and the residual come from the preceding kernel
  const __half* xrow = p.x + (size_t)min(g, M - 1) * p.ldx + 8 * t;
  const bool xlive = g < M;
  int cs = 0, buf = 0;
  for (int u0 = blockIdx.x * upc; u0 < n_units; u0 += gridDim.x * upc) {
    float acc[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[nt][i] = 0.f;
    if (u0 + slot < n_units) {
      for (int k = k_lo; k < k_hi; ++k) {
        uint4 xv[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) xv[j] = xlive ? __ldg(reinterpret_cast<const uint4*>(xrow + k * 256 + j * 32)) : make_uint4(0, 0, 0, 0);
        asm volatile("cp.async.wait_group %0;" ::"n"(S - 2) : "memory");
        __syncwarp();  // the stage is there for every lane, and the last one has been read by all: its place is free
        request();
        const uint8_t* st = my + (size_t)cs * NT * kRingTile;
        if (++cs == S) cs = 0;
        ring_step<MX, NT>(st, g, t, xv, acc);
      }
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      *reinterpret_cast<float2*>(&red_s[buf][w][nt][g][2 * t]) = make_float2(acc[nt][0], acc[nt][1]);
      *reinterpret_cast<float2*>(&red_s[buf][w][nt][g + 8][2 * t]) = make_float2(acc[nt][2], acc[nt][3]);
    }
    __syncthreads();
    write_units<SW, NT>(p, red_s[buf], u0, upc, ks, n_rows);
    buf ^= 1;  // (the next unit's sums go to the other half: one barrier a unit)
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// Routed experts for several tokens: the (token, slot) pairs grouped by expert, up to eight pairs of an expert as the columns, so
// that an expert's weights are read and decoded once for them instead of once per pair.  Every CTA groups the pairs for itself from
// the ids (at most 256: a pair's place is the number of earlier pairs of its expert; no sort, no launch of its own); a unit
// is 16 rows (SwiGLU: 16 gate and 16 up rows) of a group, and the units of all groups form one line that the warps of a grid of two
// CTAs per SM go through as above.  The K split depends on K alone and a column's sums on its own activations alone, so a
// pair's result has the same bits whatever it is grouped with.  What bounds it: the activations (their
// rows come through the L1 as often as the weights) and the grouping (its loop unrolled: 10 us less
// for 256 pairs).  FFN half of a layer, 2048 x 768 experts, 8 per token, 32 tokens, streaming -> grouped: Q4 16 experts 130 -> 60 us,
// 64 130 -> 85; MXFP4 16 191 -> 53, 64 192 -> 74, 128 193 -> 106.
constexpr int kMoePairs = 256, kMoeCols = 8;
// A part of K has at least two steps: with one the 32-token blocks above take 5 to 12 % longer, with four up to 2 %.
constexpr int kMoeSplitSteps = 2;
struct MoeMmaParams {
  const uint8_t *base0, *base1;
  uint64_t stride;
  const int32_t* ids;  // null: pairs and weights from MoeJobs
  const uint8_t *const *tab0, *const *tab1;
  int x_div, P, n_experts;
  int* status;
  int n_rows, K, mode, ksplit;
  const __half* x;
  int ldx;
  float* y32;
  __half* y16;
  int ldy;
};

template <bool MX, bool SW>
__global__ void __launch_bounds__(32 * kRingWarps, 2) moe_mma_ring_kernel(const MoeMmaParams p, const __grid_constant__ MoeJobs jobs) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int NT = SW ? 2 : 1;
  constexpr int S = SW ? kRingStagesSw : kRingStages;
  extern __shared__ __align__(16) uint8_t ring[];
  __shared__ float red_s[kRingWarps][NT][16][kMoeCols + 1];
  __shared__ const uint8_t* w_s[NT][kMoePairs];        // a group's weights
  __shared__ __align__(16) uint16_t row_s[kMoePairs][kMoeCols];  // its pairs (output rows); 0xFFFF: none
  __shared__ unsigned long long key_s[kMoePairs];
  __shared__ uint8_t group_s[kMoePairs];               // of a group's first pair: the group
  __shared__ int warp_groups[kRingWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;  // (known to be the same for the warp: 32 rows of 16 MXFP4 experts 55.7 -> 56.3 us)
  const int g = lane >> 2, t = lane & 3;
  asm volatile("griddepcontrol.wait;" ::: "memory");  // ids, activations and gathered weights come from the kernels before
  // ---- groups: thread q places pair q
  int n_groups = 0;
  {
    const int q = threadIdx.x, n = p.ids ? p.P : jobs.n;
    const uint8_t *w0 = nullptr, *w1 = nullptr;
    unsigned long long key = ~0ull;
    if (q < n) {
      if (p.ids) {
        size_t e = (size_t)(unsigned)p.ids[q];
        if (e >= (size_t)p.n_experts) {  // an id that names no expert: expert 0 stands in and the status word says so
          if (blockIdx.x == 0) raise_status(p.status, 7);
          e = 0;
        }
        key = e;
        w0 = p.tab0 ? p.tab0[e] : p.base0 + e * p.stride;
        if (SW) w1 = p.tab1 ? p.tab1[e] : p.base1 + e * p.stride;
      } else {
        w0 = jobs.w0[q];
        if (SW) w1 = jobs.w1[q];
        key = (unsigned long long)w0;
      }
    }
    key_s[q] = key;
    *reinterpret_cast<uint4*>(row_s[q]) = make_uint4(~0u, ~0u, ~0u, ~0u);
    __syncthreads();
    int place = 0, first = q;  // earlier pairs of the expert; first pair of the group
    if (32 * w < n) {
#pragma unroll 16
      for (int i = 0; i < 32 * w + 32; ++i) {
        const bool same = key_s[i] == key && i < q;
        if (same && place % kMoeCols == 0) first = i;
        place += same;
      }
    }
    const bool opens = q < n && place % kMoeCols == 0;
    const unsigned open = __ballot_sync(0xFFFFFFFFu, opens);
    if (lane == 0) warp_groups[w] = __popc(open);
    __syncthreads();
    int gi = __popc(open & ((1u << lane) - 1));
#pragma unroll
    for (int i = 0; i < kRingWarps; ++i) {
      if (i < w) gi += warp_groups[i];
      n_groups += warp_groups[i];
    }
    if (opens) {
      first = q;
      group_s[q] = (uint8_t)gi;
      w_s[0][gi] = w0;
      if (SW) w_s[NT - 1][gi] = w1;
    }
    __syncthreads();
    if (q < n) row_s[group_s[first]][place % kMoeCols] = (uint16_t)(p.ids ? q : jobs.orow[q]);
    __syncthreads();
  }
  const int K = p.K, nblk = K / 32, n_step = K / 256, n_rows = p.n_rows;
  const int per_group = (n_rows + 15) / 16, n_units = n_groups * per_group;
  const int ks = p.ksplit, upc = kRingWarps / ks, part = w % ks, slot = w / ks;
  const int per = (n_step + ks - 1) / ks, k_lo = min(part * per, n_step), k_hi = min(k_lo + per, n_step);
  uint8_t* my = ring + (size_t)w * S * NT * kRingTile;
  const uint32_t my_u = (uint32_t)__cvta_generic_to_shared(my);
  int ru = blockIdx.x * upc + slot, rk = k_lo, rs = 0;
  const uint8_t *cp[NT][4], *sp[NT];
  auto request = [&] {
    if (ru < n_units && k_lo < k_hi) {
      if (rk == k_lo) {
        const int gr = ru / per_group, r0 = 16 * (ru - gr * per_group);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {  // rows beyond the last: the last (their sums are not written)
          const uint8_t* base = w_s[nt][gr];
#pragma unroll
          for (int q = 0; q < 4; ++q) cp[nt][q] = base + (size_t)min(r0 + (lane >> 3) + 4 * q, n_rows - 1) * (K / 2) + (lane & 7) * 16;
          sp[nt] = base + (size_t)n_rows * (K / 2) + (size_t)min(r0 + (lane & 15), n_rows - 1) * nblk * 2;
        }
      }
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) ring_request(my_u + (uint32_t)((rs * NT + nt) * kRingTile), cp[nt], sp[nt], rk, lane);
      if (++rk == k_hi) rk = k_lo, ru += gridDim.x * upc;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (++rs == S) rs = 0;
  };
#pragma unroll
  for (int i = 0; i < S - 1; ++i) request();
  int cs = 0;
  for (int u0 = blockIdx.x * upc; u0 < n_units; u0 += gridDim.x * upc) {
    float acc[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[nt][i] = 0.f;
    if (u0 + slot < n_units) {
      const int row = row_s[(u0 + slot) / per_group][g];
      const bool xlive = row != 0xFFFF;
      const __half* xrow = p.x + (size_t)(xlive ? row / p.x_div : 0) * p.ldx + 8 * t;
      for (int k = k_lo; k < k_hi; ++k) {
        uint4 xv[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) xv[j] = xlive ? __ldg(reinterpret_cast<const uint4*>(xrow + k * 256 + j * 32)) : make_uint4(0, 0, 0, 0);
        asm volatile("cp.async.wait_group %0;" ::"n"(S - 2) : "memory");
        __syncwarp();  // the stage is there for every lane, and the last one has been read by all: its place is free
        request();
        ring_step<MX, NT>(my + (size_t)cs * NT * kRingTile, g, t, xv, acc);
        if (++cs == S) cs = 0;
      }
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) red_s[w][nt][g + 8 * (i >> 1)][2 * t + (i & 1)] = acc[nt][i];
    __syncthreads();
    for (int e = threadIdx.x; e < upc * 16 * kMoeCols; e += blockDim.x) {
      const int row = e % 16, m = e / 16 % kMoeCols, sl = e / (16 * kMoeCols), u = u0 + sl;
      if (u >= n_units) break;
      const int gr = u / per_group, r = 16 * (u - gr * per_group) + row, o = row_s[gr][m];
      if (o == 0xFFFF || r >= n_rows) continue;
      float s0 = 0.f, s1 = 0.f;
      for (int q = 0; q < ks; ++q) {
        s0 += red_s[sl * ks + q][0][row][m];
        if (SW) s1 += red_s[sl * ks + q][NT - 1][row][m];
      }
      const size_t at = (size_t)o * p.ldy + r;
      if (SW) p.y16[at] = __float2half_rn(s0 / (1.0f + expf(-s0)) * s1);
      else if (p.mode == GEMV_OUT_F32) p.y32[at] = s0;
      else p.y16[at] = __float2half_rn(s0);
    }
    __syncthreads();
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

}  // namespace

bool gemv_mma_eligible(const GemvParams& g) {
  if (g.w16 || g.M < 1 || g.M > 8 || g.K % 32 || g.n_seg < 1 || g.n_seg > 3) return false;
  if ((g.ldx & 7) || (reinterpret_cast<uintptr_t>(g.x) & 15)) return false;  // a lane reads its eight activations as 16 bytes
  if (g.mode == GEMV_SWIGLU_F16 && (g.n_seg != 2 || g.seg[0].n_rows != g.seg[1].n_rows)) return false;
  for (int s = 0; s < g.n_seg; ++s)
    if ((reinterpret_cast<uintptr_t>(g.seg[s].base) & 15) || (g.K / 2) % 16) return false;  // 16-byte code loads per block
  return true;
}

cudaError_t launch_gemv_mma(const GemvParams& g, cudaStream_t st, uint64_t* n_launch) {
  if (!gemv_mma_eligible(g)) return cudaErrorInvalidValue;
  MmaGemvParams p{};
  int n_rows = 0;
  for (int s = 0; s < g.n_seg; ++s) {
    p.base[s] = g.seg[s].base;
    p.n_rows[s] = g.seg[s].n_rows;
    n_rows += g.seg[s].n_rows;
  }
  const bool sw = g.mode == GEMV_SWIGLU_F16;
  if (sw) n_rows = g.seg[0].n_rows;
  p.n_seg = g.n_seg; p.K = g.K; p.M = g.M; p.mode = g.mode;
  p.x = g.x; p.ldx = g.ldx; p.y32 = g.y32; p.y16 = g.y16; p.ldy = g.ldy;
  p.res32 = g.res32; p.res16 = g.res16; p.ldres = g.ldres;
  const int n_units = (n_rows + 15) / 16, nblk = g.K / 32;
  if (g.K % 256 == 0) {
    // as many parts of K as give every warp that the machine holds two pieces of work
    int ks = 1;
    while (ks < kRingWarps && (long)n_units * ks < 2L * 148 * 2 * kRingWarps && g.K / 256 >= ks * 2) ks *= 2;
    p.ksplit = ks;
    const int ctas = (n_units + kRingWarps / ks - 1) / (kRingWarps / ks);
    const size_t smem = (size_t)kRingWarps * (sw ? 2 * kRingStagesSw : kRingStages) * kRingTile;
    static std::atomic<uint64_t> attr_done;
    const cudaError_t e = smem_limit_once(&attr_done, {reinterpret_cast<const void*>(gemv_mma_ring_kernel<false, false>), reinterpret_cast<const void*>(gemv_mma_ring_kernel<true, false>),
                                                       reinterpret_cast<const void*>(gemv_mma_ring_kernel<false, true>), reinterpret_cast<const void*>(gemv_mma_ring_kernel<true, true>)},
                                          kRingWarps * std::max(kRingStages, 2 * kRingStagesSw) * kRingTile);
    if (e != cudaSuccess) return e;
    ++*n_launch;
    auto run = [&](auto* k) { return launch_dep(k, dim3(std::min(ctas, 2 * 148)), dim3(32 * kRingWarps), smem, st, g.pdl, 1, p); };
    if (g.mx) return sw ? run(gemv_mma_ring_kernel<true, true>) : run(gemv_mma_ring_kernel<true, false>);
    return sw ? run(gemv_mma_ring_kernel<false, true>) : run(gemv_mma_ring_kernel<false, false>);
  }
  // Split K while the units alone give fewer warps than about twice what the machine holds and every part keeps at least
  // one batch of sixteen blocks.  A function of the shapes only.
  int ks = 1;
  while (ks < 8 && (long)n_units * ks <= 2 * 148L * 24 && nblk / (ks * 2) >= 16) ks *= 2;
  p.ksplit = ks;
  const int upc = 8 / ks;
  const dim3 grid(std::max(1, std::min((n_units + upc - 1) / upc, 148 * 8))), block(256);
  ++*n_launch;
  if (g.mx) {
    return sw ? launch_dep(gemv_mma_kernel<true, true>, grid, block, 0, st, g.pdl, 1, p)
              : launch_dep(gemv_mma_kernel<true, false>, grid, block, 0, st, g.pdl, 1, p);
  }
  return sw ? launch_dep(gemv_mma_kernel<false, true>, grid, block, 0, st, g.pdl, 1, p)
            : launch_dep(gemv_mma_kernel<false, false>, grid, block, 0, st, g.pdl, 1, p);
}

// The streaming kernel takes a pair at the rate of its weights, whoever else reads them, and is the faster one while the pairs share
// few experts.  Pairs per expert, streaming against grouped, us for the FFN half of a layer of 2048 x 768 experts: Q4 2: 43 / 49
// (32 experts), 70 / 70 (64), 132 / 123 (128), 4: 42.6 / 37.0 (16), 73 / 53 (32), 130 / 85 (64); MXFP4 0.5: 23 / 23.5 (16), 1:
// 38 / 37 (32), 59 / 53 (64), 104 / 81 (128), 2: 38 / 30 (16).  A function of the call's shapes, not of where experts are.
bool moe_gemv_mma_eligible(const MoeGemvParams& g) {
  return g.M > 1 && g.P >= (g.mx ? 1 : 3) * g.n_experts && g.P <= kMoePairs && g.K % 256 == 0 && !(g.ldx & 7) && !(reinterpret_cast<uintptr_t>(g.x) & 15) &&
         (g.mode == GEMV_SWIGLU_F16 || g.mode == GEMV_OUT_F32 || g.mode == GEMV_OUT_F16);
}

cudaError_t launch_moe_gemv_mma(const MoeGemvParams& g, const MoeJobs* jobs, int sm_count, int pdl, cudaStream_t st, uint64_t* n_launch) {
  const int pairs = jobs ? jobs->n : g.P;
  if (pairs <= 0) return cudaSuccess;
  if (!moe_gemv_mma_eligible(g)) return cudaErrorInvalidValue;
  const bool sw = g.mode == GEMV_SWIGLU_F16;
  MoeMmaParams p{};
  p.base0 = g.base0; p.base1 = g.base1; p.stride = g.stride; p.ids = jobs ? nullptr : g.ids;
  p.tab0 = g.tab0; p.tab1 = g.tab1; p.x_div = g.x_div; p.P = g.P; p.n_experts = g.n_experts; p.status = g.status;
  p.n_rows = g.n_rows; p.K = g.K; p.mode = g.mode; p.x = g.x; p.ldx = g.ldx;
  p.y32 = g.y32; p.y16 = g.y16; p.ldy = g.ldy;
  int ks = 1;
  while (ks < kRingWarps && g.K / 256 >= 2 * kMoeSplitSteps * ks) ks *= 2;
  p.ksplit = ks;
  MoeJobs none;
  none.n = 0;
  const size_t smem = (size_t)kRingWarps * (sw ? 2 * kRingStagesSw : kRingStages) * kRingTile;
  const long ctas = ((long)pairs * ((g.n_rows + 15) / 16) * ks + kRingWarps - 1) / kRingWarps;
  static std::atomic<uint64_t> attr_done;
  const cudaError_t e = smem_limit_once(&attr_done, {reinterpret_cast<const void*>(moe_mma_ring_kernel<false, false>), reinterpret_cast<const void*>(moe_mma_ring_kernel<true, false>),
                                                     reinterpret_cast<const void*>(moe_mma_ring_kernel<false, true>), reinterpret_cast<const void*>(moe_mma_ring_kernel<true, true>)},
                                        kRingWarps * std::max(kRingStages, 2 * kRingStagesSw) * kRingTile);
  if (e != cudaSuccess) return e;
  ++*n_launch;
  auto run = [&](auto* k) {
    return launch_dep(k, dim3((unsigned)std::min<long>(ctas, 2L * sm_count)), dim3(32 * kRingWarps), smem, st, pdl, 1, p, jobs ? *jobs : none);
  };
  if (g.mx) return sw ? run(moe_mma_ring_kernel<true, true>) : run(moe_mma_ring_kernel<true, false>);
  return sw ? run(moe_mma_ring_kernel<false, true>) : run(moe_mma_ring_kernel<false, false>);
}

}  // namespace ats
