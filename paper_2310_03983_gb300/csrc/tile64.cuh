// tile64.cuh -- (min,+) arithmetic on 64 x 64 output tiles, for work too small to fill the GPU with the
// engine's 128 x 128 tiles: the closure of small matrices (fine.cu), small products and repeated
// squaring (gemm64.cu).
#pragma once

#include "slab.cuh"
#include "tgemm.cuh"

namespace apsp {

constexpr int kFB = 64;  // block and tile edge
// A CTA (one per SM) holds up to two consumer groups of 128 threads, each with its own tickets, and
// a warpgroup with a loading and a releasing warp per group.  Thread (tm, tn) of a group holds rows
// tm + 16 i and columns 4 tn + 32 h + q of its tile.
constexpr int kFGroup = 128;
constexpr int kFGroups = 2;
constexpr int kFThreads = (kFGroups + 1) * kFGroup;
constexpr int kFTileInts = kFB * kFB;
// Per group: two buffers of operand tiles, the old output tile (then the closure's published rows).
constexpr int kFGroupInts = 5 * kFTileInts;
constexpr int kFBarBytes = 256;  // barriers and item slots of a group
constexpr int kFSmemBytes = 1024 + kFGroups * (kFGroupInts * 4 + kFBarBytes) + 16;

// Offset of the 16-byte chunk kq (k = 4 kq ..) of row r of the A tile: two [64 m][32 k] halves, each
// TMA-loaded with 128-byte swizzle (a_off).
__device__ __forceinline__ int fa_off(int r, int kq) { return (kq >> 3) * (kFTileInts / 2) + a_off(r, kq & 7); }

// acc = min(acc, A (x) B) over the first klen k.  fp32 as ArithF32::slab_full (packed pair adds over
// columns, 3-input mins over k pairs).
__device__ __forceinline__ void fine_ld_a(float4 (&a)[4], const int *As, int tm, int q) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int4 v = lds128(As + fa_off(tm + 16 * i, q));
    a[i] = make_float4(__int_as_float(v.x), __int_as_float(v.y), __int_as_float(v.z), __int_as_float(v.w));
  }
}
__device__ __forceinline__ void fine_ld_b(uint64_t (&b0)[4], uint64_t (&b1)[4], const int *r) {
  lds128_2x64(r, b0[0], b0[1]);
  lds128_2x64(r + 32, b0[2], b0[3]);
  lds128_2x64(r + kFB, b1[0], b1[1]);
  lds128_2x64(r + kFB + 32, b1[2], b1[3]);
}
__device__ __forceinline__ void fine_math(float (&acc)[4][8], const float4 (&a)[4], int kp, const uint64_t (&b0)[4],
                                          const uint64_t (&b1)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float a0 = kp ? a[i].z : a[i].x, a1 = kp ? a[i].w : a[i].y;
    const uint64_t aa0 = pack2(a0, a0), aa1 = pack2(a1, a1);
    uint64_t t0[4], t1[4];
#pragma unroll
    for (int jp = 0; jp < 4; ++jp) t0[jp] = fadd2_64(aa0, b0[jp]);
#pragma unroll
    for (int jp = 0; jp < 4; ++jp) t1[jp] = fadd2_64(aa1, b1[jp]);
#pragma unroll
    for (int jp = 0; jp < 4; ++jp) {
      acc[i][2 * jp] = Ops<float>::min3(acc[i][2 * jp], lo_of(t0[jp]), lo_of(t1[jp]));
      acc[i][2 * jp + 1] = Ops<float>::min3(acc[i][2 * jp + 1], hi_of(t0[jp]), hi_of(t1[jp]));
    }
  }
}
// Operands are read one k pair ahead of the arithmetic (two warps per scheduler do not hide the
// shared loads' latency otherwise); the last read, past the k range, stays inside the group's buffers.
__device__ __forceinline__ void fine_product_f32(const int *As, const int *Bs, int tm, int tn, int klen,
                                                 float (&acc)[4][8]) {
  const int nq = klen >> 2;
  const int *bp = Bs + 4 * tn;
  float4 a[4], an[4];
  uint64_t x0[4], x1[4], y0[4], y1[4];
  if (nq > 0) {
    fine_ld_a(a, As, tm, 0);
    fine_ld_b(x0, x1, bp);
  }
#pragma unroll 2
  for (int q = 0; q < nq; ++q) {
    fine_ld_b(y0, y1, bp + (4 * q + 2) * kFB);
    fine_ld_a(an, As, tm, q + 1);
    fine_math(acc, a, 0, x0, x1);
    fine_ld_b(x0, x1, bp + (4 * q + 4) * kFB);
    fine_math(acc, a, 1, y0, y1);
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = an[i];
  }
  for (int k = 4 * nq; k < klen; ++k) {
    const int4 u0 = lds128(Bs + k * kFB + 4 * tn), u1 = lds128(Bs + k * kFB + 4 * tn + 32);
    const int b[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float a = __int_as_float(As[fa_off(tm + 16 * i, k >> 2) + (k & 3)]);
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = fminf(acc[i][j], __fadd_rn(a, __int_as_float(b[j])));
    }
  }
}


// The same on int32 words: one DPX add-min per (i, j, k), or on packed 16-bit pairs (ArithInt<true>)
// one per two of them.
template <bool P16>
__device__ __forceinline__ void fine_product_int(const int *As, const int *Bs, int tm, int tn, int klen,
                                                 float (&acc)[4][8]) {
  typedef ArithInt<P16> AR;
  const int nq = klen >> 2;
  const int *bp = Bs + 4 * tn;
  int4 a[4], an[4], b0, b1, c0, c1;
  if (nq > 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = lds128(As + fa_off(tm + 16 * i, 0));
    b0 = lds128(bp);
    b1 = lds128(bp + 32);
  }
#pragma unroll 2
  for (int q = 0; q < nq; ++q) {
#pragma unroll
    for (int i = 0; i < 4; ++i) an[i] = lds128(As + fa_off(tm + 16 * i, q + 1));
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      const int *nx = bp + (4 * q + kk + 1) * kFB;
      c0 = lds128(nx);
      c1 = lds128(nx + 32);
      const int b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int av = kk == 0 ? a[i].x : kk == 1 ? a[i].y : kk == 2 ? a[i].z : a[i].w;
#pragma unroll
        for (int j = 0; j < 8; ++j) set_acc(acc[i][j], AR::addmin(av, b[j], acc_bits(acc[i][j])));
      }
      b0 = c0;
      b1 = c1;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = an[i];
  }
  for (int k = 4 * nq; k < klen; ++k) {
    const int4 u0 = lds128(bp + k * kFB), u1 = lds128(bp + k * kFB + 32);
    const int b[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int av = As[fa_off(tm + 16 * i, k >> 2) + (k & 3)];
#pragma unroll
      for (int j = 0; j < 8; ++j) set_acc(acc[i][j], AR::addmin(av, b[j], acc_bits(acc[i][j])));
    }
  }
}

// Named barrier among the 128 threads of a consumer group.
__device__ __forceinline__ void fine_bar_sync(int bar) {
  asm volatile("bar.sync %0, 128;" ::"r"(bar) : "memory");
}

// A thread's part of a tile [64][64] in shared memory.
__device__ __forceinline__ void fine_get(int (&d)[4][8], const int *t, int tm, int tn) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int4 v = lds128(t + (tm + 16 * i) * kFB + 4 * tn + 32 * h);
      d[i][4 * h] = v.x; d[i][4 * h + 1] = v.y; d[i][4 * h + 2] = v.z; d[i][4 * h + 3] = v.w;
    }
}
}  // namespace apsp
