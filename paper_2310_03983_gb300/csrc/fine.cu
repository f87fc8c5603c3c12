// fine.cu -- blocked Floyd-Warshall over 64-vertex blocks: the closure of matrices too small for
// the 128 x 128 tiles of the GEMM engine.
//
// What bounds a small closure is not arithmetic but the chain of dependent steps: per block of b
// vertices, close the diagonal tile (b serial steps), multiply the panels by it, update the next
// diagonal tile with them, and so on.  With 128-vertex blocks each link of that chain is a whole
// 128 x 128 x 128 product on ONE SM (2.1 M pairs, 10-15 us) or 128 closure steps over a tile that
// keeps that SM's ALU pipe busy for 256 clocks each, while most SMs idle: n = 512 took 338 us.
// 64-vertex blocks cut the work of a link by eight (262 K pairs) and spread a panel or a matrix over
// four times as many SMs.
//
// One launch runs one or two stages (a batch: up to eight).  Stage s (of S = ceil(n / 64)) is
//   A(s): D[i][j] = min(D[i][j], D[i][s-1] (x) D[s-1][j]) for every tile outside block row / column
//         s - 1 (phase 3 of block s - 1); tile (s, s) is then closed by Eq. 1 in registers (phase 1
//         of block s); A(0) is only that closure;
//   B(s): the panels of block s, in-place products with the closed tile (phase 2).
// Work items (tiles) are handed out by an atomic ticket counter in a topological order: the closing
// tile, the other tiles of block row and column s, as many other tiles as fill the grid's first
// round, B(s), the remaining tiles of A(s).  A panel item waits until the tiles of block row /
// column s are stored, an A item until all of stage s - 1 is.  An item only waits for items with
// smaller tickets, which running CTAs hold and finish in ticket order, so every wait ends whatever
// number of CTAs is resident (and each is bounded all the same).
//
// In place without copies: A(s) reads the panels of block s - 1 and writes none of them; B(s) writes
// (s, s-1) and (s-1, s), which A(s) reads only in block row / column s, and B(s) waits for those.
#include <algorithm>
#include <atomic>
#include <climits>

#include "closure.cuh"
#include "fine.cuh"
#include "tile64.cuh"

namespace apsp {

namespace {

struct FineArgs {
  int *d;
  int64_t ld;
  int n, nt;      // vertices, 64-vertex blocks
  int s0, s1;     // stages of this launch
  int groups;     // consumer groups in use per CTA
  int rest1;      // tiles of A(s) handed out before B(s), beside those of block row / column s
  int is_float;
  int inf;        // bits of the "no edge" value
  const int *wmax;
  int64_t wmult;
  int *counters;
  unsigned int *status;
};

// Many graphs in lockstep: staged one below the other in d, each padded to whole 128-vertex blocks with
// isolated vertices (grouped.cu).  Stage s runs for every graph with at least s blocks of 64.
struct FineGraphs {
  int ngroups;
  GraphGroup groups[kMaxGroups];
  const int *gsize;  // vertices of each graph (0: left alone); tiles of padding are skipped
};

struct FineItem {
  int i, j, s;           // output tile, stage
  int ai, aj, bi, bj;    // operand tiles (ai < 0: none, the item only closes its tile)
  int klen;              // k range (the last block may be partial)
  int row0;              // first row of the item's graph
  bool close, dep, panel, skip;
};

// Items of stage s of a matrix of nt blocks, by kind, in the order they are handed out: the closing tile,
// the other tiles of block row and column s, the first of the remaining tiles, the panels, the rest.
struct StageCounts {
  int close, dep, rest, panel;
  __device__ __forceinline__ int total() const { return close + dep + rest + panel; }
};
__device__ __forceinline__ StageCounts stage_counts(int nt, int s) {
  StageCounts c = {0, 0, 0, 0};
  if (s > nt) return c;
  c.close = s < nt;
  c.dep = s > 0 && s < nt ? 2 * nt - 4 : 0;
  c.rest = s == 0 ? 0 : s < nt ? (nt - 2) * (nt - 2) : (nt - 1) * (nt - 1);
  c.panel = s < nt ? 2 * (nt - 1) : 0;
  return c;
}
__device__ __forceinline__ int kind_count(const StageCounts &c, int kind) {
  return kind == 0 ? c.close : kind == 1 ? c.dep : kind == 2 ? c.rest : c.panel;
}

// Item x of one kind (0 close, 1 dep, 2 rest, 3 panel) of a matrix of nt blocks.
__device__ __forceinline__ FineItem fine_item(int nt, int s, int kind, int x) {
  FineItem it;
  it.s = s;
  it.close = kind == 0;
  it.dep = kind < 2;
  it.panel = kind == 3;
  int kblk = s - 1;
  if (kind == 0) {
    it.i = it.j = s;
  } else if (kind == 1) {
    const int u = x < nt - 2 ? x : x - (nt - 2), y = u + (u >= s - 1 ? 2 : 0);
    it.i = x < nt - 2 ? s : y;
    it.j = x < nt - 2 ? y : s;
  } else if (kind == 2) {
    const int w = s < nt ? nt - 2 : nt - 1, skip = s < nt ? 2 : 0;  // outside block rows / columns s - 1 and s
    const int ii = x / w, jj = x - ii * w;
    it.i = ii + (ii >= s - 1 ? skip : 0);
    it.j = jj + (jj >= s - 1 ? skip : 0);
  } else {
    kblk = s;
    if (x < nt - 1) {  // row panel: D[s][j] = D[s][s]* (x) D[s][j]
      it.i = s;
      it.j = x + (x >= s);
    } else {           // column panel: D[i][s] = D[i][s] (x) D[s][s]*
      it.i = (x - (nt - 1)) + ((x - (nt - 1)) >= s);
      it.j = s;
    }
  }
  it.ai = kblk < 0 ? -1 : it.i;
  it.aj = kblk;
  it.bi = kblk;
  it.bj = it.j;
  it.klen = kFB;
  it.row0 = 0;
  it.skip = false;
  return it;
}

// The counts of stage s over every matrix of the launch, and its item p.
template <bool G>
__device__ __forceinline__ StageCounts launch_counts(const FineArgs &a, const FineGraphs &gs, int s) {
  if (!G) return stage_counts(a.nt, s);
  StageCounts t = {0, 0, 0, 0};
  for (int k = 0; k < gs.ngroups; ++k) {
    const StageCounts c = stage_counts(2 * gs.groups[k].nb, s);
    const int m = gs.groups[k].count;
    t.close += m * c.close;
    t.dep += m * c.dep;
    t.rest += m * c.rest;
    t.panel += m * c.panel;
  }
  return t;
}

template <bool G>
__device__ __forceinline__ FineItem fine_decode(const FineArgs &a, const FineGraphs &gs, const StageCounts &c, int s, int p) {
  const int r1 = min(a.rest1, c.rest);
  int kind = 0, x = p;
  if (x >= c.close) { x -= c.close; kind = 1; }
  if (kind == 1 && x >= c.dep) { x -= c.dep; kind = 2; }
  if (kind == 2 && x >= r1) {
    if (x < r1 + c.panel) { x -= r1; kind = 3; }
    else x -= c.panel;
  }
  if (!G) {
    FineItem it = fine_item(a.nt, s, kind, x);
    it.klen = min(kFB, a.n - it.aj * kFB);
    return it;
  }
  int k = 0, per = 0, nt = 0;
  for (; k < gs.ngroups; ++k) {
    nt = 2 * gs.groups[k].nb;
    per = kind_count(stage_counts(nt, s), kind);
    if (x < per * gs.groups[k].count) break;
    x -= per * gs.groups[k].count;
  }
  const int q = x / per;
  FineItem it = fine_item(nt, s, kind, x - q * per);
  it.row0 = (int)gs.groups[k].row0 + q * nt * kFB;
  const int n = gs.gsize[gs.groups[k].first + q];
  it.skip = it.i * kFB >= n || it.j * kFB >= n || it.aj * kFB >= n;
  return it;
}

// Eq. 1 on the 64 x 64 register tile (entries past bk hold the "no edge" value: isolated vertices),
// two vertices k, k + 1 per step.  The lanes that hold the two rows publish them (two slots in
// turn); every thread closes its part of the pair of rows under {k, k + 1} itself,
//     r1' = min(r1, d[k+1][k] + r0),   r0' = min(r0, d[k][k+1] + r1'),
// and relaxes d[i][j] = min(d[i][j], d[i][k] + r0'[j], d[i][k+1] + r1'[j]) with its rows' entries
// of columns k and k + 1 as they stood before the step (a path that uses both vertices lies in r0' or
// r1'), taken from the lane of the same warp that holds them.  One barrier and one shared-memory
// round trip per two vertices, and on fp32 one 3-input min for two relaxations.  The steps are a
// serial chain, bound by latency: 385 clocks each on one warp per scheduler; 256 or 512 threads
// (370, 425), one vertex per step (535 per pair), selecting the published row by a branch instead of
// selects (440), four vertices per step (780 per two pairs) and publishing the next rows ahead
// of the rest of the step (530) were measured as well.
template <bool F32>
__device__ __forceinline__ void fine_close(int (&d)[4][8], int bk, int warp, int lane, int *rows, int bar0) {
  const int tn = lane & 7, sub = lane >> 3;
#pragma unroll 1
  for (int kb = 0; kb < bk; kb += 4) {
    const bool hi = kb & 32;
    const int kh = kb >> 4, src = (lane & 24) | ((kb & 31) >> 2);  // lane of this row group with columns kb .. kb + 3
    const bool own = warp == ((kb & 15) >> 2);                     // rows kb .. kb + 3: register row kh, one per 8 lanes
#pragma unroll
    for (int kp = 0; kp < 2; ++kp) {
      const int k = kb + 2 * kp;
      int *rb = rows + kp * 2 * kFB;
      if (own && (sub >> 1) == kp) {
        int e[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) e[j] = kh < 2 ? (kh == 0 ? d[0][j] : d[1][j]) : (kh == 2 ? d[2][j] : d[3][j]);
        int *o = rb + (sub & 1) * kFB + 4 * tn;
        *reinterpret_cast<int4 *>(o) = make_int4(e[0], e[1], e[2], e[3]);
        *reinterpret_cast<int4 *>(o + 32) = make_int4(e[4], e[5], e[6], e[7]);
      }
      int c0[4], c1[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        c0[i] = __shfl_sync(0xffffffffu, hi ? d[i][4 + 2 * kp] : d[i][2 * kp], src);
        c1[i] = __shfl_sync(0xffffffffu, hi ? d[i][5 + 2 * kp] : d[i][2 * kp + 1], src);
      }
      fine_bar_sync(bar0);
      const int d01 = rb[k + 1], d10 = rb[kFB + k];
      if (F32) {
        uint64_t r0[4], r1[4];
        lds128_2x64(rb + 4 * tn, r0[0], r0[1]);
        lds128_2x64(rb + 4 * tn + 32, r0[2], r0[3]);
        lds128_2x64(rb + kFB + 4 * tn, r1[0], r1[1]);
        lds128_2x64(rb + kFB + 4 * tn + 32, r1[2], r1[3]);
        const uint64_t p01 = pack2(__int_as_float(d01), __int_as_float(d01));
        const uint64_t p10 = pack2(__int_as_float(d10), __int_as_float(d10));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint64_t t = fadd2_64(p10, r0[j]);
          r1[j] = pack2(fminf(lo_of(r1[j]), lo_of(t)), fminf(hi_of(r1[j]), hi_of(t)));
          const uint64_t u = fadd2_64(p01, r1[j]);
          r0[j] = pack2(fminf(lo_of(r0[j]), lo_of(u)), fminf(hi_of(r0[j]), hi_of(u)));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint64_t q0 = pack2(__int_as_float(c0[i]), __int_as_float(c0[i]));
          const uint64_t q1 = pack2(__int_as_float(c1[i]), __int_as_float(c1[i]));
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const uint64_t t = fadd2_64(q0, r0[j]), u = fadd2_64(q1, r1[j]);
            d[i][2 * j] = __float_as_int(Ops<float>::min3(__int_as_float(d[i][2 * j]), lo_of(t), lo_of(u)));
            d[i][2 * j + 1] = __float_as_int(Ops<float>::min3(__int_as_float(d[i][2 * j + 1]), hi_of(t), hi_of(u)));
          }
        }
      } else {
        const int4 x0 = lds128(rb + 4 * tn), x1 = lds128(rb + 4 * tn + 32);
        const int4 y0 = lds128(rb + kFB + 4 * tn), y1 = lds128(rb + kFB + 4 * tn + 32);
        int r0[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
        int r1[8] = {y0.x, y0.y, y0.z, y0.w, y1.x, y1.y, y1.z, y1.w};
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          r1[j] = __viaddmin_s32(d10, r0[j], r1[j]);
          r0[j] = __viaddmin_s32(d01, r1[j], r0[j]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j)
            d[i][j] = __viaddmin_s32(c1[i], r1[j], __viaddmin_s32(c0[i], r0[j], d[i][j]));
      }
    }
  }
}

constexpr int kFClose = 1, kFDep = 2, kFStageShift = 2;  // flags of an item slot

// The consumer warps compute; a group's loading warp takes tickets, waits for an item's dependencies and
// starts the TMA copies of its operand tiles into one of two buffers (so the next item's tiles arrive
// during this one's product) and of its old output tile; its releasing warp counts stored items, so
// that the fence this needs is off the consumers' path.  mA: boxes of 64 rows x 32 columns, 128-byte
// swizzle; mB: 64 x 64.  The register split is the GEMM engine's (tgemm.cuh).
template <bool G>
__global__ void __launch_bounds__(kFThreads, 1)
    fine_fw_kernel(const __grid_constant__ FineArgs a, const __grid_constant__ FineGraphs gs,
                   const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB) {
  extern __shared__ uint8_t smem_raw[];
  int *const smem0 = reinterpret_cast<int *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int wg = threadIdx.x / kFGroup, lane = threadIdx.x & 31;
  const int g = wg < kFGroups ? wg : ((threadIdx.x >> 5) & 1);  // group of this warp
  int *const smem = smem0 + g * kFGroupInts;
  int *const old = smem + 4 * kFTileInts;
  uint64_t *full = reinterpret_cast<uint64_t *>(smem0 + kFGroups * kFGroupInts) + g * (kFBarBytes / 8), *empty = full + 2;
  uint64_t *rel_full = full + 4, *rel_empty = full + 6, *cfull = full + 8, *cempty = full + 9;
  volatile int *slot = reinterpret_cast<volatile int *>(full + 10);  // [2][4]: i (< 0: no more), j, klen, flags
  volatile int *rel = slot + 8;                                     // [2]: flags (< 0: no more)
  // Ticket of the closing item each group holds (INT_MAX: none).
  volatile int *closing = reinterpret_cast<volatile int *>(smem0 + kFGroups * kFGroupInts + kFGroups * kFBarBytes / 4);
  int *const ticket = a.counters, *const finished = a.counters + 1, *const cnt = a.counters + 2;
  // cnt[2 x]: stored tiles of block row / column s, cnt[2 x + 1]: stored items, of stage s = s0 + x.
  if (wg < kFGroups && threadIdx.x % kFGroup == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(&full[b], 1);
      mbar_init(&empty[b], 4);
      mbar_init(&rel_full[b], 4);
      mbar_init(&rel_empty[b], 1);
    }
    mbar_init(cfull, 1);
    mbar_init(cempty, 4);
    closing[g] = INT_MAX;
    fence_barrier_init();
  }
  if (threadIdx.x == 0) {
    tma_prefetch_desc(&mA);
    tma_prefetch_desc(&mB);
  }
  __syncthreads();
  pdl_wait();  // after the set-up, before any global memory access
  pdl_trigger();

  if (wg == kFGroups) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kProducerRegs));
    if (lane != 0 || g >= a.groups) return;
    if ((threadIdx.x >> 5) % 4 < 2) {  // ------------------------- loads -------------------------
      uint32_t issued = 0, pars = 0;
      int s = a.s0, base = 0, before = 0;  // current stage, its first ticket, the items of the one before it
      StageCounts sc = launch_counts<G>(a, gs, s);
      for (int n = 0;; ++n) {
        const int b = n & 1;
        const uint32_t ph = (n >> 1) & 1;
        const int t = atomicAdd(ticket, 1);
        while (s < a.s1 && t - base >= sc.total()) {
          base += before = sc.total();
          if (++s < a.s1) sc = launch_counts<G>(a, gs, s);
        }
        bool ok = true;
        FineItem it = {};
        if (s < a.s1) {
          it = fine_decode<G>(a, gs, sc, s, t - base);
          const int x = 2 * (s - a.s0);
          if (G && it.skip) {  // padding: nothing to do, but counted
            if (it.dep) atomicAdd(cnt + x, 1);
            atomicAdd(cnt + x + 1, 1);
            --n;
            continue;
          }
          // The closing item heads the chain of dependent steps: the SM's other group starts no later item
          // until it is closed (which depends on no later ticket).
          if (it.close) closing[g] = t;
          if (a.groups == 2)
            for (uint32_t w = 0; t > closing[g ^ 1] && w < kSpinLimit; ++w) __nanosleep(64);
          if (it.panel) ok = counter_wait(cnt + x, sc.close + sc.dep, a.status);
          else if (s > a.s0) ok = counter_wait(cnt + x - 1, before, a.status);
          fence_proxy_async_global();
        }
        ok = mbar_wait(&empty[b], ph ^ 1, a.status) && ok;
        if (s >= a.s1 || !ok) {
          for (int x = 0; x < 2; ++x)  // leave no copy writing into an exiting CTA's shared memory
            if (issued & (1u << x)) mbar_wait(&full[x], (pars >> x) & 1, a.status);
          if (n > 0) mbar_wait(cfull, (n - 1) & 1, a.status);
          slot[4 * b] = -1;
          mbar_arrive(&full[b]);
          break;
        }
        const int row = it.row0 / kFB;
        slot[4 * b] = row + it.i;
        slot[4 * b + 1] = it.j;
        slot[4 * b + 2] = it.ai >= 0 ? it.klen : 0;
        slot[4 * b + 3] = (it.close ? kFClose : 0) | (it.dep ? kFDep : 0) | ((it.s - a.s0) << kFStageShift);
        if (it.ai < 0) {
          mbar_arrive(&full[b]);
        } else {
          int *buf = smem + b * 2 * kFTileInts;
          mbar_arrive_expect_tx(&full[b], 2 * kFTileInts * 4);
          tma_load_2d(buf, &mA, it.aj * kFB, (row + it.ai) * kFB, &full[b]);
          tma_load_2d(buf + kFTileInts / 2, &mA, it.aj * kFB + 32, (row + it.ai) * kFB, &full[b]);
          tma_load_2d(buf + kFTileInts, &mB, it.bj * kFB, (row + it.bi) * kFB, &full[b]);
          issued |= 1u << b;
          pars = (pars & ~(1u << b)) | (ph << b);
        }
        // The old output tile is needed only after the product.
        mbar_wait(cempty, (n & 1) ^ 1, a.status);
        mbar_arrive_expect_tx(cfull, kFTileInts * 4);
        tma_load_2d(old, &mB, it.j * kFB, (row + it.i) * kFB, cfull);
      }
    } else {  // ------------------------------------------------ releases ----------------------
      for (int n = 0;; ++n) {
        const int b = n & 1;
        if (!mbar_wait(&rel_full[b], (n >> 1) & 1, a.status)) break;
        const int f = rel[b];
        if (f < 0) break;
        mbar_arrive(&rel_empty[b]);
        __threadfence();  // the consumers' stores, observed through the barrier, before the count
        int *const c = cnt + 2 * (f >> kFStageShift);
        if (f & kFDep) atomicAdd(c, 1);
        atomicAdd(c + 1, 1);
      }
      // The last group to finish has seen every other group's final ticket: it resets the words.
      __threadfence();
      if (atomicAdd(finished, 1) == (int)gridDim.x * a.groups - 1)
        for (int w = 0; w < kFineWords; ++w) a.counters[w] = 0;
    }
    return;
  }

  // -------------------------------------- products and closures ------------------------------
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kConsumerRegs));
  if (g >= a.groups) return;
  const int warp = (threadIdx.x >> 5) % 4, tm = warp * 4 + (lane >> 3), tn = lane & 7;
  const int bar0 = 1 + g;
  const bool f32 = a.is_float || (a.wmax && small_int_bound(a.wmax[0], a.wmult, a.wmax[1]));
  int n = 0;
  for (;; ++n) {
    const int b = n & 1;
    const uint32_t ph = (n >> 1) & 1;
    if (!mbar_wait(&full[b], ph, a.status)) break;
    const int ti = slot[4 * b], cj = slot[4 * b + 1] * kFB, klen = slot[4 * b + 2], flags = slot[4 * b + 3];
    if (ti < 0) break;
    const int ri = ti * kFB;
    const int *As = smem + b * 2 * kFTileInts, *Bs = As + kFTileInts;
    float acc[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = __int_as_float(a.inf);
    if (f32) fine_product_f32(As, Bs, tm, tn, klen, acc);
    else fine_product_int<false>(As, Bs, tm, tn, klen, acc);
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[b]);
    // Fold the old entries (a product with a closed tile contains them anyway).
    if (!mbar_wait(cfull, n & 1, a.status)) break;
    int d[4][8];
    fine_get(d, old, tm, tn);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j)  // non-negative values order alike as fp32 and as int32 bit patterns
        d[i][j] = min(d[i][j], __float_as_int(acc[i][j]));
    if (flags & kFClose) {
      const int bk = min(kFB, a.n - ri);
      if (bk < kFB) {  // vertices past the last one are isolated
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (tm + 16 * i >= bk || 4 * tn + 32 * (j >> 2) + (j & 3) >= bk) d[i][j] = a.inf;
      }
      fine_bar_sync(bar0);  // the old tile is read: its buffer takes the published rows
      if (f32) fine_close<true>(d, bk, warp, lane, old, bar0);
      else fine_close<false>(d, bk, warp, lane, old, bar0);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before the next tile's copy into it
      if (warp == 0 && lane == 0) closing[g] = INT_MAX;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(cempty);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = ri + tm + 16 * i;
      if (r >= a.n) continue;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int col = cj + 4 * tn + 32 * h;
        int *o = a.d + (int64_t)r * a.ld + col;
        if (col + 3 < a.n) {
          *reinterpret_cast<int4 *>(o) = make_int4(d[i][4 * h], d[i][4 * h + 1], d[i][4 * h + 2], d[i][4 * h + 3]);
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (col + q < a.n) o[q] = d[i][4 * h + q];
        }
      }
    }
    if (!mbar_wait(&rel_empty[b], ph ^ 1, a.status)) break;
    if (warp == 0 && lane == 0) rel[b] = flags;
    __syncwarp();
    if (lane == 0) mbar_arrive(&rel_full[b]);
  }
  mbar_wait(&rel_empty[n & 1], ((n >> 1) & 1) ^ 1, a.status);
  if (warp == 0 && lane == 0) rel[n & 1] = -1;
  __syncwarp();
  if (lane == 0) mbar_arrive(&rel_full[n & 1]);
}

}  // namespace

// Two consumer groups share an SM's ALUs, so each item takes longer (a 64^3 product 4.1 us against
// 2.4 us) but the SM does more: worth it once the tiles of a stage, not the chain of dependent items,
// bound it.  Measured (float32, one / two groups): n = 1024 291 / 353 us, 1448 414 / 514, 2048 851 /
// 785, 2896 2212 / 1857, 4092 5623 / 4682: the line is drawn at 4.5 tiles per SM (n = 1730 on 152 SMs).
static int fine_groups(int64_t tiles, int sms) { return 2 * tiles > 9 * sms ? 2 : 1; }

template <bool G>
static int fine_launch(const FineArgs &a, const FineGraphs &gs, int64_t most, double pairs, int trace_mode,
                       const CUtensorMap &mA, const CUtensorMap &mB, cudaStream_t s) {
  auto k = fine_fw_kernel<G>;
  static std::atomic<int> checked{0};  // 1: register split verified (see launch_one in tgemm.cu)
  if (!checked.load(std::memory_order_relaxed)) {
    cudaFuncAttributes fa;
    APSP_CUDA_TRY(cudaFuncGetAttributes(&fa, k));
    if (fa.numRegs < kLaunchRegs || fa.maxThreadsPerBlock < kFThreads) return APSP_ERR_UNSUPPORTED;
    checked.store(1, std::memory_order_relaxed);
  }
  APSP_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kFSmemBytes));
  const int grid = (int)std::min<int64_t>(most, sm_count());
  FineArgs b = a;
  b.rest1 = (int)std::max<int64_t>(0, (int64_t)grid * a.groups - a.rest1);
  void *ev = nullptr;
  if (trace_on()) trace_begin(s, &ev);
  launch_pdl(k, grid, kFThreads, kFSmemBytes, s, b, gs, mA, mB);
  APSP_LAUNCH_CHECK();
  if (ev) trace_end(s, ev, trace_mode, pairs);
  return APSP_OK;
}

static int fine_maps(CUtensorMap *mA, CUtensorMap *mB, const void *d, int64_t rows, int64_t cols, int64_t ld, int dtype) {
  int r;
  if ((r = make_tmap_2d(mA, d, rows, cols, ld, kFB, 32, dtype, true))) return r;
  return make_tmap_2d(mB, d, rows, cols, ld, kFB, kFB, dtype);
}

int fine_closure(void *d, int64_t n, int64_t ld, int dtype, int inf_i, const int *wmax, int64_t wmult,
                 int *counters, int trace_class, cudaStream_t s) {
  CUtensorMap mA, mB;
  int r;
  if ((r = fine_maps(&mA, &mB, d, n, n, ld, dtype))) return r;
  FineArgs a = {};
  a.d = reinterpret_cast<int *>(d);
  a.ld = ld;
  a.n = (int)n;
  a.nt = (int)cdiv(n, kFB);
  a.is_float = dtype == APSP_F32;
  a.inf = dtype == APSP_F32 ? 0x7f800000 : inf_i;
  a.wmax = dtype == APSP_F32 ? nullptr : wmax;
  a.wmult = wmult;
  a.counters = counters;
  a.status = status_word();
  a.groups = fine_groups((int64_t)(a.nt - 1) * (a.nt - 1), sm_count());
  a.rest1 = 2 * a.nt - 3;
  // nt + 1 stages over as many launches as the 128-vertex loop makes: two, and one per 128 vertices.
  const int stages = a.nt + 1, launches = (int)cdiv(n, kBM) + 2;
  for (int l = 0; l < launches; ++l) {
    a.s0 = (int)((int64_t)stages * l / launches);
    a.s1 = (int)((int64_t)stages * (l + 1) / launches);
    int most = 1;
    double pairs = 0.0;
    for (int st = a.s0; st < a.s1; ++st) {
      const int na = st == 0 ? 1 : (a.nt - 1) * (a.nt - 1), npan = st < a.nt ? 2 * (a.nt - 1) : 0;
      most = std::max(most, std::max(na, npan));
      if (st > 0) {
        const double k = (double)std::min<int64_t>(kFB, n - (int64_t)(st - 1) * kFB);
        pairs += ((double)n - k) * ((double)n - k) * k;
      }
    }
    if ((r = fine_launch<false>(a, FineGraphs{}, most, pairs, kModeFwRest + trace_class, mA, mB, s))) return r;
  }
  return APSP_OK;
}

int64_t fine_batch_tiles(const GraphGroup *groups, int ngroups) {
  int64_t t = 0;
  for (int k = 0; k < ngroups; ++k) {
    const int64_t m = 2 * groups[k].nb - 1;
    t += m * m * groups[k].count;
  }
  return t;
}

int fine_batch(void *d, int64_t rows, int64_t ld, const GraphGroup *groups, int ngroups, const int *gsize, int dtype,
               int inf_i, const int *wmax, int *counters, cudaStream_t s) {
  CUtensorMap mA, mB;
  int r;
  if ((r = fine_maps(&mA, &mB, d, rows, ld, ld, dtype))) return r;
  FineArgs a = {};
  a.d = reinterpret_cast<int *>(d);
  a.ld = ld;
  a.n = INT_MAX;  // the staged graphs are whole tiles
  a.is_float = dtype == APSP_F32;
  a.inf = dtype == APSP_F32 ? 0x7f800000 : inf_i;
  a.wmax = dtype == APSP_F32 ? nullptr : wmax;
  a.wmult = 1;
  a.counters = counters;
  a.status = status_word();
  const int64_t tiles = fine_batch_tiles(groups, ngroups);
  a.groups = fine_groups(tiles, sm_count());
  FineGraphs gs = {};
  gs.ngroups = ngroups;
  gs.gsize = gsize;
  int64_t dep = 0;
  for (int k = 0; k < ngroups; ++k) {
    gs.groups[k] = groups[k];
    dep += (int64_t)groups[k].count * (4 * groups[k].nb - 3);
  }
  a.rest1 = (int)dep;
  const int stages = 2 * groups[0].nb + 1;  // groups are listed by decreasing nb
  for (a.s0 = 0; a.s0 < stages; a.s0 = a.s1) {
    a.s1 = std::min(stages, a.s0 + kFineMaxStages);
    double pairs = 0.0;
    for (int st = std::max(1, a.s0); st < a.s1; ++st)
      for (int k = 0; k < ngroups; ++k) {
        const double m = (2.0 * groups[k].nb - 1) * kFB;
        if (st <= 2 * groups[k].nb) pairs += groups[k].count * m * m * kFB;
      }
    if ((r = fine_launch<true>(a, gs, tiles, pairs, kModeFwRest, mA, mB, s))) return r;
  }
  return APSP_OK;
}

}  // namespace apsp
