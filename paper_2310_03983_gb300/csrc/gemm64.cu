// gemm64.cu -- (min,+) products on 64 x 64 tiles, and repeated squaring (Sec. 3.2) as one launch.
//
// The engine's 128 x 128 tiles leave most SMs idle in a product with few of them: 1024^3 is 64 tiles on
// 152 SMs, each a chain of 2 x 10^7 pairs.  64 x 64 tiles give four times as many items, each a
// quarter of the work, and two consumer groups per SM keep its ALUs as busy as one large tile does.
// The CTA is fine.cu's: two consumer groups of 128 threads, a loading and a releasing warp per group.
//
// Squaring adds stages: stage t reads set t & 1 and writes set (t + 1) & 1.  Tiles are handed out by
// tickets, stage by stage; a tile of stage t waits until every tile of stage t - 1 is stored (one
// counter: a stage cannot start before the one before it is complete), and the loop ends at the first
// stage that changes nothing.  An item waits only for smaller tickets, held by running CTAs, so every
// wait ends.  int32 matrices whose entries stay below half the 16-bit cap run on packed 16-bit
// pairs, both packed forms of a product written by the tiles that compute it; when entries outgrow
// that, the remaining products run on 32 bits (here, or on 128 x 128 tiles in squaring.cu's loop).
#include <algorithm>
#include <atomic>

#include "gemm64.cuh"
#include "tile64.cuh"

namespace apsp {

namespace {

// Words of a squaring call (64, zeroed): [0] largest finite weight, [1] zero.
constexpr int kSPacked = 2;     // the packed forms exist (square_prep_kernel ran)
constexpr int kSAbort = 3;      // 1 + the stage at which they stopped (0: they finished)
constexpr int kSCtr16 = 4;      // ticket, unused, done (16-bit stages)
constexpr int kSCtr32 = 8;      // the same for the 32-bit stages
constexpr int kSMaxStages = 12; // products that close kSquaring64MaxN vertices
constexpr int kSChanged16 = 12; // per stage: something changed
constexpr int kSMax16 = 24;     // per stage: largest finite entry written
constexpr int kSChanged32 = 36;
static_assert(int64_t(1) << kSMaxStages >= kSquaring64MaxN - 1, "stages");
static_assert(kSChanged16 + kSMaxStages <= kSMax16 && kSMax16 + kSMaxStages <= kSChanged32 &&
                  kSChanged32 + kSMaxStages <= kSquareUnchanged && kSquareUnchanged + kSMaxStages <= kSquareSkip &&
                  kSquareSkip < 64, "squaring words");

enum { kProduct = 0, kSquare32 = 1, kSquare16 = 2, kArgChunk = 3 };

struct G64Args {
  int M, N, K;         // K in operand words
  int tiles_n, items;  // 64 x 64 tiles: per row, per stage
  int stages, groups;
  int acc, is_float, inf;
  int *out[2];         // product: out[0]; 32-bit squaring: the two sets
  int64_t ldo[2];
  int *pa[2], *pb[2];  // 16-bit squaring: the two sets
  int64_t lda16, ldb16;
  const int *wmax;
  int64_t wmult;
  const int *skip, *run_if;
  int *words;
  unsigned int *status;
};

struct G64Maps {
  CUtensorMap A[2], B[2], old;
};

constexpr int kGFirst = 1, kGLast = 2, kGStageShift = 2;

// Whether the 16-bit stages run: the packed forms exist and twice the largest weight is below the cap.
__device__ __forceinline__ bool mode16(const int *words) {
  return words[kSPacked] && 2 * (int64_t)words[0] < kCap16;
}

// The number of stages of the 32-bit squaring: all, or those the 16-bit stages left.
__device__ __forceinline__ int stages32(const int *words, int stages) {
  if (!mode16(words)) return stages;
  return words[kSAbort] ? stages - (words[kSAbort] - 1) : 0;
}

template <int KIND, bool P16>
__global__ void __launch_bounds__(kFThreads, 1) gemm64_kernel(const __grid_constant__ G64Args a,
                                                              const __grid_constant__ G64Maps maps) {
  extern __shared__ uint8_t smem_raw[];
  int *const smem0 = reinterpret_cast<int *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int wg = threadIdx.x / kFGroup, lane = threadIdx.x & 31;
  const int g = wg < kFGroups ? wg : ((threadIdx.x >> 5) & 1);
  int *const smem = smem0 + g * kFGroupInts;
  int *const old = smem + 4 * kFTileInts;
  uint64_t *full = reinterpret_cast<uint64_t *>(smem0 + kFGroups * kFGroupInts) + g * (kFBarBytes / 8), *empty = full + 2;
  uint64_t *rel_full = full + 4, *rel_empty = full + 6, *cfull = full + 8, *cempty = full + 9;
  volatile int *slot = reinterpret_cast<volatile int *>(full + 10);  // [2][4]: tile row (< 0: no more), column, klen, flags
  volatile int *rel = slot + 8;                                     // [2]: 1, or -1: no more
  const bool has_old = KIND == kSquare32 || (KIND == kProduct && a.acc);
  int *const ctr = a.words + (KIND == kSquare16 ? kSCtr16 : kSCtr32);  // ticket, unused, done
  int *const changed = a.words + (KIND == kSquare16 ? kSChanged16 : kSChanged32);
  if (wg < kFGroups && threadIdx.x % kFGroup == 0) {
    for (int b = 0; b < 2; ++b) {
      mbar_init(&full[b], 1);
      mbar_init(&empty[b], 4);
      mbar_init(&rel_full[b], 4);
      mbar_init(&rel_empty[b], 1);
    }
    mbar_init(cfull, 1);
    mbar_init(cempty, 4);
    fence_barrier_init();
  }
  __syncthreads();
  pdl_wait();  // after the set-up, before any global memory access
  pdl_trigger();
  if ((a.skip && *a.skip) || (a.run_if && !*a.run_if)) return;
  if (KIND == kSquare16 && !mode16(a.words)) return;
  const int stages = KIND == kSquare32 ? stages32(a.words, a.stages) : a.stages;
  if (stages <= 0) return;

  if (wg == kFGroups) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kProducerRegs));
    if (lane != 0 || g >= a.groups) return;
    if ((threadIdx.x >> 5) % 4 < 2) {  // ------------------------- loads -------------------------
      const int chunks = (a.K - 1) / kFB + 1, step = gridDim.x * a.groups;  // K may be INT32_MAX
      uint32_t issued = 0, pars = 0, c = 0;  // c: chunks issued so far
      int m = 0, seen = 0;                   // items so far; stages known to have changed something
      bool ok = true;
      for (int it = blockIdx.x * a.groups + g;; it += step, ++m) {
        int t = it, st = 0;
        if (KIND == kSquare32 || KIND == kSquare16) {
          t = atomicAdd(ctr, 1);
          st = t / a.items;
          t -= st * a.items;
          if (st >= stages) break;
          // Stage by stage, since the loop may have ended before this ticket's stage.
          bool go = true;
          for (; seen < st && go; ++seen) {
            go = counter_wait(ctr + 2, (seen + 1) * a.items, a.status) && __ldcg(changed + seen);
            if (KIND == kSquare16 && go && 2 * (int64_t)__ldcg(a.words + kSMax16 + seen) >= kCap16) {
              a.words[kSAbort] = seen + 2;  // every loader decides alike
              go = false;
            }
          }
          if (!go) break;
          fence_proxy_async_global();
        } else if (t >= a.items) {
          break;
        }
        const int ti = t / a.tiles_n, tj = t - ti * a.tiles_n, set = st & 1;
        for (int k = 0; k < chunks && ok; ++k, ++c) {
          const int b = c & 1;
          const uint32_t ph = (c >> 1) & 1;
          if (!mbar_wait(&empty[b], ph ^ 1, a.status)) { ok = false; break; }
          slot[4 * b] = ti;
          slot[4 * b + 1] = tj;
          slot[4 * b + 2] = min(kFB, a.K - k * kFB);
          slot[4 * b + 3] = (k == 0 ? kGFirst : 0) | (k == chunks - 1 ? kGLast : 0) |
                            ((KIND == kArgChunk ? k : st) << kGStageShift);
          int *buf = smem + b * 2 * kFTileInts;
          mbar_arrive_expect_tx(&full[b], 2 * kFTileInts * 4);
          tma_load_2d(buf, &maps.A[set], k * kFB, ti * kFB, &full[b]);
          tma_load_2d(buf + kFTileInts / 2, &maps.A[set], k * kFB + 32, ti * kFB, &full[b]);
          tma_load_2d(buf + kFTileInts, &maps.B[set], tj * kFB, k * kFB, &full[b]);
          issued |= 1u << b;
          pars = (pars & ~(1u << b)) | (ph << b);
        }
        if (!ok) break;
        if (has_old) {
          if (!mbar_wait(cempty, (m & 1) ^ 1, a.status)) { ok = false; break; }
          mbar_arrive_expect_tx(cfull, kFTileInts * 4);
          tma_load_2d(old, KIND == kProduct ? &maps.old : &maps.B[set], tj * kFB, ti * kFB, cfull);
        }
      }
      for (int x = 0; x < 2; ++x)  // leave no copy writing into an exiting CTA's shared memory
        if (issued & (1u << x)) mbar_wait(&full[x], (pars >> x) & 1, a.status);
      if (has_old && m > 0) mbar_wait(cfull, (m - 1) & 1, a.status);
      const int b = c & 1;
      mbar_wait(&empty[b], ((c >> 1) & 1) ^ 1, a.status);
      slot[4 * b] = -1;
      mbar_arrive(&full[b]);
    } else if (KIND == kSquare32 || KIND == kSquare16) {  // ------------ releases ----------------------
      for (int n = 0;; ++n) {
        const int b = n & 1;
        if (!mbar_wait(&rel_full[b], (n >> 1) & 1, a.status)) break;
        if (rel[b] < 0) break;
        mbar_arrive(&rel_empty[b]);
        __threadfence();  // the consumers' stores and flags, observed through the barrier, before the count
        atomicAdd(ctr + 2, 1);
      }
    }
    return;
  }

  // ------------------------------------------ products --------------------------------------
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kConsumerRegs));
  if (g >= a.groups) return;
  const int warp = (threadIdx.x >> 5) % 4, tm = warp * 4 + (lane >> 3), tn = lane & 7;
  const bool f32 = !P16 && (a.is_float || (a.wmax && small_int_bound(a.wmax[0], a.wmult, a.wmax[1])));
  const int init = P16 ? (kCap16 << 16) | kCap16 : a.inf;
  float acc[4][8], best[KIND == kArgChunk ? 4 : 1][8];  // kArgChunk: minima so far, and the chunks
  int arg[KIND == kArgChunk ? 4 : 1][8];                // that first reached them
  int m = 0;
  for (uint32_t c = 0;; ++c) {
    const int b = c & 1;
    if (!mbar_wait(&full[b], (c >> 1) & 1, a.status)) break;
    const int ti = slot[4 * b], tj = slot[4 * b + 1], klen = slot[4 * b + 2], flags = slot[4 * b + 3];
    if (ti < 0) break;
    if (KIND == kArgChunk || (flags & kGFirst)) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          acc[i][j] = __int_as_float(init);
          if (KIND == kArgChunk && (flags & kGFirst)) {
            best[i][j] = __int_as_float(init);
            arg[i][j] = -1;
          }
        }
    }
    const int *As = smem + b * 2 * kFTileInts, *Bs = As + kFTileInts;
    if (P16) fine_product_int<true>(As, Bs, tm, tn, klen, acc);
    else if (f32) fine_product_f32(As, Bs, tm, tn, klen, acc);
    else fine_product_int<false>(As, Bs, tm, tn, klen, acc);
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[b]);
    if (KIND == kArgChunk) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          arg[i][j] = acc[i][j] < best[i][j] ? flags >> kGStageShift : arg[i][j];
          best[i][j] = fminf(best[i][j], acc[i][j]);
        }
    }
    if (!(flags & kGLast)) continue;
    const int ri = ti * kFB, cj = tj * kFB, set = (flags >> kGStageShift) & 1, st = flags >> kGStageShift;
    int v[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int x = __float_as_int(acc[i][j]);
        if (KIND == kArgChunk) v[i][j] = arg[i][j];
        else if (KIND == kSquare16) v[i][j] = ArithI16x2::collapse_truncated(x);
        else v[i][j] = P16 ? ArithI16x2::collapse(x, a.inf) : x;
      }
    bool diff = false;
    if (has_old) {
      if (!mbar_wait(cfull, m & 1, a.status)) break;
      int o[4][8];
      fine_get(o, old, tm, tn);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const bool in = ri + tm + 16 * i < a.M && cj + 4 * tn + 32 * (j >> 2) + (j & 3) < a.N;
          if (KIND == kProduct)
            v[i][j] = a.is_float ? __float_as_int(fminf(__int_as_float(v[i][j]), __int_as_float(o[i][j])))
                                 : min(v[i][j], o[i][j]);
          else diff |= in && v[i][j] != o[i][j];
        }
      __syncwarp();
      if (lane == 0) mbar_arrive(cempty);
    }
    if (KIND == kSquare16) {
      // Both packed forms of the tile into the other set; entries past the matrix count as CAP.
      int big = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = ri + tm + 16 * i;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int col = cj + 4 * tn + 32 * h;
          int2 o = make_int2(0, 0);
          if (r < a.M && col < a.N) o = __ldcg(reinterpret_cast<const int2 *>(a.pa[set] + (int64_t)r * a.lda16 + (col >> 1)));
          int w[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const bool in = r < a.M && col + q < a.N;
            w[q] = in ? v[i][4 * h + q] : kCap16;
            const int ov = ((q & 2 ? o.y : o.x) >> (16 * (q & 1))) & 0xFFFF;
            diff |= in && w[q] != ov;
            if (w[q] < kCap16) big = max(big, w[q]);
            v[i][4 * h + q] = w[q];
          }
          if (r < a.M && col < a.N)
            *reinterpret_cast<int2 *>(a.pa[set ^ 1] + (int64_t)r * a.lda16 + (col >> 1)) =
                make_int2((w[1] << 16) | w[0], (w[3] << 16) | w[2]);
          int u[4];  // row r ^ 1 sits in lane ^ 8
#pragma unroll
          for (int q = 0; q < 4; ++q) u[q] = __shfl_xor_sync(0xffffffffu, w[q], 8);
          if (!(tm & 1) && r < a.M && col < a.N)
            *reinterpret_cast<int4 *>(a.pb[set ^ 1] + (int64_t)(r >> 1) * a.ldb16 + col) =
                make_int4((u[0] << 16) | w[0], (u[1] << 16) | w[1], (u[2] << 16) | w[2], (u[3] << 16) | w[3]);
        }
      }
      big = __reduce_max_sync(0xffffffffu, big);
      if (lane == 0) atomicMax(a.words + kSMax16 + st, big);
    } else {
      int *out = KIND == kSquare32 ? a.out[set ^ 1] : a.out[0];
      const int64_t ldo = KIND == kSquare32 ? a.ldo[set ^ 1] : a.ldo[0];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = ri + tm + 16 * i;
        if (r >= a.M) continue;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int col = cj + 4 * tn + 32 * h;
          int *o = out + (int64_t)r * ldo + col;
          if (col + 3 < a.N) {
            *reinterpret_cast<int4 *>(o) = make_int4(v[i][4 * h], v[i][4 * h + 1], v[i][4 * h + 2], v[i][4 * h + 3]);
          } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (col + q < a.N) o[q] = v[i][4 * h + q];
          }
        }
      }
    }
    if (KIND == kSquare32 || KIND == kSquare16) {
      if (__any_sync(0xffffffffu, diff) && lane == 0) atomicOr(changed + st, 1);
      if (!mbar_wait(&rel_empty[m & 1], ((m >> 1) & 1) ^ 1, a.status)) break;
      if (warp == 0 && lane == 0) rel[m & 1] = 1;
      __syncwarp();
      if (lane == 0) mbar_arrive(&rel_full[m & 1]);
    }
    ++m;
  }
  if (KIND == kSquare32 || KIND == kSquare16) {
    mbar_wait(&rel_empty[m & 1], ((m >> 1) & 1) ^ 1, a.status);
    if (warp == 0 && lane == 0) rel[m & 1] = -1;
    __syncwarp();
    if (lane == 0) mbar_arrive(&rel_full[m & 1]);
  }
}

template <int KIND, bool P16>
int launch64(const G64Args &a, const G64Maps &maps, cudaStream_t s) {
  auto k = gemm64_kernel<KIND, P16>;
  static std::atomic<int> checked{0};  // 1: register split verified (see launch_one in tgemm.cu)
  if (!checked.load(std::memory_order_relaxed)) {
    cudaFuncAttributes fa;
    APSP_CUDA_TRY(cudaFuncGetAttributes(&fa, k));
    if (fa.numRegs < kLaunchRegs || fa.maxThreadsPerBlock < kFThreads) return APSP_ERR_UNSUPPORTED;
    checked.store(1, std::memory_order_relaxed);
  }
  APSP_CUDA_TRY(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kFSmemBytes));
  const int grid = (int)std::min<int64_t>(cdiv(a.items, a.groups), sm_count());
  launch_pdl(k, grid, kFThreads, kFSmemBytes, s, a, maps);
  APSP_LAUNCH_CHECK();
  return APSP_OK;
}

int maps64(CUtensorMap *mA, CUtensorMap *mB, const void *A, int64_t M, int64_t K, int64_t lda, const void *B,
           int64_t N, int64_t ldb, int dtype) {
  int r;
  if ((r = make_tmap_2d(mA, A, M, K, lda, kFB, 32, dtype, true))) return r;
  return make_tmap_2d(mB, B, K, N, ldb, kFB, kFB, dtype);
}

// a1 for an int32 matrix (zero diagonal, entries >= inf become inf, negative entries are flagged, the
// largest finite entry into words[0]) and both packed forms of it (pairs of columns, pairs of rows,
// values capped), in one pass: each thread takes two rows and two columns.
__global__ void __launch_bounds__(256) square_prep_kernel(int *d, int64_t ld, int n, int *A16, int64_t lda16, int *B16,
                                                          int64_t ldb16, int inf, int *words, unsigned int *st) {
  pdl_wait();
  pdl_trigger();
  if (blockIdx.x == 0 && threadIdx.x == 0) words[kSPacked] = 1;
  const int h = (n + 1) >> 1;
  bool bad = false;
  int m = 0;
  for (int p = blockIdx.x; p < h; p += gridDim.x) {
    for (int w = threadIdx.x; w < h; w += blockDim.x) {
      int x[2][2];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int r = 2 * p + i, c = 2 * w + j;
          int v = inf;
          if (r < n && c < n) {
            const int old = d[(int64_t)r * ld + c];
            bad |= old < 0 && r != c;
            v = r == c ? 0 : (old >= inf ? inf : old);
            if (v != old) d[(int64_t)r * ld + c] = v;
            if (v < inf) m = max(m, v);
          }
          x[i][j] = min(v, kCap16);
        }
      A16[(int64_t)(2 * p) * lda16 + w] = (x[0][1] << 16) | x[0][0];
      if (2 * p + 1 < n) A16[(int64_t)(2 * p + 1) * lda16 + w] = (x[1][1] << 16) | x[1][0];
      B16[(int64_t)p * ldb16 + 2 * w] = (x[1][0] << 16) | x[0][0];
      if (2 * w + 1 < n) B16[(int64_t)p * ldb16 + 2 * w + 1] = (x[1][1] << 16) | x[0][1];
    }
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0 && m > 0) atomicMax(words, m);
  if (__syncthreads_or(bad) && threadIdx.x == 0) flag_status(st, APSP_ERR_DOMAIN);
}

// The last complete set of the 16-bit stages back into the int32 matrix (a set that no stage changed
// equals the one before it).  A word is two columns; rows are 16-byte aligned.  Also sets the words by
// which a loop of one launch per product (squaring.cu) skips what is done: words[kSquareSkip] for its
// first product, words[kSquareUnchanged + t] ("product t changed nothing") for product t + 1.
__global__ void __launch_bounds__(256) square_unpack_kernel(int *d, int64_t ld, int n, const int *A0, const int *A1,
                                                            int64_t lda16, int stages, int inf, int *words) {
  pdl_wait();
  pdl_trigger();
  const bool packed = mode16(words);
  const int done = !packed ? 0 : words[kSAbort] ? words[kSAbort] - 1 : stages;
  if (blockIdx.x == 0 && threadIdx.x < kSMaxStages)
    words[kSquareUnchanged + threadIdx.x] = done == stages || (int)threadIdx.x != done - 1;
  if (blockIdx.x == 0 && threadIdx.x == 0) words[kSquareSkip] = done > 0;
  if (!packed) return;
  const int *A = done & 1 ? A1 : A0;
  for (int i = blockIdx.x; i < n; i += gridDim.x)
    for (int j = 4 * threadIdx.x; j < n; j += 4 * blockDim.x) {
      const int2 u = *reinterpret_cast<const int2 *>(A + (int64_t)i * lda16 + (j >> 1));
      int v[4] = {u.x & 0xFFFF, (int)((unsigned)u.x >> 16), u.y & 0xFFFF, (int)((unsigned)u.y >> 16)};
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = v[q] >= kCap16 ? inf : v[q];
      int *o = d + (int64_t)i * ld + j;
      if (j + 3 < n) {
        *reinterpret_cast<int4 *>(o) = make_int4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (j + q < n) o[q] = v[q];
      }
    }
}

// The 32-bit stages' result back from the scratch matrix when only it holds it.
__global__ void __launch_bounds__(256) square_finish_kernel(int *d, int64_t ld, int n, const int *C, int64_t ldc,
                                                            int stages, const int *words) {
  pdl_wait();
  pdl_trigger();
  const int t = stages32(words, stages);
  if (t <= 0 || !(t & 1) || !words[kSChanged32 + t - 1]) return;
  for (int i = blockIdx.x; i < n; i += gridDim.x)
    for (int j = threadIdx.x; j < n; j += blockDim.x) d[(int64_t)i * ld + j] = C[(int64_t)i * ldc + j];
}

int64_t sq_lda16(int64_t n) { return round_up((n + 1) >> 1, 4); }
int64_t sq_ldb16(int64_t n) { return round_up(n, 4); }

// Two consumer groups per SM overlap one's loads, epilogue and waits with the other's arithmetic, but
// round the work up to pairs of tiles per SM.  Time of `items` tiles in hundredths of half the time
// a pair takes; one tile alone on an SM takes about 1.27 of that (measured, squaring: n = 1300, 441 tiles,
// 388 us with one group and 437 with two; n = 1200, 361 tiles, 362 and 332; n = 1600, 625 tiles,
// 716 and 639).
int64_t one_group(int64_t items) { return 127 * cdiv(items, sm_count()); }
int64_t two_groups(int64_t items) {
  const int64_t sms = sm_count(), left = items % (2 * sms);
  return 200 * (items / (2 * sms)) + (left == 0 ? 0 : 127 + 83 * std::min(left, sms) / sms);
}
int groups_for(int64_t items) { return items <= sm_count() || one_group(items) < two_groups(items) ? 1 : 2; }

}  // namespace

// Rounds of 128 x 128 tiles (four units of work each, one per SM) against rounds of 64 x 64 tiles.  A
// product on its own must win by 15% on paper (percent = 85): at the edge they lose (1000 x 1300 x 700
// int32, 82 us against 77; 2000^3 in 32 bits, 513 against 490), inside it they gain (1024^3 fp32 67 against
// 121 us, 512^3 22 against 62, 300 x 300 x 6000 205 against 670, 4000 x 1300 x 64 26 against 29).
bool gemm64_pays(int64_t M, int64_t N, int64_t K, int percent) {
  if (K <= 0 || M > INT32_MAX / 2 || N > INT32_MAX / 2) return false;
  const int64_t t128 = cdiv(M, kBM) * cdiv(N, kBN), t64 = cdiv(M, kFB) * cdiv(N, kFB);
  if (t64 > INT32_MAX / 2) return false;
  const int64_t c64 = groups_for(t64) == 1 ? one_group(t64) : two_groups(t64);
  return 100 * c64 < percent * 400 * cdiv(t128, sm_count());
}

int launch_gemm64(bool acc, int dtype, const void *A, int64_t lda, const void *B, int64_t ldb, const TileProblem &p,
                  cudaStream_t s) {
  G64Args a = {};
  a.M = (int)p.M; a.N = (int)p.N; a.K = (int)p.K;
  a.tiles_n = (int)cdiv(p.N, kFB);
  a.items = (int)(cdiv(p.M, kFB) * a.tiles_n);
  a.stages = 1;
  a.groups = groups_for(a.items);
  a.acc = acc;
  a.is_float = dtype == APSP_F32;
  a.inf = dtype == APSP_F32 ? 0x7f800000 : p.inf_i;
  a.out[0] = reinterpret_cast<int *>(p.C);
  a.ldo[0] = p.ldc;
  a.wmax = dtype == APSP_F32 ? nullptr : p.wmax;
  a.wmult = p.wmult;
  a.skip = p.skip;
  a.run_if = p.run_if;
  a.status = p.status;
  G64Maps m = {};
  int r;
  if ((r = maps64(&m.A[0], &m.B[0], A, p.M, p.K, lda, B, p.N, ldb, dtype))) return r;
  if ((r = make_tmap_2d(&m.old, p.C, p.M, p.N, p.ldc, kFB, kFB, dtype))) return r;
  void *ev = nullptr;
  const bool tr = trace_on() && !p.no_trace;
  if (tr) trace_begin(s, &ev);
  r = p.arith16 ? launch64<kProduct, true>(a, m, s) : launch64<kProduct, false>(a, m, s);
  if (tr) trace_end(s, ev, kModeGemm + p.trace_class, (double)p.M * (double)p.N * (double)p.K * (p.arith16 ? 2.0 : 1.0));
  return r;
}

int launch_arg_chunks(const float *A, int64_t lda, const float *B, int64_t ldb, int64_t M, int64_t N, int64_t K, int *out,
                      int64_t ldo, cudaStream_t s) {
  G64Args a = {};
  a.M = (int)M; a.N = (int)N; a.K = (int)K;
  a.tiles_n = (int)cdiv(N, kFB);
  a.items = (int)(cdiv(M, kFB) * a.tiles_n);
  a.stages = 1;
  a.groups = groups_for(a.items);
  a.is_float = 1;
  a.inf = 0x7f800000;
  a.out[0] = out;
  a.ldo[0] = ldo;
  a.status = status_word();
  G64Maps m = {};
  int r;
  if ((r = maps64(&m.A[0], &m.B[0], A, M, K, lda, B, N, ldb, APSP_F32))) return r;
  return launch64<kArgChunk, false>(a, m, s);
}

size_t squaring64_bytes(int64_t n, int dtype) {
  if (dtype != APSP_I32) return 0;
  return 2 * ((size_t)round_up(n * sq_lda16(n) * 4, 256) + (size_t)round_up(((n + 1) >> 1) * sq_ldb16(n) * 4, 256));
}

static G64Args square_args(int64_t n, int iters, int *words) {
  G64Args a = {};
  a.M = a.N = a.K = (int)n;
  a.tiles_n = (int)cdiv(n, kFB);
  a.items = a.tiles_n * a.tiles_n;
  a.stages = iters;
  a.groups = groups_for(a.items);
  a.words = words;
  a.status = status_word();
  return a;
}

int squaring64_packed(void *d, int64_t n, int64_t ld, int inf_i, int iters, int *words, void *packed, cudaStream_t s) {
  if (iters > kSMaxStages) return APSP_ERR_ARG;
  int r;
  G64Args q = square_args(n, iters, words);
  G64Maps mq = {};
  q.inf = inf_i;
  q.K = (int)((n + 1) >> 1);
  q.lda16 = sq_lda16(n);
  q.ldb16 = sq_ldb16(n);
  uint8_t *at = reinterpret_cast<uint8_t *>(packed);
  for (int k = 0; k < 2; ++k) {
    q.pa[k] = reinterpret_cast<int *>(at);
    at += round_up(n * q.lda16 * 4, 256);
    q.pb[k] = reinterpret_cast<int *>(at);
    at += round_up((int64_t)q.K * q.ldb16 * 4, 256);
    if ((r = maps64(&mq.A[k], &mq.B[k], q.pa[k], n, q.K, q.lda16, q.pb[k], n, q.ldb16, APSP_I32))) return r;
  }
  const int grid = (int)std::min<int64_t>(n, (int64_t)sm_count() * 4);
  int *D = reinterpret_cast<int *>(d);
  launch_pdl(square_prep_kernel, grid, 256, 0, s, D, ld, (int)n, q.pa[0], q.lda16, q.pb[0], q.ldb16, inf_i, words,
             status_word());
  APSP_LAUNCH_CHECK();
  if ((r = launch64<kSquare16, true>(q, mq, s))) return r;
  launch_pdl(square_unpack_kernel, grid, 256, 0, s, D, ld, (int)n, q.pa[0], q.pa[1], q.lda16, iters, inf_i, words);
  APSP_LAUNCH_CHECK();
  return APSP_OK;
}

int squaring64(void *d, int64_t n, int64_t ld, int dtype, int inf_i, int iters, int *words, int *C, int64_t ldc,
               cudaStream_t s) {
  if (iters > kSMaxStages) return APSP_ERR_ARG;
  const bool isf = dtype == APSP_F32;
  int r;
  G64Args a = square_args(n, iters, words);
  G64Maps m = {};
  a.is_float = isf;
  a.inf = isf ? 0x7f800000 : inf_i;
  a.out[0] = reinterpret_cast<int *>(d);
  a.out[1] = C;
  a.ldo[0] = ld;
  a.ldo[1] = ldc;
  a.wmax = isf ? nullptr : words;  // every entry is a simple path: <= (n - 1) * the largest weight
  a.wmult = n - 1;
  for (int k = 0; k < 2; ++k)
    if ((r = maps64(&m.A[k], &m.B[k], a.out[k], n, n, a.ldo[k], a.out[k], n, a.ldo[k], dtype))) return r;
  if ((r = launch64<kSquare32, false>(a, m, s))) return r;
  const int grid = (int)std::min<int64_t>(n, (int64_t)sm_count() * 4);
  launch_pdl(square_finish_kernel, grid, 256, 0, s, a.out[0], ld, (int)n, C, ldc, iters, words);
  APSP_LAUNCH_CHECK();
  return APSP_OK;
}

}  // namespace apsp
