// The first layer of a training step: its input (the features of the batch),
// its product, and its weight and bias gradients. The input is the largest
// array of a step (B x n_in, 604 MB at 2^18 rays of the torus object), so
//   - rays are put in order of their segment count first (order_rays_kernel,
//     from the traversal's own histogram), and a tile of 128 rays has the
//     segments of its first ray: what a ray without a segment s would hold is
//     neither written, read nor multiplied;
//   - the features are written once as the two-term BF16 operands that the
//     products multiply (hi = BF16(x), lo = BF16(x - hi): the same bytes as
//     FP32), one 8-row core matrix per four levels and warp, segment by segment
//     -- both products then take a segment as one bulk copy, read K-major
//     (rays x features) forward and MN-major (features x rays) for the weight
//     gradients, with no conversion or transposition on the way.
// Before, features were FP32 rows of all n_in columns, which each product loaded
// through registers, split and stored to shared memory (transposing for the
// weight gradients). 2^18 rays of the torus object (5.4 of 9 segments in a tile
// on average): product 363 -> 69 us, weight and bias gradients 492 -> 129 us,
// the scatter of the input gradient 952 -> 805 us, the features themselves as
// before (650 us: their corner loads keep L1 at 74% of its wavefronts, with
// rays in order of place too: 590), for 6 us of ordering.
//
// Products as in train_gemm.cu: tcgen05 kind::f16, hi.hi + hi.lo + lo.hi, FP32
// accumulation.
#include <algorithm>

#include "device.cuh"
#include "encode.cuh"
#include "tc_common.cuh"

namespace lsnif {

namespace {

constexpr int kMaxStages = 6;
constexpr int kFlush = 8;  // tiles summed in tensor memory before they are added to the gradients

struct Layer0Args {
  const DevObject *obj;
  int64_t B;
  int64_t n_tiles;
  int n_in, n_seg, chk;  // features of a ray, its segments, features of a segment
  int stages;
  const int32_t *k;      // by row
  const uint8_t *x;      // tiles: per segment hi, lo (128 x chk BF16 each, K-major core matrices)
  const uint8_t *w0t;    // per segment hi, lo (chk x W BF16 each, outputs contiguous)
  const float *bias;
  float *acts;           // B x W
  const float *dY;       // B x W
  float *gW, *gb;
  int act;
  int *err;
};

__device__ __forceinline__ void mma_l0(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// rays by falling segment count: row -> ray (order) and the row's count (k).
// hist: the traversal's counts of rays with 1, 2, ... segments. The order of
// rays of one count is that of the blocks' arrival.
__global__ void __launch_bounds__(1024) order_rays_kernel(const uint8_t *k8, int64_t B, const int32_t *hist,
                                                          int32_t *cursor, int32_t *k, int32_t *order, float *live) {
  __shared__ int cnt[kBuckets], base[kBuckets];
  const int tid = threadIdx.x;
  if (tid < kBuckets) cnt[tid] = 0;
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + tid;
  const bool in = i < B;
  const int kk = in ? k8[i] : 0;
  const unsigned active = __ballot_sync(0xffffffffu, in);
  int rank = 0;
  if (in) {
    const unsigned peers = __match_any_sync(active, kk);
    const int lane = tid & 31, leader = __ffs(peers) - 1;
    int b = 0;
    if (lane == leader) b = atomicAdd(&cnt[kk], __popc(peers));
    rank = __shfl_sync(peers, b, leader) + __popc(peers & ((1u << lane) - 1u));
  }
  __syncthreads();
  if (tid < kBuckets) {
    int before = 0, j = kBuckets - 1;
    for (; j > tid; --j) before += hist[j];
    base[tid] = before + (cnt[tid] ? atomicAdd(cursor + tid, cnt[tid]) : 0);
    if (tid == 0 && blockIdx.x == 0) *live = (float)before;
  }
  __syncthreads();
  if (in) {
    const int at = base[kk] + rank;
    order[at] = (int32_t)i;
    k[at] = kk;
  }
}

// Features of (tile blockIdx.x, segment blockIdx.y). A warp's item is 8 rows x
// 4 levels of one point each: its stores fill whole 128-byte core matrices. All
// warps of a block take the same four levels at a time (L1).
// What bounds it: the L1 wavefronts of the divergent corner loads (74% of the
// peak); levels before rows in the order of items measured the same.
template <int F>
__global__ void __launch_bounds__(256) tile_features_kernel(const DevObject *dobj, int64_t B, const int32_t *k,
                                                            const int32_t *order, const float *pts, uint8_t *X) {
  const DevObject &ob = *dobj;
  const int s = blockIdx.y;
  const int64_t r0 = (int64_t)blockIdx.x * kTileM;
  if (s >= k[r0]) return;
  const int L = ob.L, H = ob.H, LF = L * F, chk = 2 * LF;
  const uint32_t term = (uint32_t)kTileM * chk * 2, sbo = (uint32_t)(chk / 8) * 128u;
  uint8_t *tile = X + ((size_t)blockIdx.x * (H / 2) + s) * 2 * term;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane & 3;
  // items: (four levels, exit or entry, 8 rows), rows fastest
  for (int it = warp; it < (L / 4) * 32; it += 8) {
    const int row = (it & 15) * 8 + (lane >> 2), h = (it >> 4) & 1, l = (it >> 5) * 4 + sub;
    const int64_t r = r0 + row;
    const int kk = r < B ? k[r] : 0;
    // byte offset of this level's features in a term
    const int col = h * LF + l * F;
    const uint32_t o = core_off(row, col >> 3, sbo) + (uint32_t)(col & 7) * 2u;
    uint32_t hw[F / 2], lw[F / 2];
#pragma unroll
    for (int j = 0; j < F / 2; ++j) hw[j] = lw[j] = 0u;
    bool both = false;
    if (s < kk) {
      const float *pp = pts + ((size_t)order[r] * H + 2 * s + h) * 3;
      const float3 p = make_float3(pp[0], pp[1], pp[2]);
      // an entry point equal to the exit point before it has that point's
      // features, which its thread writes to both places
      if (h == 0 && s > 0 && pp[-3] == p.x && pp[-2] == p.y && pp[-1] == p.z) continue;
      both = h == 1 && s + 1 < kk && pp[3] == p.x && pp[4] == p.y && pp[5] == p.z;
      float f[F];
      encode_level_f32_if<F>(ob.tab32 + (size_t)l * (ob.mask + 1) * F, ob.mask, p, (float)ob.res[l], true, f);
#pragma unroll
      for (int j = 0; j < F / 2; ++j) {
        const __nv_bfloat162 hh = __floats2bfloat162_rn(f[2 * j], f[2 * j + 1]);
        const float2 hf = __bfloat1622float2(hh);
        const __nv_bfloat162 ll = __floats2bfloat162_rn(f[2 * j] - hf.x, f[2 * j + 1] - hf.y);
        hw[j] = *reinterpret_cast<const uint32_t *>(&hh);
        lw[j] = *reinterpret_cast<const uint32_t *>(&ll);
      }
    }
    auto put = [&](uint8_t *at) {
      if constexpr (F == 2) {
        *reinterpret_cast<uint32_t *>(at) = hw[0];
        *reinterpret_cast<uint32_t *>(at + term) = lw[0];
      } else {
        *reinterpret_cast<uint2 *>(at) = make_uint2(hw[0], hw[1]);
        *reinterpret_cast<uint2 *>(at + term) = make_uint2(lw[0], lw[1]);
      }
    };
    put(tile + o);
    // the next segment's entry point: the same row, LF columns earlier
    if (both) put(tile + 2 * term + core_off(row, (col - LF) >> 3, sbo) + (uint32_t)(col & 7) * 2u);
  }
}

// The roles of both product kernels meet on barriers: full[] (a stage's copy
// has landed), empty[] (the products that read a stage are done).
struct Ring {
  uint64_t *full, *empty;
  int n;
};

// A wait of a whole warp: its lanes go on, or give up after an abort, together
// (what follows are warp-wide loads of tensor memory).
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag) {
  return __all_sync(0xffffffffu, mbar_wait(su32(bar), parity, abort_flag)) != 0;
}

// Loader: `copy(j, t, s, slot)` for the j-th segment of this CTA. Every copy has
// landed when it returns, also after an abort.
template <typename Copy>
__device__ __forceinline__ void run_loader(const Layer0Args &a, const Ring &ring, int first, int step,
                                           volatile int *abort_flag, Copy copy) {
  int n = 0;
  for (int64_t t = blockIdx.x; t < a.n_tiles && !*abort_flag; t += gridDim.x) {
    const int kmax = a.k[t * kTileM];
    for (int s = first; s < kmax; s += step, ++n) {
      const int slot = n % ring.n, use = n / ring.n;
      if (use > 0 && !mbar_wait(su32(&ring.empty[slot]), (uint32_t)((use - 1) & 1), abort_flag)) break;
      copy(t, s, slot);
    }
    if (kmax == 0) break;  // the rest has no segments
  }
  for (int j = max(0, n - ring.n); j < n; ++j)
    if (!mbar_wait_teardown(su32(&ring.full[j % ring.n]), (uint32_t)((j / ring.n) & 1))) *abort_flag = 1;
}

// acts = act(X . W0^T + bias), row after row. A tile's segments stream through
// the ring (features and their slice of W0, which L2 holds) while the tile
// before is written from the other accumulator. What bounds it: reading X.
constexpr int kFwdThreads = 192;  // four warps of rows, the loader, the products

template <int W>
__global__ void __launch_bounds__(kFwdThreads) layer0_kernel(const __grid_constant__ Layer0Args a) {
  extern __shared__ __align__(1024) uint8_t fraw[];
  __shared__ uint64_t full[kMaxStages], empty[kMaxStages], acc_full[2], acc_empty[2], done;
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  __shared__ float s_bias[W];
  uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(fraw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t x_bytes = 4u * kTileM * a.chk, w_bytes = 4u * W * a.chk, stage = x_bytes + w_bytes;
  if (tid == 0) {
    for (int j = 0; j < a.stages; ++j) {
      mbar_init(su32(&full[j]), 1);
      mbar_init(su32(&empty[j]), 1);
    }
    for (int j = 0; j < 2; ++j) {
      mbar_init(su32(&acc_full[j]), 1);
      mbar_init(su32(&acc_empty[j]), kTileM);
    }
    mbar_init(su32(&done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
  }
  if (tid < W) s_bias[tid] = a.bias[tid];
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&s_tmem)), "r"(2 * W)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t tmem = s_tmem;
  const Ring ring{full, empty, a.stages};
  if (warp == 4) {
    if (lane == 0)
      run_loader(a, ring, 0, 1, &s_abort, [&](int64_t t, int s, int slot) {
        const uint32_t bar = su32(&full[slot]), at = su32(base) + (uint32_t)slot * stage;
        mbar_expect(bar, stage);
        bulk_load(at, a.x + ((size_t)t * a.n_seg + s) * x_bytes, x_bytes, bar);
        bulk_load(at + x_bytes, a.w0t + (size_t)s * w_bytes, w_bytes, bar);
      });
  } else if (warp == 5) {
    if (lane == 0) {
      // A: rows x features, K-major; B: features x outputs, outputs contiguous (MN-major)
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(W >> 3) << 17) |
                             ((uint32_t)(kTileM >> 4) << 24);
      const uint32_t a_sbo = (uint32_t)(a.chk / 8) * 128u, b_lbo = (uint32_t)(W / 8) * 128u;
      int n = 0, tiles = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < a.n_tiles && ok; t += gridDim.x, ++tiles) {
        const int kmax = a.k[t * kTileM];
        if (kmax == 0) break;
        const int buf = tiles & 1, use = tiles >> 1;
        if (use > 0 && !mbar_wait(su32(&acc_empty[buf]), (uint32_t)((use - 1) & 1), &s_abort)) break;
        const uint32_t d = tmem + (uint32_t)(buf * W);
        for (int s = 0; s < kmax; ++s, ++n) {
          const int slot = n % a.stages;
          ok = mbar_wait(su32(&full[slot]), (uint32_t)((n / a.stages) & 1), &s_abort);
          if (!ok) break;
          tc_after();
          const uint32_t ah = su32(base) + (uint32_t)slot * stage, al = ah + x_bytes / 2, bh = ah + x_bytes,
                         bl = bh + w_bytes / 2;
          for (int ks = 0; ks < a.chk / 16; ++ks) {
            const uint64_t dah = umma_desc(ah + ks * 256, 128, a_sbo), dal = umma_desc(al + ks * 256, 128, a_sbo);
            const uint64_t dbh = umma_desc(bh + ks * 2 * b_lbo, b_lbo, 128),
                           dbl = umma_desc(bl + ks * 2 * b_lbo, b_lbo, 128);
            mma_l0(d, dah, dbh, idesc, (s > 0 || ks > 0) ? 1u : 0u);
            mma_l0(d, dah, dbl, idesc, 1u);
            mma_l0(d, dal, dbh, idesc, 1u);
          }
          mma_commit(su32(&empty[slot]));
        }
        if (ok) mma_commit(su32(&acc_full[buf]));
      }
      mma_commit(su32(&done));
      if (!mbar_wait_teardown(su32(&done), 0u)) s_abort = 1;
    }
  } else {
    const int row = warp * 32 + lane;
    int tiles = 0;
    for (int64_t t = blockIdx.x; t < a.n_tiles; t += gridDim.x) {
      const int buf = tiles & 1, use = tiles >> 1;
      const bool any = a.k[t * kTileM] > 0;
      if (any) {
        if (!warp_wait(&acc_full[buf], (uint32_t)(use & 1), &s_abort)) break;
        ++tiles;
        tc_after();
      }
      const int64_t i = t * kTileM + row;
      float *out = a.acts + i * W;
      const uint32_t at = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(buf * W);
#pragma unroll 1
      for (int c = 0; c < W; c += 16) {
        uint32_t v[16];
        if (any) {
          TMEM_LD16(at + c, v);
          tmem_wait_ld();
        } else {
#pragma unroll
          for (int u = 0; u < 16; ++u) v[u] = 0u;
        }
        if (c + 16 == W && any) {
          tc_before();
          mbar_arrive(su32(&acc_empty[buf]));
        }
        if (i < a.B) {
          float x[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) x[u] = act_fn(__uint_as_float(v[u]) + s_bias[c + u], a.act);
#pragma unroll
          for (int u = 0; u < 16; u += 8) store8(out + c + u, x + u);
        }
      }
    }
  }
  tc_before();
  __syncthreads();
  tc_after();
  if (tid == 0 && s_abort) atomicOr(a.err, kErrWaitTimeout);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * W) : "memory");
}

// gW += dY^T . X and gb += column sums of dY. Eight warps split a tile's dY
// (rows x outputs, FP32) into two terms and sum its columns; a segment's
// product [outputs x features] has its own columns of tensor memory, which are
// added to the gradients every kFlush tiles (1024 rays: the ranges the batch
// was split into before). Tensor memory holds 512 columns: blockIdx.y takes
// every gridDim.y-th segment. W = 64 fills half of the 128 rows of an
// instruction; the other half reads on in shared memory and is not used.
// What bounds it: reading X (3 TB/s). With one of the three products 110 us
// instead of 129, with a flush every 128 tiles 116: sums stay short instead.
constexpr int kGradThreads = 320;  // eight warps of dY, the loader, the products

template <int W>
__global__ void __launch_bounds__(kGradThreads) layer0_grad_kernel(const __grid_constant__ Layer0Args a) {
  extern __shared__ __align__(1024) uint8_t graw[];
  __shared__ uint64_t full[kMaxStages], empty[kMaxStages], y_full[2], y_empty[2], acc_full, acc_empty, done;
  __shared__ uint32_t s_tmem, s_cols;
  __shared__ volatile int s_abort;
  __shared__ float s_sum[256 * 8 / W][W];  // [rows of a sweep][column]
  uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(graw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int KG = W / 8;
  constexpr uint32_t y_term = (uint32_t)kTileM * W * 2;
  const uint32_t x_bytes = 4u * kTileM * a.chk;
  const int first = blockIdx.y, step = gridDim.y;
  const int segs = (a.n_seg - first + step - 1) / step;
  uint8_t *sY = base + (size_t)a.stages * x_bytes;  // two buffers of (hi, lo), 1 KB more readable
  if (tid == 0) {
    for (int j = 0; j < a.stages; ++j) {
      mbar_init(su32(&full[j]), 1);
      mbar_init(su32(&empty[j]), 1);
    }
    for (int j = 0; j < 2; ++j) {
      mbar_init(su32(&y_full[j]), 256);
      mbar_init(su32(&y_empty[j]), 1);
    }
    mbar_init(su32(&acc_full), 1);
    mbar_init(su32(&acc_empty), 256);
    mbar_init(su32(&done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
    uint32_t cols = 32;
    while (cols < (uint32_t)(segs * a.chk)) cols *= 2;
    s_cols = cols;
  }
  __syncthreads();
  const uint32_t cols = s_cols;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&s_tmem)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t tmem = s_tmem;
  const Ring ring{full, empty, a.stages};
  if (warp == 8) {
    if (lane == 0)
      run_loader(a, ring, first, step, &s_abort, [&](int64_t t, int s, int slot) {
        const uint32_t bar = su32(&full[slot]);
        mbar_expect(bar, x_bytes);
        bulk_load(su32(base) + (uint32_t)slot * x_bytes, a.x + ((size_t)t * a.n_seg + s) * x_bytes, x_bytes, bar);
      });
  } else if (warp == 9) {
    if (lane == 0) {
      // both operands MN-major: outputs (A) and features (B) contiguous, rays along K
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                             ((uint32_t)(a.chk >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
      const uint32_t a_lbo = (uint32_t)KG * 128u, b_lbo = (uint32_t)(a.chk / 8) * 128u;
      int n = 0, tiles = 0;
      uint32_t begun = 0;  // segments whose columns hold a sum
      bool ok = true;
      for (int64_t t = blockIdx.x; t < a.n_tiles && ok; t += gridDim.x, ++tiles) {
        const int kmax = a.k[t * kTileM];
        if (kmax <= first) break;
        const int buf = tiles & 1;
        if (tiles > 0 && tiles % kFlush == 0) {
          if (!mbar_wait(su32(&acc_empty), (uint32_t)((tiles / kFlush - 1) & 1), &s_abort)) break;
          begun = 0;
        }
        if (!mbar_wait(su32(&y_full[buf]), (uint32_t)((tiles >> 1) & 1), &s_abort)) break;
        const uint32_t yh = su32(sY) + (uint32_t)buf * 2 * y_term, yl = yh + y_term;
        for (int s = first, j = 0; s < kmax; s += step, ++j, ++n) {
          const int slot = n % a.stages;
          ok = mbar_wait(su32(&full[slot]), (uint32_t)((n / a.stages) & 1), &s_abort);
          if (!ok) break;
          tc_after();
          const uint32_t xh = su32(base) + (uint32_t)slot * x_bytes, xl = xh + x_bytes / 2;
          const uint32_t d = tmem + (uint32_t)(j * a.chk);
          for (int ks = 0; ks < kTileM / 16; ++ks) {
            const uint64_t dah = umma_desc(yh + ks * 2 * a_lbo, a_lbo, 128), dal = umma_desc(yl + ks * 2 * a_lbo, a_lbo, 128);
            const uint64_t dbh = umma_desc(xh + ks * 2 * b_lbo, b_lbo, 128), dbl = umma_desc(xl + ks * 2 * b_lbo, b_lbo, 128);
            mma_l0(d, dah, dbh, idesc, ks > 0 ? 1u : (begun >> j) & 1u);
            mma_l0(d, dah, dbl, idesc, 1u);
            mma_l0(d, dal, dbh, idesc, 1u);
          }
          begun |= 1u << j;
          mma_commit(su32(&empty[slot]));
        }
        if (!ok) break;
        mma_commit(su32(&y_empty[buf]));
        if (tiles % kFlush == kFlush - 1) mma_commit(su32(&acc_full));
      }
      mma_commit(su32(&done));
      if (!mbar_wait_teardown(su32(&done), 0u)) s_abort = 1;
    }
  } else {
    // item: one row's 8 outputs; a quarter-warp stores one core matrix. The 256
    // items of a sweep are whole groups of 8 rows, so a thread keeps its columns.
    float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const int g = (tid >> 3) % KG;
    int tiles = 0, seen = 0;  // tiles taken; segments in the columns since the last flush
    // the sums of the last tiles into the gradients: warp w has outputs
    // (w & 3) 32 + lane, warps 0-3 the even groups of 16 columns, 4-7 the odd ones
    auto flush = [&]() {
      const int out = (warp & 3) * 32 + lane;
      if (out < W) {
        const uint32_t at = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        for (int c = (warp >> 2) * 16; c < seen * a.chk; c += 32) {
          uint32_t v[16];
          TMEM_LD16(at + c, v);
          tmem_wait_ld();
          const int j = c / a.chk;
          float *to = a.gW + (size_t)out * a.n_in + (size_t)(first + j * step) * a.chk + (c - j * a.chk);
#pragma unroll
          for (int u = 0; u < 16; u += 4)
            atomicAdd(reinterpret_cast<float4 *>(to + u),
                      make_float4(__uint_as_float(v[u]), __uint_as_float(v[u + 1]), __uint_as_float(v[u + 2]),
                                  __uint_as_float(v[u + 3])));
        }
      }
      tc_before();
      seen = 0;
    };
    bool ok = true;
    for (int64_t t = blockIdx.x; t < a.n_tiles; t += gridDim.x) {
      const int kmax = a.k[t * kTileM];
      if (kmax <= first) break;
      const int buf = tiles & 1, use = tiles >> 1;
      if (use > 0 && !warp_wait(&y_empty[buf], (uint32_t)((use - 1) & 1), &s_abort)) { ok = false; break; }
      seen = max(seen, (kmax - first + step - 1) / step);
      uint8_t *yb = sY + (size_t)buf * 2 * y_term;
#pragma unroll 2
      for (int it = tid; it < kTileM * KG; it += 256) {
        const int r = (it & 7) + (it / (8 * KG)) * 8;
        const int64_t i = t * kTileM + r;
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (i < a.B) {
          load8(a.dY + i * W + g * 8, v);
        }
        uint32_t hw[4], lw[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * u], v[2 * u + 1]);
          const float2 hf = __bfloat1622float2(h);
          const __nv_bfloat162 l = __floats2bfloat162_rn(v[2 * u] - hf.x, v[2 * u + 1] - hf.y);
          hw[u] = *reinterpret_cast<const uint32_t *>(&h);
          lw[u] = *reinterpret_cast<const uint32_t *>(&l);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) sum[u] += v[u];
        const uint32_t o = core_off(r, g, (uint32_t)KG * 128u);
        *reinterpret_cast<uint4 *>(yb + o) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
        *reinterpret_cast<uint4 *>(yb + y_term + o) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
      }
      fence_async_smem();
      mbar_arrive(su32(&y_full[buf]));
      if (tiles % kFlush == kFlush - 1) {
        if (!warp_wait(&acc_full, (uint32_t)((tiles / kFlush) & 1), &s_abort)) { ok = false; break; }
        tc_after();
        flush();
        mbar_arrive(su32(&acc_empty));
      }
      ++tiles;
    }
    if (ok && seen > 0) {
      if (warp_wait(&done, 0u, &s_abort)) {
        tc_after();
        flush();
      }
    }
    if (first == 0) {
      // column sums: rows of a sweep are 8 x (256 / (8 KG)) threads per column group
      const int rr = (tid & 7) + (tid / (8 * KG)) * 8;
#pragma unroll
      for (int u = 0; u < 8; ++u) s_sum[rr][g * 8 + u] = sum[u];
      named_sync(1, 256);
      if (tid < W) {
        float t = 0.f;
        for (int j = 0; j < 256 * 8 / W; ++j) t += s_sum[j][tid];
        if (tiles > 0) atomicAdd(a.gb + tid, t);
      }
    }
  }
  tc_before();
  __syncthreads();
  tc_after();
  if (tid == 0 && s_abort) atomicOr(a.err, kErrWaitTimeout);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}

int sm_count() {
  int sms = 152, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

constexpr int kSmemMax = 222 << 10;  // dynamic: the static part and the system's 1 KB come on top
constexpr int kSumBytes = 8192;     // the column sums (static, layer0_grad_kernel)

Layer0Args layer0_args(const DevObject *dobj, const DevObject &h, int64_t B, const int32_t *k, const void *x) {
  Layer0Args a{};
  a.obj = dobj;
  a.B = B;
  a.n_tiles = (B + kTileM - 1) / kTileM;
  a.n_in = h.n_in;
  a.n_seg = h.H / 2;
  a.chk = 2 * h.L * h.F;
  a.k = k;
  a.x = static_cast<const uint8_t *>(x);
  a.act = h.act;
  return a;
}

}  // namespace

cudaError_t launch_order_rays(const uint8_t *k8, int64_t B, const int32_t *hist, int32_t *cursor, int32_t *k,
                              int32_t *order, float *live, cudaStream_t st) {
  const cudaError_t e = cudaMemsetAsync(cursor, 0, kBuckets * sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  order_rays_kernel<<<(unsigned)((B + 1023) / 1024), 1024, 0, st>>>(k8, B, hist, cursor, k, order, live);
  return cudaGetLastError();
}

cudaError_t launch_tile_features(const DevObject *dobj, const DevObject &h, int64_t B, const int32_t *k,
                                 const int32_t *order, const float *pts, void *x, cudaStream_t st) {
  const dim3 grid((unsigned)((B + kTileM - 1) / kTileM), (unsigned)(h.H / 2));
  if (h.F == 2) tile_features_kernel<2><<<grid, 256, 0, st>>>(dobj, B, k, order, pts, static_cast<uint8_t *>(x));
  else tile_features_kernel<4><<<grid, 256, 0, st>>>(dobj, B, k, order, pts, static_cast<uint8_t *>(x));
  return cudaGetLastError();
}

cudaError_t launch_layer0(const DevObject *dobj, const DevObject &h, int64_t B, const int32_t *k, const void *x,
                          const void *w0t, const float *bias, float *acts, int *err, cudaStream_t st) {
  Layer0Args a = layer0_args(dobj, h, B, k, x);
  a.w0t = static_cast<const uint8_t *>(w0t);
  a.bias = bias;
  a.acts = acts;
  a.err = err;
  const size_t stage = 4 * (size_t)a.chk * (kTileM + h.width);
  a.stages = (int)std::max<size_t>(1, std::min<size_t>(kMaxStages, (kSmemMax - 1024) / stage));
  const size_t smem = a.stages * stage + 1024;
  const unsigned grid = (unsigned)std::min<int64_t>(a.n_tiles, sm_count());
  auto *kern = h.width == 64 ? layer0_kernel<64> : layer0_kernel<128>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
  if (e != cudaSuccess) return e;
  kern<<<grid, kFwdThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_layer0_grad(const DevObject *dobj, const DevObject &h, int64_t B, const int32_t *k, const void *x,
                               const float *dY, float *gW, float *gb, int *err, cudaStream_t st) {
  Layer0Args a = layer0_args(dobj, h, B, k, x);
  a.dY = dY;
  a.gW = gW;
  a.gb = gb;
  a.err = err;
  // the shares the segments are dealt to: the largest has to fit 512 columns
  int y = 1;
  while ((a.n_seg + y - 1) / y * a.chk > 512) ++y;
  const size_t stage = 4 * (size_t)a.chk * kTileM, yb = 8 * (size_t)kTileM * h.width + 1024;
  const size_t room = kSmemMax - kSumBytes - 1024 - yb;
  a.stages = (int)std::max<size_t>(1, std::min<size_t>(kMaxStages, room / stage));
  const size_t smem = a.stages * stage + yb + 1024;
  const dim3 grid((unsigned)std::min<int64_t>(a.n_tiles, std::max(1, sm_count() / y)), (unsigned)y);
  auto *kern = h.width == 64 ? layer0_grad_kernel<64> : layer0_grad_kernel<128>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax - kSumBytes);
  if (e != cudaSuccess) return e;
  kern<<<grid, kGradThreads, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace lsnif
