// Weight and bias gradients of the layers after the first, one launch for all
// of them: gW[l] += d[l]^T . acts[l - 1] and gb[l] += column sums of d[l], d[l]
// the gradients of layer l's outputs before the activation (B x outputs), the
// sums over the batch.
//
// Before, each layer took a split product (train_gemm.cu, which transposes both
// operands in register loads of 4 bytes on the way to shared memory) and a pass
// over d for the column sums: 300 us for the torus object's four layers at 2^18
// rays, 142 us here.
// What bounds it: reading d and the activations, 2 B W FP32 per layer (3.4 TB/s;
// the loads' latency: with two CTAs per SM 189 us).
//
// A CTA (blockIdx.y: the layer) takes tile after tile of 128 rays. Its threads
// read rows (32 bytes at a time: with two 16-byte loads 168 us, not 142), split them into
// two-term BF16 and store whole 8-row core matrices; both operands are then
// read MN-major (outputs and inputs contiguous, rays along K), so nothing is
// transposed. The threads that split d add up its columns on the way. The
// product [outputs x inputs] stays in tensor memory for kFlush tiles (1024
// rays, the ranges the batch was split into before). Several CTAs share an SM
// (W = 64: three), so that one reads while another multiplies.
//
// Products as in train_gemm.cu: tcgen05 kind::f16, hi.hi + hi.lo + lo.hi, FP32
// accumulation. A layer of fewer than 128 outputs fills part of an
// instruction's rows; the others read on in shared memory and are not used.
#include <algorithm>

#include "device.cuh"
#include "tc_common.cuh"

namespace lsnif {

namespace {

constexpr int kGradThreads = 256;
constexpr int kFlush = 8;

struct GradArgs {
  int64_t B;
  int64_t n_tiles;
  int n_layers;
  const int32_t *k;  // rows' segment counts in falling order, or NULL: tiles from the first 0 on have no gradients
  const float *d[LSNIF_MAX_HIDDEN];
  const float *acts[LSNIF_MAX_HIDDEN];
  float *gW[LSNIF_MAX_HIDDEN], *gb[LSNIF_MAX_HIDDEN];
  int outs[LSNIF_MAX_HIDDEN], pad[LSNIF_MAX_HIDDEN];  // outputs; rounded up to 16
  int *err;
};

__device__ __forceinline__ void mma_g(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// 128 rows from `src` (`rows` of them, `cols` wide) as two-term BF16 core
// matrices of kg groups of 8 columns (zeros past rows and cols). An item is one
// row's 8 columns, a quarter-warp stores one core matrix; a thread's items all
// have the same columns, whose sums it adds to `sum`.
template <bool SUM>
__device__ __forceinline__ void split_tile(const float *__restrict__ src, int rows, int cols, int kg, uint8_t *hi,
                                           uint8_t *lo, float (&sum)[8]) {
  const int nt = kGradThreads / (8 * kg) * (8 * kg), tid = threadIdx.x;
  if (tid >= nt) return;
  const int g = (tid >> 3) % kg;
  const bool vec = (cols & 7) == 0;
#pragma unroll 4
  for (int it = tid; it < kTileM * kg; it += nt) {
    const int r = (it & 7) + (it / (8 * kg)) * 8;
    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (r < rows) {
      const float *p = src + (size_t)r * cols + g * 8;
      if (vec) {
        load8(p, v);
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (g * 8 + u < cols) v[u] = __ldg(p + u);
      }
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
    if constexpr (SUM) {
#pragma unroll
      for (int u = 0; u < 8; ++u) sum[u] += v[u];
    }
    const uint32_t o = core_off(r, g, (uint32_t)kg * 128u);
    *reinterpret_cast<uint4 *>(hi + o) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
    *reinterpret_cast<uint4 *>(lo + o) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
  }
}

template <int W>
__global__ void __launch_bounds__(kGradThreads, W == 64 ? 3 : 1) layer_grads_kernel(const __grid_constant__ GradArgs a) {
  extern __shared__ __align__(1024) uint8_t graw[];
  __shared__ uint64_t bar;
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(graw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int l = blockIdx.y, outs = a.outs[l], kgy = a.pad[l] / 8;
  constexpr int KG = W / 8;
  constexpr uint32_t term = (uint32_t)kTileM * W * 2;
  uint8_t *yh = base, *yl = base + term, *xh = base + 2 * term, *xl = base + 3 * term;
  if (tid == 0) {
    mbar_init(su32(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&s_tmem)), "r"(W)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t tmem = s_tmem;
  float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, none[8];
  // the product into the gradients: warps w and w + 4 have outputs (w & 3) 32 +
  // lane, and the even and the odd groups of 16 inputs
  auto flush = [&]() {
    const int out = (warp & 3) * 32 + lane;
    if ((warp & 3) * 32 < outs) {
      const uint32_t at = tmem + ((uint32_t)((warp & 3) * 32) << 16);
      for (int c = (warp >> 2) * 16; c < W; c += 32) {
        uint32_t v[16];
        TMEM_LD16(at + c, v);
        tmem_wait_ld();
        if (out < outs) {
          float *to = a.gW[l] + (size_t)out * W + c;
#pragma unroll
          for (int u = 0; u < 16; u += 4)
            atomicAdd(reinterpret_cast<float4 *>(to + u),
                      make_float4(__uint_as_float(v[u]), __uint_as_float(v[u + 1]), __uint_as_float(v[u + 2]),
                                  __uint_as_float(v[u + 3])));
        }
      }
    }
    tc_before();
  };
  int tiles = 0;
  for (int64_t t = blockIdx.x; t < a.n_tiles; t += gridDim.x) {
    if (a.k && a.k[t * kTileM] == 0) break;
    if (tiles > 0) {  // the products that read the tile before
      if (tid == 0) mbar_wait(su32(&bar), (uint32_t)((tiles - 1) & 1), &s_abort);
      __syncthreads();
      if (s_abort) break;
      tc_after();
      if (tiles % kFlush == 0) flush();
    }
    const int64_t r0 = t * kTileM;
    const int rows = (int)min((int64_t)kTileM, a.B - r0);
    split_tile<false>(a.acts[l] + r0 * W, rows, W, KG, xh, xl, none);
    split_tile<true>(a.d[l] + r0 * outs, rows, outs, kgy, yh, yl, sum);
    fence_async_smem();
    tc_before();
    __syncthreads();
    if (tid == 0) {
      tc_after();
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(W >> 3) << 17) |
                             ((uint32_t)(kTileM >> 4) << 24);
      const uint32_t a_lbo = (uint32_t)kgy * 128u, b_lbo = (uint32_t)KG * 128u;
      for (int ks = 0; ks < kTileM / 16; ++ks) {
        const uint64_t dah = umma_desc(su32(yh) + ks * 2 * a_lbo, a_lbo, 128),
                       dal = umma_desc(su32(yl) + ks * 2 * a_lbo, a_lbo, 128);
        const uint64_t dbh = umma_desc(su32(xh) + ks * 2 * b_lbo, b_lbo, 128),
                       dbl = umma_desc(su32(xl) + ks * 2 * b_lbo, b_lbo, 128);
        mma_g(tmem, dah, dbh, idesc, (ks > 0 || tiles % kFlush != 0) ? 1u : 0u);
        mma_g(tmem, dah, dbl, idesc, 1u);
        mma_g(tmem, dal, dbh, idesc, 1u);
      }
      mma_commit(su32(&bar));
    }
    ++tiles;
  }
  // the last products end before shared and tensor memory are released, also after an abort
  if (tid == 0 && tiles > 0 && !mbar_wait_teardown(su32(&bar), (uint32_t)((tiles - 1) & 1))) s_abort = 1;
  __syncthreads();
  tc_after();
  if (!s_abort && tiles > 0) {
    flush();
    // column sums: the threads of a column group, row by row of a sweep
    float *part = reinterpret_cast<float *>(base);
    const int nt = kGradThreads / (8 * kgy) * (8 * kgy), cols = kgy * 8, per = nt / kgy;
    if (tid < nt) {
      const int g = (tid >> 3) % kgy, rr = (tid & 7) + (tid / (8 * kgy)) * 8;
#pragma unroll
      for (int u = 0; u < 8; ++u) part[rr * cols + g * 8 + u] = sum[u];
    }
    __syncthreads();
    if (tid < outs) {
      float s = 0.f;
      for (int j = 0; j < per; ++j) s += part[j * cols + tid];
      atomicAdd(a.gb[l] + tid, s);
    }
  }
  tc_before();
  __syncthreads();
  tc_after();
  if (tid == 0 && s_abort) atomicOr(a.err, kErrWaitTimeout);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(W) : "memory");
}

template <int W>
cudaError_t launch_shape(const GradArgs &a, cudaStream_t st) {
  constexpr int kSmem = 4 * kTileM * W * 2 + 1024;
  const cudaError_t e = cudaFuncSetAttribute(layer_grads_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) return e;
  int sms = 152, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int per_layer = std::max(1, sms * (W == 64 ? 3 : 1) / a.n_layers);
  const dim3 grid((unsigned)std::min<int64_t>(a.n_tiles, per_layer), (unsigned)a.n_layers);
  layer_grads_kernel<W><<<grid, kGradThreads, kSmem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_layer_grads(const DevObject &h, int64_t B, const int32_t *k, const float *acts, const float *grads,
                               const float *dZ, float *const *gW, float *const *gb, int *err, cudaStream_t st) {
  GradArgs a{};
  a.B = B;
  a.n_tiles = (B + kTileM - 1) / kTileM;
  a.n_layers = h.n_hidden;
  a.k = k;
  for (int j = 0; j < h.n_hidden; ++j) {  // layer j + 1
    const bool last = j + 1 == h.n_hidden;
    a.d[j] = last ? dZ : grads + (size_t)(j + 1) * B * h.width;
    a.acts[j] = acts + (size_t)j * B * h.width;
    a.outs[j] = last ? h.n_out : h.width;
    a.pad[j] = last ? h.n_out_pad : h.width;
    a.gW[j] = gW[j + 1];
    a.gb[j] = gb[j + 1];
  }
  a.err = err;
  return h.width == 64 ? launch_shape<64>(a, st) : launch_shape<128>(a, st);
}

}  // namespace lsnif
