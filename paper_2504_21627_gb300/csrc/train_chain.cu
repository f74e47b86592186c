// The part of a training step between the first layer's activations and the
// gradient of its pre-activations in one kernel: hidden layers, logits, loss
// (Sec. 5.3), and the backward pass through the layers down to the first. The
// weight gradients, whose reduction runs over the batch, stay with the
// products of train_gemm.cu.
//
// Before, each of these layers was a launch of its own in either direction: it
// read its input and wrote its output (and, forward, both the pre-activation
// and the activation) as B x W FP32 rows, and each CTA set up, converted the
// weights and multiplied one tile. Here a CTA keeps every later layer's
// two-term weights in shared memory and takes tile after tile of 128 rays; a
// layer's output goes from one TMEM accumulator through the registers of its
// row's thread into the next layer's A operand in tensor memory, and the
// derivative of an activation is kept as one bit. What remains is the reading
// of the first activations and the writing of the activations and gradients
// that the weight gradients need: 161 us for 2^18 rays of the torus object's 4
// hidden layers of 64 (the step 4.34 -> 3.72 ms), about 3.3 TB/s. A fourth CTA per
// SM (masks in local memory) changed nothing: 164 us.
//
// Products as in train_gemm.cu: tcgen05 kind::f16, two-term BF16 operands
// (hi.hi + hi.lo + lo.hi), FP32 accumulation. The weights are the query's
// copies: umma (hi) and umma_lo (lo), out x in core matrices. Forward reads
// them as K-major B operands; backward (dY . W) reads the same bytes as
// MN-major ones, so no transposed copy is needed.
#include <algorithm>

#include "device.cuh"
#include "tc_common.cuh"

namespace lsnif {

namespace {

constexpr int kChainSmemMax = 200 << 10;  // dynamic shared memory of the largest network taken
constexpr int kCThreads = 128;  // a thread per row; warp w has TMEM lane quarter w

struct ChainArgs {
  const DevObject *obj;
  int64_t B;
  int64_t n_tiles;
  const int32_t *k;
  const int32_t *order;  // ray of a row (NULL: the row itself)
  float *acts;           // n_hidden x B x W: layer 0 given, the others written
  float *grads;          // n_hidden x B x W: gradients of the pre-activations
  float *dZ;             // B x n_out
  lsnif_labels lab;
  float *loss;           // [0..5] sums, [6] live rays
  uint32_t w_bytes;      // one term of the later layers' weights
  uint32_t bias_bytes;
  int *err;
};

template <int W>
constexpr int chain_tmem() { return 2 * W; }  // accumulator, activations hi and lo

__device__ __forceinline__ void mma_ts(uint32_t tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(tmem),
      "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// 16 values -> two-term BF16 in tensor memory, two values per 32-bit column
__device__ __forceinline__ void put_operand(uint32_t hi_at, uint32_t lo_at, const float (&x)[16]) {
  uint32_t hw[8], lw[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(x[2 * u], x[2 * u + 1]);
    const float2 hf = __bfloat1622float2(h);
    const __nv_bfloat162 l = __floats2bfloat162_rn(x[2 * u] - hf.x, x[2 * u + 1] - hf.y);
    hw[u] = *reinterpret_cast<const uint32_t *>(&h);
    lw[u] = *reinterpret_cast<const uint32_t *>(&l);
  }
  TMEM_ST8(hi_at, hw);
  TMEM_ST8(lo_at, lw);
}

__device__ __forceinline__ void wait_ld(uint32_t (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                 "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]));
}

// Loss terms s[1..5] (occ, t, normal, albedo, material) of a ray with logits z
// are added to s; g = dLoss/dz for the batch mean (1 / live rays = inv_live).
template <int NZ>
__device__ __forceinline__ void loss_row(const float *z, int n_mat, const lsnif_labels &lab, int64_t i, float inv_live,
                                         float *s, float *g) {
  const float y = lab.occ[i];
  const float z0 = z[0];
  s[1] += fmaxf(z0, 0.f) - z0 * y + log1pf(expf(-fabsf(z0)));
  g[0] = (sigmoidf_(z0) - y) * inv_live;
  // remaining heads only where the reference is occluded
  const float s1 = sigmoidf_(z[1]);
  const float dt = s1 - lab.t_local[i];
  const float g1 = (dt > 0.f ? 1.f : (dt < 0.f ? -1.f : 0.f)) * s1 * (1.f - s1);
  const float zn[3] = {z[2], z[3], z[4]};
  const float *yn = lab.normal + 3 * i;
  const float nz = fmaxf(sqrtf(zn[0] * zn[0] + zn[1] * zn[1] + zn[2] * zn[2]), 1e-12f);
  const float dot = zn[0] * yn[0] + zn[1] * yn[1] + zn[2] * yn[2];
  float l_a = 0.f, ga[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float sa = sigmoidf_(z[5 + c]);
    const float den = sa * sa + 0.01f;
    const float df = sa - lab.albedo[3 * i + c];
    l_a += df * df / den;
    ga[c] = (2.f / 3.f) * df / den * sa * (1.f - sa);
  }
  constexpr int NM = NZ - 8;
  float mx = z[8];
#pragma unroll
  for (int m = 1; m < NM; ++m)
    if (m < n_mat) mx = fmaxf(mx, z[8 + m]);
  float se = 0.f;
#pragma unroll
  for (int m = 0; m < NM; ++m)
    if (m < n_mat) se += expf(z[8 + m] - mx);
  const int ym = lab.mat[i];
  float zy = z[8];
#pragma unroll
  for (int m = 1; m < NM; ++m)
    if (m == ym) zy = z[8 + m];
  g[1] = y * g1 * inv_live;
#pragma unroll
  for (int a = 0; a < 3; ++a) g[2 + a] = y * -(yn[a] / nz - dot * zn[a] / (nz * nz * nz)) * inv_live;
#pragma unroll
  for (int c = 0; c < 3; ++c) g[5 + c] = y * ga[c] * inv_live;
#pragma unroll
  for (int m = 0; m < NM; ++m)
    if (m < n_mat) g[8 + m] = y * (expf(z[8 + m] - mx) / se - (m == ym ? 1.f : 0.f)) * inv_live;
  s[2] += y * fabsf(dt);
  s[3] += y * (1.f - dot / nz);
  s[4] += y * (l_a * (1.f / 3.f));
  s[5] += y * (mx + logf(se) - zy);
}

// NZ: columns of the output layer held in registers (16 or 64, padded)
template <int W, int NZ>
__global__ void __launch_bounds__(kCThreads) train_chain_kernel(const __grid_constant__ ChainArgs a) {
  extern __shared__ __align__(1024) uint8_t craw[];
  __shared__ uint64_t bars[2];  // [0] weights, [1] products
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  __shared__ float part[6][4];
  uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(craw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const DevObject &ob = *a.obj;
  const int NH = ob.n_hidden, n_out = ob.n_out, n_pad = ob.n_out_pad, act = ob.act, n_mat = ob.n_mat;
  uint8_t *s_hi = base, *s_lo = base + a.w_bytes;
  float *s_bias = reinterpret_cast<float *>(base + 2 * (size_t)a.w_bytes);
  uint32_t *s_mask = reinterpret_cast<uint32_t *>(base + 2 * (size_t)a.w_bytes + a.bias_bytes);  // [layer][W / 32][row]
  if (tid == 0) {
    mbar_init(su32(&bars[0]), 1);
    mbar_init(su32(&bars[1]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&s_tmem)),
                 "r"(chain_tmem<W>())
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_before();
  __syncthreads();
  tc_after();
  if (tid == 0) {
    mbar_expect(su32(&bars[0]), 2 * a.w_bytes + a.bias_bytes);
    bulk_load(su32(s_hi), ob.umma + (size_t)W * ob.n_in * 2, a.w_bytes, su32(&bars[0]));
    bulk_load(su32(s_lo), ob.umma_lo, a.w_bytes, su32(&bars[0]));
    bulk_load(su32(s_bias), ob.umma + ob.umma_bias_off, a.bias_bytes, su32(&bars[0]));
    mbar_wait(su32(&bars[0]), 0u, &s_abort);
  }
  __syncthreads();
  const uint32_t tmem = s_tmem, a_hi = tmem + W, a_lo = a_hi + W / 2;  // A operand: lane 0
  const uint32_t lane_at = (uint32_t)(warp * 32) << 16;
  const uint32_t acc = tmem + lane_at, t_hi = a_hi + lane_at, t_lo = a_lo + lane_at;
  const float inv_live = 1.f / fmaxf(a.loss[6], 1.f);
  const int r = warp * 32 + lane;
  float sums[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  uint32_t phase = 0;
  constexpr uint32_t kSbo = (uint32_t)(W / 8) * 128u;  // 8 rows of a weight tile

  // D[128 x N] = A[128 x K] . op(weights at byte w): N outputs of K inputs (forward:
  // rows of the tile are N), or N inputs of K outputs (backward: rows are K).
  // All threads: their part of A is stored; the product is complete on return.
  auto multiply = [&](uint32_t w, int N, int K, bool backward) {
    tmem_wait_st();
    tc_before();
    __syncthreads();
    if (tid == 0) {
      tc_after();
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (backward ? 1u << 16 : 0u) | ((uint32_t)(N >> 3) << 17) |
                             ((uint32_t)(kTileM >> 4) << 24);
      const uint32_t bh = su32(s_hi) + w, bl = su32(s_lo) + w, step = backward ? 2u * kSbo : 256u;
      const uint32_t lbo = backward ? kSbo : 128u, sbo = backward ? 128u : kSbo;
      for (int ks = 0; ks < K / 16; ++ks) {
        const uint64_t dh = umma_desc(bh + ks * step, lbo, sbo), dl = umma_desc(bl + ks * step, lbo, sbo);
        mma_ts(tmem, a_hi + (uint32_t)(8 * ks), dh, idesc, ks > 0 ? 1u : 0u);
        mma_ts(tmem, a_hi + (uint32_t)(8 * ks), dl, idesc, 1u);
        mma_ts(tmem, a_lo + (uint32_t)(8 * ks), dh, idesc, 1u);
      }
      mma_commit(su32(&bars[1]));
      mbar_wait(su32(&bars[1]), phase, &s_abort);
    }
    phase ^= 1u;
    __syncthreads();
    tc_after();
  };

  for (int64_t t = blockIdx.x; t < a.n_tiles && !s_abort; t += gridDim.x) {
    const int64_t i = t * kTileM + r;
    const bool on = i < a.B;
    const int64_t layer_stride = a.B * W;
    // ---- forward ----
    for (int l = 0; l < NH; ++l) {
      float *arow = a.acts + (size_t)l * layer_stride + i * W;
      const float *bias = s_bias + l * W;
#pragma unroll 1
      for (int c = 0; c < W / 16; ++c) {
        float x[16];
        if (l == 0) {
#pragma unroll
          for (int u = 0; u < 16; ++u) x[u] = 0.f;
          if (on) {
            load8(arow + 16 * c, x);
            load8(arow + 16 * c + 8, x + 8);
          }
        } else {
          uint32_t v[16];
          TMEM_LD16(acc + 16 * c, v);
          wait_ld(v);
#pragma unroll
          for (int u = 0; u < 16; ++u) x[u] = act_fn(__uint_as_float(v[u]) + bias[16 * c + u], act);
          if (on) {
            store8(arow + 16 * c, x);
            store8(arow + 16 * c + 8, x + 8);
          }
        }
        uint32_t m = 0;  // an activation is positive where its input is
#pragma unroll
        for (int u = 0; u < 16; ++u) m |= (x[u] > 0.f ? 1u : 0u) << u;
        uint32_t *mw = s_mask + ((size_t)l * (W / 32) + (c >> 1)) * kTileM + r;
        *mw = (c & 1) ? (*mw | m << 16) : m;
        put_operand(t_hi + 8 * c, t_lo + 8 * c, x);
      }
      const uint32_t w = (uint32_t)l * W * W * 2u;
      multiply(w, l + 1 < NH ? W : n_pad, W, false);
    }
    // ---- logits, loss ----
    {
      float z[NZ], g[NZ];
#pragma unroll
      for (int c = 0; c < NZ / 16; ++c) {
        if (16 * c >= n_pad) break;
        uint32_t v[16];
        TMEM_LD16(acc + 16 * c, v);
        wait_ld(v);
#pragma unroll
        for (int u = 0; u < 16; ++u) z[16 * c + u] = __uint_as_float(v[u]) + s_bias[NH * W + 16 * c + u];
      }
#pragma unroll
      for (int u = 0; u < NZ; ++u) g[u] = 0.f;
      if (on && a.k[i] > 0) loss_row<NZ>(z, n_mat, a.lab, a.order ? a.order[i] : i, inv_live, sums, g);
      if (on) {
        float *d = a.dZ + i * n_out;
#pragma unroll
        for (int u = 0; u < NZ; ++u)
          if (u < n_out) d[u] = g[u];
      }
#pragma unroll
      for (int c = 0; c < NZ / 16; ++c) {
        if (16 * c >= n_pad) break;
        float x[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) x[u] = 16 * c + u < n_out ? g[16 * c + u] : 0.f;
        put_operand(t_hi + 8 * c, t_lo + 8 * c, x);
      }
      tc_before();
    }
    // ---- backward: the gradient of layer l's pre-activations ----
    for (int l = NH - 1; l >= 0; --l) {
      multiply((uint32_t)l * W * W * 2u, W, l + 1 < NH ? W : n_pad, true);
      float *grow = a.grads + (size_t)l * layer_stride + i * W;
#pragma unroll 1
      for (int c = 0; c < W / 16; ++c) {
        uint32_t v[16];
        TMEM_LD16(acc + 16 * c, v);
        wait_ld(v);
        const uint32_t m = s_mask[((size_t)l * (W / 32) + (c >> 1)) * kTileM + r] >> (16 * (c & 1));
        float x[16];
#pragma unroll
        for (int u = 0; u < 16; ++u)
          x[u] = __uint_as_float(v[u]) * ((m >> u) & 1u ? 1.f : (act == 0 ? 0.f : 0.01f));
        if (on) {
          store8(grow + 16 * c, x);
          store8(grow + 16 * c + 8, x + 8);
        }
        if (l > 0) put_operand(t_hi + 8 * c, t_lo + 8 * c, x);
      }
      tc_before();
    }
  }
  // sums of the loss terms: warp, block, one atomic per block and term
  sums[0] = sums[1] + sums[2] + sums[3] + sums[4] + sums[5];
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    float v = sums[j];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) part[j][warp] = v;
  }
  tc_before();
  __syncthreads();
  tc_after();
  if (tid < 6) atomicAdd(a.loss + tid, (part[tid][0] + part[tid][1] + part[tid][2] + part[tid][3]) * inv_live);
  if (tid == 0 && s_abort) {
    // what is still in flight ends before the memory is released
    mma_commit(su32(&bars[1]));
    mbar_wait_teardown(su32(&bars[1]), phase);
    mbar_wait_teardown(su32(&bars[0]), 0u);
    atomicOr(a.err, kErrWaitTimeout);
  }
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(chain_tmem<W>()) : "memory");
}

template <int W, int NZ>
cudaError_t launch_shape(const ChainArgs &a, size_t smem, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(train_chain_kernel<W, NZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, kChainSmemMax);
  if (e != cudaSuccess) return e;
  int sms = 152, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // the CTAs that fit an SM: shared memory (1 KB of it the system's) and TMEM
  const int per = (int)std::max<size_t>(1, std::min<size_t>({(227u << 10) / (smem + 2048), 512u / chain_tmem<W>(), 4}));
  train_chain_kernel<W, NZ><<<(unsigned)std::min<int64_t>(a.n_tiles, (int64_t)sms * per), kCThreads, smem, st>>>(a);
  return cudaGetLastError();
}

size_t chain_smem(const DevObject &h) {
  return 2 * (size_t)h.umma_lo_bytes + 4 * ((size_t)h.n_hidden * h.width + h.n_out_pad) +
         (size_t)h.n_hidden * (h.width / 32) * kTileM * 4 + 1024;
}

}  // namespace

bool train_chain_supported(const DevObject &h) {
  return (h.width == 64 || h.width == 128) && h.n_out_pad <= 64 && chain_smem(h) <= kChainSmemMax;
}

cudaError_t launch_train_chain(const DevObject *dobj, const DevObject &h, int64_t B, const int32_t *k,
                               const int32_t *order, float *acts, float *grads, float *dZ, const lsnif_labels &lab,
                               float *loss, int *err, cudaStream_t st) {
  ChainArgs a{};
  a.obj = dobj;
  a.B = B;
  a.n_tiles = (B + kTileM - 1) / kTileM;
  a.k = k;
  a.order = order;
  a.acts = acts;
  a.grads = grads;
  a.dZ = dZ;
  a.lab = lab;
  a.loss = loss;
  a.w_bytes = h.umma_lo_bytes;
  a.bias_bytes = 4 * (uint32_t)(h.n_hidden * h.width + h.n_out_pad);
  a.err = err;
  const size_t smem = chain_smem(h);
  if (h.n_out_pad == 16) return h.width == 64 ? launch_shape<64, 16>(a, smem, st) : launch_shape<128, 16>(a, smem, st);
  return h.width == 64 ? launch_shape<64, 64>(a, smem, st) : launch_shape<128, 64>(a, smem, st);
}

}  // namespace lsnif
