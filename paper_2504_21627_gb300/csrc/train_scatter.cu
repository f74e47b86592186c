// The last step of the training backward pass in one kernel: the gradient of
// the network's input, dX = dY . W0, formed on the tensor cores chunk by chunk
// and scattered from tensor memory into the table gradients (backward of the
// trilinear interpolation), never written to global memory.
//
// Before, a product wrote dX (B x n_in FP32, 604 MB on the torus batch of
// 2^18) and a kernel with a thread per (ray, point, level) read it back: 454 +
// 1244 us, against 952 us here, 805 us over rays in order of their segment count. What bounds this form: L2's reductions (68% of
// their sector rate). So
//   - the two x corners of a cell go as one 16-byte reduction where they lie in
//     one aligned pair (every even cell; F = 2): six reductions per point and
//     level on average instead of eight (0.13 ms of the step);
//   - an entry point that is the previous segment's exit adds its gradient to
//     that point's before one set of reductions;
//   - the coarsest levels, whose few corners take every ray's reductions, are
//     summed in kReplicas dense lattices (corner coordinates as the index, no
//     hash) in scratch memory, which a second kernel adds up (7 us): fewer
//     reductions meet at one address. Lattices of at most 2^17 corners: without
//     any the step took 16 us longer, with up to 2^21 corners 170 us.
//
// A CTA takes 128 rays. dY (128 x W, FP32) is staged once as two-term BF16
// (hi + lo); for each segment s, the first layer's slice comes from a two-term
// BF16 copy laid out per segment (w0t, rebuilt each step) by a bulk copy, and
// hi.hi + hi.lo + lo.hi accumulate in FP32 in one of two TMEM buffers: the
// products of the kernel it replaces, in the same order per element. Eight
// warps read the exit points of segment s - 1 and the entry points of segment
// s (lane = ray, half of the levels each); the next segment's MMAs run while
// they scatter.
#include <algorithm>

#include "device.cuh"
#include "encode.cuh"
#include "tc_common.cuh"

namespace lsnif {

namespace {

constexpr int kSThreads = 256;
constexpr int kReplicas = 8;  // copies of the dense levels

#define TMEM_LD8(taddr, r)                                                                                    \
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"                       \
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) \
               : "r"(taddr))

struct ScatterArgs {
  const DevObject *obj;
  int64_t B;
  int W, LF;             // width; features per point
  const float *dY;       // B x W
  const uint8_t *w0t;    // per segment: hi tile, lo tile (CHK x W BF16 each, K-major core matrices)
  const int32_t *k;
  const int32_t *order;  // ray of a row (NULL: the row itself)
  const float *pts;
  float *gtab;
  float *dense;          // kReplicas copies of the dense levels' lattices
  int n_dense;           // levels 0 .. n_dense - 1 are dense
  int64_t dense_stride;  // floats of one copy
  int32_t dense_off[LSNIF_MAX_LEVELS];  // a level's first float in a copy
  int *err;
};

__device__ __forceinline__ void mma_s(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// a gradient into the corners of its cell: table entries by the hash, or (DENSE)
// by the corner's place in the (N + 1)^3 lattice `gd` -- a point that rounding
// put outside the cube has corners outside it, and goes to the table
template <int F, bool DENSE>
__device__ __forceinline__ void scatter_point(float *__restrict__ gt, float *__restrict__ gd, uint32_t mask,
                                              const float3 &p, float N, const float (&v)[F]) {
  const Cell c = lattice_cell(p, N);
  const uint32_t n1 = (uint32_t)N + 1u;
  if constexpr (DENSE) {
    if (max(c.cx + (c.wx != 0.f), max(c.cy + (c.wy != 0.f), c.cz + (c.wz != 0.f))) >= n1 ||
        max(c.cx, max(c.cy, c.cz)) >= n1) {
      scatter_point<F, false>(gt, nullptr, mask, p, N, v);
      return;
    }
  }
  float *g = DENSE ? gd : gt;
  const float wx0 = 1.f - c.wx;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int dy = q & 1, dz = q >> 1;
    const float wy = dy ? c.wy : 1.f - c.wy, wz = dz ? c.wz : 1.f - c.wz;
    const float w0 = wx0 * wy * wz, w1 = c.wx * wy * wz;
    uint32_t i0, i1;
    if (DENSE) {
      i0 = ((c.cz + dz) * n1 + c.cy + dy) * n1 + c.cx;
      i1 = i0 + 1u;
    } else {
      const uint32_t b = ((c.cy + dy) * kPi2) ^ ((c.cz + dz) * kPi3);
      i0 = (c.cx ^ b) & mask;
      i1 = ((c.cx + 1u) ^ b) & mask;
    }
    if constexpr (F == 2) {
      if ((i0 ^ i1) == 1u) {
        if (w0 == 0.f && w1 == 0.f) continue;
        // a corner of weight 0 takes 0, whatever the gradient
        const float a0 = w0 == 0.f ? 0.f : w0 * v[0], a1 = w0 == 0.f ? 0.f : w0 * v[1];
        const float b0 = w1 == 0.f ? 0.f : w1 * v[0], b1 = w1 == 0.f ? 0.f : w1 * v[1];
        const bool odd = (i0 & 1u) != 0u;
        atomicAdd(reinterpret_cast<float4 *>(g + (size_t)(i0 & ~1u) * 2),
                  odd ? make_float4(b0, b1, a0, a1) : make_float4(a0, a1, b0, b1));
      } else {
        if (w0 != 0.f) atomicAdd(reinterpret_cast<float2 *>(g + (size_t)i0 * 2), make_float2(w0 * v[0], w0 * v[1]));
        if (w1 != 0.f) atomicAdd(reinterpret_cast<float2 *>(g + (size_t)i1 * 2), make_float2(w1 * v[0], w1 * v[1]));
      }
    } else {
      if (w0 != 0.f)
        atomicAdd(reinterpret_cast<float4 *>(g + (size_t)i0 * 4), make_float4(w0 * v[0], w0 * v[1], w0 * v[2], w0 * v[3]));
      if (w1 != 0.f)
        atomicAdd(reinterpret_cast<float4 *>(g + (size_t)i1 * 4), make_float4(w1 * v[0], w1 * v[1], w1 * v[2], w1 * v[3]));
    }
  }
}

// HC: columns (features) of a point that a warp scatters: half of L F
template <int F, int HC>
__global__ void __launch_bounds__(kSThreads, HC <= 16 ? 3 : 1) input_scatter_kernel(const __grid_constant__ ScatterArgs a) {
  extern __shared__ __align__(1024) uint8_t sraw[];
  __shared__ uint64_t bars[4];  // [0..1] weight slots, [2..3] accumulators
  __shared__ uint32_t s_tmem;
  __shared__ int s_kmax;
  __shared__ volatile int s_abort;
  constexpr int LF = 2 * HC, CHK = 2 * LF;  // columns of a segment
  constexpr int kTmem = 2 * CHK < 32 ? 32 : 2 * CHK;
  uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(sraw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int W = a.W, KG = W / 8;  // K groups of 8
  const int64_t r0 = (int64_t)blockIdx.x * kTileM;
  const int rows = (int)min((int64_t)kTileM, a.B - r0);
  const uint32_t a_bytes = (uint32_t)kTileM * W * 2, b_bytes = (uint32_t)CHK * W * 2;  // one term
  uint8_t *sA = base, *sB = base + 2 * a_bytes;                                        // hi, lo | two slots of (hi, lo)
  if (tid == 0) {
    for (int b = 0; b < 4; ++b) mbar_init(su32(&bars[b]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
    s_kmax = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&s_tmem)), "r"(kTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_before();
  __syncthreads();
  tc_after();
  const uint32_t tmem = s_tmem;
  const DevObject &ob = *a.obj;
  const int quarter = warp & 3, half = warp >> 2, row = quarter * 32 + lane;
  const int kk = row < rows ? a.k[r0 + row] : 0;
  {
    const int m = __reduce_max_sync(0xffffffffu, kk);
    if (lane == 0 && half == 0) atomicMax(&s_kmax, m);
  }
  // dY -> two-term BF16; an item is one row's 8 columns,
  // and a quarter-warp stores one whole core matrix
  for (int it = tid; it < kTileM * KG; it += kSThreads) {
    const int r = (it & 7) + (it / (8 * KG)) * 8, g = (it >> 3) % KG;
    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (r < rows) {
      load8(a.dY + (r0 + r) * W + g * 8, v);
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
    const uint32_t o = core_off(r, g, (uint32_t)KG * 128u);
    *reinterpret_cast<uint4 *>(sA + o) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
    *reinterpret_cast<uint4 *>(sA + a_bytes + o) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
  }
  fence_async_smem();
  __syncthreads();
  const int kmax = s_kmax;
  // thread 0: the slice of segment s into its slot
  auto load_w = [&](int s) {
    const uint32_t slot = su32(sB) + (uint32_t)(s & 1) * 2 * b_bytes, bar = su32(&bars[s & 1]);
    mbar_expect(bar, 2 * b_bytes);
    bulk_load(slot, a.w0t + (size_t)s * 2 * b_bytes, 2 * b_bytes, bar);
  };
  // thread 0: segment s's products into accumulator s & 1
  auto multiply = [&](int s) {
    if (!mbar_wait(su32(&bars[s & 1]), (uint32_t)((s >> 1) & 1), &s_abort)) return;
    tc_after();
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(CHK >> 3) << 17) | ((uint32_t)(kTileM >> 4) << 24);
    const uint32_t ah = su32(sA), al = ah + a_bytes, bh = su32(sB) + (uint32_t)(s & 1) * 2 * b_bytes, bl = bh + b_bytes;
    const uint32_t sbo = (uint32_t)KG * 128u, d = tmem + (uint32_t)((s & 1) * CHK);
    for (int ks = 0; ks < W / 16; ++ks) {
      const uint64_t dah = umma_desc(ah + ks * 256, 128, sbo), dal = umma_desc(al + ks * 256, 128, sbo);
      const uint64_t dbh = umma_desc(bh + ks * 256, 128, sbo), dbl = umma_desc(bl + ks * 256, 128, sbo);
      mma_s(d, dah, dbh, idesc, ks > 0 ? 1u : 0u);
      mma_s(d, dah, dbl, idesc, 1u);
      mma_s(d, dal, dbh, idesc, 1u);
    }
    mma_commit(su32(&bars[2 + (s & 1)]));
  };
  int loaded = 0, issued = 0;  // thread 0: slices asked for, products committed
  if (tid == 0 && kmax > 0) {
    load_w(loaded++);
    if (kmax > 1) load_w(loaded++);
    multiply(0);
    if (!s_abort) issued = 1;
  }
  float *gdense = a.dense + (size_t)(blockIdx.x % kReplicas) * a.dense_stride;
  const int64_t r = r0 + min(row, rows - 1);
  const float *P = a.pts + (a.order ? a.order[r] : r) * ob.H * 3;
  const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(half * HC);
  constexpr int LH = HC / F;  // levels of a warp
  for (int s = 0; s <= kmax && kmax > 0; ++s) {
    if (tid == 0 && s < kmax) mbar_wait(su32(&bars[2 + (s & 1)]), (uint32_t)((s >> 1) & 1), &s_abort);
    const bool ex = s > 0 && s - 1 < kk, en = s < kk;  // an exit point of s - 1, an entry point of s
    float3 px = make_float3(0.f, 0.f, 0.f), pe = px;
    if (ex) px = make_float3(P[6 * s - 3], P[6 * s - 2], P[6 * s - 1]);
    if (en) pe = make_float3(P[6 * s], P[6 * s + 1], P[6 * s + 2]);
    const bool dup = ex && en && px.x == pe.x && px.y == pe.y && px.z == pe.z;
    __syncthreads();
    if (s_abort) break;
    tc_after();
    uint32_t gx[HC], ge[HC];
    const uint32_t tx = trow + (uint32_t)(((s + 1) & 1) * CHK + LF), te = trow + (uint32_t)((s & 1) * CHK);
#pragma unroll
    for (int c = 0; c < HC; c += 8) {
      if (s > 0) TMEM_LD8(tx + c, (&gx[c]));
      if (s < kmax) TMEM_LD8(te + c, (&ge[c]));
    }
    tmem_wait_ld();
    tc_before();
    __syncthreads();  // the accumulator of segment s - 1 is read
    if (tid == 0 && s + 1 < kmax) {
      tc_after();
      multiply(s + 1);
      if (!s_abort) issued = s + 2;
      // segment s's products are done: its slot takes the slice of s + 2
      if (loaded < kmax && !s_abort) load_w(loaded++);
    }
#pragma unroll 1
    for (int u = 0; u < LH; ++u) {
      const int l = half * LH + u;
      const float N = (float)ob.res[l];
      const bool dense = l < a.n_dense;
      float *gt = a.gtab + (size_t)l * (ob.mask + 1) * F, *gd = dense ? gdense + a.dense_off[l] : nullptr;
      float vx[F], ve[F];
#pragma unroll
      for (int f = 0; f < F; ++f) {
        vx[f] = ve[f] = 0.f;
#pragma unroll
        for (int w = 0; w < LH; ++w)  // gx and ge stay in registers
          if (w == u) {
            vx[f] = __uint_as_float(gx[w * F + f]);
            ve[f] = __uint_as_float(ge[w * F + f]);
          }
        if (dup) vx[f] += ve[f];
      }
      if (dense) {
        if (ex) scatter_point<F, true>(gt, gd, ob.mask, px, N, vx);
        if (en && !dup) scatter_point<F, true>(gt, gd, ob.mask, pe, N, ve);
      } else {
        if (ex) scatter_point<F, false>(gt, gd, ob.mask, px, N, vx);
        if (en && !dup) scatter_point<F, false>(gt, gd, ob.mask, pe, N, ve);
      }
    }
  }
  // copies and products still in flight (after an abort) end before the shared
  // memory and the tensor memory are released
  if (tid == 0) {
    if (loaded > 0 && !mbar_wait_teardown(su32(&bars[(loaded - 1) & 1]), (uint32_t)(((loaded - 1) >> 1) & 1))) s_abort = 1;
    if (loaded > 1 && !mbar_wait_teardown(su32(&bars[loaded & 1]), (uint32_t)(((loaded - 2) >> 1) & 1))) s_abort = 1;
    if (issued > 0 && !mbar_wait_teardown(su32(&bars[2 + ((issued - 1) & 1)]), (uint32_t)(((issued - 1) >> 1) & 1))) s_abort = 1;
  }
  tc_before();
  __syncthreads();
  tc_after();
  if (tid == 0 && s_abort) atomicOr(a.err, kErrWaitTimeout);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmem) : "memory");
}

// the first layer (W x n_in FP32) as two-term BF16, transposed, per segment
__global__ void __launch_bounds__(256) build_w0t_kernel(const float *W0, int W, int n_in, int CHK, uint8_t *dst) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < W * n_in; e += gridDim.x * blockDim.x) {
    const int k = e / n_in, col = e - k * n_in, s = col / CHK, n = col - s * CHK;
    const float v = W0[e];
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    uint8_t *t = dst + (size_t)s * CHK * W * 4 + core_off(n, k >> 3, (uint32_t)(W / 8) * 128u) + (k & 7) * 2;
    *reinterpret_cast<__nv_bfloat16 *>(t) = h;
    *reinterpret_cast<__nv_bfloat16 *>(t + (size_t)CHK * W * 2) = __float2bfloat16_rn(v - __bfloat162float(h));
  }
}

// dense lattices, summed over the copies, into the hashed table gradients
template <int F>
__global__ void __launch_bounds__(256) dense_sum_kernel(ScatterArgs a) {
  const DevObject &ob = *a.obj;
  const int l = blockIdx.y;
  const uint32_t n1 = (uint32_t)ob.res[l] + 1u, n = n1 * n1 * n1;
  float *g = a.gtab + (size_t)l * (ob.mask + 1) * F;
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    float v[F] = {};
    for (int r = 0; r < kReplicas; ++r) {
      const float *d = a.dense + (size_t)r * a.dense_stride + a.dense_off[l] + (size_t)e * F;
#pragma unroll
      for (int f = 0; f < F; ++f) v[f] += d[f];
    }
    bool any = false;
#pragma unroll
    for (int f = 0; f < F; ++f) any |= v[f] != 0.f;
    if (!any) continue;
    const uint32_t x = e % n1, y = (e / n1) % n1, z = e / (n1 * n1);
    float *d = g + (size_t)(hash3(x, y, z) & ob.mask) * F;
    if constexpr (F == 2) atomicAdd(reinterpret_cast<float2 *>(d), make_float2(v[0], v[1]));
    else atomicAdd(reinterpret_cast<float4 *>(d), make_float4(v[0], v[1], v[2], v[3]));
  }
}

template <int F, int HC>
cudaError_t launch_shape(const ScatterArgs &a, cudaStream_t st) {
  auto smem_of = [](int W) { return 2 * (size_t)kTileM * W * 2 + 4 * (size_t)(4 * HC) * W * 2 + 1024; };
  const size_t smem = smem_of(a.W);
  const cudaError_t e = cudaFuncSetAttribute(input_scatter_kernel<F, HC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem_of(128));
  if (e != cudaSuccess) return e;
  input_scatter_kernel<F, HC><<<(unsigned)((a.B + kTileM - 1) / kTileM), kSThreads, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

InputScatterPlan input_scatter_plan(const DevObject &h) {
  InputScatterPlan p{};
  const int LF = h.L * h.F;
  if (!((h.F == 2 || h.F == 4) && (h.width == 64 || h.width == 128) && (LF == 16 || LF == 32 || LF == 64))) return p;
  p.ok = true;
  p.w0t_bytes = (size_t)h.n_in * h.width * 4;
  // dense levels: lattices of at most 2^17 corners, the coarsest first
  int64_t floats = 0;
  for (int l = 0; l < h.L; ++l) {
    const int64_t n1 = (int64_t)h.res[l] + 1, n = n1 * n1 * n1;
    if (n > (1 << 17)) break;
    p.dense_off[l] = (int32_t)floats;
    floats += (n * h.F + 7) & ~int64_t(3);  // 16-byte aligned, room for a pair past the last corner
    p.n_dense = l + 1;
  }
  p.dense_stride = floats;
  p.dense_bytes = (size_t)floats * 4 * kReplicas;
  return p;
}

cudaError_t launch_build_w0t(const DevObject &h, const float *W0, void *w0t, cudaStream_t st) {
  build_w0t_kernel<<<152, 256, 0, st>>>(W0, h.width, h.n_in, 2 * h.L * h.F, static_cast<uint8_t *>(w0t));
  return cudaGetLastError();
}

cudaError_t launch_input_scatter(const DevObject *dobj, const DevObject &h, int64_t B, const float *dY,
                                 const void *w0t, const int32_t *k, const int32_t *order, const float *pts,
                                 float *gtab, float *dense, int *err, cudaStream_t st) {
  const InputScatterPlan p = input_scatter_plan(h);
  ScatterArgs a{};
  a.obj = dobj;
  a.B = B;
  a.W = h.width;
  a.LF = h.L * h.F;
  a.dY = dY;
  a.w0t = static_cast<const uint8_t *>(w0t);
  a.k = k;
  a.order = order;
  a.pts = pts;
  a.gtab = gtab;
  a.dense = dense;
  a.n_dense = p.n_dense;
  a.dense_stride = p.dense_stride;
  for (int l = 0; l < p.n_dense; ++l) a.dense_off[l] = p.dense_off[l];
  a.err = err;
  cudaError_t e = p.dense_bytes ? cudaMemsetAsync(dense, 0, p.dense_bytes, st) : cudaSuccess;
  if (e != cudaSuccess) return e;
  if (h.F == 2) e = a.LF == 16 ? launch_shape<2, 8>(a, st) : a.LF == 32 ? launch_shape<2, 16>(a, st) : launch_shape<2, 32>(a, st);
  else e = a.LF == 16 ? launch_shape<4, 8>(a, st) : a.LF == 32 ? launch_shape<4, 16>(a, st) : launch_shape<4, 32>(a, st);
  if (e != cudaSuccess) return e;
  if (p.n_dense) {
    const dim3 grid(128, p.n_dense);
    if (h.F == 2) dense_sum_kernel<2><<<grid, 256, 0, st>>>(a);
    else dense_sum_kernel<4><<<grid, 256, 0, st>>>(a);
  }
  return cudaGetLastError();
}

}  // namespace lsnif
