// The FP32 query's network kernel for the common shapes (F = 2 or 4, width
// 64 or 128, at most 64 features a point): hash-grid gather, every layer and
// the decode in one kernel, FP32 throughout. The stage kernels in query.cu
// (features to global memory, then a SIMT network) serve the other shapes.
//
// What bounds it: FP32 multiply-adds (50k per ray on the 576-64x4-12 network)
// and the corner loads of 16 levels per point. The stage kernels reached 7
// TFLOP/s: scalar shared-memory reads (12 per 32 multiply-adds), 8-way bank
// conflicts on the staged operands, and a round trip of every feature through
// global memory. Here
//   - a CTA takes R rays; a thread holds RT rows x CT columns of the layer's
//     outputs and multiplies with packed FP32 pairs (fma.rn.f32x2: two
//     columns per instruction, each product and sum rounded as fmaf does),
//     reading rows and columns as 16-byte words without bank conflicts;
//   - features go to shared memory only, transposed ([column][row]), and the
//     layers' outputs replace their inputs there;
//   - a boundary point that the traversal marked as the previous exit point
//     takes its features from there instead of the tables, and segments that
//     no ray of the tile reaches are skipped (exact: their features are 0;
//     not skipped while the first layer holds a non-finite weight);
//   - two or three CTAs share an SM, so that one's gather overlaps another's
//     layers.
// Every output is one chain of fused multiply-adds over ascending inputs
// starting at 0, then the bias, as in the stage kernels: the same bits.
//
// Measured (GB300, 576-64x4-12 network): the 1000 x 1000 torus frame (371k
// rays reach the network) takes 1.53 ms here, 7.2 ms in the stage kernels;
// 4,096 rays on the icosphere 45 us instead of 160. L1 is the busiest unit
// (70% of its wavefronts, 60% of them the divergent corner loads), then the
// multiply-adds (46%).
#include <algorithm>

#include "device.cuh"
#include "encode.cuh"

namespace lsnif {

namespace {

__device__ __forceinline__ unsigned long long dup2(float a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}

__device__ __forceinline__ void fma2(unsigned long long &d, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// Shape of a CTA with R rows: RT x CT outputs per thread. A warp reads RT + CT
// words per lane and input, one shared-memory wavefront each, for RT CT / 2
// packed multiply-adds: 8 x 8 balances the two units (4 x 8, with 256 threads,
// took 1.61 ms instead of 1.53 for the 1000 x 1000 torus frame below).
// Tiles of 32 rows, for small requests, use more threads on fewer outputs.
template <int W, int R>
struct PlainShape {
  static constexpr int RT = R > 32 ? 8 : 2;
  static constexpr int CT = R > 32 ? 8 : W / 16;
  static constexpr int NTX = W / CT;     // column groups
  static constexpr int T = NTX * (R / RT);  // threads
  static constexpr int CTAS = R > 32 ? 3 : 2;  // per SM
  static constexpr int PK = W == 64 ? 32 : 16;  // inputs per weight sub-chunk
  static constexpr int LD = R + 4;       // row stride of the [column][row] tile
  static constexpr int SUB = kTileM / R; // CTAs' tiles per 128-ray tile
  static_assert((CT == 4 || CT == 8) && T % 32 == 0, "4 or 8 columns per thread, whole warps");
};

constexpr int plain_rows(int W) { return W == 64 ? 128 : 64; }

// columns of a gather chunk: whole segments (two points), about 64 columns
__host__ __device__ inline int plain_segs(int LF) { return 2 * LF >= 64 ? 1 : 64 / (2 * LF); }

// kn inputs of a layer: acc += in[k][rows] x w[k][columns]
template <int W, int R>
__device__ __forceinline__ void plain_mac(unsigned long long (&acc)[PlainShape<W, R>::RT][PlainShape<W, R>::CT / 2],
                                          const float *A, const float *Ws, int kn, int ty, int tx) {
  using S = PlainShape<W, R>;
  constexpr int LDW = W + 4;
#pragma unroll 4
  for (int kk = 0; kk < kn; ++kk) {
    float a[S::RT];
    if constexpr (S::RT == 8) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 v = *reinterpret_cast<const float4 *>(A + kk * S::LD + h * (R / 2) + ty * 4);
        a[4 * h] = v.x; a[4 * h + 1] = v.y; a[4 * h + 2] = v.z; a[4 * h + 3] = v.w;
      }
    } else {
      const float2 v = *reinterpret_cast<const float2 *>(A + kk * S::LD + ty * 2);
      a[0] = v.x; a[1] = v.y;
    }
    unsigned long long b[S::CT / 2];
#pragma unroll
    for (int h = 0; h < S::CT / 4; ++h) {
      const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(Ws + kk * LDW + h * (W / 2) + tx * 4);
      b[2 * h] = v.x;
      b[2 * h + 1] = v.y;
    }
#pragma unroll
    for (int i = 0; i < S::RT; ++i) {
      const unsigned long long aa = dup2(a[i]);
#pragma unroll
      for (int j = 0; j < S::CT / 2; ++j) fma2(acc[i][j], aa, b[j]);
    }
  }
}

template <int F, int W, int R>
__global__ void __launch_bounds__(PlainShape<W, R>::T, PlainShape<W, R>::CTAS)
    plain_fused_kernel(QueryLaunch q, int lf_max) {
  using S = PlainShape<W, R>;
  constexpr int RT = S::RT, CT = S::CT, LD = S::LD, LDW = W + 4, kPThreads = S::T, kPK = S::PK;
  constexpr int WV = W * kPK / 4 / kPThreads;  // 16-byte weight words per thread and sub-chunk
  extern __shared__ __align__(16) float psm[];
  const int ka = max(plain_segs(lf_max) * 2 * lf_max, W);
  float *A = psm;                      // [ka][LD]
  float *Wb = A + (size_t)ka * LD;     // two buffers of [kPK][LDW]
  int *s_ray = reinterpret_cast<int *>(Wb + 2 * kPK * LDW);
  int *s_misc = s_ray + R;             // [0] next tile, [1] largest point count
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ty = (tid & 3) | ((tid / (4 * S::NTX)) << 2), tx = (tid >> 2) % S::NTX;
  const int total = q.s.meta[1] * S::SUB;
  // the row whose features this thread gathers: the lanes of a warp take
  // neighbouring rays at the same level
  constexpr int RB = R / 32;           // row blocks of 32
  constexpr int LSTEP = kPThreads / 32 / RB;  // warps that share a row block
  const int grow = (warp % RB) * 32 + lane, glev = warp / RB;

  float4 wr[WV];
  // weights of inputs [k0, k0 + kn) of an N-column layer with K inputs
  auto load_w = [&](const float *Wp, int K, int N, int k0, int kn) {
#pragma unroll
    for (int j = 0; j < WV; ++j) {
      const int i = tid + j * kPThreads, b = i >> 5, nb = N >> 4;
      const int n = (i & 15) + 16 * (b % nb), k4 = ((i >> 4) & 1) + 2 * (b / nb);
      if (k4 * 4 < kn) wr[j] = __ldg(reinterpret_cast<const float4 *>(Wp + (int64_t)n * K + k0 + k4 * 4));
    }
  };
  // a half-warp writes 16 columns of one input, the other half those of the
  // input 4 further on: 32 distinct banks (4 LDW = 16 modulo 32)
  auto store_w = [&](float *buf, int N, int kn) {
#pragma unroll
    for (int j = 0; j < WV; ++j) {
      const int i = tid + j * kPThreads, b = i >> 5, nb = N >> 4;
      const int n = (i & 15) + 16 * (b % nb), k4 = ((i >> 4) & 1) + 2 * (b / nb);
      if (k4 * 4 < kn) {
        float *d = buf + (k4 * 4) * LDW + n;
        d[0] = wr[j].x; d[LDW] = wr[j].y; d[2 * LDW] = wr[j].z; d[3 * LDW] = wr[j].w;
      }
    }
  };

  for (int tt = blockIdx.x; tt < total;) {
    const int t = tt / S::SUB, part = tt - t * S::SUB;
    const int slot = q.s.tiles[3 * t], start = q.s.tiles[3 * t + 1] + part * R;
    const int cnt = min(R, q.s.tiles[3 * t + 2] - part * R);
    int next = 0;
    if (tid == 0) {
      next = (int)gridDim.x + atomicAdd(q.s.meta + 3, 1);
      s_misc[1] = 0;
    }
    if (cnt <= 0) {
      __syncthreads();
      if (tid == 0) s_misc[0] = next;
      __syncthreads();
      tt = s_misc[0];
      continue;
    }
    const DevObject &ob = q.objs[slot];
    const int L = ob.L, LF = L * F, n_in = ob.n_in, n_hidden = ob.n_hidden, n_out_pad = ob.n_out_pad, act = ob.act;
    const int segs = plain_segs(LF), CC = segs * 2 * LF;
    const float *w0 = ob.mlp32;
    int buf = 0;
    const int kn0 = min(kPK, min(CC, n_in));  // at least the first sub-chunk's inputs
    load_w(w0, n_in, W, 0, kn0);
    int ray = -1, kr = 0;
    uint32_t dm = 0;
    if (grow < cnt) {
      ray = q.s.order[start + grow];
      kr = q.s.k[ray];
      dm = q.s.dup[ray];
    }
    __syncthreads();  // s_misc[1] is reset; the last tile's readers are done
    if (glev == 0) {
      s_ray[grow] = ray;
      const int m = __reduce_max_sync(0xffffffffu, kr);
      if (lane == 0) atomicMax(&s_misc[1], m);
    }
    store_w(Wb, W, kn0);
    __syncthreads();
    // segments to multiply: up to the tile's largest count, or all of them
    // when a first-layer weight is not finite (0 times it is not 0)
    int kmax = s_misc[1];
    {
      const int *bad = reinterpret_cast<const int *>(ob.plain_out + (size_t)n_out_pad * (W + 1));
      int any = 0;
#pragma unroll
      for (int j = 0; j < kNonFiniteWords; ++j) any |= bad[j];
      if (any) kmax = ob.H >> 1;
    }
    const int K0 = kmax * 2 * LF;
    unsigned long long acc[RT][CT / 2];
    auto clear = [&]() {
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int j = 0; j < CT / 2; ++j) acc[i][j] = 0ull;
    };
    clear();
    // ---- first layer: gather a chunk of segments, multiply it ----
    const float *P = q.s.pts + (size_t)max(ray, 0) * q.H_max * 3;
    for (int c0 = 0; c0 < K0; c0 += CC) {
      const int s0 = c0 / (2 * LF), ns = min(segs, kmax - s0);
      for (int sg = 0; sg < ns; ++sg) {
        const int s = s0 + sg;
        const bool on = s < kr, dup = s > 0 && ((dm >> s) & 1u);
        float3 pa = make_float3(0.f, 0.f, 0.f), pb = pa;
        if (on) {
          const float2 v0 = __ldg(reinterpret_cast<const float2 *>(P + 6 * s)), v1 = __ldg(reinterpret_cast<const float2 *>(P + 6 * s) + 1),
                       v2 = __ldg(reinterpret_cast<const float2 *>(P + 6 * s) + 2);
          pa = make_float3(v0.x, v0.y, v1.x);
          pb = make_float3(v1.y, v2.x, v2.y);
        }
        float *Ae = A + (size_t)(sg * 2 * LF) * LD + grow, *Ax = Ae + (size_t)LF * LD;
        // the previous segment's exit features: the segment before in this
        // chunk, or the last one of the chunk before, which this thread wrote
        const float *Ap = A + (size_t)((sg > 0 ? sg - 1 : segs - 1) * 2 * LF + LF) * LD + grow;
        for (int l = glev; l < L; l += LSTEP) {
          const float *tl = ob.tab32 + (size_t)l * (ob.mask + 1) * F;
          const float N = (float)ob.res[l];
          float fa[F], fb[F];
          encode_level_f32_if<F>(tl, ob.mask, pa, N, on && !dup, fa);
          encode_level_f32_if<F>(tl, ob.mask, pb, N, on, fb);
          if (on && dup) {
#pragma unroll
            for (int f = 0; f < F; ++f) fa[f] = Ap[(l * F + f) * LD];
          }
#pragma unroll
          for (int f = 0; f < F; ++f) {
            Ae[(l * F + f) * LD] = fa[f];
            Ax[(l * F + f) * LD] = fb[f];
          }
        }
      }
      __syncthreads();
      const int ce = min(c0 + CC, K0);
      for (int k0 = c0; k0 < ce;) {
        const int kn = min(kPK, ce - k0), k1 = k0 + kn;
        // the next weights: this layer's, or the second layer's first
        const bool more = k1 < K0;
        const int N1 = more || n_hidden > 1 ? W : n_out_pad;
        const int kn1 = more ? min(kPK, min((k1 / CC + 1) * CC, K0) - k1) : kPK;
        const float *w1 = more ? w0 : (n_hidden > 1 ? w0 + (size_t)W * n_in + W : ob.plain_out);
        load_w(w1, more ? n_in : W, N1, more ? k1 : 0, kn1);
        plain_mac<W, R>(acc, A + (size_t)(k0 - c0) * LD, Wb + buf * kPK * LDW, kn, ty, tx);
        buf ^= 1;
        store_w(Wb + buf * kPK * LDW, N1, kn1);
        __syncthreads();
        k0 = k1;
      }
    }
    // ---- later layers; outputs replace the inputs in A ----
    const float *wl = w0, *bias = w0 + (size_t)W * n_in;
    for (int layer = 0; layer < n_hidden; ++layer) {
      // outputs of `layer` (every thread is past its reads of A)
#pragma unroll
      for (int j = 0; j < CT; j += 2) {
        const int col = (j >> 2) * (W / 2) + tx * 4 + (j & 3);
        const float b0 = bias[col], b1 = bias[col + 1];
        float x[RT], y[RT];
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          const float2 v = unpack2(acc[i][j / 2]);
          x[i] = act_fn(v.x + b0, act);
          y[i] = act_fn(v.y + b1, act);
        }
        if constexpr (RT == 8) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float *d = A + (size_t)col * LD + h * (R / 2) + ty * 4;
            *reinterpret_cast<float4 *>(d) = make_float4(x[4 * h], x[4 * h + 1], x[4 * h + 2], x[4 * h + 3]);
            *reinterpret_cast<float4 *>(d + LD) = make_float4(y[4 * h], y[4 * h + 1], y[4 * h + 2], y[4 * h + 3]);
          }
        } else {
          float *d = A + (size_t)col * LD + ty * 2;
          *reinterpret_cast<float2 *>(d) = make_float2(x[0], x[1]);
          *reinterpret_cast<float2 *>(d + LD) = make_float2(y[0], y[1]);
        }
      }
      __syncthreads();
      if (layer + 1 == n_hidden) break;
      clear();
      wl = bias + W;
      bias = wl + (size_t)W * W;
      for (int k0 = 0; k0 < W; k0 += kPK) {
        const bool more = k0 + kPK < W, hidden = layer + 2 < n_hidden;
        const int N1 = more || hidden ? W : n_out_pad;
        const float *w1 = more ? wl : (hidden ? bias + W : ob.plain_out);
        load_w(w1, W, N1, more ? k0 + kPK : 0, kPK);
        plain_mac<W, R>(acc, A + (size_t)k0 * LD, Wb + buf * kPK * LDW, kPK, ty, tx);
        buf ^= 1;
        store_w(Wb + buf * kPK * LDW, N1, kPK);
        __syncthreads();
      }
    }
    // ---- output layer: 1 row x 4 columns per thread and pass ----
    constexpr int kPasses = R / (kPThreads / 16);  // enough for the 16 groups of 64 columns
    const int ngrp = n_out_pad >> 2, pass = kPThreads / ngrp;
    unsigned long long oz[kPasses][2];
    const int og = tid % ngrp, orow = tid / ngrp;
#pragma unroll
    for (int p = 0; p < kPasses; ++p) oz[p][0] = oz[p][1] = 0ull;
    for (int k0 = 0; k0 < W; k0 += kPK) {
      const bool more = k0 + kPK < W;
      if (more) load_w(ob.plain_out, W, n_out_pad, k0 + kPK, kPK);
      const float *Wo = Wb + buf * kPK * LDW;
      if (orow < pass) {
#pragma unroll
        for (int p = 0; p < kPasses; ++p) {
          const int r = orow + p * pass;
          if (r >= R) break;
#pragma unroll 4
          for (int kk = 0; kk < kPK; ++kk) {
            const ulonglong2 b = *reinterpret_cast<const ulonglong2 *>(Wo + kk * LDW + og * 4);
            const unsigned long long aa = dup2(A[(size_t)(k0 + kk) * LD + r]);
            fma2(oz[p][0], aa, b.x);
            fma2(oz[p][1], aa, b.y);
          }
        }
      }
      buf ^= 1;
      if (more) store_w(Wb + buf * kPK * LDW, n_out_pad, kPK);
      __syncthreads();
    }
    const float *bo = ob.plain_out + (size_t)n_out_pad * W;
    if (orow < pass) {
#pragma unroll
      for (int p = 0; p < kPasses; ++p) {
        const int r = orow + p * pass;
        if (r >= R) break;
        const float2 v0 = unpack2(oz[p][0]), v1 = unpack2(oz[p][1]);
        float *d = A + (size_t)(og * 4) * LD + r;
        d[0] = v0.x + bo[og * 4];
        d[LD] = v0.y + bo[og * 4 + 1];
        d[2 * LD] = v1.x + bo[og * 4 + 2];
        d[3 * LD] = v1.y + bo[og * 4 + 3];
      }
    }
    if (tid == 0) s_misc[0] = next;
    __syncthreads();
    tt = s_misc[0];
    if (tid < cnt) {
      float z[64];
      for (int j = 0; j < ob.n_out; ++j) z[j] = A[(size_t)j * LD + tid];
      const int32_t rr = s_ray[tid];
      const float2 tt01 = reinterpret_cast<const float2 *>(q.s.t01)[rr];
      decode_store(q.hits, rr, z, ob.n_out, ob.n_mat, tt01.x, tt01.y, q.rays.tmin[rr], q.rays.tmax[rr]);
    }
  }
}

template <int W, int R>
size_t plain_smem(int lf_max) {
  const int ka = std::max(plain_segs(lf_max) * 2 * lf_max, W);
  return sizeof(float) * ((size_t)ka * PlainShape<W, R>::LD + 2 * PlainShape<W, R>::PK * (W + 4) + R + 4);
}

template <int F, int W, int R>
cudaError_t launch_rows(const QueryLaunch &q, int lf_max, int sms) {
  const size_t smem = plain_smem<W, R>(lf_max);
  // on every launch: the limit belongs to the current device
  const cudaError_t e =
      cudaFuncSetAttribute(plain_fused_kernel<F, W, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 << 10);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (int64_t)q.s.max_tiles * PlainShape<W, R>::SUB;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)PlainShape<W, R>::CTAS * sms, tiles));
  plain_fused_kernel<F, W, R><<<grid, PlainShape<W, R>::T, smem, q.stream>>>(q, lf_max);
  return cudaGetLastError();
}

template <int F, int W>
cudaError_t launch_shape(const QueryLaunch &q, int lf_max) {
  int sms = 152, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // Tiles of 32 rows while tiles of 128 could not give every SM one: a small
  // request is bound by the length of one tile's chain of chunks and layers,
  // and more and smaller CTAs shorten it. On the torus network 4,096 rays
  // take 64 us so and 137 us in the large tiles, 16,384 rays 149 and 180 us,
  // 65,536 rays 420 and 289 us.
  const bool small = q.rays.n <= (int64_t)sms * kTileM;
  return small ? launch_rows<F, W, 32>(q, lf_max, sms) : launch_rows<F, W, plain_rows(W)>(q, lf_max, sms);
}

}  // namespace

bool plain_fused_supported(int F, int width, int lf_max) {
  return (F == 2 || F == 4) && (width == 64 || width == 128) && lf_max <= 64;
}

cudaError_t launch_plain_fused(const QueryLaunch &q, int F, int width, int lf_max, int *launches) {
  *launches += 1;
  if (F == 2 && width == 64) return launch_shape<2, 64>(q, lf_max);
  if (F == 2 && width == 128) return launch_shape<2, 128>(q, lf_max);
  if (F == 4 && width == 64) return launch_shape<4, 64>(q, lf_max);
  if (F == 4 && width == 128) return launch_shape<4, 128>(q, lf_max);
  return cudaErrorNotSupported;
}

}  // namespace lsnif
