// What the fused 16-bit query kernels' four epilogue warps share: the source
// of tiles (fetched and loaded while the previous tile's layers run), the
// per-tile work lists, and the hidden layers' activations.
//
// These warps set every tile up and run its layers after the first, so their
// time bounds the kernel where a ray has few points: on a million secondary
// rays of the torus network (6.3 points each) they were busy 45 of a tile's
// 52 thousand cycles, 11 of them in the set-up and 34 in the layers, with a
// fifth of their scheduler's issue slots. So the set-up ranks with ballots
// instead of scans, no load is waited for where it is issued, and the
// activations take 4 instructions per value instead of 9: set-up 6 and layers
// 28 thousand cycles, and a tile takes 46.
#pragma once

#include "device.cuh"
#include "tc_common.cuh"

namespace lsnif {
namespace {

constexpr int kFeedThreads = 128;  // the four epilogue warps, named barrier 2

// misc words of the kernels' shared memory that the feed uses
constexpr int kMiscTile = 8;   // [8..10] slot, first row, rows of the next tile
constexpr int kMiscKmax = 12;  // [12..15] largest point count per warp

// A work item is 128 >> shift rows of a tile: with few live rays the grouping
// asks for parts of tiles, so that a small request reaches more SMs.
// The next item is fetched in five steps, each of which only issues loads
// whose values a later step uses; one step runs per layer of the tile before.
template <bool XROWS>
struct TileFeed {
  const QueryLaunch &q;
  volatile int *abort_flag;
  volatile int32_t *misc;
  int64_t xrows;  // XROWS: input rows, and segments of each
  int xk;
  int etid, shift, n_items;
  int stage = 0, idx = 0;
  int slot = 0, start = 0, cnt = 0;  // cnt < 0: no more items
  int ray = -1, kk = 0;
  uint32_t dm = 0u;

  __device__ __forceinline__ TileFeed(const QueryLaunch &q_, volatile int *abort_flag_, volatile int32_t *misc_,
                                      int64_t xrows_, int xk_, int etid_)
      : q(q_), abort_flag(abort_flag_), misc(misc_), xrows(xrows_), xk(xk_), etid(etid_) {
    shift = XROWS ? 0 : q.s.meta[kMetaShift];
    n_items = XROWS ? (int)((xrows + kTileM - 1) / kTileM) : q.s.meta[1] << shift;
  }

  __device__ __forceinline__ void load_item() {  // of item idx < n_items
    const int t = idx >> shift;
    if (XROWS) {
      slot = 0;
      start = t * kTileM;
      cnt = (int)min((int64_t)kTileM, xrows - start);
    } else {
      slot = q.s.tiles[3 * t];
      start = q.s.tiles[3 * t + 1];
      cnt = q.s.tiles[3 * t + 2];
    }
  }

  __device__ __forceinline__ void step() {
    if (stage == 0) {
      if (etid == 0) idx = atomicAdd(q.s.meta + 3, 1);
    } else if (stage == 1) {
      if (etid == 0 && idx < n_items) load_item();
    } else if (stage == 2) {
      if (etid == 0) {
        for (;;) {
          if (idx >= n_items || *abort_flag) {
            cnt = -1;
            break;
          }
          const int rows = kTileM >> shift, part = idx & ((1 << shift) - 1);
          start += part * rows;
          cnt = min(rows, cnt - part * rows);
          if (cnt > 0) break;
          idx = atomicAdd(q.s.meta + 3, 1);  // a part past its tile's rows
          if (idx < n_items) load_item();
        }
        misc[kMiscTile] = slot;
        misc[kMiscTile + 1] = start;
        misc[kMiscTile + 2] = cnt;
      }
    } else if (stage == 3) {  // a barrier lies between the steps 2 and 3
      slot = misc[kMiscTile];
      start = misc[kMiscTile + 1];
      cnt = misc[kMiscTile + 2];
      ray = -1;
      if (etid < cnt) ray = XROWS ? start + etid : q.s.order[start + etid];
    } else if (stage == 4) {
      kk = 0;
      dm = 0u;
      if (ray >= 0) {
        if (XROWS) {
          kk = xk;
        } else {
          kk = q.s.k[ray];
          dm = q.s.dup[ray];
        }
      }
    }
    ++stage;
  }

  // the steps left, so that the item's values are there
  __device__ __forceinline__ void finish() {
    while (stage < 3) step();
    if (stage == 3) named_sync(2, kFeedThreads);
    while (stage < 5) step();
  }
};

// Work lists of a tile, for each chunk s (segment s of its rows): the points to
// gather, entry and exit of every row that has a segment s, without the entry
// points that equal the previous exit (`dup`); in lst, row | exit << 7.
//   masks[4 s + w] = (rows of warp w with a segment s, those whose entry point
//   is the previous exit); counts[s] = points to gather.
// COPIES: the dup rows follow the gathers in lst (for kernels that copy the
// features). Ranks come from two ballots per chunk. Returns the largest
// segment count; the caller publishes the lists behind a barrier.
template <bool COPIES>
__device__ __forceinline__ int build_lists(int etid, int kk, uint32_t dm, uint16_t *lst, uint2 *masks,
                                           int32_t *counts, volatile int32_t *misc, int list_chunks) {
  const int lane = etid & 31, ew = etid >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int wmax = __reduce_max_sync(0xffffffffu, kk);
  for (int s = lane; s < list_chunks; s += 32)  // chunks past this warp's largest count
    if (s >= wmax) masks[s * 4 + ew] = make_uint2(0u, 0u);
  for (int s = 0; s < wmax; ++s) {
    const unsigned ml = __ballot_sync(0xffffffffu, kk > s);
    const unsigned md = __ballot_sync(0xffffffffu, kk > s && s > 0 && ((dm >> s) & 1u));
    if (lane == 0) masks[s * 4 + ew] = make_uint2(ml, md);
  }
  if (lane == 0) misc[kMiscKmax + ew] = wmax;
  named_sync(2, kFeedThreads);
  const int kmax = max(max(misc[kMiscKmax], misc[kMiscKmax + 1]), max(misc[kMiscKmax + 2], misc[kMiscKmax + 3]));
  for (int s = 0; s < kmax; ++s) {
    int first = 0, all = 0, dfirst = 0;  // gathers (and dup rows) of the warps before, and of all
    uint2 mine = make_uint2(0u, 0u);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const uint2 m = masks[s * 4 + w];
      const int d = __popc(m.y), g = 2 * __popc(m.x) - d;
      all += g;
      if (w < ew) {
        first += g;
        dfirst += d;
      }
      if (w == ew) mine = m;
    }
    if (etid == 0) counts[s] = all;
    uint16_t *Ls = lst + s * kListStride;
    if ((mine.x >> lane) & 1u) {
      const int dups = __popc(mine.y & lt), pg = first + 2 * __popc(mine.x & lt) - dups;
      if ((mine.y >> lane) & 1u) {
        Ls[pg] = (uint16_t)(etid | 128);
        if (COPIES) Ls[all + dfirst + dups] = (uint16_t)etid;
      } else {
        Ls[pg] = (uint16_t)etid;
        Ls[pg + 1] = (uint16_t)(etid | 128);
      }
    }
  }
  return kmax;
}

// wait for the TMEM loads in flight; v's users stay behind it
__device__ __forceinline__ void tmem_wait_ld16(uint32_t (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                 "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]));
}

// two FP32 sums in one instruction, each rounded as a scalar sum
__device__ __forceinline__ float2 add2(uint32_t a0, uint32_t a1, float b0, float b1) {
  float2 r;
  asm("{\n.reg .b64 a, b;\nmov.b64 a, {%2, %3};\nmov.b64 b, {%4, %5};\nadd.rn.f32x2 a, a, b;\nmov.b64 {%0, %1}, a;\n}\n"
      : "=f"(r.x), "=f"(r.y)
      : "r"(a0), "r"(a1), "f"(b0), "f"(b1));
  return r;
}

template <bool RELU>
__device__ __forceinline__ float act_as(float x) {
  return RELU ? fmaxf(x, 0.f) : (x > 0.f ? x : 0.01f * x);
}

// A layer's W accumulators of this thread's row -> the next layer's A operand
// in tensor memory: + bias, activation, 16-bit rounding, two values per
// 32-bit column. FP16 saturates at +-65504; BF16 is two-term, hi = BF16(x) at
// tact and lo = BF16(x - hi) (the difference is exact in FP32) at tact_lo.
// The next 16 columns load while these are converted; the activation is
// chosen outside the loop.
template <int W, bool H16, bool RELU>
__device__ __forceinline__ void layer_activations(uint32_t trow, uint32_t tact, uint32_t tact_lo,
                                                  const float *__restrict__ bias) {
  uint32_t v[2][16];
  TMEM_LD16(trow, v[0]);
#pragma unroll
  for (int c = 0; c < W / 16; ++c) {
    tmem_wait_ld16(v[c & 1]);
    if (c + 1 < W / 16) TMEM_LD16(trow + 16 * (c + 1), v[(c + 1) & 1]);
    const uint32_t(&x)[16] = v[c & 1];
    uint32_t hw[8], lw[8];
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      const float4 b = *reinterpret_cast<const float4 *>(bias + 16 * c + 2 * u);
      const float2 s[2] = {add2(x[2 * u], x[2 * u + 1], b.x, b.y), add2(x[2 * u + 2], x[2 * u + 3], b.z, b.w)};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float y0 = act_as<RELU>(s[h].x), y1 = act_as<RELU>(s[h].y);
        if constexpr (H16) {
          const __half2 p = __floats2half2_rn(RELU ? fminf(y0, 65504.f) : fminf(fmaxf(y0, -65504.f), 65504.f),
                                              RELU ? fminf(y1, 65504.f) : fminf(fmaxf(y1, -65504.f), 65504.f));
          hw[u + h] = *reinterpret_cast<const uint32_t *>(&p);
        } else {
          const __nv_bfloat162 hb = __floats2bfloat162_rn(y0, y1);
          hw[u + h] = *reinterpret_cast<const uint32_t *>(&hb);
          const float2 hf = make_float2(__uint_as_float(hw[u + h] << 16), __uint_as_float(hw[u + h] & 0xffff0000u));
          const __nv_bfloat162 lb = __floats2bfloat162_rn(y0 - hf.x, y1 - hf.y);
          lw[u + h] = *reinterpret_cast<const uint32_t *>(&lb);
        }
      }
    }
    TMEM_ST8(tact + (uint32_t)(8 * c), hw);
    if constexpr (!H16) TMEM_ST8(tact_lo + (uint32_t)(8 * c), lw);
  }
}

// The output layer's logits of this thread's row (n_out_pad columns) -> the
// ray's results, or row `ray` of Z.
template <bool XROWS>
__device__ __forceinline__ void store_outputs(const HitsArg &hits, float *Z, uint32_t trow, const float *bias, int ray,
                                              bool on, int n_out, int n_out_pad, int n_mat, float t0, float t1,
                                              float tmin, float tmax) {
  float z[64];
  if (n_out_pad == 16) {  // in registers
    uint32_t v[16];
    TMEM_LD16(trow, v);
    tmem_wait_ld16(v);
    if (!on) return;
#pragma unroll
    for (int u = 0; u < 16; ++u) z[u] = __uint_as_float(v[u]) + bias[u];
    if (XROWS) {
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (j < n_out) Z[(int64_t)ray * n_out + j] = z[j];
    } else {
      decode_store<16>(hits, ray, z, n_out, n_mat, t0, t1, tmin, tmax);
    }
  } else {
#pragma unroll 1
    for (int c0 = 0; c0 < n_out_pad; c0 += 16) {
      uint32_t v[16];
      TMEM_LD16(trow + c0, v);
      tmem_wait_ld16(v);
#pragma unroll
      for (int u = 0; u < 16; ++u) z[c0 + u] = __uint_as_float(v[u]) + bias[c0 + u];
    }
    if (!on) return;
    if (XROWS) {
      for (int j = 0; j < n_out; ++j) Z[(int64_t)ray * n_out + j] = z[j];
    } else {
      decode_store<64>(hits, ray, z, n_out, n_mat, t0, t1, tmin, tmax);
    }
  }
}

}  // namespace
}  // namespace lsnif
