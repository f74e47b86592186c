// Query kernels shared by both precisions (traversal, grouping) and the plain
// FP32 path (gather kernel, SIMT network + decode kernel), plus the stage
// kernels behind lsnif_trace / lsnif_encode / lsnif_corner_indices /
// lsnif_mlp.
#include <algorithm>
#include <cstdio>

#include "device.cuh"
#include "encode.cuh"

namespace lsnif {

// ---------------------------------------------------------------------------
// a1-a5: transform, slab test, 3D-DDA over occupied voxels, boundary points.
// One thread per ray; also histograms live rays by (object slot, k).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) trace_kernel(QueryLaunch q, int smem_hist) {
  extern __shared__ int sh_hist[];
  const int nb = q.n_slots * kBuckets;
  if (smem_hist) {
    for (int i = threadIdx.x; i < nb; i += blockDim.x) sh_hist[i] = 0;
    __syncthreads();
  }
  const int64_t n = q.rays.n;
  const int Hs = q.H_max;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    uint32_t h = q.rays.obj ? q.rays.obj[i] : q.rays.single_handle;
    int s = slot_of(q.objs, q.n_slots, h);
    int k = 0;
    float t0 = CUDART_NAN_F, t1 = CUDART_NAN_F;
    if (s < 0) {
      atomicOr(q.err, kErrBadHandle);
      q.s.slot[i] = -1;
      q.s.k[i] = 0;
      q.s.dup[i] = 0u;
      miss_store(q.hits, i, 0);
      continue;
    }
    const DevObject &ob = q.objs[s];
    float3 o, d;
    int ea;
    uint32_t dupm = 0u;
    float tmin = q.rays.tmin[i];
    bool live = ob.kind == 0 &&
                to_unit(ob, q.rays.ox[i], q.rays.oy[i], q.rays.oz[i], q.rays.dx[i], q.rays.dy[i], q.rays.dz[i], o,
                        d) &&
                unit_slab(o, d, tmin, t0, t1, ea);
    if (live) {
      float *P = q.s.pts + (size_t)i * Hs * 3;
      const int cap = ob.H >> 1;
      const uint32_t *occ = ob.occ;
      // exit of the previous segment: an entry with the same (t, axis, face)
      // is the same point, bit for bit
      uint32_t lt = 0u, lf = 0u;
      int la = -2;
      dda_walk(
          ob, o, d, t0, t1, ea, [&](uint32_t vid) { return occupied(occ, vid); },
          [&](const Seg &sg) {
            if (k > 0 && __float_as_uint(sg.tin) == lt && sg.ain == la && __float_as_uint(sg.fin) == lf)
              dupm |= 1u << k;
            lt = __float_as_uint(sg.tout);
            la = sg.aout;
            lf = __float_as_uint(sg.fout);
            float3 a = seg_point(o, d, sg.tin, sg.ain, sg.fin);
            float3 b = seg_point(o, d, sg.tout, sg.aout, sg.fout);
            float *w = P + 6 * k;
            reinterpret_cast<float2 *>(w)[0] = make_float2(a.x, a.y);
            reinterpret_cast<float2 *>(w)[1] = make_float2(a.z, b.x);
            reinterpret_cast<float2 *>(w)[2] = make_float2(b.y, b.z);
            ++k;
            return k < cap;
          });
    } else {
      t0 = t1 = CUDART_NAN_F;
    }
    q.s.k[i] = (uint8_t)k;
    q.s.dup[i] = dupm;
    q.s.slot[i] = (int16_t)s;
    reinterpret_cast<float2 *>(q.s.t01)[i] = make_float2(t0, t1);
    if (k == 0) miss_store(q.hits, i, ob.n_out);
    if (k > 0) {
      if (smem_hist) atomicAdd(&sh_hist[s * kBuckets + k], 1);
      else atomicAdd(&q.s.counts[s * kBuckets + k], 1);
    }
  }
  if (smem_hist) {
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += blockDim.x)
      if (sh_hist[b]) atomicAdd(&q.s.counts[b], sh_hist[b]);
  }
}

// bits 0..7 of v moved to bits 0, 3, 6, ..., 21
__device__ __forceinline__ uint32_t spread_bits3(uint32_t v) {
  v &= 0xffu;
  v = (v | (v << 8)) & 0x0300f00fu;
  v = (v | (v << 4)) & 0x030c30c3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}

// ---------------------------------------------------------------------------
// Presorted traversal (trace mode 2): before the persistent-lane kernel, a
// counting sort hands it the rays in the order (object, Morton cell of the
// point where the ray enters the object's unit cube, direction octant), so
// the lanes of a warp walk neighbouring voxels in similar directions even
// when the rays arrive shuffled (secondary rays, rays mixed across objects):
// their distance-field and occupancy loads share cache lines and their step
// counts are alike. Rays that miss their box or name an unknown object go to
// one last bin; the traversal answers them as before. The key of each ray
// is kept in q.s.dup (the traversal overwrites it later) and the order in
// q.s.order (the grouping overwrites it later).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t presort_key(const QueryLaunch &q, int64_t i, int key_bits, uint32_t last) {
  const uint32_t h = q.rays.obj ? q.rays.obj[i] : q.rays.single_handle;
  const int s = slot_of(q.objs, q.n_slots, h);
  if (s < 0) return last;
  const DevObject &ob = q.objs[s];
  float3 o, d;
  float t0, t1;
  int ea;
  if (!(ob.kind == 0 && to_unit(ob, q.rays.ox[i], q.rays.oy[i], q.rays.oz[i], q.rays.dx[i], q.rays.dy[i],
                                q.rays.dz[i], o, d) &&
        unit_slab(o, d, q.rays.tmin[i], t0, t1, ea)))
    return last;
  const int m = key_bits / 3 - 1;  // cell bits per axis; 3 bits go to the octant
  const float scale = (float)(1 << m);
  const float e[3] = {fmaf(t0, d.x, o.x), fmaf(t0, d.y, o.y), fmaf(t0, d.z, o.z)};
  uint32_t cell = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const uint32_t c = (uint32_t)min(max((int)(e[a] * scale), 0), (1 << m) - 1);
    cell |= spread_bits3(c) << a;
  }
  const uint32_t oct = (d.x < 0.f ? 1u : 0u) | (d.y < 0.f ? 2u : 0u) | (d.z < 0.f ? 4u : 0u);
  return ((uint32_t)s << key_bits) | (cell << 3) | oct;
}

__global__ void __launch_bounds__(256) presort_count_kernel(QueryLaunch q, int key_bits, uint32_t last) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = i < q.rays.n;
  const uint32_t key = in ? presort_key(q, i, key_bits, last) : 0u;
  if (in) q.s.dup[i] = key;
  const unsigned active = __ballot_sync(0xffffffffu, in);
  if (in) {
    const unsigned peers = __match_any_sync(active, key);
    if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&q.s.bins[key], __popc(peers));
  }
}

__global__ void __launch_bounds__(256) presort_scatter_kernel(QueryLaunch q) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool in = i < q.rays.n;
  const uint32_t key = in ? q.s.dup[i] : 0u;
  const unsigned active = __ballot_sync(0xffffffffu, in);
  if (in) {
    const unsigned peers = __match_any_sync(active, key);
    const int leader = __ffs(peers) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(&q.s.bins[key], __popc(peers));
    base = __shfl_sync(peers, base, leader);
    q.s.order[base + __popc(peers & ((1u << lane) - 1u))] = (int32_t)i;
  }
}

// ---------------------------------------------------------------------------
// Persistent-lane traversal: a lane whose ray finished takes another one, so
// that a warp does not run as long as its longest ray (0 to 3V DDA steps).
//
// Starting rays: a warp takes 32 rays at a time from a global counter, all
// lanes start one each (unit-cube transform, slab test, first voxel -- nine
// divisions), rays that miss their box are answered at once, and the others
// go to a queue in shared memory. Idle lanes pop from the queue. The start
// thus runs with all lanes, which a lane-by-lane refill did not (18 of 32).
//
// Empty-space skipping: every iteration crosses one cell: the cube of
// voxels within Chebyshev distance r of the current voxel, where r + 1 is
// the voxel's distance to the nearest occupied voxel (so the whole cube is
// empty; r = 0 is the voxel itself). All cells are crossed by the same
// instruction sequence (exit plane per axis, earliest axis with the lowest
// axis on ties, cross it), so lanes of a warp do not split between a voxel
// path and a skipping path. Crossing times are the same expression of the
// plane index as in the voxel-by-voxel walk (dda_walk), and when a cube is
// crossed the other axes first step over every plane the walk would cross
// before it, so the voxels visited, the boundary points and the shared-point
// marks are exactly those of the voxel-by-voxel walk (trace_kernel).
//
// What bounds it: instruction issue (75% of the slots; latency when a request
// is small). So voxel and plane indices are FP32 integers (exact: at most
// 1024), a crossing time costs two instructions and no conversion, the three
// axes run one straight-line sequence whatever the crossed axis, the voxel
// after a jump is the floor of a position wherever rounding cannot matter
// (axis_guess), a boundary point is formed once, as one cell's exit and the
// next one's entry, and the lanes that ended write their records together at
// the end of a round. Rounds are long (all lanes' rays end) while the 32 rays
// of a start enter within an eighth of the box, as a camera's do: the lanes
// then stay on neighbouring rays. Otherwise idle lanes take new rays after 16
// cells. On the torus, each measured with the form before (integer indices,
// lane-by-lane refill) and this one: a million rays from a sphere 574 -> 333 us, a million from the
// surface 335 -> 199 us, 4,096 rays 85 -> 48 us, 4.19M camera rays 588 -> 593 us.
// ---------------------------------------------------------------------------
constexpr int kOnceObjects = 32;  // group_at_once_kernel
constexpr int kQueueWords = 14;  // words of a started ray in the queue
constexpr int kShortRound = 16, kLongRound = 256;  // cells between two refills of a warp's idle lanes
constexpr int kTraceWarps = 4;
constexpr int kTraceCtas = 7;    // per SM: 28 warps at 72 registers (32 at 64 spill)

struct LaneRay {
  int i;             // ray (-1: none)
  int s;             // object slot
  float3 o, d;
  float3 inv, sg;    // 1 / d (0 when d is 0), sign of d
  float3 x;          // current voxel
  float3 in;         // boundary point where the ray entered the current cell
  float tcur, t1;
  float clear;       // see axis_guess
  int k, cap;
  float r;           // the current cell: voxels within r of x, all empty when r > 0
  bool occ;          // the current voxel is occupied (its distance is 0)
  bool adj;          // the cell before was an occupied voxel: the point `in` is its exit
  uint32_t dup;      // bit k: entry point of segment k equals the exit of segment k-1
};

__device__ __forceinline__ float sel3(int a, float x, float y, float z) { return a == 0 ? x : (a == 1 ? y : z); }

// crossing time of plane P (an integer) on one axis: the expression dda_walk
// uses (P invV is exact, V being a power of two)
__device__ __forceinline__ float plane_t(float P, float invV, float o, float inv) { return (P * invV - o) * inv; }

// Whether the voxel walk crosses a plane of time t before (ea, a): earlier,
// or at the same time when this axis wins the tie.
__device__ __forceinline__ bool crosses(float t, float ea, bool tie) { return (t < ea) | (tie & (t == ea)); }

// An axis's voxel when the cell is left at time ea through another axis: the
// planes crossed before are a prefix of those ahead (plane times are monotone,
// each operation of plane_t is), at most 2 r of them (r2). The voxel is that of
// the position at ea; `ok` says that the position keeps clear of the planes, so
// that comparing the planes' computed times with ea gives the same voxel:
// plane_t is within 3 x 2^-24 of the true time, relatively, which moves the
// crossing by at most 3 x 2^-24 (1 + |o|) V voxels, and the position has an
// error of 2^-24 (1 + |o|) V; `clear` = 1/2 - 2^-20 (2 + |o|) V leaves four
// times their sum.
__device__ __forceinline__ float axis_guess(float x, float sg, float o, float d, float r2, float V, float ea,
                                            float clear, bool &ok) {
  const float far = fmaf(sg, r2, x);
  const float v = fmaf(ea, d, o) * V, f = floorf(v);
  ok = fabsf((v - f) - 0.5f) < clear;
  return fminf(fmaxf(f, fminf(x, far)), fmaxf(x, far));
}

// the same by search from the guess, comparing plane times
__device__ __noinline__ float axis_search(float g, float x, float sg, float o, float inv, float r, float invV,
                                          float ea, bool tie) {
  const float far = fmaf(2.f * sg, r, x), up = fmaxf(sg, 0.f);
  while (g != x && !crosses(plane_t(g + 1.f - up, invV, o, inv), ea, tie)) g -= sg;
  while (g != far && crosses(plane_t(g + up, invV, o, inv), ea, tie)) g += sg;
  return g;
}

// integer of a whole FP32 value in [0, 2^23)
__device__ __forceinline__ uint32_t whole(float f) { return __float_as_uint(f + 8388608.f) & 0x7fffffu; }

// occupancy distance of voxel x: 0 when occupied, else the radius of the
// empty cube around it is D - 1 (fV: V as FP32; x inside the grid)
__device__ __forceinline__ uint32_t voxel_distance(const uint8_t *dist, uint32_t V, float fV, const float3 &x) {
  return __ldg(dist + (whole(fmaf(x.z, fV, x.y)) * V + whole(x.x)));
}

__device__ __forceinline__ float sign_of(float d) { return d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f); }

__global__ void __launch_bounds__(kTraceWarps * 32, kTraceCtas)
    trace_pool_kernel(QueryLaunch q, int smem_hist, int share, const int32_t *__restrict__ perm) {
  extern __shared__ int sh_hist[];
  __shared__ uint32_t s_queue[kTraceWarps][kQueueWords][32];
  const int nb = q.n_slots * kBuckets;
  if (smem_hist) {
    for (int i = threadIdx.x; i < nb; i += blockDim.x) sh_hist[i] = 0;
    __syncthreads();
  }
  const int64_t n = q.rays.n;
  const int Hs = q.H_max;
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  uint32_t(*sq)[32] = s_queue[threadIdx.x >> 5];
  LaneRay R;
  R.i = -1;
  bool exhausted = false;  // uniform: no rays left to start
  uint32_t next = 0, share_end = 0;  // uniform: rays taken from the counter and not started yet
  int queued = 0;          // uniform: started rays waiting
  int steps = kShortRound; // uniform: cells between two refills
  int *counter = q.s.meta + 4;

  for (;;) {
    // hand a started ray to every idle lane
    for (;;) {
      const unsigned idle = __ballot_sync(FULL, R.i < 0);
      if (!idle || (!queued && exhausted)) break;
      if (!queued) {
        // start the next 32 rays of the warp's share, or of a new one
        if (next == share_end) {
          int base = 0;
          if (lane == 0) base = atomicAdd(counter, share);
          next = (uint32_t)__shfl_sync(FULL, base, 0);
          share_end = next + share;
        }
        const int64_t pos = (int64_t)next + lane;
        next += 32;
        exhausted = (int64_t)next >= n;
        bool live = false, near = false;
        float3 o, d;
        float t0 = CUDART_NAN_F, t1 = CUDART_NAN_F;
        int ea = -1, s = -1, my = 0;
        if (pos < n) {
          my = perm ? __ldg(perm + pos) : (int)pos;  // the pos-th ray of the presorted order, if any
          s = slot_of(q.objs, q.n_slots, q.rays.obj ? q.rays.obj[my] : q.rays.single_handle);
          int n_out = 0;
          if (s < 0) {
            atomicOr(q.err, kErrBadHandle);
          } else {
            const DevObject &ob = q.objs[s];
            n_out = ob.n_out;
            live = ob.kind == 0 &&
                   to_unit(ob, q.rays.ox[my], q.rays.oy[my], q.rays.oz[my], q.rays.dx[my], q.rays.dy[my],
                           q.rays.dz[my], o, d) &&
                   unit_slab(o, d, q.rays.tmin[my], t0, t1, ea);
            if (!live) t0 = t1 = CUDART_NAN_F;
            reinterpret_cast<float2 *>(q.s.t01)[my] = make_float2(t0, t1);
          }
          q.s.slot[my] = (int16_t)s;
          if (!live) {
            q.s.k[my] = 0;
            q.s.dup[my] = 0u;
            miss_store(q.hits, my, n_out);
          }
        }
        const unsigned m = __ballot_sync(FULL, live);
        if (live) {
          const DevObject &ob = q.objs[s];
          const int V = ob.V;
          const float pp[3] = {fmaf(t0, d.x, o.x), fmaf(t0, d.y, o.y), fmaf(t0, d.z, o.z)};
          const float dd[3] = {d.x, d.y, d.z}, oo[3] = {o.x, o.y, o.z};
          const int e = __popc(m & ((1u << lane) - 1u));
          uint32_t cell = 0;
          near = true;
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            int cc = (int)floorf(pp[a] * (float)V);
            cc = min(max(cc, 0), V - 1);
            if (a == ea) cc = dd[a] > 0.f ? 0 : V - 1;
            cell |= (uint32_t)cc << (10 * a);
            // every live lane joins both reductions: V, and with it the verdict,
            // differs between the lanes of a batch that mixes grids
            const int span = __reduce_max_sync(m, cc) - __reduce_min_sync(m, cc);
            near = near & (span * 8 <= V);
            sq[a][e] = __float_as_uint(oo[a]);
            sq[3 + a][e] = __float_as_uint(dd[a]);
            sq[6 + a][e] = __float_as_uint(dd[a] != 0.f ? 1.f / dd[a] : 0.f);
          }
          sq[9][e] = __float_as_uint(t0);
          sq[10][e] = __float_as_uint(t1);
          sq[11][e] = cell;
          sq[12][e] = (uint32_t)my;
          sq[13][e] = (uint32_t)s | ((uint32_t)(ea + 1) << 16);
        }
        queued = __popc(m);
        if (queued) steps = __any_sync(FULL, near) ? kLongRound : kShortRound;
        __syncwarp();
        continue;
      }
      // pop: the j-th idle lane takes the j-th last of the queue
      const int j = __popc(idle & ((1u << lane) - 1u));
      if (R.i < 0 && j < queued) {
        const int e = queued - 1 - j;
        R.o = make_float3(__uint_as_float(sq[0][e]), __uint_as_float(sq[1][e]), __uint_as_float(sq[2][e]));
        R.d = make_float3(__uint_as_float(sq[3][e]), __uint_as_float(sq[4][e]), __uint_as_float(sq[5][e]));
        R.inv = make_float3(__uint_as_float(sq[6][e]), __uint_as_float(sq[7][e]), __uint_as_float(sq[8][e]));
        R.sg = make_float3(sign_of(R.d.x), sign_of(R.d.y), sign_of(R.d.z));
        R.tcur = __uint_as_float(sq[9][e]);
        R.t1 = __uint_as_float(sq[10][e]);
        const uint32_t cell = sq[11][e];
        R.x = make_float3((float)(cell & 1023u), (float)((cell >> 10) & 1023u), (float)(cell >> 20));
        R.i = (int)sq[12][e];
        const uint32_t se = sq[13][e];
        R.s = (int)(se & 0xffffu);
        const int ea = (int)(se >> 16) - 1;
        R.in = seg_point(R.o, R.d, R.tcur, ea,
                         ea >= 0 ? (sel3(ea, R.d.x, R.d.y, R.d.z) > 0.f ? 0.f : 1.f) : 0.f);
        R.adj = false;
        R.k = 0;
        R.dup = 0u;
        const DevObject &ob = q.objs[R.s];
        R.cap = ob.H >> 1;
        const uint32_t V = ob.V;
        R.clear = 0.5f - (fmaxf(fabsf(R.o.x), fmaxf(fabsf(R.o.y), fabsf(R.o.z))) + 2.f) * (float)V * 9.5367431640625e-7f;
        const uint32_t D = voxel_distance(ob.dist, V, (float)V, R.x);
        R.r = fmaxf((float)D - 1.f, 0.f);
        R.occ = D == 0;
      }
      queued = max(queued - __popc(idle), 0);
      __syncwarp();
    }
    if (__all_sync(FULL, R.i < 0)) break;
    if (R.i < 0) continue;
    // up to `steps` cells of this lane's ray
    const DevObject &ob = q.objs[R.s];
    const uint32_t V = ob.V;
    const float invV = ob.invV, fV = (float)V;
    const uint8_t *dist = ob.dist;  // in registers: the stores below could alias the object table
    float *P = q.s.pts + (size_t)R.i * Hs * 3;
    bool done = false;
    for (int it = 0; it < steps && !done; ++it) {
      // exit plane of the cell on each axis, and its crossing time
      const float P0 = fmaf(R.sg.x, R.r, R.x.x) + fmaxf(R.sg.x, 0.f);
      const float P1 = fmaf(R.sg.y, R.r, R.x.y) + fmaxf(R.sg.y, 0.f);
      const float P2 = fmaf(R.sg.z, R.r, R.x.z) + fmaxf(R.sg.z, 0.f);
      const float e0 = R.sg.x != 0.f ? plane_t(P0, invV, R.o.x, R.inv.x) : CUDART_INF_F;
      const float e1 = R.sg.y != 0.f ? plane_t(P1, invV, R.o.y, R.inv.y) : CUDART_INF_F;
      const float e2 = R.sg.z != 0.f ? plane_t(P2, invV, R.o.z, R.inv.z) : CUDART_INF_F;
      const int a = (e0 <= e1) ? (e0 <= e2 ? 0 : 2) : (e1 <= e2 ? 1 : 2);
      const float ea = sel3(a, e0, e1, e2);
      const float tx = fminf(ea, R.t1);
      // the cell's exit point, the next cell's entry
      const float3 out = make_float3(a == 0 ? P0 * invV : fmaf(tx, R.d.x, R.o.x),
                                     a == 1 ? P1 * invV : fmaf(tx, R.d.y, R.o.y),
                                     a == 2 ? P2 * invV : fmaf(tx, R.d.z, R.o.z));
      const bool emit = R.occ & (tx > R.tcur);
      if (emit) {
        float2 *w = reinterpret_cast<float2 *>(P + 6 * R.k);
        w[0] = make_float2(R.in.x, R.in.y);
        w[1] = make_float2(R.in.z, out.x);
        w[2] = make_float2(out.y, out.z);
        R.dup |= (R.adj ? 1u : 0u) << R.k;
        ++R.k;
      }
      R.adj = emit;
      done = (ea >= R.t1) | (R.k >= R.cap);
      if (!done) {
        // The other axes first cross the planes the voxel walk crosses
        // before (ea, a) -- at most 2 r each, none for a voxel -- then axis a
        // crosses its plane. A cube may reach past the grid: an axis whose
        // next plane is the grid's own boundary leaves the grid there, and
        // the voxel walk ends at that crossing (the slab's exit time and the
        // plane's crossing time may round differently), so the ray ends here
        // too -- the cube holds no occupied voxel, so nothing is lost.
        bool ok0, ok1, ok2;
        const float r2 = R.r + R.r;
        float g0 = axis_guess(R.x.x, R.sg.x, R.o.x, R.d.x, r2, fV, ea, R.clear, ok0);
        float g1 = axis_guess(R.x.y, R.sg.y, R.o.y, R.d.y, r2, fV, ea, R.clear, ok1);
        float g2 = axis_guess(R.x.z, R.sg.z, R.o.z, R.d.z, r2, fV, ea, R.clear, ok2);
        if (!((ok0 | (a == 0)) & (ok1 | (a == 1)) & (ok2 | (a == 2)))) {
          if (a != 0) g0 = axis_search(g0, R.x.x, R.sg.x, R.o.x, R.inv.x, R.r, invV, ea, true);
          if (a != 1) g1 = axis_search(g1, R.x.y, R.sg.y, R.o.y, R.inv.y, R.r, invV, ea, a == 2);
          if (a != 2) g2 = axis_search(g2, R.x.z, R.sg.z, R.o.z, R.inv.z, R.r, invV, ea, false);
        }
        // the voxel behind axis a's plane
        R.x.x = a == 0 ? P0 + fminf(R.sg.x, 0.f) : g0;
        R.x.y = a == 1 ? P1 + fminf(R.sg.y, 0.f) : g1;
        R.x.z = a == 2 ? P2 + fminf(R.sg.z, 0.f) : g2;
        done = (fminf(R.x.x, fminf(R.x.y, R.x.z)) < 0.f) | (fmaxf(R.x.x, fmaxf(R.x.y, R.x.z)) >= fV);
        if (!done) {
          R.tcur = ea;
          R.in = out;
          // the next cell is centred on the voxel just entered
          const uint32_t D = voxel_distance(dist, V, fV, R.x);
          R.r = fmaxf(__uint_as_float(0x4b000000u | D) - 8388609.f, 0.f);
          R.occ = D == 0;
        }
      }
    }
    if (done) {  // the lanes that ended in this round, together
      q.s.k[R.i] = (uint8_t)R.k;
      q.s.dup[R.i] = R.dup;
      if (R.k == 0) miss_store(q.hits, R.i, q.objs[R.s].n_out);
      else if (smem_hist) atomicAdd(&sh_hist[R.s * kBuckets + R.k], 1);
      else atomicAdd(&q.s.counts[R.s * kBuckets + R.k], 1);
      R.i = -1;
    }
  }
  if (smem_hist) {
    __syncthreads();
    for (int b = threadIdx.x; b < nb; b += blockDim.x)
      if (sh_hist[b]) atomicAdd(&q.s.counts[b], sh_hist[b]);
  }
}

// Exclusive scan of one value per thread over a block of 1024; `total` is the
// block's sum. ws: 33 words of shared memory, free again when the call returns.
__device__ __forceinline__ int block_scan(int v, int *ws, int &total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) ws[w] = inc;
  __syncthreads();
  if (w == 0) {
    int x = ws[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    ws[lane] = x;
  }
  __syncthreads();
  const int before = (w ? ws[w - 1] : 0) + inc - v;
  total = ws[31];
  __syncthreads();
  return before;
}

// Parts (log2) in which the 16-bit fused kernels work on each tile: 1, 2 or
// 4 of 128, 64 or 32 rows. Their time is a start plus a term per round of the
// chip (the SM with the most parts), and smaller parts have shorter starts and
// rounds but more of them. Measured on the torus network (16 levels), in us:
// 128 rows 35 + 55 per round, 64 rows 25 + 28.5, 32 rows 22 + 17.5 -- so 3,000
// rays take 39 us in 32-row parts and 88 in whole tiles, 20,000 rays 57 in
// 64-row parts and 80 in whole tiles. On the icosphere network (8 levels),
// where the layers weigh more, a smaller part gains less: it has to win by a
// tenth.
__device__ __forceinline__ int tile_shift(int n_live, int sms) {
  auto rounds = [&](int rows) { return (n_live + rows * sms - 1) / (rows * sms); };
  if (rounds(128) > 4) return 0;
  const int c0 = 350 + 550 * rounds(128), c1 = 275 + 313 * rounds(64), c2 = 242 + 192 * rounds(32);
  return c2 < c1 && c2 < c0 ? 2 : (c1 < c0 ? 1 : 0);
}

// A block of 1024: totals and the tile table from the objects' ranges in the
// order. first[s]: start of object s (the end of the last is set here); pts:
// this thread's share of the point count; tile_off, ws: shared scratch.
__device__ __forceinline__ void write_tiles(const QueryLaunch &q, int run, int pts, int *first, int *tile_off, int *ws) {
  const int ns = q.n_slots;
  int points;
  block_scan(pts, ws, points);  // also a barrier: first[] is written
  if (threadIdx.x == 0) first[ns] = run;
  __syncthreads();
  const int live = (int)threadIdx.x < ns ? first[threadIdx.x + 1] - first[threadIdx.x] : 0;
  int tiles;
  const int tile0 = block_scan((live + kTileM - 1) / kTileM, ws, tiles);
  if ((int)threadIdx.x < ns) tile_off[threadIdx.x] = tile0;
  if (tiles > q.s.max_tiles) {
    if (threadIdx.x == 0) atomicOr(q.err, kErrCheck);
    tiles = q.s.max_tiles;
  }
  if (threadIdx.x == 0) {
    q.s.meta[0] = run;
    q.s.meta[1] = tiles;
    q.s.meta[2] = points;
    q.s.meta[3] = 0;
    q.s.meta[kMetaShift] = tile_shift(run, q.sms);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < tiles; t += blockDim.x) {
    // object of tile t: last s with tile_off[s] <= t
    int lo = 0, hi = ns - 1;
    while (lo < hi) {
      int mid = (lo + hi + 1) >> 1;
      if (tile_off[mid] <= t) lo = mid; else hi = mid - 1;
    }
    const int start = first[lo] + (t - tile_off[lo]) * kTileM;
    q.s.tiles[3 * t + 0] = lo;
    q.s.tiles[3 * t + 1] = start;
    q.s.tiles[3 * t + 2] = min(kTileM, first[lo + 1] - start);
  }
}

// Single block: bucket offsets (object ascending, k descending), tiles of
// kTileM rays that never straddle objects, totals, cursors reset. A warp takes
// one object's 32 buckets at a time, so an object's range starts at the value
// its lane 0 scans to. One thread walking the buckets (a load per bucket, none
// in flight beside another) took 9.8 us on six objects; this takes 5.2.
__global__ void __launch_bounds__(1024) scan_kernel(QueryLaunch q) {
  __shared__ int ws[33];
  __shared__ int first[kMaxObjects + 1];     // start of each object's range
  __shared__ int tile_off[kMaxObjects + 1];  // and its first tile
  const int ns = q.n_slots;
  static_assert(kMaxCap == 32, "a warp per object");
  int run = 0, pts = 0;
  for (int base = 0; base < ns * kMaxCap; base += 1024) {
    const int s = (base + (int)threadIdx.x) >> 5, k = kMaxCap - (threadIdx.x & 31);
    const int c = s < ns ? q.s.counts[s * kBuckets + k] : 0;
    int total;
    const int at = run + block_scan(c, ws, total);
    // group modes 2 and 3: one bucket per object (bucket k = 1 takes all)
    const int start = __shfl_sync(0xffffffffu, at, 0);
    if (s < ns) {
      q.s.offsets[s * kBuckets + k] = q.group_mode >= 2 ? start : at;
      q.s.cursor[s * kBuckets + k] = 0;
      if (k == kMaxCap) first[s] = at;
    }
    pts += 2 * k * c;
    run += total;
  }
  write_tiles(q, run, pts, first, tile_off, ws);
}

// Scatter live rays into their bucket ranges; warp-aggregated atomics keep
// rays of one warp contiguous (spatially coherent rays stay together). In
// group mode 2 a bucket is a whole object (point counts mixed), so
// consecutive rays of an object stay close in the tile order.
__global__ void __launch_bounds__(256) scatter_kernel(QueryLaunch q) {
  const int64_t n = q.rays.n;
  const int lane = threadIdx.x & 31;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += (int64_t)gridDim.x * blockDim.x) {
    int64_t i = base + threadIdx.x;
    int bucket = -1;
    if (i < n) {
      int k = q.s.k[i];
      int s = q.s.slot[i];
      if (k > 0 && s >= 0) bucket = s * kBuckets + (q.group_mode == 2 ? 1 : k);
    }
    unsigned active = __ballot_sync(0xffffffffu, bucket >= 0);
    if (bucket >= 0) {
      unsigned peers = __match_any_sync(active, bucket);
      int leader = __ffs(peers) - 1;
      int rank = __popc(peers & ((1u << lane) - 1u));
      int basep = 0;
      if (lane == leader) basep = atomicAdd(&q.s.cursor[bucket], __popc(peers));
      basep = __shfl_sync(peers, basep, leader);
      q.s.order[q.s.offsets[bucket] + basep + rank] = (int32_t)i;
    }
  }
}

// The same with each block's counts summed in shared memory first: one
// global atomic per block and bucket instead of one per warp and bucket (a
// query's few buckets otherwise take every warp's atomics). One ray per
// thread; nb = n_slots x kBuckets counts and as many block bases in shared
// memory.
__global__ void __launch_bounds__(1024) scatter_block_kernel(QueryLaunch q, int nb) {
  extern __shared__ int sh_scatter[];
  int *s_cnt = sh_scatter, *s_base = sh_scatter + nb;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) s_cnt[b] = 0;
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  int bucket = -1;
  if (i < q.rays.n) {
    const int k = q.s.k[i];
    const int s = q.s.slot[i];
    if (k > 0 && s >= 0) bucket = s * kBuckets + (q.group_mode == 2 ? 1 : k);
  }
  const unsigned active = __ballot_sync(0xffffffffu, bucket >= 0);
  int rank = 0;
  if (bucket >= 0) {
    const unsigned peers = __match_any_sync(active, bucket);
    const int leader = __ffs(peers) - 1;
    int wbase = 0;
    if (lane == leader) wbase = atomicAdd(&s_cnt[bucket], __popc(peers));
    wbase = __shfl_sync(peers, wbase, leader);
    rank = wbase + __popc(peers & ((1u << lane) - 1u));
  }
  __syncthreads();
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    const int c = s_cnt[b];
    s_base[b] = c ? atomicAdd(&q.s.cursor[b], c) : 0;
  }
  __syncthreads();
  if (bucket >= 0) q.s.order[q.s.offsets[bucket] + s_base[bucket] + rank] = (int32_t)i;
}

// scan_kernel and scatter_block_kernel in one launch, for at most 32 objects:
// every block scans the few counts itself, the first one writes the totals and
// the tile table. The cursors were cleared with the counts (group_at_once).
// Both launches against this one, between events: 4,096 to 100,000 rays 10.9 ->
// 8.8 us, 300,000 14.5 -> 8.9, a million 22.7 -> 17.5, 4.19M 37.5 -> 31.3; the
// query of 4,096 icosphere rays 57.2 -> 54.5 us. More objects than a block's
// 1,024 threads have buckets for take the two launches.
__global__ void __launch_bounds__(1024) group_at_once_kernel(QueryLaunch q) {
  constexpr int NB = kOnceObjects * kBuckets;
  __shared__ int ws[33], first[kOnceObjects + 1], tile_off[kOnceObjects + 1], s_cnt[NB], s_base[NB];
  const int ns = q.n_slots, tid = threadIdx.x, lane = tid & 31;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + tid;
  int bucket = -1;
  if (i < q.rays.n) {
    const int k = q.s.k[i];
    const int s = q.s.slot[i];
    if (k > 0 && s >= 0) bucket = s * kBuckets + (q.group_mode == 2 ? 1 : k);
  }
  static_assert(kMaxCap == 32 && kOnceObjects * kMaxCap == 1024, "a warp per object, all objects at once");
  const int so = tid >> 5, k = kMaxCap - lane;
  const int c = so < ns ? q.s.counts[so * kBuckets + k] : 0;
  for (int b = tid; b < ns * kBuckets; b += blockDim.x) s_cnt[b] = 0;
  int run;
  const int at = block_scan(c, ws, run);
  const int start = __shfl_sync(0xffffffffu, at, 0);
  if (so < ns) {
    s_base[so * kBuckets + k] = q.group_mode >= 2 ? start : at;
    if (lane == 0) first[so] = at;
  }
  const unsigned active = __ballot_sync(0xffffffffu, bucket >= 0);
  int rank = 0;
  if (bucket >= 0) {
    const unsigned peers = __match_any_sync(active, bucket);
    const int leader = __ffs(peers) - 1;
    int wbase = 0;
    if (lane == leader) wbase = atomicAdd(&s_cnt[bucket], __popc(peers));
    wbase = __shfl_sync(peers, wbase, leader);
    rank = wbase + __popc(peers & ((1u << lane) - 1u));
  }
  __syncthreads();
  for (int b = tid; b < ns * kBuckets; b += blockDim.x)
    if (s_cnt[b]) s_base[b] += atomicAdd(&q.s.cursor[b], s_cnt[b]);
  __syncthreads();
  if (bucket >= 0) q.s.order[s_base[bucket] + rank] = (int32_t)i;
  if (blockIdx.x == 0) write_tiles(q, run, 2 * k * c, first, tile_off, ws);
}

// ---------------------------------------------------------------------------
// Order-keeping grouping for single-object queries: live rays are compacted
// in their original order, so a 128-ray tile holds neighbouring rays (for
// primary rays: neighbouring pixels, which share voxels and lattice cells).
// count: live rays and points per block of kGroupBlock rays; scan: block
// offsets, totals and the tile table; scatter: stable ranks within a block.
// ---------------------------------------------------------------------------
// The point counts of this thread's four rays (0 past n). A ray of an unknown
// object has k = 0, so the slot is not needed.
__device__ __forceinline__ uchar4 group_counts(const QueryLaunch &q) {
  static_assert(kGroupBlock == 4096, "four rays per thread");
  const int64_t i = (int64_t)blockIdx.x * kGroupBlock + 4 * threadIdx.x;
  if (i + 4 <= q.rays.n) return *reinterpret_cast<const uchar4 *>(q.s.k + i);
  uchar4 k = make_uchar4(0, 0, 0, 0);
  if (i < q.rays.n) k.x = q.s.k[i];
  if (i + 1 < q.rays.n) k.y = q.s.k[i + 1];
  if (i + 2 < q.rays.n) k.z = q.s.k[i + 2];
  return k;
}

__global__ void __launch_bounds__(1024) group_count_kernel(QueryLaunch q, int nblk) {
  __shared__ int ws[33];
  const uchar4 k = group_counts(q);
  int live, pts;
  block_scan((k.x > 0) + (k.y > 0) + (k.z > 0) + (k.w > 0), ws, live);
  block_scan(2 * (k.x + k.y + k.z + k.w), ws, pts);
  if (threadIdx.x == 0) {
    q.s.blk[blockIdx.x] = live;
    q.s.blk[nblk + blockIdx.x] = pts;
  }
}

__global__ void __launch_bounds__(1024) group_scan_kernel(QueryLaunch q, int nblk) {
  __shared__ int ws[33];
  const int per = (nblk + 1023) / 1024;
  const int b0 = threadIdx.x * per;
  int sum = 0, pts = 0;
  for (int b = b0; b < min(b0 + per, nblk); ++b) { sum += q.s.blk[b]; pts += q.s.blk[nblk + b]; }
  int n_live, points;
  int run = block_scan(sum, ws, n_live);
  block_scan(pts, ws, points);
  int tiles = (n_live + kTileM - 1) / kTileM;
  if (tiles > q.s.max_tiles) {
    if (threadIdx.x == 0) atomicOr(q.err, kErrCheck);
    tiles = q.s.max_tiles;
  }
  if (threadIdx.x == 0) {
    q.s.meta[0] = n_live;
    q.s.meta[1] = tiles;
    q.s.meta[2] = points;
    q.s.meta[3] = 0;
    q.s.meta[kMetaShift] = tile_shift(n_live, q.sms);
  }
  for (int b = b0; b < min(b0 + per, nblk); ++b) {   // block offsets replace the counts
    const int v = q.s.blk[b];
    q.s.blk[b] = run;
    run += v;
  }
  for (int t = threadIdx.x; t < tiles; t += blockDim.x) {
    q.s.tiles[3 * t + 0] = q.single_slot;
    q.s.tiles[3 * t + 1] = t * kTileM;
    q.s.tiles[3 * t + 2] = min(kTileM, n_live - t * kTileM);
  }
}

__global__ void __launch_bounds__(1024) group_scatter_kernel(QueryLaunch q) {
  __shared__ int ws[33];
  const uchar4 k = group_counts(q);
  int total;
  int at = q.s.blk[blockIdx.x] + block_scan((k.x > 0) + (k.y > 0) + (k.z > 0) + (k.w > 0), ws, total);
  const int32_t i = (int32_t)((int64_t)blockIdx.x * kGroupBlock + 4 * threadIdx.x);
  if (k.x) q.s.order[at++] = i;
  if (k.y) q.s.order[at++] = i + 1;
  if (k.z) q.s.order[at++] = i + 2;
  if (k.w) q.s.order[at++] = i + 3;
}

// exclusive scan of n int32 in place, in blocks of 1024; block totals to sums
__global__ void __launch_bounds__(1024) scan_block_kernel(int32_t *v, int64_t n, int32_t *sums) {
  __shared__ int32_t ws[32];
  const int64_t i = (int64_t)blockIdx.x * 1024 + threadIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int32_t x = i < n ? v[i] : 0;
  int32_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) ws[w] = inc;
  __syncthreads();
  if (w == 0) {
    int32_t s = ws[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    ws[lane] = s;
  }
  __syncthreads();
  const int32_t before = (w > 0 ? ws[w - 1] : 0) + inc - x;
  if (i < n) v[i] = before;
  if (threadIdx.x == 1023) sums[blockIdx.x] = ws[31];
}

// single block: exclusive scan of the block sums (any count), total at sums[nb]
__global__ void __launch_bounds__(1024) scan_sums_kernel(int32_t *sums, int nb) {
  __shared__ int32_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __shared__ int32_t ws[32];
  for (int base = 0; base < nb; base += 1024) {
    const int i = base + threadIdx.x;
    const int32_t x = i < nb ? sums[i] : 0;
    int32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) ws[w] = inc;
    __syncthreads();
    if (w == 0) {
      int32_t s = ws[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
      }
      ws[lane] = s;
    }
    __syncthreads();
    const int32_t before = carry + (w > 0 ? ws[w - 1] : 0) + inc - x;
    if (i < nb) sums[i] = before;
    __syncthreads();
    if (threadIdx.x == 0) carry += ws[31];
    __syncthreads();
  }
  if (threadIdx.x == 0) sums[nb] = carry;
}

__global__ void scan_add_kernel(int32_t *v, int64_t n, const int32_t *sums) {
  const int64_t i = (int64_t)blockIdx.x * 1024 + threadIdx.x;
  if (i < n) v[i] += sums[blockIdx.x];
}

// ---------------------------------------------------------------------------
// Spatial grouping (group mode 3): live rays sorted by object, then by the
// Morton code of the cell (2^m per axis of the object's unit cube) that
// holds their first boundary point -- a counting sort over (object, cell)
// bins: count, exclusive scan, scatter. A 128-ray tile then holds rays whose
// points lie close together whatever order the rays came in (secondary
// rays, rays shuffled across objects), so the gathers' corner loads share
// L1 and L2 lines. Objects stay in ascending slot order, so the object
// ranges and tiles of scan_kernel (one bucket per object) hold as they are.
// Rays of one bin land in any order; no result depends on it.
// ---------------------------------------------------------------------------
// (object slot, Morton cell) bin of ray i, or -1 when it is not live
__device__ __forceinline__ int spatial_bin(const QueryLaunch &q, int64_t i, int cell_bits) {
  if (q.s.k[i] == 0) return -1;
  const int s = q.s.slot[i];
  if (s < 0) return -1;
  const float *P = q.s.pts + (size_t)i * q.H_max * 3;
  const int side = 1 << (cell_bits / 3);
  const float scale = (float)side;
  uint32_t c[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) c[a] = (uint32_t)min(max((int)(P[a] * scale), 0), side - 1);
  return (s << cell_bits) | (int)(spread_bits3(c[0]) | (spread_bits3(c[1]) << 1) | (spread_bits3(c[2]) << 2));
}

__global__ void __launch_bounds__(256) spatial_count_kernel(QueryLaunch q, int cell_bits) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int bin = i < q.rays.n ? spatial_bin(q, i, cell_bits) : -1;
  const unsigned active = __ballot_sync(0xffffffffu, bin >= 0);
  if (bin >= 0) {
    const unsigned peers = __match_any_sync(active, bin);
    if ((int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&q.s.bins[bin], __popc(peers));
  }
}

// bins hold the bins' first positions; each warp takes its rays' ranks
__global__ void __launch_bounds__(256) spatial_scatter_kernel(QueryLaunch q, int cell_bits) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const int bin = i < q.rays.n ? spatial_bin(q, i, cell_bits) : -1;
  const unsigned active = __ballot_sync(0xffffffffu, bin >= 0);
  if (bin >= 0) {
    const unsigned peers = __match_any_sync(active, bin);
    const int leader = __ffs(peers) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(&q.s.bins[bin], __popc(peers));
    base = __shfl_sync(peers, base, leader);
    q.s.order[base + __popc(peers & ((1u << lane) - 1u))] = (int32_t)i;
  }
}

// ---------------------------------------------------------------------------
// FP32 path: gather into X, one chunk of tiles at a time. Row (t, r) of the
// chunk is ray r of tile t; the row stride is the largest input width.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void encode_level_any(const DevObject &ob, const float *tab, const float3 &p, int l,
                                                 float *out) {
  const float *tl = tab + (size_t)l * (ob.mask + 1) * ob.F;
  const float N = (float)ob.res[l];
  if (ob.F == 2) {
    float f[2];
    encode_level<float, 2>(tl, ob.mask, p, N, f);
    out[0] = f[0]; out[1] = f[1];
  } else if (ob.F == 4) {
    float f[4];
    encode_level<float, 4>(tl, ob.mask, p, N, f);
    out[0] = f[0]; out[1] = f[1]; out[2] = f[2]; out[3] = f[3];
  } else {
    float f[1];
    encode_level<float, 1>(tl, ob.mask, p, N, f);
    out[0] = f[0];
  }
}

__global__ void __launch_bounds__(256) gather_fp32_kernel(QueryLaunch q, int tile0, int ntile, int ldx) {
  const int Hs = q.H_max;
  const int64_t tot = (int64_t)ntile * kTileM * Hs;
  const int n_tiles = q.s.meta[1];
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int h = (int)(e % Hs);
    const int64_t rr = e / Hs;
    const int r = (int)(rr % kTileM);
    const int t = tile0 + (int)(rr / kTileM);
    if (t >= n_tiles) continue;
    const int slot = q.s.tiles[3 * t], start = q.s.tiles[3 * t + 1], cnt = q.s.tiles[3 * t + 2];
    if (r >= cnt) continue;
    const DevObject &ob = q.objs[slot];
    if (h >= ob.H) continue;
    const int32_t ray = q.s.order[start + r];
    const int k = q.s.k[ray];
    const int LF = ob.L * ob.F;
    float *xo = q.s.X + ((int64_t)(t - tile0) * kTileM + r) * ldx + (size_t)h * LF;
    if (h >= 2 * k) {
      for (int j = 0; j < LF; ++j) xo[j] = 0.f;
      continue;
    }
    const float *P = q.s.pts + ((size_t)ray * Hs + h) * 3;
    const float3 p = make_float3(P[0], P[1], P[2]);
    for (int l = 0; l < ob.L; ++l) encode_level_any(ob, ob.tab32, p, l, xo + l * ob.F);
  }
}

// ---------------------------------------------------------------------------
// FP32 SIMT network: 128-row tiles, activations stay in shared memory
// between layers; decode in the epilogue.
// ---------------------------------------------------------------------------
constexpr int kMT = kTileM;  // rows per tile
constexpr int kKC = 32;      // K chunk

// out[N][kMT] = act(W[N][K] . in + b); in is global rows (Xg, stride ldx,
// rows_valid valid) or shared [K][kMT].
template <int CPT>
__device__ __forceinline__ void simt_layer(const float *__restrict__ Ain, const float *__restrict__ Xg, int64_t ldx,
                                           int rows_valid, int K, int N, const float *__restrict__ W,
                                           const float *__restrict__ bias, int act, bool apply_act, float *As,
                                           float *Ws, float *Aout) {
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;  // 16 column groups x 16 row groups of 8
  float acc[8][CPT];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < CPT; ++j) acc[i][j] = 0.f;
  for (int kc = 0; kc < K; kc += kKC) {
    const int kn = min(kKC, K - kc);
    __syncthreads();
    if (Xg) {
      for (int e = tid; e < kMT * kKC; e += blockDim.x) {
        const int r = e / kKC, kk = e % kKC;
        As[kk * kMT + r] = (r < rows_valid && kk < kn) ? Xg[(int64_t)r * ldx + kc + kk] : 0.f;
      }
    }
    for (int e = tid; e < kKC * N; e += blockDim.x) {
      const int nn = e / kKC, kk = e % kKC;
      Ws[kk * N + nn] = kk < kn ? W[(int64_t)nn * K + kc + kk] : 0.f;
    }
    __syncthreads();
    const float *A = Xg ? As : (Ain + (size_t)kc * kMT);
    for (int kk = 0; kk < kn; ++kk) {
      float a[8], b[CPT];
#pragma unroll
      for (int i = 0; i < 8; ++i) a[i] = A[kk * kMT + ty * 8 + i];
#pragma unroll
      for (int j = 0; j < CPT; ++j) b[j] = Ws[kk * N + tx * CPT + j];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < CPT; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < CPT; ++j) {
    const int col = tx * CPT + j;
    const float bj = bias[col];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float v = acc[i][j] + bj;
      Aout[col * kMT + ty * 8 + i] = apply_act ? act_fn(v, act) : v;
    }
  }
  __syncthreads();
}

__device__ void simt_dispatch(int N, const float *Ain, const float *Xg, int64_t ldx, int rows_valid, int K,
                              const float *W, const float *bias, int act, bool apply_act, float *As, float *Ws,
                              float *Aout) {
  switch (N / 16) {
    case 1: simt_layer<1>(Ain, Xg, ldx, rows_valid, K, N, W, bias, act, apply_act, As, Ws, Aout); break;
    case 2: simt_layer<2>(Ain, Xg, ldx, rows_valid, K, N, W, bias, act, apply_act, As, Ws, Aout); break;
    case 3: simt_layer<3>(Ain, Xg, ldx, rows_valid, K, N, W, bias, act, apply_act, As, Ws, Aout); break;
    case 4: simt_layer<4>(Ain, Xg, ldx, rows_valid, K, N, W, bias, act, apply_act, As, Ws, Aout); break;
    case 8: simt_layer<8>(Ain, Xg, ldx, rows_valid, K, N, W, bias, act, apply_act, As, Ws, Aout); break;
    case 16: simt_layer<16>(Ain, Xg, ldx, rows_valid, K, N, W, bias, act, apply_act, As, Ws, Aout); break;
    default: {
      // other multiples of 16: generic path, 1 column group at a time
      for (int n0 = 0; n0 < N; n0 += 16)
        simt_layer<1>(Ain, Xg, ldx, rows_valid, K, 16, W + (int64_t)n0 * K, bias + n0, act, apply_act, As, Ws,
                      Aout + (size_t)n0 * kMT);
    }
  }
}

// One tile's network from its input rows X (stride ldx, `rows` valid) into
// logits out[n_out_pad][kMT] (a shared buffer); returns that buffer.
__device__ float *simt_network(const DevObject &ob, const float *X, int64_t ldx, int rows, float *As, float *Ws,
                               float *act0, float *act1) {
  const int W = ob.width;
  const float *p = ob.mlp32;
  simt_dispatch(W, nullptr, X, ldx, rows, ob.n_in, p, p + (size_t)W * ob.n_in, ob.act, true, As, Ws, act0);
  p += (size_t)W * ob.n_in + W;
  float *cur = act0, *nxt = act1;
  for (int l = 1; l < ob.n_hidden; ++l) {
    simt_dispatch(W, cur, nullptr, 0, kMT, W, p, p + (size_t)W * W, ob.act, true, As, Ws, nxt);
    p += (size_t)W * W + W;
    float *tmp = cur; cur = nxt; nxt = tmp;
  }
  // output layer, padded to n_out_pad rows (zero weights) by the launcher's copy
  const float *Wo = ob.plain_out, *bo = ob.plain_out + (size_t)ob.n_out_pad * W;
  simt_dispatch(ob.n_out_pad, cur, nullptr, 0, kMT, W, Wo, bo, ob.act, false, As, Ws, nxt);
  return nxt;
}

__global__ void __launch_bounds__(256) mlp_fp32_kernel(QueryLaunch q, int tile0, int ntile, int ldx) {
  extern __shared__ __align__(16) float sm[];
  const int wmax = q.s.wmax;
  float *As = sm;
  float *Ws = As + kKC * kMT;
  float *act0 = Ws + kKC * wmax;
  float *act1 = act0 + (size_t)wmax * kMT;
  const int n_tiles = q.s.meta[1];
  for (int tt = blockIdx.x; tt < ntile; tt += gridDim.x) {
    const int t = tile0 + tt;
    if (t >= n_tiles) break;
    const int slot = q.s.tiles[3 * t], start = q.s.tiles[3 * t + 1], cnt = q.s.tiles[3 * t + 2];
    const DevObject &ob = q.objs[slot];
    float *Z = simt_network(ob, q.s.X + (int64_t)tt * kMT * ldx, ldx, cnt, As, Ws, act0, act1);
    if (threadIdx.x < cnt) {
      const int r = threadIdx.x;
      float z[64];
      for (int j = 0; j < ob.n_out; ++j) z[j] = Z[j * kMT + r];
      const int32_t ray = q.s.order[start + r];
      const float2 tt01 = reinterpret_cast<const float2 *>(q.s.t01)[ray];
      decode_store(q.hits, ray, z, ob.n_out, ob.n_mat, tt01.x, tt01.y, q.rays.tmin[ray], q.rays.tmax[ray]);
    }
    __syncthreads();
  }
}

// lsnif_mlp, FP32: X rows in, logits out.
__global__ void __launch_bounds__(256) mlp_fp32_rows_kernel(const DevObject *dobj, const float *X, int64_t n,
                                                            float *Zout, int wmax) {
  extern __shared__ __align__(16) float sm[];
  const DevObject &ob = *dobj;
  float *As = sm;
  float *Ws = As + kKC * kMT;
  float *act0 = Ws + kKC * wmax;
  float *act1 = act0 + (size_t)wmax * kMT;
  for (int64_t t0 = (int64_t)blockIdx.x * kMT; t0 < n; t0 += (int64_t)gridDim.x * kMT) {
    const int rv = (int)min((int64_t)kMT, n - t0);
    float *Z = simt_network(ob, X + t0 * ob.n_in, ob.n_in, rv, As, Ws, act0, act1);
    if (threadIdx.x < rv)
      for (int j = 0; j < ob.n_out; ++j) Zout[(t0 + threadIdx.x) * ob.n_out + j] = Z[j * kMT + threadIdx.x];
    __syncthreads();
  }
}

constexpr int kMlpSmemMax = 232448;  // all a CTA may have
static size_t mlp_fp32_smem(int wmax) {
  return sizeof(float) * ((size_t)kKC * kMT + (size_t)kKC * wmax + 2 * (size_t)wmax * kMT);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static int grid_for(int64_t n, int threads, int cap) {
  int64_t g = (n + threads - 1) / threads;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (int)g;
}

// the CTAs that are resident at once
static int trace_pool_grid(int64_t n, int sms) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + kTraceWarps * 32 - 1) / (kTraceWarps * 32), (int64_t)sms * kTraceCtas));
}

// Rays a warp takes from the counter at once: 32, and up to 256 where each
// warp starts at least 8 such shares (fewer atomics on one address; within
// 2% of 32 at every size timed).
static int trace_pool_share(int64_t n, int grid) {
  return 32 * (int)std::max<int64_t>(1, std::min<int64_t>(8, n / ((int64_t)grid * kTraceWarps * 32 * 8)));
}

// The counters, the histogram and the cursors lie together in the queries'
// scratch and are cleared in one operation, up to the cursors where the
// grouping at once needs them cleared.
static bool group_at_once(const QueryLaunch &q) {
  return q.s.counts == q.s.meta + kMetaWords && q.s.cursor > q.s.counts && q.s.cursor - q.s.meta < (1 << 14) &&
         q.group_mode != 1 && q.group_mode != 3 && q.n_slots <= kOnceObjects;
}

cudaError_t launch_trace(const QueryLaunch &q, int *launches) {
  const int nb = q.n_slots * kBuckets;
  // the counters and the histogram, in one operation where they lie together
  const bool joined = q.s.counts == q.s.meta + kMetaWords;
  const size_t words = group_at_once(q) ? q.s.cursor - q.s.meta + nb : nb + (joined ? kMetaWords : 0);
  cudaError_t e0 = cudaMemsetAsync(joined ? q.s.meta : q.s.counts, 0, sizeof(int32_t) * words, q.stream);
  if (e0 == cudaSuccess && !joined) e0 = cudaMemsetAsync(q.s.meta + 4, 0, sizeof(int32_t), q.stream);
  if (e0 != cudaSuccess) return e0;
  const int smem_hist = nb <= 12288;
  const size_t smem = smem_hist ? nb * sizeof(int) : 0;
  if (q.trace_mode != 0 && smem > (32 << 10)) {  // with the queue, past the 48 KiB a launch may use unasked
    const cudaError_t e =
        cudaFuncSetAttribute(trace_pool_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 48 << 10);
    if (e != cudaSuccess) return e;
  }
  if (q.trace_mode == 1) {
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int grid = trace_pool_grid(q.rays.n, sms);
    trace_pool_kernel<<<grid, kTraceWarps * 32, smem, q.stream>>>(q, smem_hist, trace_pool_share(q.rays.n, grid), nullptr);
    *launches += 1;
    return cudaGetLastError();
  }
  if (q.trace_mode == 2) {
    const int key_bits = spatial_cell_bits(q.n_slots);
    const uint32_t last = (uint32_t)q.n_slots << key_bits;  // rays the traversal answers as misses
    const int64_t nbins = (int64_t)last + 1;
    const unsigned blocks = (unsigned)std::max<int64_t>((q.rays.n + 255) / 256, 1);
    cudaError_t e = cudaMemsetAsync(q.s.bins, 0, (size_t)nbins * 4, q.stream);
    if (e != cudaSuccess) return e;
    presort_count_kernel<<<blocks, 256, 0, q.stream>>>(q, key_bits, last);
    e = launch_exclusive_scan(q.s.bins, nbins, q.s.bin_sums, q.stream);
    if (e != cudaSuccess) return e;
    presort_scatter_kernel<<<blocks, 256, 0, q.stream>>>(q);
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int grid = trace_pool_grid(q.rays.n, sms);
    trace_pool_kernel<<<grid, kTraceWarps * 32, smem, q.stream>>>(q, smem_hist, trace_pool_share(q.rays.n, grid), q.s.order);
    *launches += 6;
    return cudaGetLastError();
  }
  const int grid = grid_for(q.rays.n, 256, 152 * 16);
  trace_kernel<<<grid, 256, smem, q.stream>>>(q, smem_hist);
  *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_group(const QueryLaunch &q, int *launches) {
  if (q.group_mode == 1) {
    const int nblk = (int)((q.rays.n + kGroupBlock - 1) / kGroupBlock);
    group_count_kernel<<<nblk, 1024, 0, q.stream>>>(q, nblk);
    group_scan_kernel<<<1, 1024, 0, q.stream>>>(q, nblk);
    group_scatter_kernel<<<nblk, 1024, 0, q.stream>>>(q);
    *launches += 3;
    return cudaGetLastError();
  }
  if (q.group_mode == 3) {
    const int bits = spatial_cell_bits(q.n_slots);
    const int64_t nbins = (int64_t)q.n_slots << bits;
    const unsigned blocks = (unsigned)std::max<int64_t>((q.rays.n + 255) / 256, 1);
    scan_kernel<<<1, 1024, 0, q.stream>>>(q);
    cudaError_t e = cudaMemsetAsync(q.s.bins, 0, (size_t)nbins * 4, q.stream);
    if (e != cudaSuccess) return e;
    spatial_count_kernel<<<blocks, 256, 0, q.stream>>>(q, bits);
    e = launch_exclusive_scan(q.s.bins, nbins, q.s.bin_sums, q.stream);
    if (e != cudaSuccess) return e;
    spatial_scatter_kernel<<<blocks, 256, 0, q.stream>>>(q, bits);
    *launches += 6;
    return cudaGetLastError();
  }
  if (group_at_once(q)) {
    group_at_once_kernel<<<(unsigned)std::max<int64_t>((q.rays.n + 1023) / 1024, 1), 1024, 0, q.stream>>>(q);
    *launches += 1;
    return cudaGetLastError();
  }
  scan_kernel<<<1, 1024, 0, q.stream>>>(q);
  const int nb = q.n_slots * kBuckets;
  if (nb <= 4096) {
    const int64_t blocks = (q.rays.n + 1023) / 1024;
    scatter_block_kernel<<<(unsigned)std::max<int64_t>(blocks, 1), 1024, 2 * nb * sizeof(int), q.stream>>>(q, nb);
  } else {
    const int grid = grid_for(q.rays.n, 256, 152 * 16);
    scatter_kernel<<<grid, 256, 0, q.stream>>>(q);
  }
  *launches += 2;
  return cudaGetLastError();
}

cudaError_t launch_exclusive_scan(int32_t *v, int64_t n, int32_t *sums, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int64_t nb = (n + 1023) / 1024;
  scan_block_kernel<<<(unsigned)nb, 1024, 0, st>>>(v, n, sums);
  scan_sums_kernel<<<1, 1024, 0, st>>>(sums, (int)nb);
  scan_add_kernel<<<(unsigned)nb, 1024, 0, st>>>(v, n, sums);
  return cudaGetLastError();
}

cudaError_t launch_plain_tail(const QueryLaunch &q, int ldx, int chunk_tiles, int *launches) {
  const size_t smem = mlp_fp32_smem(q.s.wmax);
  if (smem > kMlpSmemMax) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(mlp_fp32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMlpSmemMax);
  if (e != cudaSuccess) return e;
  for (int t0 = 0; t0 < q.s.max_tiles; t0 += chunk_tiles) {
    const int nt = min(chunk_tiles, q.s.max_tiles - t0);
    const int64_t items = (int64_t)nt * kTileM * q.H_max;
    gather_fp32_kernel<<<grid_for(items, 256, 152 * 32), 256, 0, q.stream>>>(q, t0, nt, ldx);
    mlp_fp32_kernel<<<min(nt, 152 * 4), 256, smem, q.stream>>>(q, t0, nt, ldx);
    *launches += 2;
  }
  return cudaGetLastError();
}

// ---- stage entry points ----------------------------------------------------

__global__ void trace_only_kernel(const DevObject *dobj, RaysArg r, int32_t *kout, float *t01, float *pts,
                                  int32_t *vox, int *err) {
  const DevObject &ob = *dobj;
  const int H = ob.H, cap = H >> 1;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < r.n; i += (int64_t)gridDim.x * blockDim.x) {
    float3 o, d;
    int ea;
    float t0 = CUDART_NAN_F, t1 = CUDART_NAN_F;
    int k = 0;
    bool live = to_unit(ob, r.ox[i], r.oy[i], r.oz[i], r.dx[i], r.dy[i], r.dz[i], o, d) &&
                unit_slab(o, d, r.tmin[i], t0, t1, ea);
    if (live) {
      dda_walk(
          ob, o, d, t0, t1, ea, [&](uint32_t vid) { return occupied(ob.occ, vid); },
          [&](const Seg &sg) {
            float3 a = seg_point(o, d, sg.tin, sg.ain, sg.fin);
            float3 b = seg_point(o, d, sg.tout, sg.aout, sg.fout);
            if (pts) {
              float *w = pts + ((size_t)i * H + 2 * k) * 3;
              w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = b.x; w[4] = b.y; w[5] = b.z;
            }
            if (vox) vox[(size_t)i * cap + k] = (int32_t)sg.vid;
            ++k;
            return k < cap;
          });
    } else {
      t0 = t1 = CUDART_NAN_F;
    }
    if (vox)
      for (int j = k; j < cap; ++j) vox[(size_t)i * cap + j] = -1;
    if (kout) kout[i] = k;
    if (t01) { t01[2 * i] = t0; t01[2 * i + 1] = t1; }
  }
}

cudaError_t launch_trace_only(const DevObject *dobj, const RaysArg &rays, int32_t *k, float *t01, float *pts,
                              int32_t *vox, int *err, cudaStream_t st) {
  int grid = grid_for(rays.n, 256, 152 * 16);
  trace_only_kernel<<<grid, 256, 0, st>>>(dobj, rays, k, t01, pts, vox, err);
  return cudaGetLastError();
}

template <typename T, int F>
__global__ void encode_kernel(DevObject hob, const T *tab, const float *pts, int64_t n, float *feats) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float3 p = make_float3(pts[3 * i], pts[3 * i + 1], pts[3 * i + 2]);
    for (int l = 0; l < hob.L; ++l) {
      float f[F];
      encode_level<T, F>(tab + (size_t)l * (hob.mask + 1) * F, hob.mask, p, (float)hob.res[l], f);
      for (int j = 0; j < F; ++j) feats[(i * hob.L + l) * F + j] = f[j];
    }
  }
}

cudaError_t launch_encode(const DevObject *dobj, const DevObject &h, const float *pts, int64_t n, float *feats,
                          int precision, cudaStream_t st) {
  (void)dobj;
  int grid = grid_for(n, 256, 152 * 32);
  if (precision == LSNIF_FP32_PLAIN) {
    if (h.F == 2) encode_kernel<float, 2><<<grid, 256, 0, st>>>(h, h.tab32, pts, n, feats);
    else if (h.F == 4) encode_kernel<float, 4><<<grid, 256, 0, st>>>(h, h.tab32, pts, n, feats);
    else encode_kernel<float, 1><<<grid, 256, 0, st>>>(h, h.tab32, pts, n, feats);
  } else {
    const __half *t16 = reinterpret_cast<const __half *>(h.tab16);
    if (h.F == 2) encode_kernel<__half, 2><<<grid, 256, 0, st>>>(h, t16, pts, n, feats);
    else if (h.F == 4) encode_kernel<__half, 4><<<grid, 256, 0, st>>>(h, t16, pts, n, feats);
    else encode_kernel<__half, 1><<<grid, 256, 0, st>>>(h, t16, pts, n, feats);
  }
  return cudaGetLastError();
}

__global__ void corners_kernel(DevObject hob, const float *pts, int64_t n, uint32_t *out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float3 p = make_float3(pts[3 * i], pts[3 * i + 1], pts[3 * i + 2]);
    for (int l = 0; l < hob.L; ++l) {
      Cell c = lattice_cell(p, (float)hob.res[l]);
      for (int corner = 0; corner < 8; ++corner) {
        uint32_t x = c.cx + (corner & 1), y = c.cy + ((corner >> 1) & 1), z = c.cz + ((corner >> 2) & 1);
        out[(i * hob.L + l) * 8 + corner] = hash3(x, y, z) & hob.mask;
      }
    }
  }
}

cudaError_t launch_corners(const DevObject *dobj, const DevObject &h, const float *pts, int64_t n, uint32_t *out,
                           cudaStream_t st) {
  (void)dobj;
  int grid = grid_for(n, 256, 152 * 32);
  corners_kernel<<<grid, 256, 0, st>>>(h, pts, n, out);
  return cudaGetLastError();
}

cudaError_t launch_mlp_plain(const DevObject *dobj, const DevObject &h, const float *X, int64_t n, float *Z,
                             cudaStream_t st) {
  const int wmax = max(h.width, h.n_out_pad);
  const size_t smem = mlp_fp32_smem(wmax);
  if (smem > kMlpSmemMax) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(mlp_fp32_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMlpSmemMax);
  if (e != cudaSuccess) return e;
  mlp_fp32_rows_kernel<<<grid_for(n, kMT, 152 * 4), 256, smem, st>>>(dobj, X, n, Z, wmax);
  return cudaGetLastError();
}

// ---- object preparation -----------------------------------------------------

__global__ void to_half_kernel(const float *src, __half *dst, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    dst[i] = __float2half_rn(src[i]);
}

cudaError_t launch_tables_to_half(const float *src, uint16_t *dst, int64_t n, cudaStream_t st) {
  to_half_kernel<<<grid_for(n, 256, 152 * 32), 256, 0, st>>>(src, reinterpret_cast<__half *>(dst), n);
  return cudaGetLastError();
}

// BF16 (dst) and FP16 (dst16) weights in the tcgen05 no-swizzle K-major
// core-matrix layout: element (n, k) of a layer with K inputs sits at byte
//   ((n/8)*(K/8) + k/8)*128 + (n%8)*16 + (k%8)*2
// Rows past the real output count are zero. Biases follow as FP32 in both.
// FP16 weights saturate at +-65504.
__global__ void build_umma_kernel(DevObject h, uint8_t *dst, uint8_t *dst16, uint8_t *dst_lo, uint8_t *dst_w0c) {
  const float *p = h.mlp32;
  uint32_t off = 0;
  const uint32_t off1 = (uint32_t)h.width * h.n_in * 2;  // where the layers after the first start
  int n_layers = h.n_hidden + 1;
  for (int l = 0; l < n_layers; ++l) {
    int K = l == 0 ? h.n_in : h.width;
    int Nr = l < h.n_hidden ? h.width : h.n_out;
    int Np = l < h.n_hidden ? h.width : h.n_out_pad;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)Np * K;
         e += (int64_t)gridDim.x * blockDim.x) {
      int nn = (int)(e / K), kk = (int)(e % K);
      float v = nn < Nr ? p[(int64_t)nn * K + kk] : 0.f;
      size_t o = off + ((size_t)(nn / 8) * (K / 8) + kk / 8) * 128 + (nn % 8) * 16 + (kk % 8) * 2;
      const __nv_bfloat16 hi = __float2bfloat16_rn(v);
      *reinterpret_cast<__nv_bfloat16 *>(dst + o) = hi;
      *reinterpret_cast<__half *>(dst16 + o) = __float2half_rn(fminf(fmaxf(v, -65504.f), 65504.f));
      if (l > 0) *reinterpret_cast<__nv_bfloat16 *>(dst_lo + (o - off1)) = __float2bfloat16_rn(v - __bfloat162float(hi));
      if (l == 0) {  // chunk-major copy: chunk s = kk / CHK is one contiguous W x CHK slice
        const int chk = 2 * h.L * h.F, s = kk / chk, c = kk % chk;
        const size_t oc = (size_t)s * h.width * chk * 2 + ((size_t)(nn / 8) * (chk / 8) + c / 8) * 128 + (nn % 8) * 16 +
                          (c % 8) * 2;
        *reinterpret_cast<__half *>(dst_w0c + oc) = __float2half_rn(fminf(fmaxf(v, -65504.f), 65504.f));
      }
    }
    const float *b = p + (size_t)Nr * K;
    float *bd = reinterpret_cast<float *>(dst + h.umma_bias_off) + (size_t)l * h.width;
    float *bd16 = reinterpret_cast<float *>(dst16 + h.umma_bias_off) + (size_t)l * h.width;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < Np; j += gridDim.x * blockDim.x)
      bd[j] = bd16[j] = j < Nr ? b[j] : 0.f;
    off += (uint32_t)Np * K * 2;
    p += (size_t)Nr * K + Nr;
  }
}

// FP32 output layer padded with zero rows to n_out_pad (FP32 path), and, one
// word per block, whether this block saw a first-layer weight that is not
// finite (kNonFiniteWords blocks).
__global__ void __launch_bounds__(256) build_plain_out_kernel(DevObject h, float *dst) {
  bool bad = false;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < h.width * h.n_in; i += gridDim.x * blockDim.x)
    bad |= !isfinite(h.mlp32[i]);
  const int any = __syncthreads_or(bad);
  if (threadIdx.x == 0) reinterpret_cast<int *>(dst + (size_t)h.n_out_pad * (h.width + 1))[blockIdx.x] = any;
  const float *p = h.mlp32;
  int fan_in = h.n_in;
  for (int l = 0; l < h.n_hidden; ++l) {
    p += (size_t)h.width * fan_in + h.width;
    fan_in = h.width;
  }
  const float *b = p + (size_t)h.n_out * h.width;
  const int tot = h.n_out_pad * h.width;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < tot + h.n_out_pad; i += gridDim.x * blockDim.x) {
    if (i < tot) {
      const int r = i / h.width;
      dst[i] = r < h.n_out ? p[i] : 0.f;
    } else {
      const int j = i - tot;
      dst[i] = j < h.n_out ? b[j] : 0.f;
    }
  }
}

cudaError_t launch_build_umma(const DevObject &h, cudaStream_t st) {
  build_umma_kernel<<<152, 256, 0, st>>>(h, const_cast<uint8_t *>(h.umma), const_cast<uint8_t *>(h.umma_h),
                                         const_cast<uint8_t *>(h.umma_lo), const_cast<uint8_t *>(h.w0_16c));
  build_plain_out_kernel<<<kNonFiniteWords, 256, 0, st>>>(h, const_cast<float *>(h.plain_out));
  return cudaGetLastError();
}

}  // namespace lsnif
