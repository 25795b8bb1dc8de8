// vk_voronoi3.cu -- Voronoi-neighbor rule in 3D (Sec. "Computational tools:
// Voronoi neighbor lists": neighbors are the particles whose Voronoi cells
// share a face; the relation is reciprocal) fused with the Vicsek update of
// Eq. (1) and Eq. (2) (vectorial noise, as every 3D rule here).
//
// The cell starts as the box bounded by the particle's own periodic images
// and is clipped by the bisector planes of the candidates of a ring walk of
// the uniform 3D grid (vk_voronoi3.cuh: exact predicates, dual
// triangulation).  A site at offset d can cut the cell only if |d| < 2R, R the
// distance of the farthest vertex, so the walk stops once the scanned block
// holds that ball.  When 2R reaches a quarter of the box, non-minimum images
// of other particles can cut too: the cell is then finished against every
// image of every particle within 2R.  Neighbors are the sites of faces of
// positive area, in id order.  Coincident particles latch VK_ERR_DEGENERATE
// (no cell separates them).
//
// One warp builds one cell, held in shared memory.  A cell meets about 240
// candidates, of which about 25 cut it; it has about 27 vertices.
//   * Testing: each lane holds one candidate and runs over the vertices (one
//     broadcast load and three FMAs each), so 32 candidates cost one pass.
//     The rows of a ring are pruned by their distance and dealt out to the
//     lanes evenly.
//   * Clipping: of the candidates that may cut, the nearest goes first (it
//     removes most), and the others are tested again.  The lanes hold the
//     triangles: each finds its side, the boundary edges are numbered by
//     ballots, and the new fan is linked through a table indexed by plane.
//   * The exact integer solve of a new vertex is spread over four lanes (three
//     numerators and the determinant).
//   * Headings are summed per cell (three lanes, one component each) and the
//     update runs for up to 16 finished cells at once, one per lane.
// The kernel is bound by instruction issue and the latency of its serial
// chain of clips; DRAM is idle.  Measured on GB300, one step: 262,144 uniform
// particles 9.5 ms (one thread per cell in 5.3 KB of local memory, 2.4 of 32
// lanes active: 54.8 ms), and a few thousand no longer take the 10 ms that one
// thread needs for one cell.
// Cells that outgrow 64 faces or 128 vertices on the way are rebuilt by the
// same code with twice the room.
#include <algorithm>

#include "vk_internal.cuh"
#include "vk_voronoi3.cuh"
#include "vk_voronoi3_api.cuh"

namespace vk {

namespace {

constexpr int kMaxImages = 64;

// A cell in shared memory: at most PM planes and TM triangles (8-bit indices,
// packed three to a word).  Free triangles have y = 0, which no plane cuts.
template <int PM, int TM>
struct Cell3 {
  static constexpr int P = PM, T = TM, B = TM / 2, W = TM / 32;
  float4 y[TM];       // y = 2x of the vertex (FP32 estimate)
  int4 plane[PM];     // offset d (grid units) and the site's sorted slot (-1: own image)
  uint32_t tp[TM];    // planes, det(d_a, d_b, d_c) > 0
  uint32_t tn[TM];    // byte k: triangle across the edge of planes k, k + 1
  uint32_t out[W];    // triangles beyond the plane being applied
  uint8_t bp[B], bq[B], bo[B], bt[B];  // boundary edges p -> q, kept triangle across, new triangle
  uint8_t from[PM], to[PM];            // boundary edge leaving / reaching a plane
};

using CellS = Cell3<64, 128>;
using CellL = Cell3<128, 256>;

__device__ __forceinline__ int byte_of(uint32_t v, int k) { return (int)(v >> (8 * k)) & 255; }
__device__ __forceinline__ int next3(int k) { return k == 2 ? 0 : k + 1; }

__device__ __forceinline__ float warp_max(float v) {
  return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));  // v >= 0
}

// One warp's builder; every member is called by all 32 lanes, and every value
// outside the cell is the same in all lanes unless it says otherwise.
template <class C3>
struct Builder3 {
  C3& S;
  int lane;
  uint32_t below;       // lanes below this one
  uint32_t alive[C3::W];
  int np, nt, status;
  float r2, ymax;       // upper bounds of max |x|^2 and max |y| over the vertices

  __device__ __forceinline__ const int32_t* pd(int p) const { return reinterpret_cast<const int32_t*>(&S.plane[p]); }

  __device__ __forceinline__ void refresh_radius() {
    float m = 0.f;
    for (int t = lane; t < nt; t += 32) {
      const float4 y = S.y[t];
      m = fmaxf(m, y.x * y.x + y.y * y.y + y.z * y.z);
    }
    m = warp_max(m);
    // |x| = |y| / 2; 2^-18 covers the estimate's and this sum's rounding
    r2 = 0.25f * m * (1.f + 3.8147e-6f) + 1.f;
    ymax = sqrtf(m) * (1.f + 3.8147e-6f) + 1.f;
  }

  // the box bounded by the particle's own images at +-L per axis: octant t
  // (bit a: the minus side of axis a) has planes 2a + side; across the edge
  // that leaves out axis a lies octant t ^ (1 << a)
  __device__ __forceinline__ void init(const uint32_t* L) {
    status = v3::kOk;
    np = 6;
    nt = 8;
#pragma unroll
    for (int i = 0; i < C3::W; ++i) alive[i] = i == 0 ? 0xFFu : 0u;
    if (lane < 6) {
      const int a = lane >> 1;
      const int32_t v = lane & 1 ? -(int32_t)L[a] : (int32_t)L[a];
      S.plane[lane] = make_int4(a == 0 ? v : 0, a == 1 ? v : 0, a == 2 ? v : 0, -1);
    }
    if (lane < 8) {
      const int t = lane;
      const uint32_t px = t & 1, py = 2 + ((t >> 1) & 1), pz = 4 + ((t >> 2) & 1);
      // the determinant's sign flips with every minus side
      if (__popc(t) & 1) {
        S.tp[t] = px | pz << 8 | py << 16;
        S.tn[t] = (uint32_t)(t ^ 2) | (uint32_t)(t ^ 1) << 8 | (uint32_t)(t ^ 4) << 16;
      } else {
        S.tp[t] = px | py << 8 | pz << 16;
        S.tn[t] = (uint32_t)(t ^ 4) | (uint32_t)(t ^ 1) << 8 | (uint32_t)(t ^ 2) << 16;
      }
      const float x = (float)L[0], y = (float)L[1], z = (float)L[2];
      S.y[t] = make_float4(t & 1 ? -x : x, t & 2 ? -y : y, t & 4 ? -z : z, 0.f);
    }
    __syncwarp();
    refresh_radius();
  }

  // 2^-19 (|d| ymax + w): bound of the error of the FP32 side estimate (see
  // v3::side_band)
  __device__ __forceinline__ float band(float wf) const {
    return 1.9073486e-6f * (sqrtf(wf) * 1.0001f * ymax + wf);
  }
  __device__ __forceinline__ float side_est(int t, float dx, float dy, float dz, float wf) const {
    const float4 y = S.y[t];
    return fmaf(dx, y.x, fmaf(dy, y.y, fmaf(dz, y.z, -wf)));
  }
  // (per lane) exact-sign side of triangle t for plane d
  __device__ __forceinline__ int side(int t, const int32_t* d, float wf, float bd) const {
    const float s = side_est(t, (float)d[0], (float)d[1], (float)d[2], wf);
    if (s > bd) return 1;
    if (s < -bd) return -1;
    const uint32_t tp = S.tp[t];
    return v3::side_exact(pd(byte_of(tp, 0)), pd(byte_of(tp, 1)), pd(byte_of(tp, 2)), d);
  }

  // (per lane) may the site at offset d cut or touch the cell?
  __device__ __forceinline__ bool may_cut(const int32_t* d, float wf) const {
    const float dx = (float)d[0], dy = (float)d[1], dz = (float)d[2];
    float m0 = -3.0e38f, m1 = -3.0e38f;
    int t = 0;
    for (; t + 1 < nt; t += 2) {
      const float4 a = S.y[t], b = S.y[t + 1];
      m0 = fmaxf(m0, fmaf(dx, a.x, fmaf(dy, a.y, dz * a.z)));
      m1 = fmaxf(m1, fmaf(dx, b.x, fmaf(dy, b.y, dz * b.z)));
    }
    if (t < nt) {
      const float4 a = S.y[t];
      m0 = fmaxf(m0, fmaf(dx, a.x, fmaf(dy, a.y, dz * a.z)));
    }
    // (the sum is rounded once more than side_est's: twice its band)
    return fmaxf(m0, m1) - wf >= -2.f * band(wf);
  }

  // the points of the new triangles bt[0..nb): Cramer's rule on exact
  // integers, lanes 0..2 of four the numerators, lane 3 the determinant
  __device__ __forceinline__ void solve(int nb) {
    const int c = lane & 3;
    const int k = c == 3 ? 0 : c, k1 = next3(k), k2 = next3(k1);
    for (int j0 = 0; j0 < nb; j0 += 8) {
      const int j = j0 + (lane >> 2);
      const int t = S.bt[min(j, nb - 1)];
      const uint32_t tp = S.tp[t];
      const int32_t* M[3] = {pd(byte_of(tp, 0)), pd(byte_of(tp, 1)), pd(byte_of(tp, 2))};
      v3::i128 num = 0;
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int32_t *A = M[(r + 1) % 3], *Bq = M[(r + 2) % 3];
        const int64_t cf = v3::minor2(A[k1], A[k2], Bq[k1], Bq[k2]);
        const int64_t f = c == 3 ? (int64_t)M[r][0] : v3::norm2(M[r]);
        num += (v3::i128)f * cf;
      }
      const float v = v3::i128_to_float(num);
      const float det = __shfl_sync(0xffffffffu, v, lane | 3);
      if (j < nb) reinterpret_cast<float*>(&S.y[t])[c] = c == 3 ? 0.f : v / det;
    }
    __syncwarp();
  }

  // Clip by the plane of the site at offset d (slot: its sorted slot).
  __device__ __forceinline__ void clip(const int32_t* d, int32_t slot, float wf) {
    const float bd = band(wf);
    uint32_t om[C3::W];
    uint32_t any = 0;
#pragma unroll
    for (int i = 0; i < C3::W; ++i) {
      om[i] = 0;
      if (i * 32 >= nt) continue;
      const bool o = (alive[i] >> lane & 1u) && side(i * 32 + lane, d, wf, bd) > 0;
      om[i] = __ballot_sync(0xffffffffu, o);
      any |= om[i];
    }
    if (!any) return;
    int e = np;  // the new plane
    if (np < C3::P) {
      ++np;
    } else {
      // reuse a plane that no triangle holds any more
      for (int p = lane; p < C3::P; p += 32) S.to[p] = 0;
      __syncwarp();
#pragma unroll
      for (int i = 0; i < C3::W; ++i)
        if (alive[i] >> lane & 1u) {
          const uint32_t tp = S.tp[i * 32 + lane];
          S.to[byte_of(tp, 0)] = S.to[byte_of(tp, 1)] = S.to[byte_of(tp, 2)] = 1;
        }
      __syncwarp();
      e = -1;
      for (int p0 = 0; p0 < C3::P && e < 0; p0 += 32) {
        const uint32_t m = __ballot_sync(0xffffffffu, S.to[p0 + lane] == 0);
        if (m) e = p0 + __ffs(m) - 1;
      }
      if (e < 0) {
        status = v3::kCapacity;
        return;
      }
    }
    if (lane == 0) {
#pragma unroll
      for (int i = 0; i < C3::W; ++i) S.out[i] = om[i];
      S.plane[e] = make_int4(d[0], d[1], d[2], slot);
    }
    __syncwarp();
    // boundary edges (p -> q) of the removed region, with the kept triangle across
    int nb = 0;
#pragma unroll
    for (int i = 0; i < C3::W; ++i) {
      if (om[i] == 0) continue;
      const bool mine = om[i] >> lane & 1u;
      const uint32_t tp = mine ? S.tp[i * 32 + lane] : 0u, tn = mine ? S.tn[i * 32 + lane] : 0u;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int o = byte_of(tn, k);
        const bool b = mine && !(S.out[o >> 5] >> (o & 31) & 1u);
        const uint32_t m = __ballot_sync(0xffffffffu, b);
        const int j = nb + __popc(m & below);
        if (b && j < C3::B) {
          S.bp[j] = (uint8_t)byte_of(tp, k);
          S.bq[j] = (uint8_t)byte_of(tp, next3(k));
          S.bo[j] = (uint8_t)o;
        }
        nb += __popc(m);
      }
    }
    if (nb < 3 || nb > C3::B) {
      status = nb < 3 ? v3::kInternal : v3::kCapacity;
      return;
    }
    // the removed triangles' places are taken first, then the next free ones
    int got = 0;
    nt = 0;
#pragma unroll
    for (int i = 0; i < C3::W; ++i) {
      alive[i] &= ~om[i];
      const uint32_t fr = ~alive[i];
      const int r = got + __popc(fr & below);
      const bool f = (fr >> lane & 1u) && r < nb;
      if (f) S.bt[r] = (uint8_t)(i * 32 + lane);
      const uint32_t m = __ballot_sync(0xffffffffu, f);
      if ((om[i] & ~m) >> lane & 1u) S.y[i * 32 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
      alive[i] |= m;
      got += __popc(m);
      if (alive[i]) nt = i * 32 + 32 - __clz(alive[i]);
    }
    if (got < nb) {
      status = v3::kCapacity;
      return;
    }
    __syncwarp();
    // link the fan: the triangle of an edge p -> q borders those of the edges
    // leaving q and reaching p
    for (int j = lane; j < nb; j += 32) {
      S.from[S.bp[j]] = (uint8_t)j;
      S.to[S.bq[j]] = (uint8_t)j;
    }
    __syncwarp();
    bool ok = true;
    for (int j = lane; j < nb; j += 32) {
      const int p = S.bp[j], q = S.bq[j], o = S.bo[j], t = S.bt[j];
      const int nx = S.from[q], pv = S.to[p];
      ok = ok && S.from[p] == j && S.to[q] == j && nx < nb && pv < nb && S.bp[nx] == q && S.bq[pv] == p;
      if (!ok) break;
      S.tp[t] = (uint32_t)p | (uint32_t)q << 8 | (uint32_t)e << 16;
      S.tn[t] = (uint32_t)o | (uint32_t)S.bt[nx] << 8 | (uint32_t)S.bt[pv] << 16;
      const uint32_t to = S.tp[o];
      const int k = byte_of(to, 0) == q ? 0 : (byte_of(to, 1) == q ? 1 : 2);
      reinterpret_cast<uint8_t*>(&S.tn[o])[k] = (uint8_t)t;
    }
    if (!__all_sync(0xffffffffu, ok)) {
      status = v3::kInternal;
      return;
    }
    __syncwarp();
    solve(nb);
    refresh_radius();
  }

  // one candidate per lane (offset d, slot q): clip by those that cut, nearest first
  __device__ __forceinline__ void batch(bool valid, const int32_t* d, int32_t q) {
    if (__any_sync(0xffffffffu, valid && d[0] == 0 && d[1] == 0 && d[2] == 0)) {
      status = v3::kCoincident;
      return;
    }
    const float wf = (float)v3::norm2(d);
    // |d| / 2 beyond every vertex: cannot cut
    bool flag = valid && wf < 4.f * r2 && may_cut(d, wf);
    while (__any_sync(0xffffffffu, flag) && status == v3::kOk) {
      const uint32_t key = flag ? __float_as_uint(wf) : 0xFFFFFFFFu;
      const uint32_t best = __reduce_min_sync(0xffffffffu, key);
      const int src = __ffs(__ballot_sync(0xffffffffu, flag && key == best)) - 1;
      const int32_t dd[3] = {__shfl_sync(0xffffffffu, d[0], src), __shfl_sync(0xffffffffu, d[1], src),
                             __shfl_sync(0xffffffffu, d[2], src)};
      clip(dd, __shfl_sync(0xffffffffu, q, src), __uint_as_float(best));
      flag = flag && lane != src;
      if (flag) flag = wf < 4.f * r2 && may_cut(d, wf);
    }
  }

  // distance of the slab of cells at offset o along an axis from the particle
  // (the nearer of its two images); (per lane)
  static __device__ __forceinline__ float slab(int64_t p, int c, int o, int n, const uint32_t* __restrict__ bnd,
                                               int64_t L) {
    if (o == 0) return 0.f;
    const int64_t lo = cell_lo_tab(c + o, n, bnd, L) - p, hi = cell_lo_tab(c + o + 1, n, bnd, L) - 1 - p;
    return (float)(o > 0 ? min(lo, L - hi) : min(-hi, L + lo));
  }

  // The cell of the particle at sorted slot `self`; false when it could not be
  // built (status says why).
  __device__ __forceinline__ bool build(const Rep& R, int64_t self, const int32_t* pi, const int4* __restrict__ S_pos,
                                        const GridView& G, const uint32_t* __restrict__ bounds, uint32_t* n_cand) {
    init(R.L);
    int c[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) c[a] = cell_of_tab((uint32_t)pi[a], R.nc[a], bounds + R.bnd[a], R.inv_w[a]);
    const int nx = R.nc[0], ny = R.nc[1], nz = R.nc[2];
    // One loop feeds the only copy of the clipping code: the rings of cells
    // (0 and 1 together, then outwards), then, in a tiny box, all images.
    bool images = false;
    int K[3] = {0, 0, 0};
    for (int r = 1;; ++r) {
      int lo[3], hi[3], plo[3], phi[3];
      bool full = true, any_new = r == 1;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        lo[a] = ring_lo(r, R.nc[a]);
        hi[a] = ring_hi(r, R.nc[a]);
        plo[a] = r > 1 ? ring_lo(r - 1, R.nc[a]) : 1;
        phi[a] = r > 1 ? ring_hi(r - 1, R.nc[a]) : 0;
        full = full && hi[a] - lo[a] + 1 == R.nc[a];
        any_new = any_new || lo[a] < plo[a] || hi[a] > phi[a];
      }
      // the rows of the ring: one x segment, or two where the row crosses the
      // scanned block (the second ones are numbered after all first ones)
      const int ry = hi[1] - lo[1] + 1, rows = ry * (hi[2] - lo[2] + 1);
      const int sx = 2 * K[0] + 1, sy = 2 * K[1] + 1, per = sx * sy * (2 * K[2] + 1);
      const int items = images ? 1 : !any_new ? 0 : r > 1 ? 2 * rows : rows;
      for (int i0 = 0; i0 < items; i0 += 32) {
        const int it = i0 + lane;
        const bool second = it >= rows;
        const int row = second ? it - rows : it;
        const int oz = lo[2] + row / ry, oy = lo[1] + row % ry;
        const bool old = oz >= plo[2] && oz <= phi[2] && oy >= plo[1] && oy <= phi[1];
        const int xa = second ? phi[0] + 1 : lo[0], xb = old && !second ? plo[0] - 1 : hi[0];
        uint32_t q0 = 0, q1 = 0;
        int l0 = 0, len = 0;
        if (!images && row < rows && xa <= xb && (old || !second)) {
          const float dy = slab(pi[1], c[1], oy, ny, bounds + R.bnd[1], R.L[1]);
          const float dz = slab(pi[2], c[2], oz, nz, bounds + R.bnd[2], R.L[2]);
          if ((dy * dy + dz * dz) * 0.99999f < 4.f * r2) {
            const int64_t rb = R.c0 + ((int64_t)wrap_index(c[2] + oz, nz) * ny + wrap_index(c[1] + oy, ny)) * nx;
            const int xs = wrap_index(c[0] + xa, nx), xe = xs + (xb - xa) + 1;
            q0 = __ldg(G.off + rb + xs);
            l0 = (int)(__ldg(G.off + rb + min(xe, nx)) - q0);
            len = l0;
            if (xe > nx) {  // the segment goes on at the other side of the period
              q1 = __ldg(G.off + rb);
              len += (int)(__ldg(G.off + rb + xe - nx) - q1);
            }
          }
        }
        // deal the candidates of the 32 segments out to the lanes
        int incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += v;
        }
        const int64_t total = images ? (int64_t)R.n * per : __shfl_sync(0xffffffffu, incl, 31);
        *n_cand += images ? 0u : (uint32_t)total;
        for (int64_t b0 = 0; b0 < total; b0 += 32) {
          const int64_t idx = b0 + lane;
          int64_t q;
          int k[3] = {0, 0, 0};
          if (images) {
            q = R.p0 + idx / per;
            const int im = (int)(idx % per);
            k[0] = im % sx - K[0];
            k[1] = im / sx % sy - K[1];
            k[2] = im / (sx * sy) - K[2];
          } else {
            int own = 0;
#pragma unroll
            for (int st = 16; st > 0; st >>= 1)
              if (__shfl_sync(0xffffffffu, incl, own + st - 1) <= (int)idx) own += st;
            own = min(own, 31);
            const int at = (int)idx - (__shfl_sync(0xffffffffu, incl, own) - __shfl_sync(0xffffffffu, len, own));
            const int s0 = __shfl_sync(0xffffffffu, l0, own);
            const uint32_t b = __shfl_sync(0xffffffffu, q0, own), b1 = __shfl_sync(0xffffffffu, q1, own);
            q = at < s0 ? b + (uint32_t)at : b1 + (uint32_t)(at - s0);
          }
          const bool valid = idx < total && q != self;
          int32_t d[3] = {1, 0, 0};
          if (valid) {
            const int4 pj = __ldg(S_pos + q);
            d[0] = (int32_t)(min_image((int64_t)pj.x - pi[0], (int64_t)R.L[0]) + (int64_t)k[0] * R.L[0]);
            d[1] = (int32_t)(min_image((int64_t)pj.y - pi[1], (int64_t)R.L[1]) + (int64_t)k[1] * R.L[1]);
            d[2] = (int32_t)(min_image((int64_t)pj.z - pi[2], (int64_t)R.L[2]) + (int64_t)k[2] * R.L[2]);
          }
          batch(valid, d, (int32_t)q);
          if (status != v3::kOk) return false;
        }
      }
      if (images) return true;
      if (any_new && !full) {
        // every unscanned site is at squared distance >= B^2; none can cut once
        // B^2 >= 4 R^2 (lowered by 2^-22 to stay below the exact value)
        int64_t Bd = INT64_MAX;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          if (hi[a] - lo[a] + 1 == R.nc[a]) continue;
          const uint32_t* bnd = bounds + R.bnd[a];
          Bd = min(Bd, min((int64_t)pi[a] - cell_lo_tab(c[a] - r, R.nc[a], bnd, R.L[a]) + 1,
                           cell_lo_tab(c[a] + r + 1, R.nc[a], bnd, R.L[a]) - (int64_t)pi[a]));
        }
        if ((float)((uint64_t)Bd * (uint64_t)Bd) * 0.99999976f < 4.f * r2) continue;
      }
      // other images lie at >= L_min / 2: they matter only when 2R > L_min / 2
      const float Lmin = (float)min(R.L[0], min(R.L[1], R.L[2]));
      if (!(16.f * r2 > Lmin * Lmin) || R.n <= 1) return true;
      const float Rr = sqrtf(r2);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const float kk = floorf((2.f * Rr + 0.5f * (float)R.L[a]) / (float)R.L[a]) + 1.f;
        // more than kMaxImages images per axis (a box far longer than wide
        // holding a handful of particles) is outside the supported range
        if (!(kk <= (float)kMaxImages)) {
          status = v3::kCapacity;
          return false;
        }
        K[a] = (int)kk;
      }
      images = true;
    }
  }

  // (per lane) does the face of plane p have positive area, t0 one of its triangles?
  __device__ __forceinline__ bool face_positive(int p, int t0) const {
    int t = t0, first = -1;
    for (int guard = 0; guard < C3::T; ++guard) {
      // t = (p, q, r) in cyclic order from p; the next triangle around p is
      // across the edge (p, q) and reads (q, p, s)
      const uint32_t tp = S.tp[t];
      const int k = byte_of(tp, 0) == p ? 0 : (byte_of(tp, 1) == p ? 1 : 2);
      const int q = byte_of(tp, next3(k)), u = byte_of(S.tn[t], k);
      const uint32_t up = S.tp[u];
      const int ku = byte_of(up, 0) == p ? 0 : (byte_of(up, 1) == p ? 1 : 2);
      const int s = byte_of(up, next3(ku));
      // the edge t -> u on line p^q has zero length iff t's point is on plane s
      const float ws = (float)v3::norm2(pd(s));
      if (side(t, pd(s), ws, band(ws)) != 0) {
        if (first < 0) first = q;
        else if (v3::det3(pd(p), pd(first), pd(q)) != 0) return true;
      }
      t = u;
      if (t == t0) break;
    }
    return false;
  }

  // neighbor slots in id order, each id once, into slots[0..count); ids in
  // ids[].  Both are scratch of C3::P entries in shared memory.
  __device__ __forceinline__ int neighbors(const int32_t* __restrict__ S_id, int32_t* ids, int32_t* slots) {
    // a triangle of every live plane
    for (int p = lane; p < np; p += 32) S.to[p] = 0;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < C3::W; ++i)
      if (alive[i] >> lane & 1u) {
        const int t = i * 32 + lane;
        const uint32_t tp = S.tp[t];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          S.from[byte_of(tp, k)] = (uint8_t)t;
          S.to[byte_of(tp, k)] = 1;
        }
      }
    __syncwarp();
    int cnt = 0;
    int32_t id[C3::P / 32], sl[C3::P / 32];
#pragma unroll
    for (int i = 0; i < C3::P / 32; ++i) {
      const int p = i * 32 + lane;
      if (i * 32 >= np) break;
      sl[i] = p < np ? S.plane[p].w : -1;
      const bool is = p < np && S.to[p] && sl[i] >= 0 && face_positive(p, S.from[p]);
      id[i] = is ? __ldg(S_id + sl[i]) : -1;
      const uint32_t m = __ballot_sync(0xffffffffu, is);
      if (is) {
        const int at = cnt + __popc(m & below);
        ids[at] = id[i];
        slots[at] = sl[i];
      }
      cnt += __popc(m);
    }
    __syncwarp();
    // order by id; of two images of one site the first counts
    int rank[C3::P / 32];
    int32_t mine[C3::P / 32];
    int kept = 0;
#pragma unroll
    for (int i = 0; i < C3::P / 32; ++i) {
      rank[i] = -1;
      if (i * 32 >= cnt) break;
      const int at = i * 32 + lane;
      bool keep = at < cnt;
      if (keep) {
        const int32_t v = ids[at];
        mine[i] = slots[at];
        int r = 0;
        for (int j = 0; j < cnt; ++j) {
          const int32_t w = ids[j];
          keep = keep && !(w == v && j < at);
          r += w < v ? 1 : 0;
        }
        rank[i] = r;
      }
      if (!keep) rank[i] = -1;
      kept += __popc(__ballot_sync(0xffffffffu, keep));
    }
    __syncwarp();
    if (kept < cnt) {
      // some id was listed twice (tiny boxes): count its predecessors once
#pragma unroll
      for (int i = 0; i < C3::P / 32; ++i) {
        if (i * 32 >= cnt) break;
        if (rank[i] >= 0) {
          const int32_t v = ids[i * 32 + lane];
          int r = 0;
          for (int j = 0; j < cnt; ++j) {
            bool dup = false;
            for (int h = 0; h < j; ++h) dup = dup || ids[h] == ids[j];
            r += !dup && ids[j] < v ? 1 : 0;
          }
          rank[i] = r;
        }
      }
      __syncwarp();
    }
#pragma unroll
    for (int i = 0; i < C3::P / 32; ++i) {
      if (i * 32 >= cnt) break;
      if (rank[i] >= 0) slots[rank[i]] = mine[i];
    }
    __syncwarp();
    return kept;
  }
};

__device__ __forceinline__ int32_t status_of(int st) {
  return st == v3::kCoincident ? kStDegenerate : kStCapacity;
}

// finished cells of a warp waiting for their update
constexpr int kPend = 16;

// WPB warps per block
template <class C3>
struct Warp3 {
  C3 cell;
  int32_t ids[C3::P], slots[C3::P];
  HeadSum<1> sum[kPend][3];     // per axis
  int32_t m[kPend];             // neighbors; -1: state carried over; -2: on the overflow list
};

constexpr int kV3Warps = 4;
// resident blocks per SM the kernels are compiled for: 4 (128 registers)
// measured 9.5 ms at 262,144 cells, 5, 6 and 7 (more spills) 12.1, 11.7, 11.3
#ifndef VK_V3_BLOCKS
#define VK_V3_BLOCKS 4
#endif

// Search + update.  LIST: the particles of the overflow list; otherwise all,
// taken `chunk` at a time from a work counter, so that slow cells (void rims)
// hold back one warp only.
template <class C3, bool LIST>
__global__ void __launch_bounds__(32 * kV3Warps, VK_V3_BLOCKS) voronoi3_step_kernel(
    const Rep* __restrict__ reps, const BlockTask* __restrict__ tasks, int n_items, int chunk,
    const uint32_t* __restrict__ bounds, const int4* __restrict__ S_pos, const float4* __restrict__ S_dir,
    const int32_t* __restrict__ S_id, GridView G, int4* __restrict__ U_pos, float4* __restrict__ U_dir,
    int32_t* __restrict__ U_id, uint32_t* __restrict__ U_rank, uint32_t* __restrict__ counts,
    PhiAcc* __restrict__ phi_acc,
    const int64_t* __restrict__ d_step, StepParams Pm, int32_t* status, int2* __restrict__ ovf_list,
    int32_t* __restrict__ ovf_count) {
  extern __shared__ __align__(16) unsigned char v3_smem[];
  Warp3<C3>& W = reinterpret_cast<Warp3<C3>*>(v3_smem)[threadIdx.x >> 5];
  const int lane = (int)(threadIdx.x & 31);
  const int64_t step = *d_step;
  if (LIST) n_items = *ovf_count;
  int next = (int)(blockIdx.x * kV3Warps + (threadIdx.x >> 5)) * chunk;
  const int stride = (int)gridDim.x * kV3Warps * chunk;
  for (;; next += stride) {
    int base = next;
    if (!LIST) {
      if (lane == 0) base = atomicAdd(ovf_count + 1, chunk);
      base = __shfl_sync(0xffffffffu, base, 0);
    }
    if (base >= n_items) break;
    const int todo = min(chunk, n_items - base);
    auto particle = [&](int i, int* rep) -> int64_t {
      if (LIST) {
        const int2 e = ovf_list[base + i];
        *rep = e.y;
        return e.x;
      }
      const BlockTask t = tasks[(base + i) / kBlock];
      *rep = t.rep;
      const int li = t.first + (base + i) % kBlock;
      return li < reps[t.rep].n ? reps[t.rep].p0 + li : -1;
    };
    for (int i = 0; i < todo; ++i) {
      int rep;
      const int64_t s = particle(i, &rep);
      if (s < 0) {
        if (lane == 0) W.m[i] = -2;
        continue;
      }
      const Rep& R = reps[rep];
      const int4 p = S_pos[s];
      const int32_t pi[3] = {p.x, p.y, p.z};
      Builder3<C3> b{W.cell, lane, (1u << lane) - 1u};
      uint32_t n_cand = 0;
      if (b.build(R, s, pi, S_pos, G, bounds, &n_cand)) {
        const int cnt = b.neighbors(S_id, W.ids, W.slots);
        // neighbor headings in id order, in the place of the finished cell's points
        float4* dir = W.cell.y;
        for (int j = lane; j < cnt; j += 32) dir[j] = __ldg(S_dir + W.slots[j]);
        __syncwarp();
        if (lane < 3) {
          HeadSum<1> H;
          H.init();
          const float* own = reinterpret_cast<const float*>(S_dir + s) + lane;
          if (Pm.include_self) H.add(own, Pm.sum_mode);
          for (int j = 0; j < cnt; ++j) H.add(reinterpret_cast<const float*>(&dir[j]) + lane, Pm.sum_mode);
          W.sum[i][lane] = H;
        }
        if (lane == 0) W.m[i] = cnt;
      } else if (!LIST && b.status == v3::kCapacity) {
        if (lane == 0) {  // finished by the overflow launch (its heading enters phi there)
          ovf_list[atomicAdd(ovf_count, 1)] = make_int2((int)s, rep);
          W.m[i] = -2;
        }
      } else if (lane == 0) {
        // no cell: the state is carried over and the status latched (the host reports it)
        set_status(status, status_of(b.status));
        W.m[i] = -1;
      }
      if (Pm.stats && lane == 0) {
        atomicAdd(Pm.stats + 0, (unsigned long long)n_cand);
        atomicMax(Pm.stats + 2, (unsigned long long)n_cand);
        atomicAdd(Pm.stats + 3, 1ull);
      }
      __syncwarp();
    }
    __syncwarp();
    // Eq. (2) + Eq. (1), one finished cell per lane
    const int m = lane < todo ? W.m[lane] : -2;
    int rep = 0;
    float nnew[3] = {0.f, 0.f, 0.f};
    if (m > -2) {
      const int64_t s = particle(lane, &rep);
      const Rep& R = reps[rep];
      const int4 p = S_pos[s];
      const float4 nv = S_dir[s];
      const int32_t pi[3] = {p.x, p.y, p.z};
      const float ni[3] = {nv.x, nv.y, nv.z};
      const int32_t id = S_id[s];
      int32_t pout[3] = {p.x, p.y, p.z};
      if (m >= 0) {
        HeadSum<3> H;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          H.s[a] = W.sum[lane][a].s[0];
          H.c[a] = W.sum[lane][a].c[0];
          H.d[a] = W.sum[lane][a].d[0];
        }
        align_advect<3>(R, Pm, (uint32_t)step, id, ni, H, m + (Pm.include_self ? 1 : 0), pi, pout, nnew);
      } else {
#pragma unroll
        for (int a = 0; a < 3; ++a) nnew[a] = ni[a];
      }
      U_pos[s] = make_int4(pout[0], pout[1], pout[2], 0);
      U_dir[s] = make_float4(nnew[0], nnew[1], nnew[2], 0.f);
      U_id[s] = id;
      U_rank[s] = atomicAdd(counts + linear_cell<3>(R, pout), 1u);
    }
    phi_add_warp<3>(phi_acc + (size_t)(step % Pm.phi_cap) * (size_t)Pm.n_rep * 3, rep, nnew, m > -2);
    __syncwarp();
  }
}

// Neighbor lists: pass 0 writes the degree of every particle (by id), pass 1
// the sorted ids at out_off[id].
__global__ void __launch_bounds__(32 * kV3Warps) voronoi3_export_kernel(
    const Rep* __restrict__ reps, int rep, const uint32_t* __restrict__ bounds, const int4* __restrict__ S_pos,
    const int32_t* __restrict__ S_id, GridView G, int pass, int32_t* __restrict__ deg,
    const int64_t* __restrict__ out_off, int32_t* __restrict__ out_ids, int32_t* status) {
  extern __shared__ __align__(16) unsigned char v3_smem[];
  Warp3<CellL>& W = reinterpret_cast<Warp3<CellL>*>(v3_smem)[threadIdx.x >> 5];
  const int lane = (int)(threadIdx.x & 31);
  const Rep& R = reps[rep];
  for (int li = blockIdx.x * kV3Warps + (int)(threadIdx.x >> 5); li < R.n; li += gridDim.x * kV3Warps) {
    const int64_t s = R.p0 + li;
    const int4 p = S_pos[s];
    const int32_t pi[3] = {p.x, p.y, p.z};
    const int32_t id = S_id[s];
    Builder3<CellL> b{W.cell, lane, (1u << lane) - 1u};
    uint32_t n_cand = 0;
    int cnt = 0;
    if (b.build(R, s, pi, S_pos, G, bounds, &n_cand)) cnt = b.neighbors(S_id, W.ids, W.slots);
    else if (lane == 0) set_status(status, status_of(b.status));
    if (pass == 0) {
      if (lane == 0) deg[id] = cnt;
    } else {
      for (int j = lane; j < cnt; j += 32) out_ids[out_off[id] + j] = __ldg(S_id + W.slots[j]);
    }
    __syncwarp();
  }
}

GridView grid_view3(const Buffers& b) {
  GridView G;
  G.off = b.offsets;
  G.sub_s = b.sub_s;
  G.sub_base = b.sub_base;
  G.sub_off = b.sub_off;
  return G;
}

}  // namespace

cudaError_t prepare_voronoi3() {
  cudaError_t e = cudaFuncSetAttribute(voronoi3_step_kernel<CellL, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(sizeof(Warp3<CellL>) * kV3Warps));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(voronoi3_export_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(sizeof(Warp3<CellL>) * kV3Warps));
  return e;
}

cudaError_t launch_voronoi3_step(const Geometry& g, const Buffers& b, const StepParams& P, cudaStream_t st) {
  // Persistent: as many blocks as fit at once; warps take particles from the
  // work counter (ovf_count[1], cleared by every scatter).  (The occupancy is
  // looked up once, thread-safely; one block per SM if the query fails.)
  static const int per_sm = [] {
    int blocks = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, voronoi3_step_kernel<CellS, false>, 32 * kV3Warps,
                                                      sizeof(Warp3<CellS>) * kV3Warps) != cudaSuccess)
      blocks = 1;
    return std::max(blocks, 1);
  }();
  const int n_items = g.n_tasks * kBlock;
  const int sms = device_sm_count();
  const int blocks = std::min(sms * per_sm, (n_items + kV3Warps - 1) / kV3Warps);
  // up to 16 cells share one update; fewer where that would leave warps idle
  const int chunk = std::max(1, std::min(kPend, n_items / (blocks * kV3Warps * 4)));
  voronoi3_step_kernel<CellS, false><<<blocks, 32 * kV3Warps, sizeof(Warp3<CellS>) * kV3Warps, st>>>(
      g.reps, g.tasks, n_items, chunk, b.bounds, (const int4*)b.S_pos, (const float4*)b.S_dir, b.S_id, grid_view3(b),
      (int4*)b.U_pos, (float4*)b.U_dir, b.U_id, b.U_rank, b.counts, b.phi_acc, b.d_step, P, b.d_status, b.ovf_list,
      b.ovf_count);
  voronoi3_step_kernel<CellL, true><<<sms, 32 * kV3Warps, sizeof(Warp3<CellL>) * kV3Warps, st>>>(
      g.reps, g.tasks, 0, 1, b.bounds, (const int4*)b.S_pos, (const float4*)b.S_dir, b.S_id, grid_view3(b),
      (int4*)b.U_pos, (float4*)b.U_dir, b.U_id, b.U_rank, b.counts, b.phi_acc, b.d_step, P, b.d_status, b.ovf_list,
      b.ovf_count);
  return cudaGetLastError();
}

cudaError_t launch_voronoi3_export(const Geometry& g, const Buffers& b, int rep, int n, int pass, int32_t* deg,
                                   const int64_t* out_off, int32_t* out_ids, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const int nb = std::min((n + kV3Warps - 1) / kV3Warps, device_sm_count() * 4);
  voronoi3_export_kernel<<<nb, 32 * kV3Warps, sizeof(Warp3<CellL>) * kV3Warps, st>>>(
      g.reps, rep, b.bounds, (const int4*)b.S_pos, b.S_id, grid_view3(b), pass, deg, out_off, out_ids, b.d_status);
  return cudaGetLastError();
}

}  // namespace vk
