// vk_metric.cu -- the metric rule (Sec. "Metric and topological flocking
// models": each particle aligns with every particle within the interaction
// radius r0, the original Vicsek rule; Eq. 1 and Eq. 2), 2D and 3D.
//
// 2D: one warp steps 32 consecutive particles of the cell-sorted order
// together.  Particles of one coarse cell share a rectangle, the union of
// their squares [p - r0q, p + r0q]: the warp stages its candidates 32 at a time
// in shared memory, each with its heading already in fixed point, and every
// lane tests every candidate from broadcast reads.  In a dense cluster the
// squares overlap almost entirely (281 candidates per particle at 4M clustered,
// r0 = 1); one thread walking its own square read each of them from its own
// address and converted its heading again for every neighbor.  Measured there
// (GB300, us per step): 6103 with one thread per square, 2240 with the warp,
// although its rectangles hold 687 candidates per particle; bound by the issue
// of the tests.  3D: the rows of cells that the ball's cube meets, one thread per
// particle, or rings of cells where the cube is too wide.
// A candidate is a neighbor iff its exact int64 squared minimum-image
// distance is <= r0q^2.  The neighbor count has no bound, so nothing is
// buffered: the headings are summed as they are found, each component
// rounded to 2^-32 and added in int64.  Integer addition is associative, so
// the sum does not depend on the visiting order (which the atomic ranks of
// the cell sort leave free) and a step is bit-identical run to run; the
// rounding errs by at most 2^-33 per neighbor.  The sum is converted to
// FP64 for the update.
#include <algorithm>

#include "vk_box2d.cuh"

namespace vk {

namespace {

// slot runs one listing buffers per thread (shared memory)
struct MetricRuns {
  static constexpr int kRuns = VK_KNN2_BOX_RUNS;
  uint2 run[kRuns][kBlock];
};

// heading sum and count of the neighbors found so far
template <int DIM>
struct MetricSum {
  long long s[DIM];
  int m;
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int a = 0; a < DIM; ++a) s[a] = 0;
    m = 0;
  }
  __device__ __forceinline__ void add(const float* v) {
#pragma unroll
    for (int a = 0; a < DIM; ++a) s[a] += phi_fixed(v[a]);
    ++m;
  }
};

// (export) every neighbor of a slot (2D), found by the square walk, or by a
// scan of the whole replica when the square is too wide for it (r0 near a
// quarter of the box, or a coarse grid too small for the square)
struct MetricList2 {
  const Ctx& C;
  uint64_t r2;
  int32_t* out;
  int w;
  __device__ __forceinline__ void group(uint32_t q, uint32_t n, const int2* pj, uint32_t ox, uint32_t oy) {
#pragma unroll
    for (int u = 0; u < kGroup; ++u) {
      const int32_t dx = (int32_t)((uint32_t)pj[u].x - ox), dy = (int32_t)((uint32_t)pj[u].y - oy);
      const uint64_t D = (uint64_t)((int64_t)dx * dx) + (uint64_t)((int64_t)dy * dy);
      if ((uint32_t)u < n && D <= r2 && (int64_t)(q + (uint32_t)u) != C.self) {
        if (out) out[w] = (int32_t)(q + (uint32_t)u);
        ++w;
      }
    }
  }
};

// the whole replica, one candidate at a time (the fallback of the 2D walk)
template <class V>
__device__ __forceinline__ void metric_scan_all2(const Rep& R, const int2* __restrict__ pos, const Ctx& C, V& v) {
  for (int64_t q = R.p0; q < R.p0 + R.n; ++q) {
    int32_t dx, dy;
    box_offset(C, __ldg(pos + q), dx, dy);
    // offsets relative to the particle itself: ox = x_i - 0 in the same image
    const int2 pj = make_int2((int32_t)((uint32_t)C.px + (uint32_t)dx), (int32_t)((uint32_t)C.py + (uint32_t)dy));
    int2 g[kGroup] = {pj, pj, pj, pj};
    v.group((uint32_t)q, 1u, g, C.px, C.py);
  }
}

// Eq. (2) alignment + noise and Eq. (1) advection from the exact sum
template <int DIM>
__device__ __forceinline__ void metric_update(const Rep& R, const StepParams& P, uint32_t step, int32_t id,
                                              const float* ni, MetricSum<DIM>& S, const int32_t* pi,
                                              int32_t* pout, float* nout) {
  if (P.include_self) S.add(ni);
  HeadSum<DIM> H;
  H.init();
#pragma unroll
  for (int a = 0; a < DIM; ++a) H.d[a] = ldexp((double)S.s[a], -32);
  align_advect_mode<DIM>(R, P, 2, step, id, ni, H, S.m, pi, pout, nout);
}

// 32 candidates of a warp: position and fixed-point heading
struct MetricStage {
  int2 pos[32];
  longlong2 head[32];
};

constexpr int kMetricBlk = 128;

// WIDE: rectangles that reach half a period or meet a coarse cell twice are to be
// expected (metric_wide).  Such a one is then cut per axis, and minimum images are
// taken one by one (20,000 particles, r0 a fifth and a quarter of the box: 464 and 682
// us per step; the whole replica for such rectangles 2148 and 3424, one thread per
// square 1179 and 1459).  The narrow kernel takes the whole replica: with the other
// code in it, it loses 5 to 10 %.
template <bool WIDE>
__global__ void __launch_bounds__(kMetricBlk) metric2_step_kernel(
    const Rep* __restrict__ reps, const BlockTask* __restrict__ tasks, const int2* __restrict__ S_pos,
    const float2* __restrict__ S_dir, const int32_t* __restrict__ S_id, GridView G, int2* __restrict__ U_pos,
    float2* __restrict__ U_dir, int32_t* __restrict__ U_id, uint32_t* __restrict__ counts,
    PhiAcc* __restrict__ phi_acc, const int64_t* __restrict__ d_step, StepParams P) {
  __shared__ MetricStage stages[kMetricBlk / 32];
  __shared__ PhiShared phs;
  phi_block_begin(phs);
  MetricStage& M = stages[threadIdx.x >> 5];
  constexpr int kSplit = kBlock / kMetricBlk;
  const int lane = (int)(threadIdx.x & 31);
  const BlockTask t = tasks[blockIdx.x / kSplit];
  const Rep R = reps[t.rep];
  const int li = t.first + (int)(blockIdx.x % kSplit) * kMetricBlk + (int)threadIdx.x;
  const int64_t step = *d_step;
  float nnew[3] = {0.f, 0.f, 0.f};
  uint32_t n_cand = 0;
  const bool valid = li < R.n;
  const int64_t s = R.p0 + (valid ? li : 0);
  const int2 p = S_pos[s];
  const int nx = R.nc[0], ny = R.nc[1], shx = R.sh[0], shy = R.sh[1];
  const int64_t Lx = R.L[0], Ly = R.L[1], r = R.r0q;
  const int cx = (int)((uint32_t)p.x >> shx), cy = (int)((uint32_t)p.y >> shy);
  const int64_t r2 = r * r;
  MetricSum<2> S;
  S.init();
  unsigned left = __ballot_sync(0xffffffffu, valid);
  while (left) {
    // the lanes of one coarse cell
    const int lead = __ffs(left) - 1;
    const int lx = __shfl_sync(0xffffffffu, cx, lead), ly = __shfl_sync(0xffffffffu, cy, lead);
    const bool on = valid && cx == lx && cy == ly;
    left &= ~__ballot_sync(0xffffffffu, on);
    const int32_t x0 = __reduce_min_sync(0xffffffffu, on ? p.x : INT_MAX), x1 = __reduce_max_sync(0xffffffffu, on ? p.x : -1);
    const int32_t y0 = __reduce_min_sync(0xffffffffu, on ? p.y : INT_MAX), y1 = __reduce_max_sync(0xffffffffu, on ? p.y : -1);
    // their rectangle.  Offsets within it are exact in one image while it is
    // narrower than half a period and meets no coarse cell twice.  Otherwise
    // minimum images are taken one by one, of the whole replica, or (WIDE) of
    // the axes that it covers or meets a cell twice on and its part of the others.
    const int64_t ax = x0 - r, bx = x1 + r, ay = y0 - r, by = y1 + r;
    const long long lim = on ? r2 : -1;  // squared distances are >= 0: the other lanes find nothing
    bool image = 2 * (bx - ax + 1) >= Lx || 2 * (by - ay + 1) >= Ly;
    bool fullx = WIDE ? bx - ax + 1 >= Lx : image, fully = WIDE ? by - ay + 1 >= Ly : image;
    int ux0 = 0, ux1 = nx - 1, uy0 = 0, uy1 = ny - 1;
    if (!fullx) {
      ux0 = ucell2(ax, nx, shx, Lx);
      ux1 = ucell2(bx, nx, shx, Lx);
      fullx = ux1 - ux0 >= nx;
    }
    if (!fully) {
      uy0 = ucell2(ay, ny, shy, Ly);
      uy1 = ucell2(by, ny, shy, Ly);
      fully = uy1 - uy0 >= ny;
    }
    image = image || fullx || fully;
    if (WIDE) {
      if (fullx) ux0 = 0, ux1 = nx - 1;
      if (fully) uy0 = 0, uy1 = ny - 1;
    }
    // candidates [qb, qe); (ox, oy): the period added to their coordinates, or
    // (wrap) minimum images taken one by one
    auto scan = [&](int64_t qb, int64_t qe, uint32_t ox, uint32_t oy, bool wrap) {
      n_cand += on ? (uint32_t)(qe - qb) : 0u;
      for (int64_t q0 = qb; q0 < qe; q0 += 32) {
        const int n = (int)min(qe - q0, (int64_t)32);
        __syncwarp();
        if (lane < n) {
          const int2 pj = __ldg(S_pos + q0 + lane);
          const float2 d = __ldg(S_dir + q0 + lane);
          M.pos[lane] = make_int2((int32_t)((uint32_t)pj.x + ox), (int32_t)((uint32_t)pj.y + oy));
          M.head[lane] = make_longlong2(phi_fixed(d.x), phi_fixed(d.y));
        }
        __syncwarp();
        auto test = [&](int j, bool image_j) {
          const int2 pj = M.pos[j];
          int32_t dx = (int32_t)((uint32_t)pj.x - (uint32_t)p.x), dy = (int32_t)((uint32_t)pj.y - (uint32_t)p.y);
          if (image_j && !WIDE) {  // (seldom; short code for it costs the other loop registers)
            dx = (int32_t)min_image((int64_t)pj.x - p.x, Lx);
            dy = (int32_t)min_image((int64_t)pj.y - p.y, Ly);
          } else if (image_j) {  // a distance of half a period is the same in both images
            dx = (uint32_t)abs(dx) > R.L[0] / 2 ? (int32_t)(R.L[0] - (uint32_t)abs(dx)) : dx;
            dy = (uint32_t)abs(dy) > R.L[1] / 2 ? (int32_t)(R.L[1] - (uint32_t)abs(dy)) : dy;
          }
          if ((int64_t)dx * dx + (int64_t)dy * dy <= lim) {
            const longlong2 h = M.head[j];
            S.s[0] += h.x;
            S.s[1] += h.y;
            ++S.m;
          }
        };
        if (wrap && !WIDE) {
          for (int j = 0; j < n; ++j) test(j, true);
        } else if (wrap) {
#pragma unroll 4
          for (int j = 0; j < n; ++j) test(j, true);
        } else {
#pragma unroll 4
          for (int j = 0; j < n; ++j) test(j, false);
        }
      }
    };
    if (WIDE ? fullx && fully : image) {
      scan(R.p0, R.p0 + R.n, 0u, 0u, true);
      continue;
    }
    const bool wrap = WIDE && image;
    const uint32_t fx0 = cell_frac((uint32_t)(ax < 0 ? ax + Lx : ax), shx);
    const uint32_t fx1 = cell_frac((uint32_t)(bx >= Lx ? bx - Lx : bx), shx);
    const uint32_t fy0 = cell_frac((uint32_t)(ay < 0 ? ay + Ly : ay), shy);
    const uint32_t fy1 = cell_frac((uint32_t)(by >= Ly ? by - Ly : by), shy);
    for (int uy = uy0; uy <= uy1; ++uy)
      for (int ux = ux0; ux <= ux1; ++ux) {
        const int wy = uy < 0 ? uy + ny : (uy >= ny ? uy - ny : uy);
        const int wx = ux < 0 ? ux + nx : (ux >= nx ? ux - nx : ux);
        const uint32_t ox = wrap ? 0u : ux < 0 ? 0u - R.L[0] : (ux >= nx ? R.L[0] : 0u);
        const uint32_t oy = wrap ? 0u : uy < 0 ? 0u - R.L[1] : (uy >= ny ? R.L[1] : 0u);
        const int64_t gc = R.c0 + (int64_t)wy * nx + wx;
        const uint32_t base = __ldg(G.sub_base + gc);
        const int sd = __ldg(G.sub_s + gc);
        const bool allx = WIDE && fullx, ally = WIDE && fully;
        const int c0 = ux == ux0 && !allx ? sub_of(fx0, sd) : 0, c1 = ux == ux1 && !allx ? sub_of(fx1, sd) : sd - 1;
        const int r0 = uy == uy0 && !ally ? sub_of(fy0, sd) : 0, r1 = uy == uy1 && !ally ? sub_of(fy1, sd) : sd - 1;
        if (c0 == 0 && c1 == sd - 1) {  // whole rows follow one another
          scan(__ldg(G.sub_off + base + r0 * sd), __ldg(G.sub_off + base + (r1 + 1) * sd), ox, oy, wrap);
          continue;
        }
        for (int rr = r0; rr <= r1; rr += 32) {
          uint32_t qb = 0, qe = 0;  // each lane looks up one row of sub-cells
          if (rr + lane <= r1) {
            const uint32_t lo = base + (uint32_t)((rr + lane) * sd);
            qb = __ldg(G.sub_off + lo + c0);
            qe = __ldg(G.sub_off + lo + c1 + 1);
          }
          unsigned rows = __ballot_sync(0xffffffffu, qe > qb);
          while (rows) {
            const int j = __ffs(rows) - 1;
            rows &= rows - 1u;
            scan(__shfl_sync(0xffffffffu, qb, j), __shfl_sync(0xffffffffu, qe, j), ox, oy, wrap);
          }
        }
      }
  }
  if (valid) {
    const float2 nv = S_dir[s];
    const float ni[3] = {nv.x, nv.y, 0.f};
    // the particle met itself once, at distance zero
    S.s[0] -= phi_fixed(nv.x);
    S.s[1] -= phi_fixed(nv.y);
    --S.m;
    const int32_t id = S_id[s];
    const int32_t pi[3] = {p.x, p.y, 0};
    int32_t pout[3] = {0, 0, 0};
    metric_update<2>(R, P, (uint32_t)step, id, ni, S, pi, pout, nnew);
    U_pos[s] = make_int2(pout[0], pout[1]);
    U_dir[s] = make_float2(nnew[0], nnew[1]);
    U_id[s] = id;
    atomicAdd(counts + linear_cell<2>(R, pout), 1u);
  }
  record_search_stats(P.stats, valid, n_cand, 1u);
  phi_block_end<2>(phs, nnew, phi_acc + ((size_t)(step % P.phi_cap) * (size_t)P.n_rep + (size_t)t.rep) * 3);
}

// 3D: every particle within r0q of slot self, from the rows of cells that the
// cube [p - r0q, p + r0q]^3 meets (contiguous runs, each in one periodic
// image); where the cube is too wide for that, from rings of cells until every
// unscanned particle is farther.  (64-bit divisions for the ring bounds and
// minimum images cost more than the distances.)
template <class F>
__device__ __forceinline__ void metric_walk3(const Rep& R, int64_t self, const int32_t* pi,
                                             const int4* __restrict__ pos, const GridView& G,
                                             const uint32_t* __restrict__ bounds, uint32_t* n_cand, uint32_t* n_runs,
                                             F& f) {
  const int64_t r = R.r0q;
  const uint64_t r2 = (uint64_t)r * (uint64_t)r;
  int lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
  bool fits = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int64_t L = R.L[a];
    fits = fits && 4 * r + 2 < L;
    if (fits) {
      const uint32_t* bnd = bounds + R.bnd[a];
      const int64_t x0 = pi[a] - r, x1 = pi[a] + r;
      lo[a] = cell_of_tab((uint32_t)(x0 < 0 ? x0 + L : x0), R.nc[a], bnd, R.inv_w[a]) - (x0 < 0 ? R.nc[a] : 0);
      hi[a] = cell_of_tab((uint32_t)(x1 >= L ? x1 - L : x1), R.nc[a], bnd, R.inv_w[a]) + (x1 >= L ? R.nc[a] : 0);
      fits = hi[a] - lo[a] < R.nc[a];
    }
  }
  if (!fits) {
    auto run = [&](uint32_t qb, uint32_t qe) {
      *n_cand += qe - qb;
      *n_runs += 1;
      for (uint32_t q = qb; q < qe; ++q) {
        if ((int64_t)q == self) continue;
        const int4 pj = __ldg(pos + q);
        const int32_t pjv[3] = {pj.x, pj.y, pj.z};
        uint64_t D = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int64_t d = min_image((int64_t)pjv[a] - (int64_t)pi[a], (int64_t)R.L[a]);
          D += (uint64_t)(d * d);
        }
        if (D <= r2) f(q);
      }
    };
    auto stop = [&](uint64_t B2) { return B2 > r2; };
    grid_walk3(R, pi, G, run, stop);
    return;
  }
  const int nx = R.nc[0], ny = R.nc[1], nz = R.nc[2];
  for (int uz = lo[2]; uz <= hi[2]; ++uz) {
    const int cz = uz < 0 ? uz + nz : (uz >= nz ? uz - nz : uz);
    const uint32_t oz = (uint32_t)pi[2] + (uz < 0 ? R.L[2] : 0u) - (uz >= nz ? R.L[2] : 0u);
    for (int uy = lo[1]; uy <= hi[1]; ++uy) {
      const int cy = uy < 0 ? uy + ny : (uy >= ny ? uy - ny : uy);
      const uint32_t oy = (uint32_t)pi[1] + (uy < 0 ? R.L[1] : 0u) - (uy >= ny ? R.L[1] : 0u);
      const int64_t row = R.c0 + ((int64_t)cz * ny + cy) * nx;
      for (int xs = lo[0]; xs <= hi[0];) {  // the x range splits at the period
        const int wx = xs < 0 ? xs + nx : (xs >= nx ? xs - nx : xs);
        const int xe = min(hi[0], xs < 0 ? -1 : (xs < nx ? nx - 1 : INT_MAX));
        const uint32_t ox = (uint32_t)pi[0] + (xs < 0 ? R.L[0] : 0u) - (xs >= nx ? R.L[0] : 0u);
        const uint32_t qb = __ldg(G.off + row + wx), qe = __ldg(G.off + row + wx + (xe - xs) + 1);
        xs = xe + 1;
        *n_cand += qe - qb;
        *n_runs += 1;
        for (uint32_t q = qb; q < qe; ++q) {
          const int4 pj = __ldg(pos + q);
          const int32_t dx = (int32_t)((uint32_t)pj.x - ox), dy = (int32_t)((uint32_t)pj.y - oy),
                        dz = (int32_t)((uint32_t)pj.z - oz);
          const uint64_t D = (uint64_t)((int64_t)dx * dx) + (uint64_t)((int64_t)dy * dy) +
                             (uint64_t)((int64_t)dz * dz);
          if (D <= r2 && (int64_t)q != self) f(q);
        }
      }
    }
  }
}

__global__ void __launch_bounds__(kBlock) metric3_step_kernel(
    const Rep* __restrict__ reps, const BlockTask* __restrict__ tasks, const uint32_t* __restrict__ bounds, const int4* __restrict__ S_pos,
    const float4* __restrict__ S_dir, const int32_t* __restrict__ S_id, GridView G, int4* __restrict__ U_pos,
    float4* __restrict__ U_dir, int32_t* __restrict__ U_id, uint32_t* __restrict__ U_rank, uint32_t* __restrict__ counts,
    PhiAcc* __restrict__ phi_acc, const int64_t* __restrict__ d_step, StepParams P) {
  const BlockTask t = tasks[blockIdx.x];
  const Rep R = reps[t.rep];
  const int li = t.first + (int)threadIdx.x;
  const int64_t step = *d_step;
  float nnew[3] = {0.f, 0.f, 0.f};
  uint32_t n_cand = 0, n_runs = 0;
  if (li < R.n) {
    const int64_t s = R.p0 + li;
    int32_t pi[3];
    float ni[3];
    unpack(S_pos[s], pi);
    unpack(S_dir[s], ni);
    const int32_t id = S_id[s];
    MetricSum<3> S;
    S.init();
    auto add = [&](uint32_t q) {
      float v[3];
      unpack(__ldg(S_dir + q), v);
      S.add(v);
    };
    metric_walk3(R, s, pi, S_pos, G, bounds, &n_cand, &n_runs, add);
    int32_t pout[3] = {0, 0, 0};
    metric_update<3>(R, P, (uint32_t)step, id, ni, S, pi, pout, nnew);
    U_pos[s] = make_int4(pout[0], pout[1], pout[2], 0);
    U_dir[s] = make_float4(nnew[0], nnew[1], nnew[2], 0.f);
    U_id[s] = id;
    int64_t lin = 0;
#pragma unroll
    for (int a = 2; a >= 0; --a)
      lin = lin * R.nc[a] + cell_of_tab((uint32_t)pout[a], R.nc[a], bounds + R.bnd[a], R.inv_w[a]);
    U_rank[s] = atomicAdd(counts + R.c0 + lin, 1u);
  }
  record_search_stats(P.stats, li < R.n, n_cand, n_runs);
  block_phi_accumulate<3>(nnew, phi_acc + ((size_t)(step % P.phi_cap) * (size_t)P.n_rep + (size_t)t.rep) * 3);
}

// sort row [b, e) of ids in place (insertion sort: rows are short, and the
// export is off the step path)
__device__ __forceinline__ void sort_row(int32_t* __restrict__ ids, int64_t b, int64_t e) {
  for (int64_t i = b + 1; i < e; ++i) {
    const int32_t x = ids[i];
    int64_t j = i;
    while (j > b && ids[j - 1] > x) {
      ids[j] = ids[j - 1];
      --j;
    }
    ids[j] = x;
  }
}

// Neighbor lists of one replica by id.  Pass 0: deg[id] = count.  Pass 1:
// the neighbor ids of row id at out_off[id] (the slots are collected in
// out_ids first, then mapped to ids and sorted).
__global__ void __launch_bounds__(kBlock) metric2_export_kernel(const Rep* __restrict__ reps, int rep,
                                                                const int2* __restrict__ S_pos,
                                                                const int32_t* __restrict__ S_id, GridView G,
                                                                int pass, int32_t* __restrict__ deg,
                                                                const int64_t* __restrict__ out_off,
                                                                int32_t* __restrict__ out_ids) {
  __shared__ MetricRuns H;
  const Rep R = reps[rep];
  const int li = blockIdx.x * kBlock + (int)threadIdx.x;
  // no early return: every thread of the block reaches the end together
  if (li < R.n) {
    const int64_t s = R.p0 + li;
    const int32_t id = S_id[s];
    Ctx C;
    init_ctx(C, R, s, S_pos[s]);
    int32_t* row = pass == 1 ? out_ids + out_off[id] : nullptr;
    MetricList2 v{C, (uint64_t)R.r0q * (uint64_t)R.r0q, row, 0};
    BoxCount bc;
    if (!box_walk(H, R, G, S_pos, C, (int64_t)R.r0q, bc, v)) {
      v.w = 0;
      metric_scan_all2(R, S_pos, C, v);
    }
    if (pass == 0) {
      deg[id] = v.w;
    } else {
      for (int j = 0; j < v.w; ++j) row[j] = __ldg(S_id + row[j]);
      sort_row(row, 0, v.w);
    }
  }
}

__global__ void __launch_bounds__(kBlock) metric3_export_kernel(const Rep* __restrict__ reps, int rep,
                                                                const uint32_t* __restrict__ bounds,
                                                                const int4* __restrict__ S_pos,
                                                                const int32_t* __restrict__ S_id, GridView G,
                                                                int pass, int32_t* __restrict__ deg,
                                                                const int64_t* __restrict__ out_off,
                                                                int32_t* __restrict__ out_ids) {
  const Rep R = reps[rep];
  const int li = blockIdx.x * kBlock + (int)threadIdx.x;
  if (li >= R.n) return;
  const int64_t s = R.p0 + li;
  const int32_t id = S_id[s];
  int32_t pi[3];
  unpack(S_pos[s], pi);
  int32_t* row = pass == 1 ? out_ids + out_off[id] : nullptr;
  int w = 0;
  auto put = [&](uint32_t q) {
    if (row) row[w] = __ldg(S_id + q);
    ++w;
  };
  uint32_t n_cand = 0, n_runs = 0;
  metric_walk3(R, s, pi, S_pos, G, bounds, &n_cand, &n_runs, put);
  if (pass == 0) deg[id] = w;
  else sort_row(row, 0, w);
}

GridView metric_view(const Buffers& b) {
  GridView G;
  G.off = b.offsets;
  G.sub_s = b.sub_s;
  G.sub_base = b.sub_base;
  G.sub_off = b.sub_off;
  return G;
}

}  // namespace

cudaError_t launch_metric_step(const Geometry& g, const Buffers& b, const StepParams& P, cudaStream_t st) {
  if (g.dim == 2) {
    auto kernel = g.metric_wide ? metric2_step_kernel<true> : metric2_step_kernel<false>;
    kernel<<<g.n_tasks * (kBlock / kMetricBlk), kMetricBlk, 0, st>>>(
        g.reps, g.tasks, (const int2*)b.S_pos, (const float2*)b.S_dir, b.S_id, metric_view(b), (int2*)b.U_pos,
        (float2*)b.U_dir, b.U_id, b.counts, b.phi_acc, b.d_step, P);
  } else {
    metric3_step_kernel<<<g.n_tasks, kBlock, 0, st>>>(g.reps, g.tasks, b.bounds, (const int4*)b.S_pos,
                                                      (const float4*)b.S_dir, b.S_id, metric_view(b),
                                                      (int4*)b.U_pos, (float4*)b.U_dir, b.U_id, b.U_rank, b.counts,
                                                      b.phi_acc, b.d_step, P);
  }
  return cudaGetLastError();
}

cudaError_t launch_metric_export(const Geometry& g, const Buffers& b, int rep, int n, int pass, int32_t* deg,
                                 const int64_t* out_off, int32_t* out_ids, cudaStream_t st) {
  const int nb = (n + kBlock - 1) / kBlock;
  if (nb == 0) return cudaSuccess;
  if (g.dim == 2) {
    metric2_export_kernel<<<nb, kBlock, 0, st>>>(g.reps, rep, (const int2*)b.S_pos, b.S_id,
                                                 metric_view(b), pass, deg, out_off, out_ids);
  } else {
    metric3_export_kernel<<<nb, kBlock, 0, st>>>(g.reps, rep, b.bounds, (const int4*)b.S_pos, b.S_id, metric_view(b), pass,
                                                 deg, out_off, out_ids);
  }
  return cudaGetLastError();
}

}  // namespace vk
