// vk_voronoi_fast.cuh -- the Voronoi cell builder of the 2D kernels (the
// Voronoi rule's main kernel and the tissue model's cell pass), for the
// ordinary cell: up to 16 edges, inside half a period, no coincident
// particles.  Anything else is reported, and built by the general code of
// vk_voronoi.cuh, whose predicates this builder shares.
//
// Eight lanes build one cell, four cells per warp, in step: lane j holds edges
// j and j + 8 of the polygon (site, vertex estimate and its error bound) in
// registers.  A candidate is tested against all vertices at once and its cut
// run read off a ballot; clipping is a rotation of the polygon (shuffles) with
// the new site at its end and two new vertices, solved side by side.  Up to 24
// candidates at a time, three per lane, are filtered against the cell, and the
// nearest of those that may cut goes first.
//
// The search goes in stages: a small square around the particle, larger ones
// while the cell is still wide (or last step's neighbors, where the last cell
// was a large one), then the cell's relevance box: a site can cut the cell only
// inside the union of the disks through the particle centred at the vertices.
//
// The kernels are bound by instruction issue and fetch.  One thread per cell,
// with the polygon in shared memory, kept 5.6 to 7.5 of 32 lanes busy, because
// lanes clip at different times and run loops of different lengths; eight
// lanes per cell keep 24 busy.  Measured (GB300, us per step, one thread per
// cell with the polygon in thread-local memory / this): 65,536 particles beside
// a lattice 889 / 306, 1M uniform 10751 / 3176.
#pragma once
#include "vk_voronoi.cuh"

namespace vk {

namespace {

// half-width of the first square in sub-cells (0.75, 1.0, 1.3: 65,536 particles
// 4969, 3515, 3719 us per 10 steps, 1M 8167, 7473, 7076 per 2)
#ifndef VK_VOR_SQUARE
#define VK_VOR_SQUARE 1.0f
#endif
// a cell that reaches farther than this many half-widths gets a larger square first
// seeds that leave a cell this many times as wide as the one they come from are
// followed by the squares (1.25, 2, 4: 65,536 particles 3717, 3727, 3733 us, 150 to
// 8000 within 4 %)
#ifndef VK_VOR_STALE
#define VK_VOR_STALE 2.0f
#endif
#ifndef VK_VOR_REACH
#define VK_VOR_REACH 4.0f
#endif

constexpr int kEdges = 16;  // edges of an ordinary cell, also on the way
constexpr int kCG = 8;      // lanes per cell
constexpr int kPer = 3;     // candidates per lane and batch

// Cursor over the slot runs of a rectangle [x0, x1] x [y0, y1] of offsets
// around a particle: the rows of sub-cells of the coarse cells it meets, each
// with the periodic image its cell lies in.
struct RowCursor {
  int ucx0, ucx1, ucy1, ucx, ucy;   // unwrapped coarse cells
  uint32_t fx0, fx1, fy0, fy1;      // in-cell fractions of the corners
  int ucy0, row, row_end, s;
  uint32_t lo, hi;                  // first and one-past-last sub-cell of the row
  uint32_t code;                    // image of the current cell: 4 / 8 at -L / +L in x, 1 / 2 in y

  // false when the rectangle reaches half a period or meets a coarse cell twice
  __device__ __forceinline__ bool init(const Rep& R, int2 p, int32_t x0, int32_t x1, int32_t y0, int32_t y1) {
    const int32_t hx = (int32_t)(R.L[0] / 2) - 2, hy = (int32_t)(R.L[1] / 2) - 2;
    if (x0 <= -hx || x1 >= hx || y0 <= -hy || y1 >= hy) return false;
    const int64_t ax = (int64_t)p.x + x0, bx = (int64_t)p.x + x1, ay = (int64_t)p.y + y0, by = (int64_t)p.y + y1;
    const int64_t Lx = R.L[0], Ly = R.L[1];
    ucx0 = ucell2(ax, R.nc[0], R.sh[0], Lx);
    ucx1 = ucell2(bx, R.nc[0], R.sh[0], Lx);
    ucy0 = ucell2(ay, R.nc[1], R.sh[1], Ly);
    ucy1 = ucell2(by, R.nc[1], R.sh[1], Ly);
    if (ucx1 - ucx0 >= R.nc[0] || ucy1 - ucy0 >= R.nc[1]) return false;
    fx0 = cell_frac((uint32_t)(ax < 0 ? ax + Lx : ax), R.sh[0]);
    fx1 = cell_frac((uint32_t)(bx >= Lx ? bx - Lx : bx), R.sh[0]);
    fy0 = cell_frac((uint32_t)(ay < 0 ? ay + Ly : ay), R.sh[1]);
    fy1 = cell_frac((uint32_t)(by >= Ly ? by - Ly : by), R.sh[1]);
    ucx = ucx0;
    ucy = ucy0;
    row = 0;
    row_end = -1;
    return true;
  }

  // next run [*qb, *qe); false at the end (runs may be empty)
  __device__ __forceinline__ bool next(const Rep& R, const GridView& G, uint32_t* qb, uint32_t* qe) {
    if (row > row_end) {
      if (ucx > ucx1) {
        ucx = ucx0;
        ++ucy;
      }
      if (ucy > ucy1) return false;
      const int nx = R.nc[0], ny = R.nc[1];
      const int cy = ucy < 0 ? ucy + ny : (ucy >= ny ? ucy - ny : ucy);
      const int cx = ucx < 0 ? ucx + nx : (ucx >= nx ? ucx - nx : ucx);
      code = (ucx < 0 ? 4u : (ucx >= nx ? 8u : 0u)) | (ucy < 0 ? 1u : (ucy >= ny ? 2u : 0u));
      const int64_t gc = R.c0 + (int64_t)cy * nx + cx;
      const uint32_t base = __ldg(G.sub_base + gc);
      s = __ldg(G.sub_s + gc);
      if (s == 1) {
        // unsplit cells of a row follow one another: take all of them up to
        // the rectangle's end or the period's in one run
        const int last = min(ucx1, ucx < 0 ? -1 : (ucx < nx ? nx - 1 : 2 * nx - 1));
        const int64_t ge = gc + (last - ucx);
        const uint32_t be = __ldg(G.sub_base + ge + 1);
        if (be - base == (uint32_t)(last - ucx + 1)) {
          *qb = __ldg(G.sub_off + base);
          *qe = __ldg(G.sub_off + be);
          ucx = last + 1;
          return true;
        }
      }
      const int sx0 = ucx == ucx0 ? sub_of(fx0, s) : 0, sx1 = ucx == ucx1 ? sub_of(fx1, s) : s - 1;
      row = ucy == ucy0 ? sub_of(fy0, s) : 0;
      row_end = ucy == ucy1 ? sub_of(fy1, s) : s - 1;
      lo = base + (uint32_t)(row * s + sx0);
      hi = lo + (uint32_t)(sx1 - sx0 + 1);
      ++ucx;
    }
    *qb = __ldg(G.sub_off + lo);
    *qe = __ldg(G.sub_off + hi);
    ++row;
    lo += (uint32_t)s;
    hi += (uint32_t)s;
    return true;
  }
};

// Vertex estimate as vertex_geom's, with one reciprocal for its quotients:
// the three roundings left (of the doubled determinant, its reciprocal and the
// product) stay within the four units that its error bound allows for.
__device__ __forceinline__ bool vertex_est(int2 a, int2 b, float2* v, float* e) {
  const int64_t dh = (int64_t)a.x * b.y - (int64_t)a.y * b.x;  // exact, > 0 for consecutive sites
  if (dh <= 0) return false;
  const float fax = (float)a.x, fay = (float)a.y, fbx = (float)b.x, fby = (float)b.y;
  const float al = fax * fax + fay * fay, bl = fbx * fbx + fby * fby;
  const float p1 = fby * al, p2 = fay * bl, p3 = fax * bl, p4 = fbx * al;
  const float inv = __frcp_rn(2.0f * (float)dh);
  // numerator errors: 16 ulps of the magnitudes (inputs, squares, products, difference)
  const float ex = (fabsf(p1) + fabsf(p2)) * 9.5367431640625e-07f;
  const float ey = (fabsf(p3) + fabsf(p4)) * 9.5367431640625e-07f;
  v->x = (p1 - p2) * inv;
  v->y = (p3 - p4) * inv;
  const float up = inv * (1.0f + 4.76837158203125e-07f);
  const float ax = (fabsf(p1 - p2) + ex) * up, ay = (fabsf(p3 - p4) + ey) * up;  // bounds of |Vx|, |Vy|
  const float e0 = (fmaxf(ex, ey) * up + fmaxf(ax, ay) * 4.76837158203125e-07f) * 1.5f;
  *e = e0 < 3.0e38f ? e0 : 3.0e38f;  // (also of an infinity or NaN)
  return true;
}


constexpr unsigned kAll = 0xffffffffu;

__device__ __forceinline__ float group_max(float v) {
#pragma unroll
  for (int o = 1; o < kCG; o <<= 1) v = fmaxf(v, __shfl_xor_sync(kAll, v, o));
  return v;
}
__device__ __forceinline__ float group_min(float v) { return -group_max(-v); }

// One group's cell.  Every member is called by the whole warp (the four groups
// stay in step); "group" values are the same in a group's eight lanes.
struct Cell8 {
  int gl, base;            // lane within the group, the group's first lane
  int m;                   // edges (group)
  bool other;              // the general code has to build the cell (group)
  float r2max, k1;         // largest |V|^2; tolerance per |mx| + |my| of a candidate (group)
  uint32_t n_seen;         // candidates met (group)
  int2 q[2];               // edge gl + 8 i: site offset, sorted slot, vertex to the next edge, error bound
  int32_t slot[2];
  float2 v[2];
  float e[2];

  __device__ __forceinline__ bool has(int i) const { return gl + 8 * i < m; }
  __device__ __forceinline__ unsigned group_bits(bool b) const { return (__ballot_sync(kAll, b) >> base) & 255u; }

  // the site after each of the lane's edges
  __device__ __forceinline__ void next_sites(bool big, int2* nq) const {
    const int a = gl + 1 == m ? 0 : gl + 1;
    nq[0].x = __shfl_sync(kAll, q[0].x, base + (a & 7));
    nq[0].y = __shfl_sync(kAll, q[0].y, base + (a & 7));
    if (big) {
      const int x8 = __shfl_sync(kAll, q[1].x, base), y8 = __shfl_sync(kAll, q[1].y, base);
      const int x0 = __shfl_sync(kAll, q[0].x, base), y0 = __shfl_sync(kAll, q[0].y, base);
      if (a == 8) nq[0] = make_int2(x8, y8);
      const int b = gl + 9 == m ? 0 : gl + 9;
      nq[1].x = __shfl_sync(kAll, q[1].x, base + (b & 7));
      nq[1].y = __shfl_sync(kAll, q[1].y, base + (b & 7));
      if (b == 0) nq[1] = make_int2(x0, y0);
    }
  }

  // the square of the particle's own images
  __device__ __forceinline__ void init(uint32_t Lx, uint32_t Ly) {
    const int32_t X = (int32_t)Lx, Y = (int32_t)Ly;
    const float fx = 0.5f * (float)X, fy = 0.5f * (float)Y;
    m = 4;
    other = false;
    n_seen = 0;
    q[0] = make_int2(gl == 0 ? X : gl == 2 ? -X : 0, gl == 1 ? Y : gl == 3 ? -Y : 0);
    v[0] = make_float2(gl == 0 || gl == 3 ? fx : -fx, gl < 2 ? fy : -fy);
    e[0] = fmaxf(fx, fy) * 1.1920929e-07f;
    slot[0] = slot[1] = -1;
    q[1] = make_int2(0, 0);
    v[1] = make_float2(0.f, 0.f);
    e[1] = 0.f;
    bounds();
  }

  __device__ __forceinline__ void bounds() {
    float mx = 0.f, em = 0.f;
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (has(i)) {
        const float x = fabsf(v[i].x) + e[i], y = fabsf(v[i].y) + e[i];
        mx = fmaxf(mx, x * x + y * y);
        em = fmaxf(em, e[i]);
      }
    r2max = group_max(mx) * (1.0f + 9.5367431640625e-07f);
    // |V| <= sqrt(r2max); as vertex_cut_fast's tolerance, for the worst vertex
    k1 = 3.0f * group_max(em) + 2.9e-06f * sqrtf(r2max);
  }

  // the relevance box
  __device__ __forceinline__ void box(float* x0, float* x1, float* y0, float* y1) const {
    *x0 = *y0 = 3.0e38f;
    *x1 = *y1 = -3.0e38f;
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (has(i)) {
        const float x = fabsf(v[i].x) + e[i], y = fabsf(v[i].y) + e[i];
        const float r = __fadd_ru(__fsqrt_ru((x * x + y * y) * (1.0f + 9.5367431640625e-07f)), e[i]);
        *x0 = fminf(*x0, __fsub_rd(v[i].x, r));
        *x1 = fmaxf(*x1, __fadd_ru(v[i].x, r));
        *y0 = fminf(*y0, __fsub_rd(v[i].y, r));
        *y1 = fmaxf(*y1, __fadd_ru(v[i].y, r));
      }
    *x0 = group_min(*x0);
    *x1 = group_max(*x1);
    *y0 = group_min(*y0);
    *y1 = group_max(*y1);
  }

  // (kPer candidates per lane) drop the flags of those that cannot cut or touch the group's cell
  __device__ __forceinline__ void filter(bool* flag, const int32_t* mx, const int32_t* my) const {
    float fx[kPer], fy[kPer], t[kPer];
#pragma unroll
    for (int s = 0; s < kPer; ++s) {
      fx[s] = (float)mx[s];
      fy[s] = (float)my[s];
      t[s] = -3.0e38f;
    }
    const int most = __reduce_max_sync(kAll, m);
#pragma unroll 1
    for (int a = 0; a < most; ++a) {
      const float x = __shfl_sync(kAll, a < 8 ? v[0].x : v[1].x, base + (a & 7));
      const float y = __shfl_sync(kAll, a < 8 ? v[0].y : v[1].y, base + (a & 7));
      if (a < m)
#pragma unroll
        for (int s = 0; s < kPer; ++s) t[s] = fmaxf(t[s], fmaf(fx[s], x, fy[s] * y));
    }
#pragma unroll
    for (int s = 0; s < kPer; ++s) {
      const float D = fx[s] * fx[s] + fy[s] * fy[s];
      flag[s] = flag[s] && D * (1.0f - 4.76837158203125e-07f) <= 4.0f * r2max &&
                2.0f * t[s] - D >= -((fabsf(fx[s]) + fabsf(fy[s])) * k1 + D * 1.9073486328125e-06f);
    }
  }

  // clip by the site at offset (mx, my) in sorted slot sl (group; `on`: this group has one)
  __device__ __forceinline__ void clip(bool on, int32_t mx, int32_t my, int32_t sl) {
    const bool big = __any_sync(kAll, m > 8);
    unsigned mask = 0, open = 0;
    int f[2] = {-1, -1};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (i == 1 && !big) break;
      if (on && has(i)) f[i] = vertex_cut_fast(v[i].x, v[i].y, e[i], mx, my);
      mask |= group_bits(f[i] > 0) << (8 * i);
      open |= __ballot_sync(kAll, f[i] == 0);
    }
    if (open) {  // vertices that the estimate leaves undecided: exactly
      // (no work for a site that is an edge already: a seed that comes round again)
      const bool edge = group_bits((has(0) && slot[0] == sl) || (has(1) && slot[1] == sl)) != 0;
      if (edge) f[0] = f[1] = -1;
      int2 nq[2];
      next_sites(big, nq);
      bool touch = false;
      mask = 0;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (i == 1 && !big) break;
        if (f[i] == 0) {
          f[i] = vertex_cut_sign(q[i].x, q[i].y, nq[i].x, nq[i].y, mx, my);
          touch = touch || f[i] == 0;
        }
        mask |= group_bits(f[i] > 0) << (8 * i);
      }
      // no vertex cut, some on the bisector: a second particle at an edge site's place?
      const bool touched = group_bits(touch) != 0 && mask == 0;
      bool twin = false;
#pragma unroll
      for (int i = 0; i < 2; ++i) twin = twin || (has(i) && q[i].x == mx && q[i].y == my && slot[i] != sl);
      if (group_bits(touched && twin)) other = true;
    }
    bool cut = on && !other && mask != 0;
    // the vertices strictly beyond the bisector form one cyclic run [s, s + c)
    const int c = __popc(mask);
    const unsigned starts = mask & ~(mask << 1 | mask >> (m - 1));
    const int kept = m - c + 1;  // sites that stay
    if (cut && (__popc(starts) != 1 || c >= m || kept >= kEdges)) {
      other = true;  // outgrown (or an inconsistency, for the general code to report)
      cut = false;
    }
    if (!__any_sync(kAll, cut)) return;
    int first = __ffs(starts) - 1 + c;  // the first site that stays
    if (first >= m) first -= m;
    const int old = m;
    if (cut) m = kept + 1;
    const bool grown = big || __any_sync(kAll, m > 8);
    // edge a of the new polygon is edge (first + a) mod old
    const int2 oq[2] = {q[0], q[1]};
    const float2 ov[2] = {v[0], v[1]};
    const int32_t os[2] = {slot[0], slot[1]};
    const float oe[2] = {e[0], e[1]};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (i == 1 && !grown) break;
      int j = first + gl + 8 * i;
      if (j >= old) j -= old;
      const int from = base + (j & 7);
      int2 nq = make_int2(__shfl_sync(kAll, oq[0].x, from), __shfl_sync(kAll, oq[0].y, from));
      float2 nv = make_float2(__shfl_sync(kAll, ov[0].x, from), __shfl_sync(kAll, ov[0].y, from));
      int32_t ns = __shfl_sync(kAll, os[0], from);
      float ne = __shfl_sync(kAll, oe[0], from);
      if (big) {
        const int2 hq = make_int2(__shfl_sync(kAll, oq[1].x, from), __shfl_sync(kAll, oq[1].y, from));
        const float2 hv = make_float2(__shfl_sync(kAll, ov[1].x, from), __shfl_sync(kAll, ov[1].y, from));
        const int32_t hs = __shfl_sync(kAll, os[1], from);
        const float he = __shfl_sync(kAll, oe[1], from);
        if (j >= 8) {
          nq = hq;
          nv = hv;
          ns = hs;
          ne = he;
        }
      }
      if (cut && gl + 8 * i < kept) {
        q[i] = nq;
        v[i] = nv;
        slot[i] = ns;
        e[i] = ne;
      } else if (cut && gl + 8 * i == kept) {
        q[i] = make_int2(mx, my);
        slot[i] = sl;
      }
    }
    // the two new vertices, before and after the new site
    int2 nq[2];
    next_sites(grown, nq);
    bool bad = false;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (i == 1 && !grown) break;
      const int a = gl + 8 * i;
      if (cut && (a == kept || a == kept - 1)) bad = bad || !vertex_est(q[i], nq[i], &v[i], &e[i]);
    }
    if (group_bits(bad)) other = true;
  }

  // The cell of the particle at slot `self` (group; `on`: the group has one).
  // More than `budget` candidates also leave the cell to the general code.
  __device__ __forceinline__ void build(bool on, const Rep& R, int64_t self, int2 p, const int2* __restrict__ pos,
                                        const GridView& G, const Seeds& sd, uint32_t budget) {
    const int32_t X = (int32_t)R.L[0], Y = (int32_t)R.L[1];
    init(R.L[0], R.L[1]);
    RowCursor rc;
    int32_t skip = 0;  // sites with both offsets below it have been visited
    enum : int { kSeeds, kSquare, kBox };
    int stage = sd.n > 0 ? kSeeds : kSquare;
    float w = 0.f;  // half-width of the square of the stage
    const float wmax = 0.125f * fminf((float)X, (float)Y);
    if (on) {
      const int32_t pi[2] = {p.x, p.y};
      const int64_t gc = linear_cell<2>(R, pi);
      w = (float)((uint64_t)1 << min(R.sh[0], R.sh[1])) * VK_VOR_SQUARE / (float)__ldg(G.sub_s + gc);
      if (w > wmax && stage == kSquare) stage = kBox;
    }
    bool going = on;
    while (__any_sync(kAll, going)) {
      const int32_t first_new = skip;  // this stage passes over what the last one visited
      const bool fresh = n_seen == 0 && stage == kSquare;  // (everything near cuts the first square)
      float x0, x1, y0, y1;
      box(&x0, &x1, &y0, &y1);
      if (going && stage == kSquare) {
        const int32_t h = (int32_t)w;
        if (rc.init(R, p, -h, h, -h, h)) skip = h + 1;
        else stage = kBox;
      }
      if (going && stage == kBox) {
        const float far = 1.0e9f;
        if (!(x0 > -far && x1 < far && y0 > -far && y1 < far) ||
            !rc.init(R, p, (int32_t)floorf(x0) - 2, (int32_t)ceilf(x1) + 2, (int32_t)floorf(y0) - 2,
                     (int32_t)ceilf(y1) + 2))
          other = true;
      }
      bool left = going && !other;  // runs left
      bool seeds_left = stage == kSeeds;
      uint32_t qb = 0, qe = 0;
      for (;;) {
        // gather kPer candidates per lane from the runs
        uint32_t at[kPer] = {};
        int n = 0;
        while (__any_sync(kAll, left && n < kCG * kPer)) {
          if (left && n < kCG * kPer) {
            if (qb == qe) {
              if (stage == kSeeds) {
                left = seeds_left;
                seeds_left = false;
                qb = 0;
                qe = (uint32_t)sd.n;
              } else {
                left = rc.next(R, G, &qb, &qe);
              }
              if (!left) qb = qe = 0;
              n_seen += qe - qb;
            }
            const int take = min((int)(qe - qb), kCG * kPer - n);
#pragma unroll
            for (int s = 0; s < kPer; ++s) {
              const int j = kCG * s + gl - n;
              if (j >= 0 && j < take) at[s] = qb + (uint32_t)j;
            }
            n += take;
            qb += (uint32_t)take;
          }
        }
        if (n_seen > budget) {
          other = true;
          left = false;
          n = 0;
        }
        if (!__any_sync(kAll, n > 0)) break;
        bool flag[kPer];
        int32_t mx[kPer], my[kPer];
        float D[kPer];
        bool on_top = false;
#pragma unroll
        for (int s = 0; s < kPer; ++s) {
          flag[s] = kCG * s + gl < n;
          mx[s] = my[s] = 0;
          if (flag[s]) {
            if (stage == kSeeds) at[s] = (uint32_t)sd.slot_of[R.p0 + sd.ids[at[s]]];
            const int2 pj = __ldg(pos + at[s]);
            // the stages lie within half a period: minimum images
            mx[s] = (int32_t)((uint32_t)pj.x - (uint32_t)p.x);
            my[s] = (int32_t)((uint32_t)pj.y - (uint32_t)p.y);
            mx[s] += mx[s] > X / 2 ? -X : (mx[s] < -(X / 2) ? X : 0);
            my[s] += my[s] > Y / 2 ? -Y : (my[s] < -(Y / 2) ? Y : 0);
            flag[s] = (int64_t)at[s] != self && !(abs(mx[s]) < first_new && abs(my[s]) < first_new);
          }
          D[s] = (float)mx[s] * (float)mx[s] + (float)my[s] * (float)my[s];
          on_top = on_top || (flag[s] && mx[s] == 0 && my[s] == 0);
        }
        if (group_bits(on_top)) {  // coincident with the particle
          other = true;
          left = false;
        }
        // clip, nearest first; the candidates are filtered before the first
        // clip (in the first square, which a few have to close, after four) and
        // after every third
#pragma unroll 1
        for (int done = fresh ? -4 : 0;; ++done) {
          if (__any_sync(kAll, done >= 0 && done % 3 == 0)) {
            bounds();
            filter(flag, mx, my);
          }
          float near = 3.0e38f;
#pragma unroll
          for (int s = 0; s < kPer; ++s) near = fminf(near, flag[s] && !other ? D[s] : 3.0e38f);
          const float own = near;
#pragma unroll
          for (int o = 1; o < kCG; o <<= 1) near = fminf(near, __shfl_xor_sync(kAll, near, o));
          const bool on = near < 3.0e38f;
          if (!__any_sync(kAll, on)) break;
          const int src = base + __ffs(group_bits(own == near)) - 1;
          int32_t cx = 0, cy = 0;
          uint32_t ca = 0;
          int pick = -1;
#pragma unroll
          for (int s = kPer - 1; s >= 0; --s)
            if (flag[s] && D[s] == near) {
              cx = mx[s];
              cy = my[s];
              ca = at[s];
              pick = s;
            }
          if (base + gl == src)
#pragma unroll
            for (int s = 0; s < kPer; ++s) flag[s] = flag[s] && s != pick;
          clip(on, __shfl_sync(kAll, cx, src), __shfl_sync(kAll, cy, src), (int32_t)__shfl_sync(kAll, ca, src));
        }
        bounds();
        if (other) left = false;
      }
      if (other || stage == kBox) going = false;
      // a cell still much wider than the square: the box would hold far more
      // particles than a larger square needs to close the cell.  (Seeds leave a
      // cell about as wide as it was, unless they are of a state long past.)
      if (stage == kSeeds && reach() > VK_VOR_STALE * sd.reach && w < wmax) {
        stage = kSquare;
      } else if (stage == kSquare && reach() > VK_VOR_REACH * w && 2.0f * w < wmax) {
        w *= 2.0f;
      } else {
        stage = kBox;
      }
    }
  }

  // twice the largest distance of a vertex: no site farther away can cut the cell (group)
  __device__ __forceinline__ float reach() const { return 2.0f * sqrtf(r2max); }

  // bit a: edge a is of positive length, i.e. its two vertices lie apart (group)
  __device__ __forceinline__ unsigned positive_edges() const {
    const bool big = __any_sync(kAll, m > 8);
    int2 nq[2];
    next_sites(big, nq);
    // site and vertex before each of the lane's edges
    unsigned kept = 0;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (i == 1 && !big) break;
      const int a = gl + 8 * i, j = a == 0 ? m - 1 : a - 1;
      const int from = base + (j & 7);
      int2 b = make_int2(__shfl_sync(kAll, q[0].x, from), __shfl_sync(kAll, q[0].y, from));
      float2 bv = make_float2(__shfl_sync(kAll, v[0].x, from), __shfl_sync(kAll, v[0].y, from));
      float be = __shfl_sync(kAll, e[0], from);
      if (big) {
        const int2 hb = make_int2(__shfl_sync(kAll, q[1].x, from), __shfl_sync(kAll, q[1].y, from));
        const float2 hv = make_float2(__shfl_sync(kAll, v[1].x, from), __shfl_sync(kAll, v[1].y, from));
        const float he = __shfl_sync(kAll, e[1], from);
        if (j >= 8) {
          b = hb;
          bv = hv;
          be = he;
        }
      }
      const bool is = has(i) && (vertex_cut_fast(bv.x, bv.y, be, nq[i].x, nq[i].y) != 0 ||
                                 vertex_cut_sign(b.x, b.y, q[i].x, q[i].y, nq[i].x, nq[i].y) != 0);
      kept |= group_bits(is) << (8 * i);
    }
    return kept;
  }
  // ... and belongs to another particle
  __device__ __forceinline__ unsigned neighbor_edges() const {
    unsigned kept = positive_edges();
#pragma unroll
    for (int i = 0; i < 2; ++i) kept &= ~(group_bits(has(i) && slot[i] < 0) << (8 * i));
    return kept;
  }

  // Neighbors, the sites of edges of positive length, ordered by id: of each of
  // the lane's edges the id (INT_MAX: none) and its place in the order (-1).
  // Returns their number (group).
  __device__ __forceinline__ int neighbors(bool ok, const int32_t* __restrict__ ids, int32_t* nid, int* rank) const {
    const unsigned kept = neighbor_edges();
    const bool big = __any_sync(kAll, m > 8);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      rank[i] = 0;
      nid[i] = ok && (kept >> (gl + 8 * i) & 1u) ? __ldg(ids + slot[i]) : INT_MAX;
    }
#pragma unroll
    for (int j = 0; j < kCG; ++j) {
      const int32_t o = __shfl_sync(kAll, nid[0], base + j);
#pragma unroll
      for (int i = 0; i < 2; ++i) rank[i] += o < nid[i] ? 1 : 0;
    }
    if (big)
#pragma unroll
      for (int j = 0; j < kCG; ++j) {
        const int32_t o = __shfl_sync(kAll, nid[1], base + j);
#pragma unroll
        for (int i = 0; i < 2; ++i) rank[i] += o < nid[i] ? 1 : 0;
      }
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (nid[i] == INT_MAX) rank[i] = -1;
    return __popc(kept);
  }
};

}  // namespace

}  // namespace vk
