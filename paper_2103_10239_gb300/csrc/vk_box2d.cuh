// vk_box2d.cuh -- a particle's search context and the exact field-of-view test
// of the 2D kNN rule (vk_knn2d.cu), and the square walk of the two-level grid
// that exports the metric rule's lists (vk_metric.cu): every particle of the
// square [p - a, p + a] around a particle, as contiguous runs of the
// cell-sorted arrays, with exact minimum-image offsets.
#pragma once
#include <climits>

#include "vk_internal.cuh"

// slot runs one square listing may buffer per thread
#ifndef VK_KNN2_BOX_RUNS
#define VK_KNN2_BOX_RUNS 16
#endif

namespace vk {

// The field of view of the kNN rule (reading of Sec. "Metric and topological
// flocking models": the k nearest neighbors within an angular field of
// view): offset d is in view iff d.nq >= cq |d|, with the heading and the
// cosine of the half-angle rounded to 2^-24 (nq = rint(n 2^24), cq =
// rint(c 2^24), round half to even), compared exactly through squares in
// 128-bit integers; d = 0 is in view, and everything is when c <= -1.
struct View {
  int32_t nxq, nyq, cq;
};

__device__ __forceinline__ View make_view(float2 n, int32_t cq) {
  View w;
  w.nxq = (int32_t)__float2ll_rn(n.x * 16777216.0f);
  w.nyq = (int32_t)__float2ll_rn(n.y * 16777216.0f);
  w.cq = cq;
  return w;
}

__device__ __forceinline__ bool in_view(const View& w, int32_t dx, int32_t dy, uint64_t D) {
  if (w.cq <= -(1 << 24)) return true;  // a full circle
  const long long sdot = (long long)dx * w.nxq + (long long)dy * w.nyq;
  const __int128 lhs = (__int128)sdot * sdot;
  const __int128 rhs = (__int128)((long long)w.cq * w.cq) * (__int128)D;
  if (w.cq >= 0) return sdot >= 0 && lhs >= rhs;
  return sdot >= 0 || lhs <= rhs;
}


struct Ctx {
  int64_t self;
  uint32_t px, py;
  uint32_t Lx, Ly;
  int32_t hix, lox, hiy, loy;  // minimum image: d > hi -> d - L, d <= lo -> d + L
  View view;  // field of view of the kNN rule (everything when view.cq <= -2^24)
};

__device__ __forceinline__ void init_ctx(Ctx& C, const Rep& R, int64_t self, int2 p) {
  C.self = self;
  C.px = (uint32_t)p.x;
  C.py = (uint32_t)p.y;
  C.Lx = R.L[0];
  C.Ly = R.L[1];
  C.hix = (int32_t)(R.L[0] / 2);
  C.lox = -(int32_t)((R.L[0] + 1) / 2);
  C.hiy = (int32_t)(R.L[1] / 2);
  C.loy = -(int32_t)((R.L[1] + 1) / 2);
  C.view.nxq = 0;
  C.view.nyq = 0;
  C.view.cq = kViewAll;
}

// tracing counters of the radius-first search
struct BoxCount {
  uint32_t cand = 0;   // candidates examined
  uint32_t tries = 0;  // squares scanned
  uint32_t runs = 0;   // contiguous slot runs read
  uint32_t hits = 0;   // hits merged
  uint32_t cells = 0;  // coarse cells visited
  uint32_t why = 0;    // fallback reason: 0 none, 1 square too wide, 2 too few hits, 3 close distances
};

// exact minimum-image offset and squared distance of pj from the particle
__device__ __forceinline__ uint64_t box_offset(const Ctx& C, int2 pj, int32_t& dx, int32_t& dy) {
  dx = (int32_t)((uint32_t)pj.x - C.px);
  dy = (int32_t)((uint32_t)pj.y - C.py);
  if (dx > C.hix) dx = (int32_t)((uint32_t)dx - C.Lx);
  else if (dx <= C.lox) dx = (int32_t)((uint32_t)dx + C.Lx);
  if (dy > C.hiy) dy = (int32_t)((uint32_t)dy - C.Ly);
  else if (dy <= C.loy) dy = (int32_t)((uint32_t)dy + C.Ly);
  return (uint64_t)((int64_t)dx * dx) + (uint64_t)((int64_t)dy * dy);
}

// Walk the slot runs of the square [p - a, p + a] (the sub-cell rows of the
// coarse cells it meets), each with the periodic image its cell lies in.
// Runs are listed up to HB::kRuns at a time into the thread's column of
// H.run (uint2 run[kRuns][kBlock]); one
// flat loop walks each batch, so that threads of a warp whose squares split
// into different numbers of runs still scan candidates together.  The
// visitor gets the candidates four at a time (their loads are independent,
// so they are in flight together; a group never crosses a run):
// v.group(q, n, pj, ox, oy) for slots q..q+n-1 at positions pj[0..n), whose
// exact offsets from the particle are pj - (ox, oy) in wrapping 32-bit
// arithmetic.  False when the square is too wide for the minimum image or
// meets a coarse cell through two periodic images (nothing was visited).
constexpr int kGroup = 4;

template <class HB, class V>
__device__ __forceinline__ bool box_walk(HB& H, const Rep& R, const GridView& G, const int2* __restrict__ pos,
                                         const Ctx& C, int64_t a, BoxCount& bc, V& v) {
  const int64_t Lx = C.Lx, Ly = C.Ly;
  if (2 * (2 * a + 1) >= Lx || 2 * (2 * a + 1) >= Ly) return false;
  const int nx = R.nc[0], ny = R.nc[1];
  const int64_t qx0 = (int64_t)C.px - a, qx1 = (int64_t)C.px + a;
  const int64_t qy0 = (int64_t)C.py - a, qy1 = (int64_t)C.py + a;
  const int ucx0 = ucell2(qx0, nx, R.sh[0], Lx), ucx1 = ucell2(qx1, nx, R.sh[0], Lx);
  const int ucy0 = ucell2(qy0, ny, R.sh[1], Ly), ucy1 = ucell2(qy1, ny, R.sh[1], Ly);
  // in-cell offsets of the square's corners in their own cells
  const uint32_t fx0 = cell_frac((uint32_t)(qx0 < 0 ? qx0 + Lx : qx0), R.sh[0]);
  const uint32_t fx1 = cell_frac((uint32_t)(qx1 >= Lx ? qx1 - Lx : qx1), R.sh[0]);
  const uint32_t fy0 = cell_frac((uint32_t)(qy0 < 0 ? qy0 + Ly : qy0), R.sh[1]);
  const uint32_t fy1 = cell_frac((uint32_t)(qy1 >= Ly ? qy1 - Ly : qy1), R.sh[1]);
  if (ucx1 - ucx0 + 1 > nx || ucy1 - ucy0 + 1 > ny) return false;
  bc.tries += 1;
  // enumeration cursor over (coarse cell, row of sub-cells): runs are listed
  // kRuns at a time, each batch is scanned, then listing resumes
  int ucx = ucx0, ucy = ucy0;
  int row = 0, row_end = -1;  // rows of the current cell still to list
  int64_t gc = 0;
  uint32_t sb0 = 0, code = 0;
  int s = 1, sx0 = 0, sx1 = 0;
  bool split = false, listed_all = false;
  while (!listed_all) {
    int nrun = 0;
    while (nrun < HB::kRuns) {
      if (row > row_end) {  // next coarse cell
        if (ucx > ucx1) {
          ucx = ucx0;
          ++ucy;
        }
        if (ucy > ucy1) {
          listed_all = true;
          break;
        }
        const int cy = ucy < 0 ? ucy + ny : (ucy >= ny ? ucy - ny : ucy);
        const int cx = ucx < 0 ? ucx + nx : (ucx >= nx ? ucx - nx : ucx);
        // shift code per axis: 0 same image, 1 the image at -L, 2 at +L
        code = (ucx < 0 ? 1u : (ucx >= nx ? 2u : 0u)) << 2 | (ucy < 0 ? 1u : (ucy >= ny ? 2u : 0u));
        gc = R.c0 + (int64_t)cy * nx + cx;
        sb0 = __ldg(G.sub_base + gc);
        split = __ldg(G.sub_base + gc + 1) - sb0 > 1;
        bc.cells += 1;
        row = 0;
        row_end = 0;
        if (split) {
          s = __ldg(G.sub_s + gc);
          sx0 = ucx == ucx0 ? sub_of(fx0, s) : 0;
          sx1 = ucx == ucx1 ? sub_of(fx1, s) : s - 1;
          row = ucy == ucy0 ? sub_of(fy0, s) : 0;
          row_end = ucy == ucy1 ? sub_of(fy1, s) : s - 1;
        }
        ++ucx;
      }
      uint32_t qb, qe;
      if (split) {
        const uint32_t rb = sb0 + (uint32_t)row * (uint32_t)s;
        qb = __ldg(G.sub_off + rb + sx0);
        qe = __ldg(G.sub_off + rb + sx1 + 1);
      } else {
        qb = __ldg(G.off + gc);
        qe = __ldg(G.off + gc + 1);
      }
      ++row;
      if (qe > qb) H.run[nrun++][threadIdx.x] = make_uint2(qb, (qe - qb) << 4 | code);
    }
    bc.runs += (uint32_t)nrun;
    int r = -1;
    uint32_t q = 0, qe = 0, ox = 0, oy = 0;
    for (;;) {
      if (q == qe) {
        if (++r == nrun) break;
        const uint2 e = H.run[r][threadIdx.x];
        q = e.x;
        qe = e.x + (e.y >> 4);
        // reference shifted into the run's periodic image: dx = x_j - ox exactly
        const uint32_t cxd = (e.y >> 2) & 3u, cyd = e.y & 3u;
        ox = C.px + (cxd == 1u ? (uint32_t)C.Lx : 0u) - (cxd == 2u ? (uint32_t)C.Lx : 0u);
        oy = C.py + (cyd == 1u ? (uint32_t)C.Ly : 0u) - (cyd == 2u ? (uint32_t)C.Ly : 0u);
        bc.cand += qe - q;
      }
      const uint32_t n = min(qe - q, (uint32_t)kGroup);
      int2 pj[kGroup];
#pragma unroll
      for (int u = 0; u < kGroup; ++u) pj[u] = __ldg(pos + q + min((uint32_t)u, n - 1));
      v.group(q, n, pj, ox, oy);
      q += n;
    }
  }
  return true;
}

}  // namespace vk
