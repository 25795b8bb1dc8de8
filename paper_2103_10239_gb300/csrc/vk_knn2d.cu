// vk_knn2d.cu -- the 2D k-nearest-neighbor rule fused with the Vicsek update
// (Sec. "Metric and topological flocking models": each particle aligns with
// its k nearest neighbors at any distance; Eq. 1 and Eq. 2).
//
// Radius first: each particle knows roughly how far its k-th neighbor is (its
// k-th distance at the last step, kept as a hint in the state), so it scans,
// once, the square [p - a, p + a] with a a little above that distance: the
// sub-cell rows of the one to four coarse cells that the square meets, each a
// contiguous run of the sorted arrays.  Nothing outside the square is closer
// than a + 1, so k hits within it are the k nearest.
//
//   * knn2_box_step_kernel: one thread per particle, one square each.  The
//     kernel is bound by instruction issue (a few cache lines of data per
//     particle, DRAM below 2 % of its rate), so the whole selection runs on
//     32-bit keys: the FP32 squared distance with its low bits replaced by
//     the hit's number, inserted into a register list by min / max (two
//     instructions an entry).  A key orders two candidates with certainty
//     when the keys differ by two steps or more (2^-18 relative); a list with
//     a closer pair (about one particle in 5000) or with fewer than k hits is
//     handed on.
//   * knn2_second_kernel: long lists of handed-on particles get larger squares
//     by the same one-thread search.
//   * knn2_group_kernel: short lists, and what is left: 16 lanes per particle
//     scan the rows of larger squares together and rank the hits exactly, by
//     (int64 squared distance, id).
//
// Measured (GB300, us per step, 64-bit list / 32-bit keys and power-of-two
// cells): 4M clustered, k = 7, ten steps from a set state: first square 2372 /
// 1175 (913 in cells of 64 particles, with the guess of first radii out of line), listed
// particles 1232 / 594; 50,021 uniform, k = 16, vectorial noise: 178 / 34, 183 / 35.  2048
// uniform: 45 + 48 / 26 + 26, and 25 by the groups alone.
#include <algorithm>
#include <climits>
#include <type_traits>

#include "vk_box2d.cuh"
#include "vk_group.cuh"

namespace vk {

namespace {

constexpr int kBlk = 128;  // threads per block of the step kernel (a block task is split)
constexpr int kSplit = kBlock / kBlk;

// KC keys per thread: room for k <= KC - 1 neighbors and the one after them.
// CAP hits buffered per thread (about 1.3 k + 1 are expected), numbered in
// BITS bits, and RUNS slot runs listed before they are scanned.  What they do not
// take of shared memory caches positions: for k <= 7, 24 hits and 8 runs / 20 and
// 6: 512 replicas 1634 / 1563 us per step, 4M clustered 943 / 905; 16 hits (956)
// fill too often, and 6 runs for k = 16 (448 against 431 at 1M) are too few.
template <int KC> struct BoxCfg;
template <> struct BoxCfg<8> { static constexpr int CAP = 20, BITS = 5, BLOCKS = 6, RUNS = 6; };
template <> struct BoxCfg<12> { static constexpr int CAP = 32, BITS = 5, BLOCKS = 5, RUNS = 8; };
template <> struct BoxCfg<17> { static constexpr int CAP = 48, BITS = 6, BLOCKS = 3, RUNS = 8; };
template <> struct BoxCfg<33> { static constexpr int CAP = 64, BITS = 6, BLOCKS = 2, RUNS = 8; };

template <int KC>
struct BoxShared {
  uint2 hit[BoxCfg<KC>::CAP][kBlk];  // (slot, bits of the FP32 squared distance), one column per thread
  uint2 run[BoxCfg<KC>::RUNS][kBlk];  // (first slot, length << 4 | image shift codes)
};

// A thread does not take a square of more coarse cells than these (per axis): a
// particle outside a cluster has a wide square, most of it empty cells, and the whole
// launch waits for it.  The groups look at 16 cells at a time.  Ordinary squares meet
// one to four.  Measured (us per step, 200,000 particles in a wide cluster; no limit /
// 12 / 8 / 5): 210, 231, 203, 189.  Not in a field of view, whose squares are wider for
// every particle that faces a void (1M 4.1 ms a pass without, 4.5 with).
constexpr int kMaxCells = 5;

// the slot behind a key of the list
template <int KC>
__device__ __forceinline__ int32_t key_slot(const BoxShared<KC>& H, uint32_t key) {
  return (int32_t)H.hit[key & ((1u << BoxCfg<KC>::BITS) - 1u)][threadIdx.x].x;
}

// The k nearest of the particle at slot `self` from the square of half-width
// a = ceil(r), as keys t[KC-1-k .. KC-2] in order (the first entries are
// sentinels, so that no register array is indexed dynamically); false when
// the square cannot decide, with the radius to try next.
//
// Every slot of the square with FP32 squared distance <= tau goes to the
// thread's hit column, and the column is merged into t after the scan, where
// the warp's threads have met again (and whenever the column is full: the KC
// best then stay, and tau shrinks to the k-th).  With a field of view of at
// most a half-plane, candidates behind the particle are dropped in the scan
// (exactly); the rest of the view test is the merge's.
template <int KC, bool FOV>
__device__ __forceinline__ bool box_search(BoxShared<KC>& H, const Rep& R, const GridView& G,
                                           const int2* __restrict__ pos, int32_t self, int2 p, const View& vw,
                                           float radius, int k, uint32_t* t, float* r_next, BoxCount& bc) {
  constexpr int B = BoxCfg<KC>::BITS, CAP = BoxCfg<KC>::CAP;
  const int32_t a = (int32_t)ceilf(fminf(radius, 1.0e9f));
  *r_next = (float)a;
  const uint32_t Lx = R.L[0], Ly = R.L[1];
  bc.why = 1u;  // too wide for the minimum image, a coarse cell met through two periodic images, or too many cells
  if (4ll * a + 2 >= (int64_t)Lx || 4ll * a + 2 >= (int64_t)Ly) return false;
  const int nx = R.nc[0], ny = R.nc[1], shx = R.sh[0], shy = R.sh[1];
  const int tid = (int)threadIdx.x;
  // corners wrapped into the box, their unwrapped coarse cells and in-cell fractions
  const bool wx0 = p.x < a, wy0 = p.y < a;
  const bool wx1 = (uint32_t)p.x + (uint32_t)a >= Lx, wy1 = (uint32_t)p.y + (uint32_t)a >= Ly;
  const uint32_t x0 = (uint32_t)p.x - (uint32_t)a + (wx0 ? Lx : 0u), x1 = (uint32_t)p.x + (uint32_t)a - (wx1 ? Lx : 0u);
  const uint32_t y0 = (uint32_t)p.y - (uint32_t)a + (wy0 ? Ly : 0u), y1 = (uint32_t)p.y + (uint32_t)a - (wy1 ? Ly : 0u);
  const int ucx0 = (int)(x0 >> shx) - (wx0 ? nx : 0), ucx1 = (int)(x1 >> shx) + (wx1 ? nx : 0);
  const int ucy0 = (int)(y0 >> shy) - (wy0 ? ny : 0), ucy1 = (int)(y1 >> shy) + (wy1 ? ny : 0);
  if (ucx1 - ucx0 >= (FOV ? nx : min(nx, kMaxCells)) || ucy1 - ucy0 >= (FOV ? ny : min(ny, kMaxCells))) return false;
  const uint32_t fx0 = cell_frac(x0, shx), fx1 = cell_frac(x1, shx);
  const uint32_t fy0 = cell_frac(y0, shy), fy1 = cell_frac(y1, shy);
  bc.tries += 1;
  // below (a + 1)^2 by more than the rounding of the distances
  const float a1 = (float)a + 1.0f;
  float tau = a1 * a1 * (1.0f - 9.5367431640625e-07f);
  const uint32_t edge = __float_as_uint(tau) >> B;
#pragma unroll
  for (int s = 0; s < KC; ++s) t[s] = s < KC - 1 - k ? 0u : 0xFFFFFFFFu;
  int cnt = 0, merged = 0, got = 0;
  // cursors over (coarse cell, row of sub-cells) and over the listed runs
  int ucx = ucx0, ucy = ucy0, row = 0, row_end = -1, s = 1, nrun = 0, r = 0;
  uint32_t lo = 0, hi = 0, code = 0;  // first and one-past-last sub-cell of the row
  uint32_t q = 0, qb = 0, len = 0, ox = 0, oy = 0;
  bool more = true, done = false;
  for (;;) {
    while (cnt <= CAP - 4) {
      if (q - qb >= len) {  // next run
        if (r == nrun) {
          // list up to RUNS runs, so that one flat loop scans them and the
          // threads of a warp scan candidates together however their squares split
          nrun = r = 0;
          while (more && nrun <= BoxCfg<KC>::RUNS - 2) {
            if (row > row_end) {  // next coarse cell
              if (ucx > ucx1) {
                ucx = ucx0;
                ++ucy;
              }
              if (ucy > ucy1) {
                more = false;
                break;
              }
              const int cy = ucy < 0 ? ucy + ny : (ucy >= ny ? ucy - ny : ucy);
              const int cx = ucx < 0 ? ucx + nx : (ucx >= nx ? ucx - nx : ucx);
              // shift code per axis: 0 same image, 1 the image at -L, 2 at +L
              code = (ucx < 0 ? 4u : (ucx >= nx ? 8u : 0u)) | (ucy < 0 ? 1u : (ucy >= ny ? 2u : 0u));
              const int64_t gc = R.c0 + (int64_t)cy * nx + cx;
              const uint32_t base = __ldg(G.sub_base + gc);
              s = __ldg(G.sub_s + gc);
              const int sx0 = ucx == ucx0 ? sub_of(fx0, s) : 0, sx1 = ucx == ucx1 ? sub_of(fx1, s) : s - 1;
              row = ucy == ucy0 ? sub_of(fy0, s) : 0;
              row_end = ucy == ucy1 ? sub_of(fy1, s) : s - 1;
              lo = base + (uint32_t)(row * s + sx0);
              hi = lo + (uint32_t)(sx1 - sx0 + 1);
              bc.cells += 1;
              ++ucx;
            }
            // two rows at a time: their four loads are in flight together
            const uint32_t step = row < row_end ? (uint32_t)s : 0u;
            const uint32_t b0 = __ldg(G.sub_off + lo), e0 = __ldg(G.sub_off + hi);
            const uint32_t b1 = __ldg(G.sub_off + lo + step), e1 = __ldg(G.sub_off + hi + step);
            if (e0 > b0) H.run[nrun++][tid] = make_uint2(b0, (e0 - b0) << 4 | code);
            if (step && e1 > b1) H.run[nrun++][tid] = make_uint2(b1, (e1 - b1) << 4 | code);
            row += 2;
            lo += 2u * (uint32_t)s;
            hi += 2u * (uint32_t)s;
          }
          bc.runs += (uint32_t)nrun;
          if (nrun == 0) {
            done = true;
            break;
          }
        }
        const uint2 e = H.run[r++][tid];
        qb = e.x;
        len = e.y >> 4;
        q = qb & ~1u;  // 16-byte aligned pairs; the slot before the run is masked
        // reference shifted into the run's periodic image: dx = x_j - ox exactly
        ox = (uint32_t)p.x + (e.y & 4u ? Lx : 0u) - (e.y & 8u ? Lx : 0u);
        oy = (uint32_t)p.y + (e.y & 1u ? Ly : 0u) - (e.y & 2u ? Ly : 0u);
        bc.cand += len;
      }
      // four candidates from two 16-byte loads (the arrays are padded by four slots)
      const int4 A = __ldg(reinterpret_cast<const int4*>(pos + q));
      const int4 C = __ldg(reinterpret_cast<const int4*>(pos + q + 2));
      const int32_t xs[4] = {A.x, A.z, C.x, C.z}, ys[4] = {A.y, A.w, C.y, C.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        // branch-free append: written at the next free place, kept only for a hit
        const int32_t dx = (int32_t)((uint32_t)xs[u] - ox), dy = (int32_t)((uint32_t)ys[u] - oy);
        const float fx = (float)dx, fy = (float)dy;
        const float D = __fmaf_rn(fx, fx, __fmul_rn(fy, fy));
        bool hit = D <= tau && q + (uint32_t)u - qb < len;
        if (FOV) hit = hit && (vw.cq < 0 || (long long)dx * vw.nxq + (long long)dy * vw.nyq >= 0);
        H.hit[cnt][tid] = make_uint2(q + (uint32_t)u, __float_as_uint(D));
        cnt += hit ? 1 : 0;
      }
      q += 4;
      if (q - qb >= len && r == nrun && !more) {
        done = true;
        break;
      }
    }
#pragma unroll 2
    for (int b = merged; b < cnt; ++b) {
      const uint2 h = H.hit[b][tid];
      bool keep = (int32_t)h.x != self;
      if (FOV && vw.cq != 0) {  // (cq = 0: the scan's test was the whole test)
        const int2 pj = __ldg(pos + h.x);
        const int64_t dx = min_image((int64_t)pj.x - p.x, Lx), dy = min_image((int64_t)pj.y - p.y, Ly);
        keep = keep && in_view(vw, (int32_t)dx, (int32_t)dy, (uint64_t)(dx * dx) + (uint64_t)(dy * dy));
      }
      got += keep ? 1 : 0;
      uint32_t x = keep ? (h.y & ~((1u << B) - 1u)) | (uint32_t)b : 0xFFFFFFFFu;
#pragma unroll
      for (int e = 0; e < KC; ++e) {
        const uint32_t m = min(t[e], x);
        x = max(t[e], x);
        t[e] = m;
      }
    }
    if (done) break;
    // full column: its KC best move to the front and keep their order
    merged = 0;
    uint2 best[KC];
#pragma unroll
    for (int e = 0; e < KC; ++e)
      if (e >= KC - 1 - k && t[e] != 0xFFFFFFFFu) best[e] = H.hit[t[e] & ((1u << B) - 1u)][tid];
#pragma unroll
    for (int e = 0; e < KC; ++e)
      if (e >= KC - 1 - k && t[e] != 0xFFFFFFFFu) {
        H.hit[merged][tid] = best[e];
        t[e] = (t[e] & ~((1u << B) - 1u)) | (uint32_t)merged;
        ++merged;
      }
    cnt = merged;
    if (t[KC - 2] < 0xFF000000u) tau = fminf(tau, __uint_as_float(((t[KC - 2] >> B) + 3u) << B));
  }
  bc.hits += (uint32_t)got;
  if ((t[KC - 2] >> B) + 1u < edge) {
    bool close = false;  // a pair whose order the keys leave open
#pragma unroll
    for (int e = 0; e < KC - 1; ++e) close |= e >= KC - 1 - k && (t[e + 1] >> B) - (t[e] >> B) <= 1u;
    bc.why = close ? 3u : 0u;
    return !close;
  }
  // too few: scale the radius towards about 1.5 k expected hits
  const float want = 1.5f * (float)k + 1.f;
  *r_next = (float)a * (got > 0 ? fminf(sqrtf(want / (float)got), 2.f) : 2.f);
  bc.why = 2u;
  return false;
}

// A group of GS lanes searches for one particle, exactly (vk_group.cuh).
template <int GS, int CAP, bool FOV>
struct Group : GroupTop<GS, CAP> {
  using Top = GroupTop<GS, CAP>;
  using Top::mask;
  using Top::shift;
  using Top::gl;
  using Top::tau;
  const int2* __restrict__ pos;
  Ctx C;

  // the candidates of slots [qb, qe)
  __device__ __forceinline__ void run(int64_t qb, int64_t qe) {
    Top::n_cand += (uint32_t)(qe - qb);
    for (int64_t b = qb; b < qe; b += GS) {
      const int64_t q = b + gl;
      bool hit = false;
      unsigned long long D = 0;
      if (q < qe && (int32_t)q != Top::self) {
        int32_t dx, dy;
        D = box_offset(C, __ldg(pos + q), dx, dy);
        hit = D <= tau;
        if (FOV) hit = hit && in_view(C.view, dx, dy, D);
      }
      Top::append(hit, D, q);
    }
  }

  // does the square of half-width a meet some coarse cell of an axis twice
  // (then the axis is covered whole)?
  static __device__ __forceinline__ bool spans(uint32_t p, int64_t a, int n, int sh, int64_t L) {
    return 2 * a + 1 >= L || ucell2((int64_t)p + a, n, sh, L) - ucell2((int64_t)p - a, n, sh, L) >= n;
  }
  // sub-cells [*i0, *i1] of unwrapped cell u that meet [p - w, p + w]; false if none does
  static __device__ __forceinline__ bool clip(uint32_t p, int64_t w, int u, int n, int sh, int64_t L, int s, int* i0,
                                              int* i1) {
    const int64_t lo = (int64_t)p - w - cell_lo2(u, n, sh, L), hi = lo + 2 * w;
    if (hi < 0 || lo >> sh > 0) return false;
    *i0 = lo <= 0 ? 0 : sub_of(cell_frac((uint32_t)lo, sh), s);
    *i1 = hi >> sh > 0 ? s - 1 : sub_of(cell_frac((uint32_t)hi, sh), s);
    return true;
  }

  // The candidates of the square of half-width a (an axis that it spans is
  // covered whole).  The lanes look at GS coarse cells at a time, so that
  // empty ones cost little; a non-empty one is scanned by rows of the
  // sub-cells that meet the square of half-width min(a, sqrt(tau)): a list
  // that has filled up on the way leaves little to scan.  Near cells and rows
  // go first: of a cluster that the square reaches from outside, met from its far
  // side, every particle would be nearer than the last (all lists of 65,536 particles
  // around one point, k = 32, before first radii looked at their cells: 7890 / 634 us).
  // True when the square is the whole box.
  __device__ __forceinline__ bool square(const Rep& R, const GridView& G, int64_t a) {
    const int64_t Lx = C.Lx, Ly = C.Ly;
    const int nx = R.nc[0], ny = R.nc[1], shx = R.sh[0], shy = R.sh[1];
    const bool fullx = spans(C.px, a, nx, shx, Lx), fully = spans(C.py, a, ny, shy, Ly);
    const int ux0 = fullx ? 0 : ucell2((int64_t)C.px - a, nx, shx, Lx);
    const int ux1 = fullx ? nx - 1 : ucell2((int64_t)C.px + a, nx, shx, Lx);
    const int uy0 = fully ? 0 : ucell2((int64_t)C.py - a, ny, shy, Ly);
    const int uy1 = fully ? ny - 1 : ucell2((int64_t)C.py + a, ny, shy, Ly);
    tau = fullx && fully ? ~0ull : (unsigned long long)(a + 1) * (unsigned long long)(a + 1) - 1;
    unsigned long long at = ~0ull;  // the tau that w was taken for
    int64_t w = a;
    const int ownx = (int)(C.px >> shx), owny = (int)(C.py >> shy);
    for (int iy = uy0; iy <= uy1; ++iy) {
      const int uy = iy <= owny ? owny + uy0 - iy : iy;  // down from the particle's own, then up
      const bool below = uy < owny;
      const int cy = uy < 0 ? uy + ny : (uy >= ny ? uy - ny : uy);
      const int64_t rb = R.c0 + (int64_t)cy * nx;
      for (int uc = ux0; uc <= ux1; uc += GS) {
        const int lx = uc + gl;
        const int64_t lc = rb + (lx < 0 ? lx + nx : (lx >= nx ? lx - nx : lx));
        const bool some = lx <= ux1 && __ldg(G.off + lc) != __ldg(G.off + lc + 1);
        unsigned cells = (__ballot_sync(mask, some) & mask) >> shift;
        const unsigned left = ownx < uc ? 0u : ownx - uc >= GS ? ~0u : (2u << (ownx - uc)) - 1u;
        while (cells) {
          const int bit = cells & left ? 31 - __clz(cells & left) : __ffs(cells) - 1;
          const int ux = uc + bit;
          cells &= ~(1u << bit);
          const int64_t gc = rb + (ux < 0 ? ux + nx : (ux >= nx ? ux - nx : ux));
          const uint32_t base = __ldg(G.sub_base + gc);
          const int s = __ldg(G.sub_s + gc);
          if (tau != at) {
            at = tau;
            if (tau < (unsigned long long)a * (unsigned long long)a)
              w = min(a, (int64_t)(sqrtf((float)tau) * 1.000001f) + 1);
          }
          int sx0 = 0, sx1 = s - 1, r0 = 0, r1 = s - 1;
          if (!fullx && !clip(C.px, w, ux, nx, shx, Lx, s, &sx0, &sx1)) continue;
          if (!fully && !clip(C.py, w, uy, ny, shy, Ly, s, &r0, &r1)) continue;
          for (int rr = r0; rr <= r1; rr += GS) {
            // each lane looks up one row of sub-cells
            uint32_t qb = 0, qe = 0;
            if (rr + gl <= r1) {
              const uint32_t lo = base + (uint32_t)((below ? r0 + r1 - rr - gl : rr + gl) * s);
              qb = __ldg(G.sub_off + lo + sx0);
              qe = __ldg(G.sub_off + lo + sx1 + 1);
            }
            unsigned rows = (__ballot_sync(mask, qe > qb) & mask) >> shift;
            while (rows) {
              const int j = shift + __ffs(rows) - 1;
              rows &= rows - 1u;
              run(__shfl_sync(mask, qb, j), __shfl_sync(mask, qe, j));
            }
          }
        }
      }
    }
    return fullx && fully;
  }
};

// the general update (vectorial noise, FP64 sums), kept out of line
__device__ __noinline__ void align_advect_general(const Rep& R, const StepParams& P, uint32_t step, int32_t id,
                                                  const float* ni, const HeadSum<2>& H, int m, const int32_t* pi,
                                                  int32_t* pout, float* nout) {
  align_advect<2>(R, P, step, id, ni, H, m, pi, pout, nout);
}

// Eq. (2) alignment + noise and Eq. (1) advection of one particle; at(j) is
// the slot of list entry j in [KC-1-k, KC-1) in (D, id) order, -1 where a
// field of view holds fewer than k.  Writes the next state and counts the new
// coarse cell.
template <int KC, class At>
__device__ __forceinline__ void knn2_update(const Rep& R, const StepParams& P, int64_t step, int64_t s, int2 p,
                                            float2 nv, int32_t id, At at, const float2* __restrict__ S_dir,
                                            int2* __restrict__ U_pos, float2* __restrict__ U_dir,
                                            int32_t* __restrict__ U_id, uint32_t* __restrict__ counts, float* nnew) {
  HeadSum<2> H;
  H.init();
  const float ni[3] = {nv.x, nv.y, 0.f};
  int m = P.include_self ? 1 : 0;
  if (P.include_self) H.add(ni, P.sum_mode);
#pragma unroll
  for (int c = 0; c < KC - 1; c += 8) {
    // eight headings in flight, then summed in order; a missing entry adds
    // zero, which changes neither sum nor compensation
    float2 d[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = c + u;
      d[u] = make_float2(0.f, 0.f);
      if (j < KC - 1 && j >= KC - 1 - P.k) {
        const int32_t q = at(j);
        if (q >= 0) {
          d[u] = __ldg(S_dir + q);
          ++m;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (c + u >= KC - 1) break;
      const float v[2] = {d[u].x, d[u].y};
      H.add(v, P.sum_mode);
    }
  }
  const int32_t pi[3] = {p.x, p.y, 0};
  int32_t pout[3] = {0, 0, 0};
  if (P.noise == 0 && P.sum_mode != 2) {
    // angular noise, FP32 sums (the default) inline
    const uint4 w = philox4x32_10(make_uint4((uint32_t)id, (uint32_t)step, R.replica, 0u),
                                  make_uint2(P.seed_lo, P.seed_hi));
    const float u = unit24(w.x);
    const float Sx = P.sum_mode == 1 ? __fadd_rn(H.s[0], H.c[0]) : H.s[0];
    const float Sy = P.sum_mode == 1 ? __fadd_rn(H.s[1], H.c[1]) : H.s[1];
    // Eq. (2) with angular noise: the direction of S (the own heading when
    // S = 0) turned by eta (u - 1/2), as a rotation of the unit vector
    float ex = nv.x, ey = nv.y;
    if (Sx != 0.f || Sy != 0.f) {
      const float inv = rsqrtf(Sx * Sx + Sy * Sy);
      ex = Sx * inv;
      ey = Sy * inv;
    }
    float sn, cs;
    sincosf(R.eta * (u - 0.5f), &sn, &cs);
    nnew[0] = cs * ex - sn * ey;
    nnew[1] = sn * ex + cs * ey;
    pout[0] = wrap_add(p.x, grid_step(R.s, P.advect_new ? nnew[0] : nv.x), R.L[0]);
    pout[1] = wrap_add(p.y, grid_step(R.s, P.advect_new ? nnew[1] : nv.y), R.L[1]);
  } else {
    align_advect_general(R, P, (uint32_t)step, id, ni, H, m, pi, pout, nnew);
  }
  U_pos[s] = make_int2(pout[0], pout[1]);
  U_dir[s] = make_float2(nnew[0], nnew[1]);
  U_id[s] = id;
  atomicAdd(counts + linear_cell<2>(R, pout), 1u);
}

// Search radius without a hint: a multiple of the k-th distance expected from
// the density of the particle's own sub-cell.  Outside a cluster that is the
// density of a nearly empty cell, and the square may hold the whole cluster, for
// which one thread needs milliseconds: a square of more than kMaxCand particles, by
// the counts of the coarse cells that it meets, shrinks to about 1.5 k of them.
// Measured (all lists of 65,536 particles around one point, k = 7 and 32): 2896 and
// 11,680 us without, 195 and 413 with it; with a limit on the thread's scan instead, which
// every particle has to check, 289 and 534, and 0.5 % on all steps.  Out of line: inlined it
// takes registers from the search (4M clustered 17.9 ms a pass, 17.1 so).
constexpr float kMaxCand = 512.f;

__device__ __forceinline__ float axis_share(int64_t p, int64_t a, int u, int n, int sh, int64_t L) {
  const int64_t lo = cell_lo2(u, n, sh, L) - p, hi = lo + ((int64_t)1 << sh);
  return (float)(min(a + 1, hi) - max(-a, lo)) / (float)((int64_t)1 << sh);
}

__device__ __noinline__ float box_radius_estimate(const Rep* __restrict__ rep, GridView G, int2 p, int k) {
  const Rep& R = *rep;
  const int32_t pi[2] = {p.x, p.y};
  int64_t gc, gs;
  locate<2>(R, G, nullptr, pi, &gc, &gs);
  const float s = (float)__ldg(G.sub_s + gc);
  const uint32_t cnt = __ldg(G.sub_off + gs + 1) - __ldg(G.sub_off + gs);
  const float area = (float)(1ull << R.sh[0]) * (float)(1ull << R.sh[1]) / (s * s);
  const float r = 1.6f * sqrtf((float)k * area / (3.14159265f * (float)max(cnt, 1u)));
  const int64_t a = (int64_t)ceilf(fminf(r, 1.0e9f)), Lx = R.L[0], Ly = R.L[1];
  if (4 * a + 2 >= Lx || 4 * a + 2 >= Ly) return r;
  const int nx = R.nc[0], ny = R.nc[1];
  const int ux0 = ucell2(p.x - a, nx, R.sh[0], Lx), ux1 = ucell2(p.x + a, nx, R.sh[0], Lx);
  const int uy0 = ucell2(p.y - a, ny, R.sh[1], Ly), uy1 = ucell2(p.y + a, ny, R.sh[1], Ly);
  if (ux1 - ux0 > kMaxCells || uy1 - uy0 > kMaxCells) return r;
  if (ux0 >= 0 && ux1 < nx && uy1 - uy0 <= 1) {  // (the usual case: whole cells hold no more)
    const int64_t c0 = R.c0 + (int64_t)(uy0 < 0 ? uy0 + ny : uy0) * nx, c1 = R.c0 + (int64_t)(uy1 >= ny ? uy1 - ny : uy1) * nx;
    const uint32_t m0 = __ldg(G.off + c0 + ux1 + 1) - __ldg(G.off + c0 + ux0);
    const uint32_t m1 = __ldg(G.off + c1 + ux1 + 1) - __ldg(G.off + c1 + ux0);
    if (m0 + m1 <= (uint32_t)kMaxCand) return r;
  }
  float n = 0.f;
  for (int uy = uy0; uy <= uy1; ++uy)
    for (int ux = ux0; ux <= ux1; ++ux) {
      const int64_t c = R.c0 + (int64_t)(uy < 0 ? uy + ny : (uy >= ny ? uy - ny : uy)) * nx +
                        (ux < 0 ? ux + nx : (ux >= nx ? ux - nx : ux));
      const uint32_t m = __ldg(G.off + c + 1) - __ldg(G.off + c);
      if (m > 0)
        n += (float)m * axis_share(p.x, a, ux, nx, R.sh[0], Lx) * axis_share(p.y, a, uy, ny, R.sh[1], Ly);
    }
  return n > kMaxCand ? r * sqrtf((1.5f * (float)k + 1.f) / n) : r;
}

// Tracing: totals of the radius-first counters (stats[5..12]; the squares also count
// in stats[1]).
__device__ __forceinline__ void record_box_stats(unsigned long long* stats, const BoxCount& bc) {
  if (!stats) return;
  unsigned long long v[8] = {bc.tries, bc.runs, bc.cand, bc.cells, bc.hits, bc.why == 1u, bc.why == 2u, bc.why == 3u};
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(stats + 1, v[0]);
#pragma unroll
    for (int i = 0; i < 8; ++i) atomicAdd(stats + 5 + i, v[i]);
  }
}

// Append (slot, replica) to a device list, one atomic per warp: the
// warp's entries land next to each other, so the kernel that consumes the
// list reads spatially close particles in one warp.  Every lane of the warp
// must call it.
__device__ __forceinline__ void warp_append(bool put, int2 e, int2* __restrict__ list, int32_t* __restrict__ count) {
  const unsigned m = __ballot_sync(0xffffffffu, put);
  if (m == 0u) return;
  const int lane = (int)(threadIdx.x & 31);
  int base = 0;
  if (lane == __ffs(m) - 1) base = atomicAdd(count, __popc(m));
  base = __shfl_sync(0xffffffffu, base, __ffs(m) - 1);
  if (put) list[base + __popc(m & ((1u << lane) - 1u))] = e;
}

// what a search hands its result to: the Vicsek update of a step ...
template <int KC>
struct StepOut {
  const float2* __restrict__ S_dir;
  int2* __restrict__ U_pos;
  float2* __restrict__ U_dir;
  int32_t* __restrict__ U_id;
  float* __restrict__ U_hint;
  uint32_t* __restrict__ counts;
  PhiAcc* __restrict__ phi_acc;
  const int64_t* __restrict__ d_step;
  StepParams P;
  static constexpr bool kStep = true;
  // by slot: the radius a handed-on particle tries next, negative where only a
  // group can serve it (its hint replaces it in the end)
  __device__ __forceinline__ float* radius() const { return U_hint; }
  template <class At>
  __device__ __forceinline__ void put(const Rep& R, int64_t step, int64_t s, int2 p, int32_t id, At at, float dk,
                                      float* nnew) const {
    knn2_update<KC>(R, P, step, s, p, S_dir[s], id, at, S_dir, U_pos, U_dir, U_id, counts, nnew);
    U_hint[s] = sqrtf(dk) * 1.0001f + 1.f;
  }
};
// ... or the particle's row of an export table, by id (-1 past the count found)
template <int KC>
struct RowOut {
  const float2* __restrict__ S_dir;
  const int32_t* __restrict__ S_id;
  int32_t* __restrict__ out;
  float* __restrict__ r_next;
  StepParams P;
  static constexpr bool kStep = false;
  __device__ __forceinline__ float* radius() const { return r_next; }
  template <class At>
  __device__ __forceinline__ void put(const Rep&, int64_t, int64_t, int2, int32_t id, At at, float, float*) const {
#pragma unroll
    for (int j = 0; j < KC - 1; ++j)
      if (j >= KC - 1 - P.k) {
        const int32_t q = at(j);
        out[(int64_t)id * P.k + (j - (KC - 1 - P.k))] = q >= 0 ? __ldg(S_id + q) : -1;
      }
  }
};

// what a particle that a thread could not serve is left with: close distances
// and squares too wide stay what they are, so that another thread would fail too
__device__ __forceinline__ float left_radius(float r, const BoxCount& bc) {
  return bc.why == 1u || bc.why == 3u ? -r : r;
}

// the first radius of a particle
__device__ __forceinline__ float box_radius(const Rep* __restrict__ rep, const GridView& G, int2 p, float hint,
                                            const StepParams& P) {
  return hint > 0.f ? P.halo_alpha * hint + P.halo_beta * fabsf(rep->s) : box_radius_estimate(rep, G, p, P.k);
}

// the search of one thread's particle with the square of half-width ceil(r)
template <int KC, bool FOV, class Out>
__device__ __forceinline__ bool box_particle(BoxShared<KC>& H, const Rep& R, const GridView& G,
                                             const int2* __restrict__ S_pos, const int32_t* __restrict__ S_id,
                                             float r, int64_t s, int64_t step, const Out& out, float* r_next,
                                             BoxCount& bc, float* nnew) {
  const int2 p = S_pos[s];
  View vw;
  if (FOV) vw = make_view(out.S_dir[s], out.P.fov_cq);
  uint32_t t[KC];
  if (!box_search<KC, FOV>(H, R, G, S_pos, (int32_t)s, p, vw, r, out.P.k, t, r_next, bc)) return false;
  out.put(R, step, s, p, S_id[s], [&](int j) { return key_slot<KC>(H, t[j]); }, __uint_as_float(t[KC - 2]), nnew);
  return true;
}

// Search + update, one square per particle.  Particles it cannot serve go on
// the deferred list (slot, replica) with the radius to try next in U_hint.
template <int KC, bool FOV>
__global__ void __launch_bounds__(kBlk, BoxCfg<KC>::BLOCKS) knn2_box_step_kernel(
    const Rep* __restrict__ reps, const BlockTask* __restrict__ tasks, const int2* __restrict__ S_pos,
    const int32_t* __restrict__ S_id, const float* __restrict__ S_hint, GridView G, StepOut<KC> out,
    int2* __restrict__ defer_list, int32_t* __restrict__ defer_count) {
  extern __shared__ __align__(16) unsigned char box_smem[];
  BoxShared<KC>& H = *reinterpret_cast<BoxShared<KC>*>(box_smem);
  __shared__ PhiShared phs;
  phi_block_begin(phs);
  const BlockTask t = tasks[blockIdx.x / kSplit];
  const Rep R = reps[t.rep];
  const int li = t.first + (int)(blockIdx.x % kSplit) * kBlk + (int)threadIdx.x;
  const bool valid = li < R.n;
  const int64_t step = *out.d_step;
  float nnew[3] = {0.f, 0.f, 0.f};
  BoxCount bc;
  bool served = false;
  if (valid) {
    const int64_t s = R.p0 + li;
    float r = box_radius(reps + t.rep, G, S_pos[s], S_hint[s], out.P);
    served = box_particle<KC, FOV>(H, R, G, S_pos, S_id, r, s, step, out, &r, bc, nnew);
    if (!served) out.radius()[s] = left_radius(r, bc);
  }
  warp_append(valid && !served, make_int2((int)(R.p0 + li), t.rep), defer_list, defer_count);
  record_search_stats(out.P.stats, served, bc.cand, 0u, false);
  record_box_stats(out.P.stats, bc);
  phi_block_end<2>(phs, nnew,
                   out.phi_acc + ((size_t)(step % out.P.phi_cap) * (size_t)out.P.n_rep + (size_t)t.rep) * 3);
}

template <int KC, bool FOV>
__global__ void __launch_bounds__(kBlk, BoxCfg<KC>::BLOCKS) knn2_box_export_kernel(
    const Rep* __restrict__ reps, int rep, const int2* __restrict__ S_pos, const int32_t* __restrict__ S_id,
    const float* __restrict__ S_hint, GridView G, RowOut<KC> out, int2* __restrict__ defer_list,
    int32_t* __restrict__ defer_count) {
  extern __shared__ __align__(16) unsigned char box_smem[];
  BoxShared<KC>& H = *reinterpret_cast<BoxShared<KC>*>(box_smem);
  const Rep R = reps[rep];
  const int li = blockIdx.x * kBlk + (int)threadIdx.x;
  const bool valid = li < R.n;
  const int64_t s = R.p0 + li;
  bool served = false;
  if (valid) {
    BoxCount bc;
    float r = box_radius(reps + rep, G, S_pos[s], S_hint ? S_hint[s] : 0.f, out.P);
    served = box_particle<KC, FOV>(H, R, G, S_pos, S_id, r, s, 0, out, &r, bc, nullptr);
    if (!served) out.radius()[s] = left_radius(r, bc);
  }
  warp_append(valid && !served, make_int2((int)s, rep), defer_list, defer_count);
}

// Handed-on particles, long lists: one thread each, up to two larger squares;
// what is left goes on the second list.  A list that would leave most of the
// chip idle at one thread per particle is left whole to the groups of the
// next kernel (which serve a particle at 1.4 ns when they fill the chip, a
// thread at 0.45 ns, but a thread takes about 30 us from start to end).
constexpr int kLongList = 24576;
constexpr int kSecondTries = 2;

template <int KC, bool FOV, class Out>
__global__ void __launch_bounds__(kBlk, BoxCfg<KC>::BLOCKS) knn2_second_kernel(
    const Rep* __restrict__ reps, const int2* __restrict__ S_pos, const int32_t* __restrict__ S_id, GridView G,
    Out out, const int2* __restrict__ list, const int32_t* __restrict__ count, int2* __restrict__ left_list,
    int32_t* __restrict__ left_count) {
  extern __shared__ __align__(16) unsigned char box_smem[];
  BoxShared<KC>& H = *reinterpret_cast<BoxShared<KC>*>(box_smem);
  const int total = *count;
  if (total < kLongList) return;
  int64_t step = 0;
  if constexpr (Out::kStep) step = *out.d_step;
  for (int base = blockIdx.x * kBlk; base < total; base += gridDim.x * kBlk) {
    const int i = base + (int)threadIdx.x;
    const bool valid = i < total;
    int2 e = make_int2(0, 0);
    float nnew[3] = {0.f, 0.f, 0.f};
    BoxCount bc;
    bool served = false;
    if (valid) {
      e = list[i];
      const Rep R = reps[e.y];
      float r = out.radius()[e.x];
      for (int tr = 0; tr < kSecondTries && !served && r > 0.f; ++tr) {
        served = box_particle<KC, FOV>(H, R, G, S_pos, S_id, r, e.x, step, out, &r, bc, nnew);
        if (!served) r = left_radius(r, bc);
      }
      if (!served) out.radius()[e.x] = r;
    }
    warp_append(valid && !served, e, left_list, left_count);
    if constexpr (Out::kStep) {
      phi_add_warp<2>(out.phi_acc + (size_t)(step % out.P.phi_cap) * (size_t)out.P.n_rep * 3, e.y, nnew, served);
      record_search_stats(out.P.stats, served, bc.cand, 0u, false);
      if (out.P.stats && bc.tries) atomicAdd(out.P.stats + 1, (unsigned long long)bc.tries);
    }
  }
}

// The rest: GS lanes each, larger squares until k hits are in one.  A warp
// takes up to 32 particles, its groups search them one after another, and
// then every lane updates one, so that the update runs on full warps.  Takes
// the first list where the kernel above left it (its length is read on the
// device, so that the launch can sit in a CUDA graph).
//
// ALL: small systems (and the general search) come here at once, every particle
// (n_all of them, by the tasks of a step or those of one replica): the thread
// kernel's time is one particle's, from start to end, however few there are, and
// the listed ones wait for it.
constexpr int kGS = 16;
constexpr int kGroupBlk = 128;
// resident blocks per SM that the kernel is compiled for, for long lists and for small systems
template <int KC> constexpr int kListBlocks = KC <= 12 ? 6 : 3;
template <int KC> constexpr int kSmallBlocks = KC <= 12 ? 4 : 3;
constexpr float kWholeBox = 4.6e18f;  // squared distance beyond every box's

template <int KC, bool FOV, bool ALL, int BLOCKS, class Out>
__global__ void __launch_bounds__(kGroupBlk, BLOCKS) knn2_group_kernel(
    const Rep* __restrict__ reps, const int2* __restrict__ S_pos, const int32_t* __restrict__ S_id, GridView G,
    Out out, const int2* __restrict__ first_list, const int2* __restrict__ left_list,
    const int32_t* __restrict__ counts, int64_t n_all, const BlockTask* __restrict__ tasks, int one_rep,
    const float* __restrict__ S_hint) {
  constexpr int CAP = GroupCfg<KC>::CAP, NG = 32 / kGS, NW = kGroupBlk / 32;
  __shared__ GroupList<CAP> lists[kGroupBlk / kGS];
  __shared__ int32_t res[NW][32][KC - 1];  // slots of the k nearest of the warp's particles
  __shared__ float res_d[NW][32];          // their k-th squared distance
  const bool first = !ALL && counts[0] < kLongList;
  const int2* __restrict__ list = first ? first_list : left_list;
  const int64_t total = ALL ? n_all : first ? counts[0] : counts[1];
  // (slot, replica) of entry i; slot -1 where a replica's last task has no particle
  auto entry = [&](int64_t i) -> int2 {
    if (!ALL) return list[i];
    if (!tasks) return make_int2((int)(reps[one_rep].p0 + i), one_rep);
    const BlockTask t = tasks[i / kBlock];
    const int li = t.first + (int)(i % kBlock);
    return make_int2(li < reps[t.rep].n ? (int)(reps[t.rep].p0 + li) : -1, t.rep);
  };
  const int lane = (int)(threadIdx.x & 31), wid = (int)(threadIdx.x >> 5);
  const int nw = (int)gridDim.x * NW, w = (int)blockIdx.x * NW + wid;
  // short lists are spread over all warps, long ones taken 32 at a time
  const int chunk = (int)min((int64_t)32, (total + (int64_t)nw * NG - 1) / ((int64_t)nw * NG) * NG);
  int64_t step = 0;
  if constexpr (Out::kStep) step = *out.d_step;
  const int k = out.P.k;
  for (int64_t base = (int64_t)w * chunk; base < total; base += (int64_t)nw * chunk) {
    const int todo = (int)min((int64_t)chunk, total - base);
    for (int i = lane / kGS; i < todo; i += NG) {
      const int2 e = entry(base + i);
      if (e.x < 0) continue;
      const Rep& R = reps[e.y];
      Group<kGS, CAP, FOV> g{{lists[threadIdx.x / kGS], S_id, ((1u << kGS) - 1u) << (lane / kGS * kGS),
                              lane / kGS * kGS, lane % kGS, e.x},
                             S_pos};
      const int2 p = S_pos[e.x];
      init_ctx(g.C, R, e.x, p);
      if (FOV) g.C.view = make_view(out.S_dir[e.x], out.P.fov_cq);
      g.k = k;
      float r = ALL ? box_radius(reps + e.y, G, p, S_hint ? S_hint[e.x] : 0.f, out.P) : fabsf(out.radius()[e.x]);
      uint32_t tries = 1;
      g.n_cand = 0;
      for (;; ++tries) {
        const int64_t a = (int64_t)ceilf(fminf(r, 4.0e9f));
        g.cnt = 0;
        if (g.square(R, G, a) || g.cnt >= k) break;
        const float want = 1.5f * (float)k + 1.f;
        r = (float)a * (g.cnt > 0 ? fminf(sqrtf(want / (float)g.cnt), 2.f) : 2.f) + 1.f;
      }
      for (int j = g.cnt + g.gl; j < k; j += kGS) res[wid][i][j] = -1;
      // (a view that holds fewer than k: the next search begins with the whole box)
      if (g.gl == 0) res_d[wid][i] = FOV && g.cnt < k ? kWholeBox : 0.f;
      __syncwarp(g.mask);
      g.rank([&](int, int rk, unsigned long long D, int32_t q) {
        if (rk < k) res[wid][i][rk] = q;
        if (rk == k - 1) res_d[wid][i] = (float)D;
      });
      __syncwarp(g.mask);
      if constexpr (Out::kStep)
        if (out.P.stats && g.gl == 0) {
          atomicAdd(out.P.stats + 0, (unsigned long long)g.n_cand);
          atomicAdd(out.P.stats + 1, (unsigned long long)tries);
          atomicMax(out.P.stats + 2, (unsigned long long)g.n_cand);
          atomicAdd(out.P.stats + 3, 1ull);
          atomicAdd(out.P.stats + 4, 1ull);
        }
    }
    __syncwarp();
    // every lane one particle
    int2 e = make_int2(0, 0);
    float nnew[3] = {0.f, 0.f, 0.f};
    bool mine = lane < todo;
    if (mine) {
      e = entry(base + lane);
      mine = e.x >= 0;
    }
    if (mine) {
      out.put(reps[e.y], step, e.x, S_pos[e.x], S_id[e.x],
              [&](int j) { return res[wid][lane][j - (KC - 1 - k)]; }, res_d[wid][lane], nnew);
    }
    if constexpr (Out::kStep)
      phi_add_warp<2>(out.phi_acc + (size_t)(step % out.P.phi_cap) * (size_t)out.P.n_rep * 3, e.y, nnew, mine);
    __syncwarp();
  }
}

GridView view_of(const Buffers& b) {
  GridView G;
  G.off = b.offsets;
  G.sub_s = b.sub_s;
  G.sub_base = b.sub_base;
  G.sub_off = b.sub_off;
  return G;
}

// blocks of the group kernel: as many as fit at once, fewer for small systems
int group_blocks(int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + 7) / 8, (int64_t)device_sm_count() * 6));
}
// blocks of the second-square kernel (strides over lists of any length)
template <int KC>
int second_blocks(int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + kBlk - 1) / kBlk, (int64_t)device_sm_count() * BoxCfg<KC>::BLOCKS));
}

// Systems of up to this many particles: the groups alone.  us per step, all
// three kernels / groups (up to here the sort also became one launch): 256,
// k = 7 69 / 23; 2048, k = 7 78 / 31, k = 32 125 / 98; 4096, k = 7 89 / 40, k = 32
// 142 / 126; 8192, k = 7 97 / 80, k = 16 105 / 114, k = 32 173 / 268.
constexpr int64_t kDirect2 = 4096;

template <int KC>
StepOut<KC> step_out(const Buffers& b, const StepParams& P) {
  return {(const float2*)b.S_dir, (int2*)b.U_pos, (float2*)b.U_dir, b.U_id, b.U_hint, b.counts, b.phi_acc, b.d_step, P};
}

// every particle by the group kernel: those of the tasks (n of them with the
// tasks' unused places), or of one replica
template <int KC, bool FOV, class Out>
cudaError_t group_all(const Geometry& g, const Buffers& b, const Out& out, int64_t n, const BlockTask* tasks, int rep,
                      cudaStream_t st) {
  // a launch that four blocks per SM hold takes more registers (2048 particles, k = 7: 36.0 us
  // per step with room for six, 34.3 for four; 100,000 by the general search 191 and 213)
  const int blocks = group_blocks(n);
  auto kernel = KC <= 12 && blocks > 4 * device_sm_count() ? knn2_group_kernel<KC, FOV, true, kListBlocks<KC>, Out>
                                                           : knn2_group_kernel<KC, FOV, true, kSmallBlocks<KC>, Out>;
  kernel<<<blocks, kGroupBlk, 0, st>>>(g.reps, (const int2*)b.S_pos, b.S_id, view_of(b), out, nullptr, nullptr, nullptr, n,
                                       tasks, rep, b.S_hint);
  return cudaGetLastError();
}

template <int KC, bool FOV>
cudaError_t step2(const Geometry& g, const Buffers& b, const StepParams& P, cudaStream_t st) {
  if (knn2_direct(g.n_total, P))
    return group_all<KC, FOV>(g, b, step_out<KC>(b, P), (int64_t)g.n_tasks * kBlock, g.tasks, 0, st);
  // the lists are empty here: the previous scatter (or init) cleared them
  knn2_box_step_kernel<KC, FOV><<<g.n_tasks * kSplit, kBlk, sizeof(BoxShared<KC>), st>>>(
      g.reps, g.tasks, (const int2*)b.S_pos, b.S_id, b.S_hint, view_of(b), step_out<KC>(b, P), b.ovf_list,
      b.ovf_count);
  return cudaGetLastError();
}

// the listed particles: the first list in the first half of ovf_list, what the
// second squares leave in the second half
template <int KC, bool FOV, class Out>
void finish_lists(const Geometry& g, const Buffers& b, const Out& out, int64_t n, cudaStream_t st) {
  int2* left = b.ovf_list + g.n_total;
  knn2_second_kernel<KC, FOV><<<second_blocks<KC>(n), kBlk, sizeof(BoxShared<KC>), st>>>(
        g.reps, (const int2*)b.S_pos, b.S_id, view_of(b), out, b.ovf_list, b.ovf_count, left, b.ovf_count + 1);
  knn2_group_kernel<KC, FOV, false, kListBlocks<KC>><<<group_blocks(n), kGroupBlk, 0, st>>>(
      g.reps, (const int2*)b.S_pos, b.S_id, view_of(b), out, b.ovf_list, left, b.ovf_count, 0, nullptr, 0, nullptr);
}

template <int KC, bool FOV>
cudaError_t finish2(const Geometry& g, const Buffers& b, const StepParams& P, cudaStream_t st) {
  finish_lists<KC, FOV>(g, b, step_out<KC>(b, P), g.n_total, st);
  return cudaGetLastError();
}

template <int KC, bool FOV>
cudaError_t export2(const Geometry& g, const Buffers& b, int rep, int n, int32_t* out_ids, cudaStream_t st,
                    const StepParams& P) {
  if (n == 0) return cudaSuccess;
  // the lists are empty between steps; the caller clears what the export used
  const RowOut<KC> out{(const float2*)b.S_dir, b.S_id, out_ids, b.U_hint, P};
  if (knn2_direct(n, P)) return group_all<KC, FOV>(g, b, out, n, nullptr, rep, st);
  knn2_box_export_kernel<KC, FOV><<<(n + kBlk - 1) / kBlk, kBlk, sizeof(BoxShared<KC>), st>>>(
      g.reps, rep, (const int2*)b.S_pos, b.S_id, b.S_hint, view_of(b), out, b.ovf_list, b.ovf_count);
  finish_lists<KC, FOV>(g, b, out, n, st);
  return cudaGetLastError();
}

template <int KC>
cudaError_t prepare2() {
  const int bytes = (int)sizeof(BoxShared<KC>);
  const void* f[] = {(const void*)knn2_box_step_kernel<KC, false>, (const void*)knn2_box_step_kernel<KC, true>,
                      (const void*)knn2_box_export_kernel<KC, false>, (const void*)knn2_box_export_kernel<KC, true>,
                     (const void*)knn2_second_kernel<KC, false, StepOut<KC>>,
                     (const void*)knn2_second_kernel<KC, true, StepOut<KC>>,
                     (const void*)knn2_second_kernel<KC, false, RowOut<KC>>,
                     (const void*)knn2_second_kernel<KC, true, RowOut<KC>>};
  for (const void* k : f) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// f(the list size the kernels for k are compiled for, field of view or not)
template <int KC> using KeyCount = std::integral_constant<int, KC>;

template <class F>
cudaError_t for_k(const StepParams& P, F f) {
  auto view = [&](auto kc) { return P.fov_cq != kViewAll ? f(kc, std::true_type{}) : f(kc, std::false_type{}); };
  if (P.k <= 7) return view(KeyCount<8>{});
  if (P.k <= 11) return view(KeyCount<12>{});
  if (P.k <= 16) return view(KeyCount<17>{});
  return view(KeyCount<33>{});
}

}  // namespace

bool knn2_direct(int64_t n, const StepParams& P) { return P.knn_search == 1 || n <= kDirect2; }

cudaError_t prepare_knn2(int k) {
  if (k <= 7) return prepare2<8>();
  if (k <= 11) return prepare2<12>();
  if (k <= 16) return prepare2<17>();
  return prepare2<33>();
}

cudaError_t launch_knn2_step(const Geometry& g, const Buffers& b, const StepParams& P, cudaStream_t st) {
  return for_k(P, [&](auto kc, auto view) { return step2<kc(), view()>(g, b, P, st); });
}

cudaError_t launch_knn2_finish(const Geometry& g, const Buffers& b, const StepParams& P, cudaStream_t st) {
  return for_k(P, [&](auto kc, auto view) { return finish2<kc(), view()>(g, b, P, st); });
}

cudaError_t launch_knn2_export(const Geometry& g, const Buffers& b, int rep, int n, int32_t* out, cudaStream_t st,
                               const StepParams& P) {
  return for_k(P, [&](auto kc, auto view) { return export2<kc(), view()>(g, b, rep, n, out, st, P); });
}

}  // namespace vk
