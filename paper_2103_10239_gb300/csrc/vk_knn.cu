// vk_knn.cu -- k-nearest-neighbor rule (Sec. "Metric and topological flocking
// models": each particle aligns with its k nearest neighbors, at any distance,
// so the relation is not reciprocal) fused with the Vicsek update of Eq. (1)
// and Eq. (2), in 3D (the 2D rule, the benchmark's, is in vk_knn2d.cu).
//
// One thread per particle, in cell-sorted order, radius first: the cube around
// the particle a little wider than its k-th distance at the last step; 16 lanes
// each for the particles that this cube cannot serve.  Lists are exported by the
// same searches (a ring walk by one thread with a 64-bit list took 326 us for 5000
// particles, k = 7, 3.9 ms for 200,000, k = 32, and 28.4 ms for 60,000 in a cluster; this
// 67 us, 1.4 and 14.5 ms, with the copies).
#include <algorithm>
#include <climits>

#include "vk_group.cuh"
#include "vk_internal.cuh"

namespace vk {

namespace {

// ---------------------------------------------------------------------------
// Radius first (3D): each particle scans the cube [p - a, p + a]^3, a a
// little above its k-th neighbor distance at the previous step, as the
// x-row segments of the cells it meets (each a contiguous run of the sorted
// arrays, with the periodic image it lies in).  Nothing outside the cube is
// closer than a + 1.  As in 2D (vk_knn2d.cu) the selection runs on 32-bit
// keys, the FP32 squared distance with the hit's number in its low bits: a
// 64-bit list with ids cost eight compares and moves per hit, run by the few
// lanes that had one: 1943 us per step at 1M particles; this takes 906 with the
// particles handed on (1144 in cells of 1.5 particles and cubes of 1.3).
// Candidates within the cube's inscribed ball are buffered and merged after
// the scan by min / max; a list whose order the keys leave open, or with too
// few hits, is handed on.
// ---------------------------------------------------------------------------
constexpr int kBlk3 = 128;
constexpr int kSplit3 = kBlock / kBlk3;
constexpr int kRuns3 = 8;

// KC keys (k <= KC - 1 and the one after them), CAP buffered hits (about 2.2 k
// + 1 are expected) numbered in BITS bits
template <int KC> struct CubeCfg;
template <> struct CubeCfg<8> { static constexpr int CAP = 32, BITS = 5, BLOCKS = 5; };
template <> struct CubeCfg<17> { static constexpr int CAP = 64, BITS = 6, BLOCKS = 3; };
template <> struct CubeCfg<33> { static constexpr int CAP = 96, BITS = 7, BLOCKS = 2; };

template <int KC>
struct CubeShared {
  uint2 hit[CubeCfg<KC>::CAP][kBlk3];  // (slot, bits of the FP32 squared distance), one column per thread
  uint2 run[kRuns3][kBlk3];            // (first slot, length << 6 | image codes)
};

// unwrapped cell index of an unwrapped coordinate, -L <= x < 2L
__device__ __forceinline__ int ucell3(int64_t x, int n, const uint32_t* __restrict__ bnd, float inv_w, int64_t L) {
  if (x < 0) return cell_of_tab((uint32_t)(x + L), n, bnd, inv_w) - n;
  if (x >= L) return cell_of_tab((uint32_t)(x - L), n, bnd, inv_w) + n;
  return cell_of_tab((uint32_t)x, n, bnd, inv_w);
}

// Put the k nearest of the hits 0..cnt-1 of a thread's column (all of a cube's
// ball) in its first places, in order: by FP32 distances where these are far
// enough apart, else exactly, by (int64 squared distance, id).  Lattices of 64,000
// and of 56,000 particles, k = 7, us per step: all by groups 305 (simple cubic), 195
// (bcc), 176 (fcc), this 185, 119, 102.
__device__ __noinline__ void order_column(uint2 (*hit)[kBlk3], int cnt, int k, int32_t self,
                                          const int4* __restrict__ pos, const int32_t* __restrict__ ids,
                                          const Rep* __restrict__ rep) {
  const int tid = (int)threadIdx.x;
  const int4 p = pos[self];
  const int64_t Lx = rep->L[0], Ly = rep->L[1], Lz = rep->L[2];
  auto exact = [&](uint32_t q) {
    const int4 o = pos[q];
    const int64_t dx = min_image((int64_t)o.x - p.x, Lx), dy = min_image((int64_t)o.y - p.y, Ly),
                  dz = min_image((int64_t)o.z - p.z, Lz);
    return (uint64_t)(dx * dx) + (uint64_t)(dy * dy) + (uint64_t)(dz * dz);
  };
  for (int b = 0; b < cnt; ++b)
    if ((int32_t)hit[b][tid].x == self) hit[b][tid] = hit[--cnt][tid];
  for (int j = 0; j < k; ++j) {
    int best = j;
    uint2 h = hit[j][tid];
    uint64_t Dh = ~0ull;  // h's exact distance, once one was needed
    for (int b = j + 1; b < cnt; ++b) {
      const uint2 o = hit[b][tid];
      const float fo = __uint_as_float(o.y), fh = __uint_as_float(h.y);
      bool before = fo < fh;
      uint64_t Do = ~0ull;
      if (fabsf(fo - fh) <= fh * 3.814697265625e-06f) {  // 2^-18, eight times the FP32 error and more
        Do = exact(o.x);
        if (Dh == ~0ull) Dh = exact(h.x);
        before = Do < Dh || (Do == Dh && ids[o.x] < ids[h.x]);
      }
      if (before) {
        best = b;
        h = o;
        Dh = Do;
      }
    }
    hit[best][tid] = hit[j][tid];
    hit[j][tid] = h;
  }
}

// the k nearest from the cube of half-width ceil(radius), as keys
// t[KC-1-k .. KC-2] in order; false when it cannot decide, with the radius to
// try next
template <int KC>
__device__ __forceinline__ bool cube_search(CubeShared<KC>& H, const Rep& R, const Rep* __restrict__ rep,
                                            const uint32_t* __restrict__ bounds, const GridView& G,
                                            const int4* __restrict__ pos, const int32_t* __restrict__ ids,
                                            int32_t self, const int32_t* pi, float radius, int k, uint32_t* t, float* r_next,
                                            uint32_t* n_cand, uint32_t* n_runs) {
  constexpr int B = CubeCfg<KC>::BITS, CAP = CubeCfg<KC>::CAP;
  const int tid = (int)threadIdx.x;
  const int32_t a = (int32_t)ceilf(fminf(radius, 1.0e9f));
  *r_next = (float)a;
  int lo[3], hi[3];
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    const int64_t L = R.L[ax];
    if (4ll * a + 2 >= L) return false;
    const uint32_t* bnd = bounds + R.bnd[ax];
    lo[ax] = ucell3((int64_t)pi[ax] - a, R.nc[ax], bnd, R.inv_w[ax], L);
    hi[ax] = ucell3((int64_t)pi[ax] + a, R.nc[ax], bnd, R.inv_w[ax], L);
    if (hi[ax] - lo[ax] + 1 > R.nc[ax]) return false;
  }
  const float a1 = (float)a + 1.0f;
  float tau = a1 * a1 * (1.0f - 9.5367431640625e-07f);
  const uint32_t edge = __float_as_uint(tau) >> B;
#pragma unroll
  for (int e = 0; e < KC; ++e) t[e] = e < KC - 1 - k ? 0u : 0xFFFFFFFFu;
  const int nx = R.nc[0], ny = R.nc[1], nz = R.nc[2];
  int cnt = 0, merged = 0, got = 0;
  int uy = lo[1], uz = lo[2], seg = 0, nrun = 0, r = 0;
  uint32_t q = 0, qe = 0, ox = 0, oy = 0, oz = 0;
  bool more = true, done = false, wide = false, kept = true;
  for (;;) {
    while (cnt <= CAP - 2) {
      if (q == qe) {
        if (r == nrun) {
          nrun = r = 0;
          while (more && nrun < kRuns3) {
            const int cz = uz < 0 ? uz + nz : (uz >= nz ? uz - nz : uz);
            const int cy = uy < 0 ? uy + ny : (uy >= ny ? uy - ny : uy);
            const int64_t row = R.c0 + ((int64_t)cz * ny + cy) * nx;
            // the x range splits at the period into up to three segments
            const int xs = seg == 0 ? lo[0] : (seg == 1 ? max(lo[0], 0) : max(lo[0], nx));
            const int xe = seg == 0 ? min(hi[0], -1) : (seg == 1 ? min(hi[0], nx - 1) : hi[0]);
            if (xs <= xe) {
              const int wx = xs < 0 ? xs + nx : (xs >= nx ? xs - nx : xs);
              const uint32_t qb = __ldg(G.off + row + wx), qf = __ldg(G.off + row + wx + (xe - xs) + 1);
              // image codes per axis: 0 same, 1 at -L, 2 at +L
              const uint32_t code = (xs < 0 ? 1u : xs >= nx ? 2u : 0u) | (uy < 0 ? 4u : uy >= ny ? 8u : 0u) |
                                    (uz < 0 ? 16u : uz >= nz ? 32u : 0u);
              // longer than a run's length can say (no return from here: the warp's threads have to meet again)
              wide = wide || qf - qb >= 1u << 26;
              if (qf > qb) H.run[nrun++][tid] = make_uint2(qb, (qf - qb) << 6 | code);
            }
            if (++seg == 3 || (lo[0] >= 0 && hi[0] < nx && seg == 2)) {
              seg = lo[0] >= 0 && hi[0] < nx ? 1 : 0;
              if (++uy > hi[1]) {
                uy = lo[1];
                if (++uz > hi[2]) more = false;
              }
            }
          }
          *n_runs += (uint32_t)nrun;
          if (nrun == 0) {
            done = true;
            break;
          }
        }
        const uint2 e = H.run[r++][tid];
        q = e.x;
        qe = e.x + (e.y >> 6);
        *n_cand += e.y >> 6;
        // the particle shifted into the run's periodic image: offsets x_j - ox exactly
        ox = (uint32_t)pi[0] + (e.y & 1u ? R.L[0] : 0u) - (e.y & 2u ? R.L[0] : 0u);
        oy = (uint32_t)pi[1] + (e.y & 4u ? R.L[1] : 0u) - (e.y & 8u ? R.L[1] : 0u);
        oz = (uint32_t)pi[2] + (e.y & 16u ? R.L[2] : 0u) - (e.y & 32u ? R.L[2] : 0u);
      }
      // two candidates at a time (the second of an odd run's end is masked)
      const int4 p0 = __ldg(pos + q), p1 = __ldg(pos + min(q + 1, qe - 1));
      const int4 ps[2] = {p0, p1};
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float fx = (float)(int32_t)((uint32_t)ps[u].x - ox), fy = (float)(int32_t)((uint32_t)ps[u].y - oy),
                    fz = (float)(int32_t)((uint32_t)ps[u].z - oz);
        const float D = __fmaf_rn(fx, fx, __fmaf_rn(fy, fy, __fmul_rn(fz, fz)));
        H.hit[cnt][tid] = make_uint2(q + (uint32_t)u, __float_as_uint(D));
        cnt += D <= tau && q + (uint32_t)u < qe ? 1 : 0;
      }
      q = min(q + 2, qe);
      if (q == qe && r == nrun && !more) {
        done = true;
        break;
      }
    }
#pragma unroll 2
    for (int b = merged; b < cnt; ++b) {
      const uint2 h = H.hit[b][tid];
      const bool keep = (int32_t)h.x != self;
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
    kept = false;
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
  if ((t[KC - 2] >> B) + 1u < edge) {
    bool close = wide;  // a pair whose order the keys leave open
#pragma unroll
    for (int e = 0; e < KC - 1; ++e) close |= e >= KC - 1 - k && (t[e + 1] >> B) - (t[e] >> B) <= 1u;
    // The column holds all that come into question: order it exactly (lattices;
    // groups would take twice as long).  Not where keys are so many that chance
    // alone leaves some pair open in most warps (200,000 particles, k = 32: 1066 us per
    // step without, 1204 with).
    if (KC <= 17 && close && kept && !wide) {
      order_column(H.hit, cnt, k, self, pos, ids, rep);
#pragma unroll
      for (int e = 0; e < KC - 1; ++e)
        if (e >= KC - 1 - k) {
          const int j = e - (KC - 1 - k);
          t[e] = (H.hit[j][tid].y & ~((1u << B) - 1u)) | (uint32_t)j;
        }
      return true;
    }
    return !close;
  }
  // too few: scale the radius towards about 1.6 k expected hits
  *r_next = (float)a * (got > 0 ? fminf(cbrtf(1.6f * (float)(k + 1) / (float)got), 2.f) : 2.f);
  return false;
}

// search radius without a hint: from the density of the particle's own cell
__device__ __forceinline__ float cube_radius_estimate(const Rep& R, const uint32_t* __restrict__ bounds,
                                                      const GridView& G, const int32_t* pi, int k) {
  int c[3];
  float vol = 1.f;
#pragma unroll
  for (int ax = 0; ax < 3; ++ax) {
    const uint32_t* bnd = bounds + R.bnd[ax];
    c[ax] = cell_of_tab((uint32_t)pi[ax], R.nc[ax], bnd, R.inv_w[ax]);
    vol *= (float)(__ldg(bnd + c[ax] + 1) - __ldg(bnd + c[ax]));
  }
  const int64_t gc = R.c0 + ((int64_t)c[2] * R.nc[1] + c[1]) * R.nc[0] + c[0];
  const float m = (float)max(__ldg(G.off + gc + 1) - __ldg(G.off + gc), 1u);
  return 1.3f * cbrtf(3.f * (float)k * vol / (4.f * 3.14159265f * m));
}

// the first radius of a particle
__device__ __forceinline__ float cube_radius(const Rep& R, const uint32_t* __restrict__ bounds, const GridView& G,
                                             const int32_t* pi, float hint, const StepParams& P) {
  return hint > 0.f ? P.halo_alpha * hint : cube_radius_estimate(R, bounds, G, pi, P.k);
}

// Eq. (2) + Eq. (1) of one particle; at(j) is the slot of list entry j in
// [KC-1-k, KC-1), in (D, id) order.  Writes the next state and counts the new cell.
template <int KC, class At>
__device__ __forceinline__ void knn3_update(const Rep& R, const StepParams& P, int64_t step, int64_t s,
                                            const int32_t* pi, int32_t id, At at, const float4* __restrict__ S_dir,
                                            int4* __restrict__ U_pos, float4* __restrict__ U_dir,
                                            int32_t* __restrict__ U_id, uint32_t* __restrict__ U_rank,
                                            uint32_t* __restrict__ counts, const uint32_t* __restrict__ bounds,
                                            float* nnew) {
  float ni[3];
  unpack(S_dir[s], ni);
  HeadSum<3> H;
  H.init();
  if (P.include_self) H.add(ni, P.sum_mode);
#pragma unroll
  for (int c = 0; c < KC - 1; c += 4) {
    float4 d[4];  // four headings in flight, then summed in order
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c + u < KC - 1 && c + u >= KC - 1 - P.k) d[u] = __ldg(S_dir + at(c + u));
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (c + u < KC - 1 && c + u >= KC - 1 - P.k) {
        const float v[3] = {d[u].x, d[u].y, d[u].z};
        H.add(v, P.sum_mode);
      }
  }
  int32_t pout[3] = {0, 0, 0};
  align_advect<3>(R, P, (uint32_t)step, id, ni, H, P.k + (P.include_self ? 1 : 0), pi, pout, nnew);
  U_pos[s] = make_int4(pout[0], pout[1], pout[2], 0);
  U_dir[s] = make_float4(nnew[0], nnew[1], nnew[2], 0.f);
  U_id[s] = id;
  int64_t lin = 0;
#pragma unroll
  for (int ax = 2; ax >= 0; --ax)
    lin = lin * R.nc[ax] + cell_of_tab((uint32_t)pout[ax], R.nc[ax], bounds + R.bnd[ax], R.inv_w[ax]);
  U_rank[s] = atomicAdd(counts + R.c0 + lin, 1u);
}

// Search + update, one cube per particle.  Particles it cannot serve go on the
// list (slot, replica), with the radius to try next in U_hint.
template <int KC>
__global__ void __launch_bounds__(kBlk3, CubeCfg<KC>::BLOCKS) knn3_step_kernel(
    const Rep* __restrict__ reps, const BlockTask* __restrict__ tasks, const int4* __restrict__ S_pos,
    const float4* __restrict__ S_dir, const int32_t* __restrict__ S_id, GridView G, int4* __restrict__ U_pos,
    float4* __restrict__ U_dir, int32_t* __restrict__ U_id, uint32_t* __restrict__ U_rank,
    uint32_t* __restrict__ counts, PhiAcc* __restrict__ phi_acc, const int64_t* __restrict__ d_step, StepParams P,
    const uint32_t* __restrict__ bounds, const float* __restrict__ S_hint, float* __restrict__ U_hint,
    int2* __restrict__ list, int32_t* __restrict__ count) {
  extern __shared__ __align__(16) unsigned char cube_smem[];
  CubeShared<KC>& H = *reinterpret_cast<CubeShared<KC>*>(cube_smem);
  __shared__ PhiShared phs;
  phi_block_begin(phs);
  const BlockTask t = tasks[blockIdx.x / kSplit3];
  const Rep R = reps[t.rep];
  const int li = t.first + (int)(blockIdx.x % kSplit3) * kBlk3 + (int)threadIdx.x;
  const int64_t step = *d_step;
  float nnew[3] = {0.f, 0.f, 0.f};
  uint32_t n_cand = 0, n_runs = 0;
  bool served = false;
  if (li < R.n) {
    const int64_t s = R.p0 + li;
    int32_t pi[3];
    unpack(S_pos[s], pi);
    const float r = cube_radius(R, bounds, G, pi, S_hint[s], P);
    float r_next = r;
    uint32_t key[KC];
    served = cube_search<KC>(H, R, reps + t.rep, bounds, G, S_pos, S_id, (int32_t)s, pi, r, P.k, key, &r_next, &n_cand, &n_runs);
    if (served) {
      knn3_update<KC>(R, P, step, s, pi, S_id[s],
                      [&](int j) { return H.hit[key[j] & ((1u << CubeCfg<KC>::BITS) - 1u)][threadIdx.x].x; }, S_dir,
                      U_pos, U_dir, U_id, U_rank, counts, bounds, nnew);
      U_hint[s] = sqrtf(__uint_as_float(key[KC - 2])) * 1.0001f + 1.f;
    } else {
      U_hint[s] = r_next;
    }
  }
  // one atomic per warp: its entries stay neighbors in the list
  const unsigned m = __ballot_sync(0xffffffffu, li < R.n && !served);
  if (m) {
    const int lane = (int)(threadIdx.x & 31);
    int base = 0;
    if (lane == 0) base = atomicAdd(count, __popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (m >> lane & 1u) list[base + __popc(m & ((1u << lane) - 1u))] = make_int2((int)(R.p0 + li), t.rep);
  }
  record_search_stats(P.stats, served, n_cand, n_runs);
  phi_block_end<3>(phs, nnew, phi_acc + ((size_t)(step % P.phi_cap) * (size_t)P.n_rep + (size_t)t.rep) * 3);
}

// A group of GS lanes searches for one particle, exactly (vk_group.cuh): the
// lanes look up the rows of a cube's cells and scan them together.
template <int GS, int CAP>
struct Group3 : GroupTop<GS, CAP> {
  using Top = GroupTop<GS, CAP>;
  using Top::mask;
  using Top::shift;
  using Top::gl;
  using Top::tau;
  const int4* __restrict__ pos;
  const uint32_t* __restrict__ bounds;
  int32_t p[3];

  __device__ __forceinline__ void run(const Rep& R, uint32_t qb, uint32_t qe) {
    Top::n_cand += qe - qb;
    for (uint32_t b = qb; b < qe; b += GS) {
      const uint32_t q = b + (uint32_t)gl;
      bool hit = false;
      unsigned long long D = 0;
      if (q < qe && (int32_t)q != Top::self) {
        int32_t pj[3];
        unpack(__ldg(pos + q), pj);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int64_t d = min_image((int64_t)pj[a] - p[a], (int64_t)R.L[a]);
          D += (unsigned long long)(d * d);
        }
        hit = D <= tau;
      }
      Top::append(hit, D, q);
    }
  }

  // Every candidate of the cube of half-width a (an axis along which it meets
  // some cell twice is covered whole); true when it is the whole box.  Rows
  // farther than tau are passed over: a list that has filled up on the way
  // leaves little to scan.
  __device__ __forceinline__ bool cube(const Rep& R, const GridView& G, int64_t a) {
    int lo[3], hi[3];
    bool all = true;
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const int64_t L = R.L[x];
      lo[x] = 0;
      hi[x] = R.nc[x] - 1;
      if (2 * a + 1 < L) {
        const int l = ucell3((int64_t)p[x] - a, R.nc[x], bounds + R.bnd[x], R.inv_w[x], L);
        const int h = ucell3((int64_t)p[x] + a, R.nc[x], bounds + R.bnd[x], R.inv_w[x], L);
        if (h - l < R.nc[x]) {
          lo[x] = l;
          hi[x] = h;
          all = false;
        }
      }
    }
    tau = all ? ~0ull : (unsigned long long)(a + 1) * (unsigned long long)(a + 1) - 1;
    const int nx = R.nc[0], ny = R.nc[1], nz = R.nc[2];
    const int ry = hi[1] - lo[1] + 1, rows = ry * (hi[2] - lo[2] + 1);
    for (int xs = lo[0]; xs <= hi[0];) {  // the x range splits at the period
      const int wx = xs < 0 ? xs + nx : (xs >= nx ? xs - nx : xs);
      const int xe = min(hi[0], xs < 0 ? -1 : (xs < nx ? nx - 1 : INT_MAX));
      for (int r0 = 0; r0 < rows; r0 += GS) {
        const int row = r0 + gl;
        uint32_t qb = 0, qe = 0;
        if (row < rows) {
          const int uy = lo[1] + row % ry, uz = lo[2] + row / ry;
          const int cy = uy < 0 ? uy + ny : (uy >= ny ? uy - ny : uy), cz = uz < 0 ? uz + nz : (uz >= nz ? uz - nz : uz);
          const float dy = slab(1, cy, R), dz = slab(2, cz, R);
          if ((dy * dy + dz * dz) * 0.99999f <= (float)tau) {
            const int64_t rb = R.c0 + ((int64_t)cz * ny + cy) * nx;
            qb = __ldg(G.off + rb + wx);
            qe = __ldg(G.off + rb + wx + (xe - xs) + 1);
          }
        }
        unsigned m = (__ballot_sync(mask, qe > qb) & mask) >> shift;
        while (m) {
          const int j = shift + __ffs(m) - 1;
          m &= m - 1u;
          run(R, __shfl_sync(mask, qb, j), __shfl_sync(mask, qe, j));
        }
      }
      xs = xe + 1;
    }
    return all;
  }

  // larger cubes, from half-width r, until k hits are in one; the number of cubes
  __device__ __forceinline__ uint32_t search(const Rep& R, const GridView& G, float r) {
    for (uint32_t tries = 1;; ++tries) {
      const int64_t a = (int64_t)ceilf(fminf(r, 4.0e9f));
      Top::cnt = 0;
      if (cube(R, G, a) || Top::cnt >= Top::k) return tries;
      r = (float)a * (Top::cnt > 0 ? fminf(cbrtf(1.6f * (float)(Top::k + 1) / (float)Top::cnt), 2.f) : 2.f) + 1.f;
    }
  }

  // (per lane) distance of cell slab c of axis x from the particle, over both images
  __device__ __forceinline__ float slab(int x, int c, const Rep& R) const {
    const uint32_t* bnd = bounds + R.bnd[x];
    const int64_t l = (int64_t)__ldg(bnd + c) - p[x], h = (int64_t)__ldg(bnd + c + 1) - 1 - p[x], L = R.L[x];
    if (l > 0) return (float)min(l, L - h);
    if (h < 0) return (float)min(-h, L + l);
    return 0.f;
  }
};

// The listed particles: 16 lanes each, larger cubes until k hits are in one
// (one thread each, with the ring walk as its last resort, took 500 us for the
// few particles of a small system).  A warp takes up to 32 of them, its groups
// search one after another, and then every lane updates one.  Small systems
// (and the general search) come here at once, every particle (n_all of them, by
// the tasks): the thread kernel's time is one particle's however few there are.
constexpr int kGS3 = 16, kGroupBlk3 = 128;

template <int KC>
__global__ void __launch_bounds__(kGroupBlk3, KC <= 8 ? 5 : 3) knn3_group_kernel(
    const Rep* __restrict__ reps, const int4* __restrict__ S_pos, const float4* __restrict__ S_dir,
    const int32_t* __restrict__ S_id, GridView G, int4* __restrict__ U_pos, float4* __restrict__ U_dir,
    int32_t* __restrict__ U_id, uint32_t* __restrict__ U_rank, uint32_t* __restrict__ counts,
    PhiAcc* __restrict__ phi_acc, const int64_t* __restrict__ d_step, StepParams P,
    const uint32_t* __restrict__ bounds, float* U_hint,
    const int2* __restrict__ list, const int32_t* __restrict__ count, int64_t n_all,
    const BlockTask* __restrict__ tasks, const float* __restrict__ S_hint) {
  constexpr int CAP = GroupCfg<KC>::CAP, NG = 32 / kGS3, NW = kGroupBlk3 / 32;
  __shared__ GroupList<CAP> lists[kGroupBlk3 / kGS3];
  __shared__ int32_t res[NW][32][KC - 1];
  __shared__ float res_d[NW][32];
  const bool all = n_all > 0;
  const int64_t total = all ? n_all : *count;
  // (slot, replica) of entry i; slot -1 where a replica's last task has no particle
  auto entry = [&](int64_t i) -> int2 {
    if (!all) return list[i];
    const BlockTask t = tasks[i / kBlock];
    const int li = t.first + (int)(i % kBlock);
    return make_int2(li < reps[t.rep].n ? (int)(reps[t.rep].p0 + li) : -1, t.rep);
  };
  const int lane = (int)(threadIdx.x & 31), wid = (int)(threadIdx.x >> 5);
  const int nw = (int)gridDim.x * NW, w = (int)blockIdx.x * NW + wid;
  const int chunk = (int)min((int64_t)32, (total + (int64_t)nw * NG - 1) / ((int64_t)nw * NG) * NG);
  const int64_t step = *d_step;
  const int k = P.k;
  for (int64_t base = (int64_t)w * chunk; base < total; base += (int64_t)nw * chunk) {
    const int todo = (int)min((int64_t)chunk, total - base);
    for (int i = lane / kGS3; i < todo; i += NG) {
      const int2 e = entry(base + i);
      if (e.x < 0) continue;
      const Rep& R = reps[e.y];
      const int4 p = S_pos[e.x];
      Group3<kGS3, CAP> g{{lists[threadIdx.x / kGS3], S_id, ((1u << kGS3) - 1u) << (lane / kGS3 * kGS3),
                           lane / kGS3 * kGS3, lane % kGS3, e.x},
                          S_pos, bounds, {p.x, p.y, p.z}};
      g.k = k;
      g.n_cand = 0;
      const uint32_t tries = g.search(R, G, all ? cube_radius(R, bounds, G, g.p, S_hint[e.x], P) : U_hint[e.x]);
      __syncwarp(g.mask);
      g.rank([&](int, int rk, unsigned long long D, int32_t q) {
        if (rk < k) res[wid][i][rk] = q;
        if (rk == k - 1) res_d[wid][i] = (float)D;
      });
      __syncwarp(g.mask);
      if (P.stats && g.gl == 0) {
        atomicAdd(P.stats + 0, (unsigned long long)g.n_cand);
        atomicAdd(P.stats + 1, (unsigned long long)tries);
        atomicMax(P.stats + 2, (unsigned long long)g.n_cand);
        atomicAdd(P.stats + 3, 1ull);
      }
    }
    __syncwarp();
    int2 e = make_int2(0, 0);
    float nnew[3] = {0.f, 0.f, 0.f};
    bool mine = lane < todo;
    if (mine) {
      e = entry(base + lane);
      mine = e.x >= 0;
    }
    if (mine) {
      int32_t pi[3];
      unpack(S_pos[e.x], pi);
      knn3_update<KC>(reps[e.y], P, step, e.x, pi, S_id[e.x], [&](int j) { return res[wid][lane][j - (KC - 1 - k)]; },
                      S_dir, U_pos, U_dir, U_id, U_rank, counts, bounds, nnew);
      U_hint[e.x] = sqrtf(res_d[wid][lane]) * 1.0001f + 1.f;
    }
    phi_add_warp<3>(phi_acc + (size_t)(step % P.phi_cap) * (size_t)P.n_rep * 3, e.y, nnew, mine);
    __syncwarp();
  }
}

// Neighbor lists of one replica, written by id: one cube per particle, as in a
// step; those that it cannot serve go on the list ...
template <int KC>
__global__ void __launch_bounds__(kBlk3, CubeCfg<KC>::BLOCKS) knn3_cube_export_kernel(
    const Rep* __restrict__ reps, int rep, const int4* __restrict__ S_pos, const int32_t* __restrict__ S_id, GridView G,
    StepParams P, const uint32_t* __restrict__ bounds, const float* __restrict__ S_hint, float* __restrict__ radius,
    int32_t* __restrict__ out, int2* __restrict__ list, int32_t* __restrict__ count) {
  extern __shared__ __align__(16) unsigned char cube_smem[];
  CubeShared<KC>& H = *reinterpret_cast<CubeShared<KC>*>(cube_smem);
  const Rep R = reps[rep];
  const int li = blockIdx.x * kBlk3 + (int)threadIdx.x;
  if (li >= R.n) return;
  const int64_t s = R.p0 + li;
  int32_t pi[3];
  unpack(S_pos[s], pi);
  float r_next;
  uint32_t key[KC], n_cand = 0, n_runs = 0;
  const float r = cube_radius(R, bounds, G, pi, S_hint[s], P);
  if (cube_search<KC>(H, R, reps + rep, bounds, G, S_pos, S_id, (int32_t)s, pi, r, P.k, key, &r_next, &n_cand, &n_runs)) {
    int32_t* row = out + (int64_t)S_id[s] * P.k;
#pragma unroll
    for (int j = 0; j < KC - 1; ++j)
      if (j >= KC - 1 - P.k)
        row[j - (KC - 1 - P.k)] = __ldg(S_id + H.hit[key[j] & ((1u << CubeCfg<KC>::BITS) - 1u)][threadIdx.x].x);
  } else {
    radius[s] = r_next;
    list[atomicAdd(count, 1)] = make_int2((int)s, rep);
  }
}

// ... of the groups (n_all > 0: every particle, small systems)
template <int KC>
__global__ void __launch_bounds__(kGroupBlk3, KC <= 8 ? 5 : 3) knn3_group_export_kernel(
    const Rep* __restrict__ reps, int rep, const int4* __restrict__ S_pos, const int32_t* __restrict__ S_id, GridView G,
    StepParams P, const uint32_t* __restrict__ bounds, const float* __restrict__ S_hint,
    const float* __restrict__ radius, int32_t* __restrict__ out, const int2* __restrict__ list,
    const int32_t* __restrict__ count, int n_all) {
  constexpr int CAP = GroupCfg<KC>::CAP, kGroups = kGroupBlk3 / kGS3;
  __shared__ GroupList<CAP> lists[kGroups];
  const int lane = (int)(threadIdx.x & 31), total = n_all > 0 ? n_all : *count, k = P.k;
  const Rep& R = reps[rep];
  for (int i = blockIdx.x * kGroups + (int)threadIdx.x / kGS3; i < total; i += gridDim.x * kGroups) {
    const int32_t s = n_all > 0 ? (int32_t)(R.p0 + i) : list[i].x;
    const int4 p = S_pos[s];
    Group3<kGS3, CAP> g{{lists[threadIdx.x / kGS3], S_id, ((1u << kGS3) - 1u) << (lane / kGS3 * kGS3),
                         lane / kGS3 * kGS3, lane % kGS3, s},
                        S_pos, bounds, {p.x, p.y, p.z}};
    g.k = k;
    g.n_cand = 0;
    g.search(R, G, n_all > 0 ? cube_radius(R, bounds, G, g.p, S_hint[s], P) : radius[s]);
    int32_t* row = out + (int64_t)S_id[s] * k;
    g.rank([&](int, int rk, unsigned long long, int32_t q) {
      if (rk < k) row[rk] = __ldg(S_id + q);
    });
    __syncwarp(g.mask);
  }
}

GridView grid_view(const Buffers& b) {
  GridView G;
  G.off = b.offsets;
  G.sub_s = b.sub_s;
  G.sub_base = b.sub_base;
  G.sub_off = b.sub_off;
  return G;
}

// Systems of up to this many particles: the groups alone.  us per step, both
// kernels / groups: 2048, k = 7 159 / 51; 16384 185 / 121, k = 32 664 / 441;
// 32768, k = 7 207 / 161, k = 32 752 / 740.
constexpr int64_t kDirect3 = 32768;
bool knn3_direct(int64_t n, const StepParams& P) { return P.knn_search == 1 || n <= kDirect3; }

template <int KC>
cudaError_t step_dispatch(const Geometry& g, const Buffers& b, const StepParams& P, cudaStream_t st) {
  const size_t smem = sizeof(CubeShared<KC>);
  const bool all = knn3_direct(g.n_total, P);
  if (!all)
    knn3_step_kernel<KC><<<g.n_tasks * kSplit3, kBlk3, smem, st>>>(
        g.reps, g.tasks, (const int4*)b.S_pos, (const float4*)b.S_dir, b.S_id, grid_view(b), (int4*)b.U_pos,
        (float4*)b.U_dir, b.U_id, b.U_rank, b.counts, b.phi_acc, b.d_step, P, b.bounds, b.S_hint, b.U_hint, b.ovf_list,
        b.ovf_count);
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((g.n_total + 7) / 8, (int64_t)device_sm_count() * 5));
  knn3_group_kernel<KC><<<blocks, kGroupBlk3, 0, st>>>(
      g.reps, (const int4*)b.S_pos, (const float4*)b.S_dir, b.S_id, grid_view(b), (int4*)b.U_pos, (float4*)b.U_dir,
      b.U_id, b.U_rank, b.counts, b.phi_acc, b.d_step, P, b.bounds, b.U_hint, b.ovf_list, b.ovf_count,
      all ? (int64_t)g.n_tasks * kBlock : 0, g.tasks, b.S_hint);
  return cudaGetLastError();
}

template <int KC>
cudaError_t prepare3() {
  cudaError_t e = cudaFuncSetAttribute(knn3_step_kernel<KC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(CubeShared<KC>));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(knn3_cube_export_kernel<KC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(CubeShared<KC>));
  return e;
}

template <int KC>
cudaError_t export_dispatch(const Geometry& g, const Buffers& b, int rep, int n, int32_t* out, cudaStream_t st,
                            const StepParams& P) {
  if (n == 0) return cudaSuccess;
  // the list is empty between steps; the export clears what it used
  const bool all = knn3_direct(n, P);
  if (!all)
    knn3_cube_export_kernel<KC><<<(n + kBlk3 - 1) / kBlk3, kBlk3, sizeof(CubeShared<KC>), st>>>(
        g.reps, rep, (const int4*)b.S_pos, b.S_id, grid_view(b), P, b.bounds, b.S_hint, b.U_hint, out, b.ovf_list,
        b.ovf_count);
  const int blocks = std::max(1, std::min((n + 7) / 8, device_sm_count() * 5));
  knn3_group_export_kernel<KC><<<blocks, kGroupBlk3, 0, st>>>(g.reps, rep, (const int4*)b.S_pos, b.S_id, grid_view(b), P,
                                                              b.bounds, b.S_hint, b.U_hint, out, b.ovf_list,
                                                              b.ovf_count, all ? n : 0);
  const cudaError_t e = all ? cudaSuccess : cudaMemsetAsync(b.ovf_count, 0, sizeof(int32_t), st);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace

int knn3_launches(int64_t n, const StepParams& P) { return knn3_direct(n, P) ? 1 : 2; }

cudaError_t prepare_knn3() {
  cudaError_t e = prepare3<8>();
  if (e == cudaSuccess) e = prepare3<17>();
  if (e == cudaSuccess) e = prepare3<33>();
  return e;
}

cudaError_t launch_knn_step(const Geometry& g, const Buffers& b, const StepParams& P, cudaStream_t st) {
  if (g.dim != 3) return cudaErrorInvalidValue;  // 2D: launch_knn2_step
  if (P.k <= 7) return step_dispatch<8>(g, b, P, st);
  if (P.k <= 16) return step_dispatch<17>(g, b, P, st);
  return step_dispatch<33>(g, b, P, st);
}

cudaError_t launch_knn_export(const Geometry& g, const Buffers& b, int rep, int n, int32_t* out, cudaStream_t st,
                              const StepParams& P) {
  if (g.dim != 3) return cudaErrorInvalidValue;  // 2D: launch_knn2_export
  if (P.k <= 7) return export_dispatch<8>(g, b, rep, n, out, st, P);
  if (P.k <= 16) return export_dispatch<17>(g, b, rep, n, out, st, P);
  return export_dispatch<33>(g, b, rep, n, out, st, P);
}

}  // namespace vk
