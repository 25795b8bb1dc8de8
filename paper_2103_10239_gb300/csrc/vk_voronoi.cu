// vk_voronoi.cu -- Voronoi-neighbor rule (Sec. "Computational tools: Voronoi
// neighbor lists": the Voronoi cell is the region closer to a particle than to
// any other; Voronoi and Delaunay neighbors are dual, and the relation is
// reciprocal) fused with the Vicsek update of Eq. (1) and Eq. (2).
//
// Instead of a global (serial) triangulation, every particle builds its own
// Voronoi cell by half-plane clipping, which is embarrassingly parallel:
//   * the cell starts as the square bounded by the particle's own periodic
//     images (+-L_x, 0), (0, +-L_y), and every candidate of the cell grid clips
//     it by its bisector.  The polygon is a cyclic list of the sites that define
//     its edges; a vertex is the circumcenter of the particle (at the origin)
//     and two consecutive sites.  "Vertex beyond the bisector of m" is exactly
//     incircle(0, a, b, m) > 0, i.e. 2 m.V > |m|^2: decided from an FP32
//     estimate of V with a rigorous error bound, else by an FP32 filter of the
//     incircle determinant, else exactly in int128;
//   * a site can still cut the cell only inside the union of the disks
//     through the particle centred at the vertices (the disk of V holds the
//     points closer to V than the particle is); its bounding box, the
//     relevance box, only shrinks;
//   * ordinary cells: vk_voronoi_fast.cuh.  A cell that outgrows 16 edges, meets
//     too many candidates (a particle bordering a void), reaches half a
//     period or has coincident particles is finished by the overflow kernel,
//     one warp per cell: the lanes test 32 candidates at a time against the
//     current cell and one lane applies the few that cut it;
//   * neighbors are the sites of edges with positive length (an edge between
//     two coincident vertices, i.e. four cocircular points, is dropped);
//   * coincident particles form one site (see Poly).
// Exact predicates need |relative coordinates| < 1.5 * 2^30, hence L_q <= 2^30.
#include "vk_voronoi_fast.cuh"

namespace vk {

namespace {

// the Vicsek update of one particle from its finished cell
template <int CAP>
__device__ __forceinline__ void voronoi_update(const Rep& R, const StepParams& Pm, int64_t step, int64_t s,
                                               const Poly<CAP>& P, const int32_t* pi, const float* ni,
                                               int32_t id, const float2* __restrict__ S_dir,
                                               int2* __restrict__ U_pos, float2* __restrict__ U_dir,
                                               int32_t* __restrict__ U_id, uint32_t* __restrict__ counts,
                                               float* nnew, int32_t* __restrict__ seed_out,
                                               int32_t* __restrict__ seed_n_out, bool heavy_next) {
  int32_t nid[CAP + Poly<CAP>::TW], nslot[CAP + Poly<CAP>::TW];
  const int cnt = voronoi_neighbors(P, id, nid, nslot);
  if (seed_out) {
    // the next step's seeds (any subset of sites would do)
    const int ns = min(cnt, kVorSeed);
    for (int j = 0; j < ns; ++j) seed_out[j] = nid[j];
    *seed_n_out = seed_word(ns, heavy_next, 2.0f * sqrtf(P.max_r2));
  }
  HeadSum<2> H;
  H.init();
  if (Pm.include_self) H.add(ni, Pm.sum_mode);
  for (int j = 0; j < cnt; ++j) {
    const float2 d = S_dir[nslot[j]];
    const float v[2] = {d.x, d.y};
    H.add(v, Pm.sum_mode);
  }
  int32_t pout[3] = {0, 0, 0};
  align_advect<2>(R, Pm, (uint32_t)step, id, ni, H, cnt + (Pm.include_self ? 1 : 0), pi, pout, nnew);
  U_pos[s] = make_int2(pout[0], pout[1]);
  U_dir[s] = make_float2(nnew[0], nnew[1]);
  U_id[s] = id;
  atomicAdd(counts + linear_cell<2>(R, pout), 1u);
}

// Heavy-cell hint: a cell that needed more than heavy_hint candidates in the
// main kernel, or half as many in the warp kernel, is flagged in its seed word,
// and the next step sends it to the warp kernel at once (particles on the rim of
// a void stay there for many steps).  Speed only.
__device__ __forceinline__ uint32_t heavy_hint(uint32_t heavy) { return heavy / 6u * 5u; }

// Main kernel: the ordinary cells, eight lanes each (vk_voronoi_fast.cuh).
// The others go on the overflow list.  A warp builds the cells of 4 x ROUNDS
// consecutive particles, four at a time, and then updates them, one per lane.
// A cell that met more than kSeedMin candidates keeps its neighbors as the
// next step's seeds, until it has shrunk to half the reach it had then: a
// particle beside a void has a wide box until its own neighbors bound the cell,
// while the nearest particles bound an ordinary one as well, and are one load
// away instead of three.  Measured (us per step, no seeds / these / seeds for
// every cell): 65,536 particles beside a lattice, steps 100 on, 1645 / 1534 / 1493,
// 1000 particles with voids 186 / 138 / 121, 512k 4682 / 3980 / 3435, but 20,000 in a
// random state 171 / 169 / 263 and the first ten steps beside the lattice 344 / 343 /
// 540.  (kSeedMin of 96 and 256: 512k 3863 and 4318, beside the lattice 352 and 375.)
constexpr uint32_t kSeedMin = 160;
constexpr int kCellBlk = 128;
// resident blocks per SM the main kernel is compiled for
#ifndef VK_VOR_MIN_BLOCKS
#define VK_VOR_MIN_BLOCKS 4
#endif

template <int ROUNDS>
__global__ void __launch_bounds__(kCellBlk, VK_VOR_MIN_BLOCKS) voronoi_step_kernel(
    const Rep* __restrict__ reps, const BlockTask* __restrict__ tasks, const int2* __restrict__ S_pos,
    const float2* __restrict__ S_dir, const int32_t* __restrict__ S_id, GridView G,
    int2* __restrict__ U_pos, float2* __restrict__ U_dir, int32_t* __restrict__ U_id,
    uint32_t* __restrict__ counts, PhiAcc* __restrict__ phi_acc, const int64_t* __restrict__ d_step, StepParams Pm,
    int2* __restrict__ ovf_list, int32_t* __restrict__ ovf_count, int32_t* __restrict__ vor_seed,
    int32_t* __restrict__ vor_seed_n, const int32_t* __restrict__ slot_of, uint32_t heavy) {
  __shared__ PhiShared phs;
  phi_block_begin(phs);
  constexpr int kPerBlock = kCellBlk / kCG * ROUNDS, kPerWarp = 4 * ROUNDS, kBlocks = kBlock / kPerBlock;
  const int lane = (int)(threadIdx.x & 31), wid = (int)(threadIdx.x >> 5);
  const BlockTask t = tasks[blockIdx.x / kBlocks];
  const Rep& R = reps[t.rep];
  const int li0 = t.first + (int)(blockIdx.x % kBlocks) * kPerBlock + wid * kPerWarp;
  const int64_t step = *d_step;
  Cell8 c;
  c.gl = lane & (kCG - 1);
  c.base = lane & ~(kCG - 1);
  // of the warp's particle number `lane`
  HeadSum<2> sum;
  sum.init();
  int my_m = -1;
  uint32_t my_seen = 0;
#pragma unroll 1
  for (int r = 0; r < ROUNDS; ++r) {
    const int li = li0 + 4 * r + lane / kCG;
    const bool on = li < R.n;
    if (!__any_sync(kAll, on)) break;
    const int64_t s = R.p0 + (on ? li : 0);
    const int2 p = S_pos[s];
    const int32_t id = S_id[s];
    const int64_t gi = R.p0 + id;
    const int32_t sw = vor_seed && on ? vor_seed_n[gi] : 0;
    const Seeds sd = seeds_of(vor_seed, sw, gi, slot_of);
    // a cell that was heavy at the last step goes straight to the warp kernel
    const bool mine = on && !(sw & kSeedHeavy);
    c.build(mine, R, s, p, S_pos, G, sd, heavy);
    const bool ok = mine && !c.other;
    if (on && !ok && c.gl == 0) ovf_list[atomicAdd(ovf_count, 1)] = make_int2((int)s, t.rep);
    // neighbors: the sites of edges of positive length, ordered by id
    int32_t nid[2];
    int rank[2];
    const int cnt = c.neighbors(ok, S_id, nid, rank);
    float2 d[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (rank[i] >= 0) d[i] = __ldg(S_dir + c.slot[i]);
    HeadSum<2> H;
    H.init();
    if (Pm.include_self) {
      const float2 nv = S_dir[s];
      const float ni[2] = {nv.x, nv.y};
      H.add(ni, Pm.sum_mode);
    }
    for (int k = 0; __any_sync(kAll, ok && k < cnt); ++k) {
      const bool second = rank[1] == k;
      const unsigned who = c.group_bits(rank[0] == k || second);
      const int from = c.base + (who ? __ffs(who) - 1 : 0);
      const float v[2] = {__shfl_sync(kAll, second ? d[1].x : d[0].x, from),
                          __shfl_sync(kAll, second ? d[1].y : d[0].y, from)};
      if (who) H.add(v, Pm.sum_mode);
    }
    if (vor_seed && ok) {
      const bool far = c.n_seen > kSeedMin, keep = far || (sd.n > 0 && c.reach() > 0.5f * sd.reach);
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (keep && rank[i] >= 0 && rank[i] < kVorSeed) vor_seed[gi * kVorSeed + rank[i]] = nid[i];
      if (c.gl == 0)
        vor_seed_n[gi] =
            keep ? seed_word(min(cnt, kVorSeed), c.n_seen > heavy_hint(heavy), far ? c.reach() : sd.reach) : 0;
    }
    // hand the sums to the lanes of these four particles
    const int from = (lane & 3) * kCG;
    const bool take = lane >> 2 == r;
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const float ts = __shfl_sync(kAll, H.s[a], from), tc = __shfl_sync(kAll, H.c[a], from);
      const double td = Pm.sum_mode == 2 ? __shfl_sync(kAll, H.d[a], from) : 0.0;
      if (take) {
        sum.s[a] = ts;
        sum.c[a] = tc;
        sum.d[a] = td;
      }
    }
    const int tm = __shfl_sync(kAll, ok ? cnt : -1, from);
    const uint32_t tn = __shfl_sync(kAll, c.n_seen, from);
    if (take) {
      my_m = tm;
      my_seen = tn;
    }
  }
  float nnew[3] = {0.f, 0.f, 0.f};
  const bool valid = lane < kPerWarp && li0 + lane < R.n;
  if (my_m >= 0) {
    const int64_t s = R.p0 + li0 + lane;
    const int2 p = S_pos[s];
    const float2 nv = S_dir[s];
    const int32_t id = S_id[s];
    const int32_t pi[3] = {p.x, p.y, 0};
    const float ni[3] = {nv.x, nv.y, 0.f};
    int32_t pout[3] = {0, 0, 0};
    align_advect<2>(R, Pm, (uint32_t)step, id, ni, sum, my_m + (Pm.include_self ? 1 : 0), pi, pout, nnew);
    U_pos[s] = make_int2(pout[0], pout[1]);
    U_dir[s] = make_float2(nnew[0], nnew[1]);
    U_id[s] = id;
    atomicAdd(counts + linear_cell<2>(R, pout), 1u);
  }
  record_search_stats(Pm.stats, valid, my_seen, 0, my_m < 0);
  phi_block_end<2>(phs, nnew, phi_acc + ((size_t)(step % Pm.phi_cap) * (size_t)Pm.n_rep + (size_t)t.rep) * 3);
}

// Overflow kernel: the few particles whose cell outgrew the main kernel's
// polygon (a particle bordering a void can have dozens of Voronoi
// neighbors) or needed too many candidates; one warp per particle.
constexpr int kOvfWarps = 4;

__global__ void __launch_bounds__(32 * kOvfWarps) voronoi_overflow_kernel(
    const Rep* __restrict__ reps, const int2* __restrict__ S_pos, const float2* __restrict__ S_dir,
    const int32_t* __restrict__ S_id, GridView G, int2* __restrict__ U_pos,
    float2* __restrict__ U_dir, int32_t* __restrict__ U_id,
    uint32_t* __restrict__ counts, PhiAcc* __restrict__ phi_acc, const int64_t* __restrict__ d_step, StepParams Pm,
    const int2* __restrict__ ovf_list, const int32_t* __restrict__ ovf_count, int32_t* status,
    int32_t* __restrict__ vor_seed, int32_t* __restrict__ vor_seed_n, const int32_t* __restrict__ slot_of,
    uint32_t heavy) {
  __shared__ Poly<kSlowCap> poly[kOvfWarps];
  Poly<kSlowCap>& P = poly[threadIdx.x >> 5];
  const int total = *ovf_count;
  const int64_t step = *d_step;
  const int nwarps = gridDim.x * kOvfWarps;
  for (int q = blockIdx.x * kOvfWarps + (int)(threadIdx.x >> 5); q < total; q += nwarps) {
    const int2 e = ovf_list[q];
    const Rep R = reps[e.y];
    const int64_t s = e.x;
    const int2 p = S_pos[s];
    const int32_t pi[3] = {p.x, p.y, 0};
    const int32_t id = S_id[s];
    const int64_t gi = R.p0 + id;
    const Seeds sd = seeds_of(vor_seed, vor_seed ? vor_seed_n[gi] : 0, gi, slot_of);
    uint32_t seen = 0;
    const bool ok = voronoi_cell_warp(R, s, pi, id, S_pos, S_id, G, P, status, sd, &seen);
    if ((threadIdx.x & 31) == 0) {
      if (!ok) {
        set_status(status, kStCapacity);
      } else {
        const float2 nv = S_dir[s];
        const float ni[3] = {nv.x, nv.y, 0.f};
        float nnew[3] = {0.f, 0.f, 0.f};
        voronoi_update(R, Pm, step, s, P, pi, ni, id, S_dir, U_pos, U_dir, U_id, counts, nnew,
                       vor_seed ? vor_seed + gi * kVorSeed : nullptr, vor_seed_n + gi, seen > heavy_hint(heavy) / 2u);
        PhiAcc* acc = phi_acc + ((size_t)(step % Pm.phi_cap) * (size_t)Pm.n_rep + (size_t)e.y) * 3;
        atomicAdd(acc + 0, (PhiAcc)phi_fixed(nnew[0]));
        atomicAdd(acc + 1, (PhiAcc)phi_fixed(nnew[1]));
      }
    }
    __syncwarp();
  }
}

// Lists: pass 0 writes the degree of every particle (by id), pass 1 the sorted
// ids at out_off[id].  As in a step, eight lanes build a cell, and a warp each of
// the others, which go on the list.  Measured (us for both passes with the copies to
// the host, one thread per cell with a polygon of 256 edges in local memory / this):
// 1000 particles 1770 / 420, 10,000 2530 / 228, a lattice of 40,000 813 / 351, 500,000
// 19,600 / 5570.
__global__ void __launch_bounds__(kCellBlk, VK_VOR_MIN_BLOCKS) voronoi_export_kernel(
    const Rep* __restrict__ reps, int rep, const int2* __restrict__ S_pos, const int32_t* __restrict__ S_id, GridView G,
    int pass, int32_t* __restrict__ deg, const int64_t* __restrict__ out_off, int32_t* __restrict__ out_ids,
    int2* __restrict__ ovf_list, int32_t* __restrict__ ovf_count, const int32_t* __restrict__ vor_seed,
    const int32_t* __restrict__ vor_seed_n, const int32_t* __restrict__ slot_of, uint32_t heavy) {
  const Rep& R = reps[rep];
  const int lane = (int)(threadIdx.x & 31);
  Cell8 c;
  c.gl = lane & (kCG - 1);
  c.base = lane & ~(kCG - 1);
  constexpr int kPerBlock = kCellBlk / kCG;
#pragma unroll 1
  for (int l0 = blockIdx.x * kPerBlock + (int)(threadIdx.x >> 5) * 4; l0 < R.n; l0 += gridDim.x * kPerBlock) {
    const int li = l0 + lane / kCG;
    const bool on = li < R.n;
    const int64_t s = R.p0 + (on ? li : 0);
    const int2 p = S_pos[s];
    const int32_t id = S_id[s];
    const int64_t gi = R.p0 + id;
    const Seeds sd = seeds_of(vor_seed, vor_seed && on ? vor_seed_n[gi] : 0, gi, slot_of);
    c.build(on, R, s, p, S_pos, G, sd, heavy);
    const bool ok = on && !c.other;
    if (on && !ok && c.gl == 0) ovf_list[atomicAdd(ovf_count, 1)] = make_int2((int)s, rep);
    int32_t nid[2];
    int rank[2];
    const int cnt = c.neighbors(ok, S_id, nid, rank);
    if (pass == 0) {
      if (ok && c.gl == 0) deg[id] = cnt;
    } else {
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (rank[i] >= 0) out_ids[out_off[id] + rank[i]] = nid[i];
    }
  }
}

__global__ void __launch_bounds__(32 * kOvfWarps) voronoi_overflow_export_kernel(
    const Rep* __restrict__ reps, const int2* __restrict__ S_pos, const int32_t* __restrict__ S_id, GridView G,
    int pass, int32_t* __restrict__ deg, const int64_t* __restrict__ out_off, int32_t* __restrict__ out_ids,
    const int2* __restrict__ ovf_list, const int32_t* __restrict__ ovf_count, int32_t* status,
    const int32_t* __restrict__ vor_seed, const int32_t* __restrict__ vor_seed_n,
    const int32_t* __restrict__ slot_of) {
  __shared__ Poly<kSlowCap> poly[kOvfWarps];
  Poly<kSlowCap>& P = poly[threadIdx.x >> 5];
  const int total = *ovf_count;
  for (int q = blockIdx.x * kOvfWarps + (int)(threadIdx.x >> 5); q < total; q += gridDim.x * kOvfWarps) {
    const int2 e = ovf_list[q];
    const Rep R = reps[e.y];
    const int2 p = S_pos[e.x];
    const int32_t pi[3] = {p.x, p.y, 0};
    const int32_t id = S_id[e.x];
    const int64_t gi = R.p0 + id;
    const Seeds sd = seeds_of(vor_seed, vor_seed ? vor_seed_n[gi] : 0, gi, slot_of);
    uint32_t seen = 0;
    const bool ok = voronoi_cell_warp(R, e.x, pi, id, S_pos, S_id, G, P, status, sd, &seen);
    if ((threadIdx.x & 31) == 0) {
      int32_t nid[kSlowCap + Poly<kSlowCap>::TW], nslot[kSlowCap + Poly<kSlowCap>::TW];
      if (!ok) set_status(status, kStCapacity);
      const int cnt = ok ? voronoi_neighbors(P, id, nid, nslot) : 0;
      if (pass == 0) {
        deg[id] = cnt;
      } else {
        for (int j = 0; j < cnt; ++j) out_ids[out_off[id] + j] = nid[j];
      }
    }
    __syncwarp();
  }
}

}  // namespace

static GridView grid_view(const Buffers& b) {
  GridView G;
  G.off = b.offsets;
  G.sub_s = b.sub_s;
  G.sub_base = b.sub_base;
  G.sub_off = b.sub_off;
  return G;
}

cudaError_t launch_voronoi_step(const Geometry& g, const Buffers& b, const StepParams& P, cudaStream_t st) {
  const GridView G = grid_view(b);
  const uint32_t heavy = g.n_total < kHeavyLine ? kHeavySmall : kHeavy;
  // 32 cells per warp (one full update) where that still fills the chip, 4 in small systems
  auto step = [&](auto kernel, int rounds) {
    kernel<<<g.n_tasks * (kBlock / (kCellBlk / kCG * rounds)), kCellBlk, 0, st>>>(
        g.reps, g.tasks, (const int2*)b.S_pos, (const float2*)b.S_dir, b.S_id, G, (int2*)b.U_pos, (float2*)b.U_dir,
        b.U_id, b.counts, b.phi_acc, b.d_step, P, b.ovf_list, b.ovf_count, b.vor_seed, b.vor_seed_n, b.slot_of,
        heavy);
  };
  const int64_t fill = (int64_t)device_sm_count() * VK_VOR_MIN_BLOCKS * (kCellBlk / kCG) * 3;
  if (g.n_total >= 8 * fill) step(voronoi_step_kernel<8>, 8);
  else if (g.n_total >= 2 * fill) step(voronoi_step_kernel<2>, 2);
  else step(voronoi_step_kernel<1>, 1);
  voronoi_overflow_kernel<<<device_sm_count() * 4, 32 * kOvfWarps, 0, st>>>(g.reps, (const int2*)b.S_pos, (const float2*)b.S_dir, b.S_id,
                                              G, (int2*)b.U_pos, (float2*)b.U_dir, b.U_id,
                                              b.counts, b.phi_acc, b.d_step, P, b.ovf_list, b.ovf_count,
                                              b.d_status, b.vor_seed, b.vor_seed_n, b.slot_of, heavy);
  return cudaGetLastError();
}

cudaError_t launch_voronoi_export(const Geometry& g, const Buffers& b, int rep, int n, int pass, int32_t* deg,
                                  const int64_t* out_off, int32_t* out_ids, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  // the list is empty between steps; the export clears what it used
  const GridView G = grid_view(b);
  const int per = kCellBlk / kCG;
  voronoi_export_kernel<<<std::min((n + per - 1) / per, device_sm_count() * 16), kCellBlk, 0, st>>>(
      g.reps, rep, (const int2*)b.S_pos, b.S_id, G, pass, deg, out_off, out_ids, b.ovf_list, b.ovf_count, b.vor_seed,
      b.vor_seed_n, b.slot_of, n < kHeavyLine ? kHeavySmall : kHeavy);
  voronoi_overflow_export_kernel<<<device_sm_count() * 4, 32 * kOvfWarps, 0, st>>>(
      g.reps, (const int2*)b.S_pos, b.S_id, G, pass, deg, out_off, out_ids, b.ovf_list, b.ovf_count, b.d_status,
      b.vor_seed, b.vor_seed_n, b.slot_of);
  const cudaError_t e = cudaMemsetAsync(b.ovf_count, 0, sizeof(int32_t), st);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace vk
