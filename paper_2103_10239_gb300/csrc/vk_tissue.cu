// vk_tissue.cu -- the Voronoi tissue model (Sec. "Geometric models of dense
// tissue": each particle generates its Voronoi cell, of area A_i and
// perimeter P_i, with the energy of Eq. (vmEnergy)
//   E = sum_i KA (A_i - A0)^2 + KP (P_i - P0)^2;
// Sec. "Voronoi model forces": F_i = -dE/dr_i by the chain rule through the
// Voronoi vertices h, the circumcenters of the Delaunay triangles).
//
// Three passes over one replica, FP64 geometry from exact integer offsets:
//   1. cells: every particle builds its cell with the Voronoi rule's builder
//      (vk_voronoi_fast.cuh, eight lanes each; vk_voronoi.cuh where that one
//      cannot) and stores its edge sites in counter-clockwise order (sorted
//      slot and exact offset), its edges as vectors with their inverse lengths,
//      its area and its perimeter; the edges of all cells are packed (36 bytes
//      each, 6 a cell on average);
//   2. forces, eight lanes per particle: for every vertex h of cell i (edge
//      sites a, b) the three cells i, a, b that share h contribute dE_c/dh; the
//      vertex's place in cells a and b comes from their stored edge lists
//      (found by slot and offset, so periodic images of the same particle stay
//      apart), and dh/dr_i is the Jacobian of the circumcenter in the paper's
//      notation (c, d, beta d, gamma d, z);
//   3. energy: the blocks sum the cells' terms, one block the blocks' sums, in
//      a fixed order.
// The FP64 units are few (about 0.6 Tops/s): recomputing circumcenters, edge
// lengths and quotients at every vertex took 780 FP64 operations per vertex and
// cell; with the stored edges it is about 110.  Measured (GB300, 1M uniform
// particles, ms, recomputed by one thread per cell / stored): cells 13.6 / 3.74,
// forces 11.1 / 2.32, energy 3.1 / 0.03.  Packed rows in place of 32 entries per
// cell: 273 instead of 1185 bytes a particle, and 6.45 / 6.11 ms for all three.
#include "vk_voronoi_fast.cuh"

namespace vk {

namespace {

struct TissueParams {
  double KA, KP, A0, P0;
  double unit;  // length of one grid unit, 2^-F
};

// circumcenter of (0, a, b), FP64
__device__ __forceinline__ double2 circum64(double ax, double ay, double bx, double by) {
  const double D = 2.0 * (ax * by - ay * bx);
  const double a2 = ax * ax + ay * ay, b2 = bx * bx + by * by;
  return make_double2((by * a2 - ay * b2) / D, (ax * b2 - bx * a2) / D);
}

__device__ __forceinline__ double2 circum_off(int2 a, int2 b, double u) {
  return circum64((double)a.x * u, (double)a.y * u, (double)b.x * u, (double)b.y * u);
}

// first entry and edges of a stored cell
__device__ __forceinline__ int64_t row_first(int64_t row) { return row >> kRowShift; }
__device__ __forceinline__ int row_edges(int64_t row) { return (int)(row & ((1 << kRowShift) - 1)); }

// Store edge a of a cell, from the vertex of sites (a - 1, a) to that of (a, a + 1).
__device__ __forceinline__ void put_edge(const TissueScratch& w, int64_t at, int32_t slot, int2 off, double2 h0,
                                         double2 h1, double* area, double* perim) {
  const double2 d = make_double2(h1.x - h0.x, h1.y - h0.y);
  const double len = sqrt(d.x * d.x + d.y * d.y);
  w.nb_slot[at] = slot;
  w.nb_off[at] = off;
  w.edge[at] = d;
  w.inv_len[at] = 1.0 / len;
  *area += 0.5 * (h0.x * h1.y - h1.x * h0.y);
  *perim += len;
}

// the cell of one particle by the general code, one thread
__device__ __noinline__ void tissue_cell_general(const Rep& R, int64_t s, const int2* __restrict__ S_pos,
                                                 const int32_t* __restrict__ S_id, const GridView& G, double unit,
                                                 const TissueScratch& w, int32_t* status, const Seeds& sd) {
  const int2 p = S_pos[s];
  const int32_t pi[3] = {p.x, p.y, 0};
  Poly<kFastCap> P;
  int m = 0;
  double A = 0.0, Pm = 0.0;
  int64_t first = 0;
  if (!voronoi_cell(R, s, pi, S_id[s], S_pos, S_id, G, P, status, sd) || P.m > kTissueCap) {
    set_status(status, kStCapacity);
  } else if (P.nt > 0) {
    set_status(status, kStDegenerate);  // coincident particles: one site, no cell each
  } else if ((first = (int64_t)atomicAdd(w.used, (unsigned long long)P.m)) + P.m > w.cap) {
    set_status(status, kStDegenerate);  // more than 6 N edges: some are of zero length
  } else {
    m = P.m;
    double2 h0 = circum_off(make_int2(P.qx[m - 1], P.qy[m - 1]), make_int2(P.qx[0], P.qy[0]), unit);
    for (int a = 0; a < m; ++a) {
      const int pa = a == 0 ? m - 1 : a - 1, na = a + 1 == m ? 0 : a + 1;
      // an edge of zero length (four cocircular particles): no derivative
      if (vertex_cut_sign(P.qx[pa], P.qy[pa], P.qx[a], P.qy[a], P.qx[na], P.qy[na]) == 0)
        set_status(status, kStDegenerate);
      const double2 h1 = circum_off(make_int2(P.qx[a], P.qy[a]), make_int2(P.qx[na], P.qy[na]), unit);
      // an edge to an image of the particle itself (tiny boxes) is kept with
      // the particle's own slot and the image's offset
      put_edge(w, first + a, P.slot[a] >= 0 ? P.slot[a] : (int32_t)s, make_int2(P.qx[a], P.qy[a]), h0, h1, &A,
               &Pm);
      h0 = h1;
    }
  }
  w.row[s] = m ? first << kRowShift | m : 0;
  w.area[s] = A;
  w.perim[s] = Pm;
}

__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int o = 1; o < kCG; o <<= 1) v += __shfl_xor_sync(kAll, v, o);
  return v;
}
__device__ __forceinline__ double2 shfl2(double2 v, int from) {
  return make_double2(__shfl_sync(kAll, v.x, from), __shfl_sync(kAll, v.y, from));
}

constexpr int kTissueBlk = 128;

// Pass 1: the cell of every particle of the replica, eight lanes each
__global__ void __launch_bounds__(kTissueBlk, 4) tissue_cells_kernel(
    const Rep* __restrict__ reps, int rep, const int2* __restrict__ S_pos, const int32_t* __restrict__ S_id,
    GridView G, double unit, TissueScratch w, int32_t* status, const int32_t* __restrict__ vor_seed,
    const int32_t* __restrict__ vor_seed_n, const int32_t* __restrict__ slot_of) {
  const Rep& R = reps[rep];
  const int lane = (int)(threadIdx.x & 31);
  Cell8 c;
  c.gl = lane & (kCG - 1);
  c.base = lane & ~(kCG - 1);
  constexpr int kPer4 = kTissueBlk / kCG;
#pragma unroll 1
  for (int l0 = blockIdx.x * kPer4 + (int)(threadIdx.x >> 5) * 4; l0 < R.n; l0 += gridDim.x * kPer4) {
    const int li = l0 + lane / kCG;
    const bool on = li < R.n;
    const int64_t s = R.p0 + (on ? li : 0);
    const int2 p = S_pos[s];
    // a Voronoi-rule sim's last neighbors seed the cell (any seeds give the same cell)
    const int64_t gi = R.p0 + S_id[s];
    const Seeds sd = seeds_of(vor_seed, vor_seed ? vor_seed_n[gi] : 0, gi, slot_of);
    c.build(on, R, s, p, S_pos, G, sd, 2 * kHeavy);
    bool ok = on && !c.other;
    // entries for the four cells' edges
    const int mine = ok ? c.m : 0;
    int before = 0, all = 0;
#pragma unroll
    for (int g = 0; g < 32; g += kCG) {
      const int v = __shfl_sync(kAll, mine, g);
      before += g < c.base ? v : 0;
      all += v;
    }
    unsigned long long taken = 0;
    if (lane == 0) taken = atomicAdd(w.used, (unsigned long long)all);
    const int64_t first = (int64_t)__shfl_sync(kAll, taken, 0) + before;
    const bool fits = first + mine <= w.cap;  // if not, some edges are of zero length
    if (ok && !fits) ok = false;
    // an edge of zero length (four cocircular particles): no derivative
    const unsigned positive = c.positive_edges();
    if (on && !c.other && c.gl == 0 && (!fits || positive != (1u << c.m) - 1u)) set_status(status, kStDegenerate);
    // vertex after each of the lane's edges, and the one before
    const bool big = __any_sync(kAll, c.m > 8);
    int2 nq[2];
    c.next_sites(big, nq);
    double2 h[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
    double A = 0.0, Pm = 0.0;
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (ok && c.has(i)) h[i] = circum_off(c.q[i], nq[i], unit);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (i == 1 && !big) break;
      const int a = c.gl + 8 * i, j = a == 0 ? c.m - 1 : a - 1;
      double2 h0 = shfl2(h[0], c.base + (j & 7));
      if (big) {
        const double2 h8 = shfl2(h[1], c.base + (j & 7));
        if (j >= 8) h0 = h8;
      }
      if (ok && c.has(i))
        put_edge(w, first + a, c.slot[i] >= 0 ? c.slot[i] : (int32_t)s, c.q[i], h0, h[i], &A, &Pm);
    }
    A = group_sum(A);
    Pm = group_sum(Pm);
    if (on && c.gl == 0) {
      if (!c.other) {
        w.row[s] = ok ? first << kRowShift | c.m : 0;
        w.area[s] = A;
        w.perim[s] = Pm;
      } else {
        tissue_cell_general(R, s, S_pos, S_id, G, unit, w, status, sd);
      }
    }
    __syncwarp();
  }
}

// dE_c/dh for the vertex h between edges `in` and `out` of cell c: from the
// shoelace area, dA/dh = (1/2)(y_next - y_prev, x_prev - x_next); from the
// perimeter, dP/dh = t_in - t_out with the edges' unit vectors
__device__ __forceinline__ double2 cell_grad(const TissueScratch& w, int64_t in, int64_t out, double gA, double gP) {
  const double2 d0 = w.edge[in], d1 = w.edge[out];
  const double i0 = w.inv_len[in], i1 = w.inv_len[out];
  return make_double2(gA * 0.5 * (d0.y + d1.y) + gP * (d0.x * i0 - d1.x * i1),
                      -gA * 0.5 * (d0.x + d1.x) + gP * (d0.y * i0 - d1.y * i1));
}

// position of the entry (slot, offset) in a stored edge list, or -1
__device__ __forceinline__ int find_entry(const int32_t* __restrict__ sl, const int2* __restrict__ off, int m,
                                          int32_t slot, int2 o) {
  for (int t = 0; t < m; ++t) {
    if (sl[t] != slot) continue;
    const int2 e = off[t];
    if (e.x == o.x && e.y == o.y) return t;
  }
  return -1;
}

// Pass 2: F_i = -sum over the vertices h of cell i of (dh/dr_i)^T (dE_i/dh +
// dE_a/dh + dE_b/dh), eight lanes per particle, one vertex each at a time
__global__ void __launch_bounds__(kTissueBlk) tissue_force_kernel(
    const Rep* __restrict__ reps, int rep, const int32_t* __restrict__ S_id, TissueParams T, TissueScratch w,
    double* __restrict__ force_out, double* __restrict__ area_out, double* __restrict__ perim_out, int32_t* status) {
  // place of particle i in the lists of its edge sites
  __shared__ int8_t place[kTissueBlk / kCG][kTissueCap];
  const Rep& R = reps[rep];
  const double u = T.unit;
  const int lane = (int)(threadIdx.x & 31), gl = lane & (kCG - 1), grp = (int)threadIdx.x / kCG;
  constexpr int kPer4 = kTissueBlk / kCG;
  for (int l0 = blockIdx.x * kPer4 + (int)(threadIdx.x >> 5) * 4; l0 < R.n; l0 += gridDim.x * kPer4) {
    const int li = l0 + lane / kCG;
    const bool on = li < R.n;
    const int64_t s = R.p0 + (on ? li : 0);
    const int32_t id = S_id[s];
    const int64_t own = on ? w.row[s] : 0, row = row_first(own);
    const int m = row_edges(own);
    const double area = w.area[s], perim = w.perim[s];
    if (on && gl == 0 && area_out) area_out[id] = area;
    if (on && gl == 0 && perim_out) perim_out[id] = perim;
    if (!force_out) continue;
    for (int k = gl; k < m; k += kCG) {
      const int64_t wa = w.row[w.nb_slot[row + k]], ra = row_first(wa);
      const int2 d = w.nb_off[row + k];
      place[grp][k] = (int8_t)find_entry(w.nb_slot + ra, w.nb_off + ra, row_edges(wa), (int32_t)s,
                                         make_int2(-d.x, -d.y));
    }
    __syncwarp();
    double Fx = 0.0, Fy = 0.0;
    const double gA = 2.0 * T.KA * (area - T.A0), gP = 2.0 * T.KP * (perim - T.P0);
    bool ok = true;
    for (int k = gl; k < m; k += kCG) {
      const int kn = k + 1 == m ? 0 : k + 1;
      const int32_t sa = w.nb_slot[row + k], sb = w.nb_slot[row + kn];
      const int2 da = w.nb_off[row + k], db = w.nb_off[row + kn];
      const int64_t wa = w.row[sa], wb = w.row[sb], ra = row_first(wa), rb = row_first(wb);
      // cell a: around a the sites run ... b, i ...; cell b: ... i, a ...
      const int ma = row_edges(wa), mb = row_edges(wb), ta = place[grp][k], tb = place[grp][kn];
      const int tp = ta <= 0 ? ma - 1 : ta - 1, tn = tb < 0 || tb + 1 == mb ? 0 : tb + 1;
      ok = ta >= 0 && tb >= 0;
      if (ok) {
        const int2 oa = w.nb_off[ra + tp], ob = w.nb_off[rb + tn];
        ok = w.nb_slot[ra + tp] == sb && oa.x == db.x - da.x && oa.y == db.y - da.y && w.nb_slot[rb + tn] == sa &&
             ob.x == da.x - db.x && ob.y == da.y - db.y;
      }
      if (!ok) break;
      // the vertex h lies between edges k and kn of cell i, tp and ta of cell a, tb and tn of cell b
      double2 g = cell_grad(w, row + k, row + kn, gA, gP);
      const double2 g1 = cell_grad(w, ra + tp, ra + ta, 2.0 * T.KA * (w.area[sa] - T.A0), 2.0 * T.KP * (w.perim[sa] - T.P0));
      const double2 g2 = cell_grad(w, rb + tb, rb + tn, 2.0 * T.KA * (w.area[sb] - T.A0), 2.0 * T.KP * (w.perim[sb] - T.P0));
      g.x += g1.x + g2.x;
      g.y += g1.y + g2.y;
      // dh/dr_i (Sec. "Voronoi model forces"; j = a, k = b): r_ij, r_ik from
      // i, r_jk = r_k - r_j; c, d = 2 c^2, beta d, gamma d, z = beta d r_ij +
      // gamma d r_ik (so h - r_i = z / d), and
      //   dh/dr_i = I + [r_ij (x) d(beta d)/dr_i + r_ik (x) d(gamma d)/dr_i
      //                  - (beta d + gamma d) I - z (x) (1/d) dd/dr_i] / d
      // with the derivatives of beta d, gamma d and d as they follow from
      // their definitions
      const double ijx = da.x * u, ijy = da.y * u, ikx = db.x * u, iky = db.y * u;
      const double jkx = ikx - ijx, jky = iky - ijy;
      const double c = ijx * (-jky) - ijy * (-jkx);  // r_ij x r_kj
      const double ic = 1.0 / c, id2 = 0.5 * ic * ic;  // 1 / d
      const double ij_jk = ijx * jkx + ijy * jky, ik_jk = ikx * jkx + iky * jky;
      const double ij2 = ijx * ijx + ijy * ijy, ik2 = ikx * ikx + iky * iky;
      const double bd = -ik2 * ij_jk, gd = ij2 * ik_jk;
      const double zx = bd * ijx + gd * ikx, zy = bd * ijy + gd * iky;
      const double dbx = 2.0 * ij_jk * ikx + ik2 * jkx, dby = 2.0 * ij_jk * iky + ik2 * jky;
      const double dgx = -2.0 * ik_jk * ijx - ij2 * jkx, dgy = -2.0 * ik_jk * ijy - ij2 * jky;
      const double ddx = 2.0 * ic * jky, ddy = -2.0 * ic * jkx;
      const double J00 = 1.0 + (ijx * dbx + ikx * dgx - (bd + gd) - zx * ddx) * id2;
      const double J01 = (ijx * dby + ikx * dgy - zx * ddy) * id2;
      const double J10 = (ijy * dbx + iky * dgx - zy * ddx) * id2;
      const double J11 = 1.0 + (ijy * dby + iky * dgy - (bd + gd) - zy * ddy) * id2;
      Fx -= g.x * J00 + g.y * J10;
      Fy -= g.x * J01 + g.y * J11;
    }
    __syncwarp();
    // the cells around a vertex do not fit together as three: with exact
    // predicates only where four or more particles are cocircular (a vertex
    // shared by more than three cells), where the energy has no derivative.
    // (m < 3: the cell pass failed, its status is latched)
    const bool bad = (__ballot_sync(kAll, !ok) >> (lane & ~(kCG - 1)) & 255u) != 0;
    Fx = group_sum(Fx);
    Fy = group_sum(Fy);
    if (on && gl == 0) {
      if (bad) set_status(status, kStDegenerate);
      force_out[2 * (int64_t)id] = bad || m < 3 ? 0.0 : Fx;
      force_out[2 * (int64_t)id + 1] = bad || m < 3 ? 0.0 : Fy;
    }
  }
}

// Pass 3: the energy, per block and then over the blocks, each in a fixed order
// (one block over a million cells took 3.1 ms)
constexpr int kEnergyBlk = 256;

__device__ __forceinline__ double block_sum(double e, double* part) {
  part[threadIdx.x] = e;
  __syncthreads();
  for (int h = kEnergyBlk / 2; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) part[threadIdx.x] += part[threadIdx.x + h];
    __syncthreads();
  }
  return part[0];
}

__global__ void __launch_bounds__(kEnergyBlk) tissue_energy_kernel(const Rep* __restrict__ reps, int rep,
                                                                   TissueParams T, const double* __restrict__ area,
                                                                   const double* __restrict__ perim,
                                                                   double* __restrict__ blocks) {
  __shared__ double part[kEnergyBlk];
  const Rep& R = reps[rep];
  double e = 0.0;
  for (int64_t li = blockIdx.x * kEnergyBlk + (int)threadIdx.x; li < R.n; li += (int64_t)gridDim.x * kEnergyBlk) {
    const double dA = area[R.p0 + li] - T.A0, dP = perim[R.p0 + li] - T.P0;
    e += T.KA * dA * dA + T.KP * dP * dP;
  }
  e = block_sum(e, part);
  if (threadIdx.x == 0) blocks[blockIdx.x] = e;
}

__global__ void __launch_bounds__(kEnergyBlk) tissue_energy_total_kernel(const double* __restrict__ blocks, int n,
                                                                         double* __restrict__ energy) {
  __shared__ double part[kEnergyBlk];
  double e = 0.0;
  for (int i = threadIdx.x; i < n; i += kEnergyBlk) e += blocks[i];
  e = block_sum(e, part);
  if (threadIdx.x == 0) *energy = e;
}

GridView tissue_view(const Buffers& b) {
  GridView G;
  G.off = b.offsets;
  G.sub_s = b.sub_s;
  G.sub_base = b.sub_base;
  G.sub_off = b.sub_off;
  return G;
}

}  // namespace

cudaError_t launch_tissue(const Geometry& g, const Buffers& b, int rep, int n, double KA, double KP, double A0,
                          double P0, double unit, TissueScratch w, double* area_out, double* perim_out,
                          double* force_out, double* energy_out, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const TissueParams T{KA, KP, A0, P0, unit};
  const int sms = device_sm_count(), per = kTissueBlk / kCG;
  const cudaError_t e = cudaMemsetAsync(w.used, 0, sizeof(*w.used), st);
  if (e != cudaSuccess) return e;
  tissue_cells_kernel<<<std::min((n + per - 1) / per, sms * 16), kTissueBlk, 0, st>>>(
      g.reps, rep, (const int2*)b.S_pos, b.S_id, tissue_view(b), unit, w, b.d_status, b.vor_seed, b.vor_seed_n,
      b.slot_of);
  if (force_out || area_out || perim_out)
    tissue_force_kernel<<<std::min((n + per - 1) / per, sms * 32), kTissueBlk, 0, st>>>(
        g.reps, rep, b.S_id, T, w, force_out, area_out, perim_out, b.d_status);
  if (energy_out) {
    const int blocks = std::min((n + kEnergyBlk - 1) / kEnergyBlk, kTissueBlocks);
    tissue_energy_kernel<<<blocks, kEnergyBlk, 0, st>>>(g.reps, rep, T, w.area, w.perim, w.blocks);
    tissue_energy_total_kernel<<<1, kEnergyBlk, 0, st>>>(w.blocks, blocks, energy_out);
  }
  return cudaGetLastError();
}

}  // namespace vk
