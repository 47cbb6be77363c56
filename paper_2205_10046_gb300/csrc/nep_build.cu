// Neighbour-list construction, atom reordering, velocity-Verlet drift and reductions.
//
// The paper takes its neighbour lists as given (Appendix B lists NN_i^R, NN_i^A, NL_im^R,
// NL_im^A); here they are built on the GPU from a cell list at every rebuild:
//   bin_atoms      validate, wrap positions into the cell (FP64), cell index, cell counts;
//   sum_cells,
//   scan_cells     exclusive prefix sum of the counts;
//   scatter        atoms into their cells, in any order;
//   reorder        move every per-atom array into cell order, each cell by atom index (the
//                  internal order, deterministic), so a
//                  warp's atoms are spatial neighbours and their neighbour data is shared in
//                  L1; perm keeps the caller's index of each internal atom;
//   commit         cell-local FP32 coordinates, cell origins, reference positions;
//   build_lists    per atom: scan the (2R+1)^3 neighbouring cells (all periodic images when
//                  the cell is thin), keep pairs within r_c + skin, group the radial list by
//                  neighbour type and put the pairs inside r_c before the skin pairs (which
//                  keeps warps convergent in the pair loops); two passes, count then write;
//   build_rev      for every angular pair (i, j, image), the slot of (j, i, -image) in the list
//                  of j, so forces are gathered without atomics (Algorithm 4's "index
//                  manipulations").
// Up to kWideBuildAtoms atoms one cooperative kernel (build_kernel) runs all steps, above they are
// kernels of their own. Every builder returns early unless a rebuild is pending, so the whole sequence sits in the
// captured MD step graph and only works when an atom moved more than skin/2. In the serving
// engine's batch a build that was not forced covers only the structures whose atoms moved that
// far (per-structure flags); the others keep their cells, atom order, lists and x_ref.
#include <cuda_bf16.h>

#include <cooperative_groups.h>

#include <algorithm>

#include "nep_internal.cuh"

namespace nep {

// Grid of the structure that atom i belongs to.
__device__ __forceinline__ const Grid &grid_of(const Batch &B, const Grid &g, int i) {
  return B.grids ? B.grids[B.sid[i]] : g;
}

__device__ __forceinline__ bool rebuild_pending(const BuildStatus *st) {
  return *(volatile const int *)&st->rebuild != 0;
}

// Atom (or internal position) i belongs to a structure that this build leaves as it is: a
// build requested by the serving engine's drift kernel, not forced, and i's structure not
// flagged. Such atoms keep their cell, their place in the order, their lists and x_ref.
__device__ __forceinline__ bool kept_by_build(const Batch &B, const BuildStatus *st, int i) {
  return B.sflag && !*(volatile const int *)&st->full && B.sflag[B.sid[i]] == 0;
}

__global__ void zero_cells_kernel(int ncell, int *count, int *cursor, unsigned long long *part, BuildStatus *st) {
  if (!rebuild_pending(st)) return;
  if (blockIdx.x == 0)  // per-build sums (the maxima are kept over the run)
    for (int k = threadIdx.x; k < 4 * kStatSlots; k += blockDim.x) part[k] = 0ull;
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x) {
    count[c] = 0;
    cursor[c] = 0;
  }
}

// Validates position r and type ti of an atom (flags in st; replaced by 0), wraps r into the cell
// (FP64; only atoms outside it are moved, so a position is not re-rounded by every build) and
// returns its cell. *moved: r or ti changed.
__device__ __forceinline__ int bin_position(const Grid &g, int T, double *r, int *ti, bool *moved, BuildStatus *st) {
  *moved = false;
  if (*ti < 0 || *ti >= T) {
    atomicOr(&st->bad_input, 1);
    *ti = 0;
    *moved = true;
  }
  bool inside = true;
  if (!isfinite(r[0]) || !isfinite(r[1]) || !isfinite(r[2])) {
    atomicOr(&st->bad_input, 2);
    r[0] = r[1] = r[2] = 0.0;
    inside = false;  // overwrite the position
  }
  double s[3];
  int c[3];
  for (int b = 0; b < 3; ++b) {
    s[b] = r[0] * g.Hinv[0][b] + r[1] * g.Hinv[1][b] + r[2] * g.Hinv[2][b];
    const double f = floor(s[b]);
    inside = inside && f == 0.0;
    s[b] -= f;
    const int cb = (int)(s[b] * g.nc[b]);
    c[b] = cb < 0 ? 0 : (cb >= g.nc[b] ? g.nc[b] - 1 : cb);
  }
  if (!inside) {
    for (int b = 0; b < 3; ++b) r[b] = s[0] * g.H[0][b] + s[1] * g.H[1][b] + s[2] * g.H[2][b];
    *moved = true;
  }
  return g.cell_off + (c[0] * g.nc[1] + c[1]) * g.nc[2] + c[2];
}

// Writes the coordinates of internal atom p derived from its position r and cell gid:
// reference position, cell origin, cell-local and cell-frame FP32 coordinates.
__device__ __forceinline__ void commit_position(const Grid &g, int gid, int tag, const double *r, size_t p,
                                                const AtomState &a) {
  const int id = gid - g.cell_off;
  const int c0 = id / (g.nc[1] * g.nc[2]), c1 = (id / g.nc[2]) % g.nc[1], c2 = id % g.nc[2];
  double o[3];
  for (int b = 0; b < 3; ++b) {
    o[b] = c0 * g.Hc[0][b] + c1 * g.Hc[1][b] + c2 * g.Hc[2][b];
    a.x[3 * p + b] = r[b];
    a.x_ref[3 * p + b] = r[b];
    a.origin[3 * p + b] = o[b];
  }
  a.pos4[p] = make_float4((float)(r[0] - o[0]), (float)(r[1] - o[1]), (float)(r[2] - o[2]), __int_as_float(tag));
  a.posA[p] = make_float4((float)r[0], (float)r[1], (float)r[2], __int_as_float(tag));
}

__device__ __forceinline__ void arm_status(BuildStatus *st) {
  st->overflow = 0;
  st->max_r = 0;
  st->max_a = 0;
  st->rev_missing = 0;
  st->bad_input = 0;
  st->tc_timeout = 0;
  st->rebuild = 1;
  st->full = 1;
}

// Shift vector of image code `code` (zero for codes outside the range); the explicitly rounded
// FP64 operations give the same values on every path that forms the table.
__device__ __forceinline__ float4 shift_vector(const Grid &g, int code) {
  const int om = (1 << g.obits) - 1;
  const int o[3] = {(code & om) - g.R[0], ((code >> g.obits) & om) - g.R[1], ((code >> (2 * g.obits)) & om) - g.R[2]};
  if (abs(o[0]) > g.R[0] || abs(o[1]) > g.R[1] || abs(o[2]) > g.R[2]) return make_float4(0.f, 0.f, 0.f, 0.f);
  double d[3];
  for (int b = 0; b < 3; ++b)
    d[b] = __dadd_rn(__dadd_rn(__dmul_rn(o[0], g.Hc[0][b]), __dmul_rn(o[1], g.Hc[1][b])), __dmul_rn(o[2], g.Hc[2][b]));
  return make_float4((float)d[0], (float)d[1], (float)d[2], 0.f);
}

// Takes a structure over from the caller: positions, types, caller order, the shift table of a
// single structure (src.dtab), and a forced build requested.
__global__ void load_kernel(int N, const LoadSrc src, AtomState a, const Grid g, BuildStatus *st) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) arm_status(st);
  if (src.dtab)
    for (int c = i; c < g.ncode; c += gridDim.x * blockDim.x) src.dtab[c] = shift_vector(g, c);
  for (int k = i; k < 3 * N; k += gridDim.x * blockDim.x) a.x[k] = src.pos[k];
  for (int k = i; k < N; k += gridDim.x * blockDim.x) {
    a.types[k] = src.types[k];
    a.perm[k] = k;
  }
}

__global__ void bin_atoms_kernel(int N, int T, AtomState a, int *count, const Grid g0, const Batch B,
                                 BuildStatus *st) {
  if (!rebuild_pending(st)) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  if (kept_by_build(B, st, i)) {  // counted in its old cell: its structure's order stays
    atomicAdd(count + a.cell_of[i], 1);
    return;
  }
  double *x = a.x + 3 * (size_t)i;
  double r[3] = {x[0], x[1], x[2]};
  int ti = a.types[i];
  bool moved;
  const int id = bin_position(grid_of(B, g0, i), T, r, &ti, &moved, st);
  if (moved) {
    a.types[i] = ti;
    for (int b = 0; b < 3; ++b) x[b] = r[b];
  }
  a.cell_of[i] = id;
  atomicAdd(count + id, 1);
}

// Sum of v over a block of kScanBlock threads, on every thread.
constexpr int kScanBlock = 256;
__device__ __forceinline__ int block_sum(int v, int *wsum) {
  v = __reduce_add_sync(0xffffffffu, v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
  __syncthreads();
  v = 0;
#pragma unroll
  for (int w = 0; w < kScanBlock / 32; ++w) v += wsum[w];
  return v;
}

// Exclusive prefix sum of count[c0..c1) from `before` on, by a block of kScanBlock threads.
__device__ __forceinline__ void block_scan(const int *count, int *start, int c0, int c1, int before, int *wsum,
                                           int *carry) {
  const int tid = threadIdx.x;
  for (int cb = c0; cb < c1; cb += kScanBlock) {
    const int c = cb + tid, v = c < c1 ? count[c] : 0;
    int x = v;  // inclusive scan over the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if ((tid & 31) >= o) x += y;
    }
    __syncthreads();
    if ((tid & 31) == 31) wsum[tid >> 5] = x;
    __syncthreads();
    int off = before;
    for (int w = 0; w < (tid >> 5); ++w) off += wsum[w];
    if (c < c1) start[c] = off + x - v;
    if (tid == kScanBlock - 1) *carry = off + x;
    __syncthreads();
    before = *carry;
  }
}

// Exclusive prefix sum of the cell counts: block b sums the b-th part of the cells (sums), then
// scans it from the sum of the parts before (scan). One block for all cells took 42 us in a batch of
// 4096 structures and 31 us for 512,000 atoms, the two kernels 9 us, for 8,000,000 atoms 15.
__global__ void __launch_bounds__(kScanBlock)
    sum_cells_kernel(int ncell, const int *count, unsigned *sums, const BuildStatus *st) {
  if (!rebuild_pending(st)) return;
  __shared__ int wsum[kScanBlock / 32];
  const int part = (ncell + gridDim.x - 1) / gridDim.x, c0 = blockIdx.x * part, c1 = min(ncell, c0 + part);
  int v = 0;
  for (int c = c0 + threadIdx.x; c < c1; c += kScanBlock) v += count[c];
  v = block_sum(v, wsum);
  if (threadIdx.x == 0) sums[blockIdx.x] = (unsigned)v;
}

__global__ void __launch_bounds__(kScanBlock)
    scan_cells_kernel(int N, int ncell, const int *count, int *start, const unsigned *sums, const BuildStatus *st) {
  if (!rebuild_pending(st)) return;
  __shared__ int wsum[kScanBlock / 32], carry;
  const int part = (ncell + gridDim.x - 1) / gridDim.x, c0 = blockIdx.x * part, c1 = min(ncell, c0 + part);
  int before = 0;
  for (int b = threadIdx.x; b < (int)blockIdx.x; b += kScanBlock) before += (int)sums[b];
  before = block_sum(before, wsum);
  block_scan(count, start, c0, c1, before, wsum, &carry);
  if (blockIdx.x == 0 && threadIdx.x == 0) start[ncell] = N;
}

__global__ void scatter_atoms_kernel(int N, const int *cell_of, const int *start, int *cursor, int *cell_atoms,
                                     const Batch B, const BuildStatus *st) {
  if (!rebuild_pending(st)) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N || kept_by_build(B, st, i)) return;
  const int c = cell_of[i];
  cell_atoms[start[c] + atomicAdd(cursor + c, 1)] = i;
}

// Every cell's atoms in the order of their index, and their data moved to those places (into
// the scratch arrays). Thread p takes entry p of the unsorted cell list: its place inside the
// cell is the number of smaller entries of the cell (a cell holds ~10 atoms, whose entries the
// neighbouring threads read too), so no kernel sorts the cells first (thread-per-cell insertion
// sort in global memory: 137 us of the 4.65 ms of a 4096-structure batch, 20 us of a 216-atom
// build). `move`: bit 0 the velocities, bit 1 the forces (unneeded where the caller keeps none
// or computes new ones before reading them).
__global__ void reorder_gather_kernel(int N, const int *start, const int *cell_atoms, AtomState a, int move,
                                      const Batch B, const BuildStatus *st) {
  if (!rebuild_pending(st)) return;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N || kept_by_build(B, st, p)) return;
  const int o = cell_atoms[p];
  const int c = a.cell_of[o];
  const int b0 = start[c], b1 = start[c + 1];
  int rank = 0;
  for (int q = b0; q < b1; ++q) rank += __ldg(cell_atoms + q) < o ? 1 : 0;
  const size_t d = 3 * (size_t)(b0 + rank), f = 3 * (size_t)o;
#pragma unroll
  for (int b = 0; b < 3; ++b) a.x2[d + b] = a.x[f + b];
  if (move & 1)
#pragma unroll
    for (int b = 0; b < 3; ++b) a.v2[d + b] = a.v[f + b];
  if (move & 2)
#pragma unroll
    for (int b = 0; b < 3; ++b) a.F2[d + b] = a.F[f + b];
  a.types2[b0 + rank] = a.types[o];
  a.perm2[b0 + rank] = a.perm[o];
  a.cell2[b0 + rank] = c;
}

// Copy the reordered data back and derive the cell-local coordinates.
__global__ void reorder_commit_kernel(int N, AtomState a, int move, const Grid g0, const Batch B,
                                      const BuildStatus *st) {
  if (!rebuild_pending(st)) return;
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= N || kept_by_build(B, st, p)) return;
  // cells are numbered structure by structure, so atom p stays inside its structure's range
  const int gid = a.cell2[p];
  double r[3];
  for (int b = 0; b < 3; ++b) {
    r[b] = a.x2[3 * (size_t)p + b];
    if (move & 1) a.v[3 * (size_t)p + b] = a.v2[3 * (size_t)p + b];
    if (move & 2) a.F[3 * (size_t)p + b] = a.F2[3 * (size_t)p + b];
  }
  const int t = a.types2[p];
  a.types[p] = t;
  a.perm[p] = a.perm2[p];
  a.cell_of[p] = gid;
  commit_position(grid_of(B, g0, p), gid, t | ((B.grids ? B.sid[p] : 0) << 8), r, p, a);
}

// floor(x / n) and the remainder, for n >= 1 and x > -n * 8
__device__ __forceinline__ int floor_div(int x, int n) { return (x + 8 * n) / n - 8; }

// List statistics of one build: summed over the warp, then added to one of kStatSlots partial
// sums by block (every warp updating the same words serialises in the L2 atomic unit);
// finish_build_kernel adds the partial sums up. nr, nA: list lengths; inr, ina: the part inside
// the cutoffs. Called by whole warps.
__device__ __forceinline__ void add_list_stats(int nr, int nA, int inr, int ina, unsigned long long *part,
                                               BuildStatus *st) {
  constexpr unsigned kAll = 0xffffffffu;
  const int mr = __reduce_max_sync(kAll, nr), ma = __reduce_max_sync(kAll, nA);
  const unsigned v[4] = {__reduce_add_sync(kAll, (unsigned)nr), __reduce_add_sync(kAll, (unsigned)nA),
                         __reduce_add_sync(kAll, (unsigned)inr), __reduce_add_sync(kAll, (unsigned)ina)};
  if ((threadIdx.x & 31) == 0) {
    if (mr > *(volatile int *)&st->max_r) atomicMax(&st->max_r, mr);
    if (ma > *(volatile int *)&st->max_a) atomicMax(&st->max_a, ma);
    unsigned long long *p = part + 4 * (blockIdx.x % kStatSlots);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (v[k]) atomicAdd(p + k, (unsigned long long)v[k]);
  }
}

// Visit every neighbour candidate (j, image) of atom i: f(j, entry, r2, type_j). Atoms are in
// cell order, so the atoms of cell c are j in [start[c], start[c+1]). For each (x, y) column of
// neighbouring cells the z cells are walked as runs that share one periodic image, so the
// shift S is formed once per run and the distance comes from the FP32 positions in the cell
// frame: d = (r_j - r_i) + S, exactly antisymmetric like pair_vector. The image code of an
// entry is the cell offset (ox, oy, oz), as the force kernels' shift tables expect.
//
// Cells that cannot hold a pair are skipped: along axis a, atom i sits at the fraction u_a of
// its cell's width, so every point of the cell at offset o >= 1 lies (o - u_a) cell
// thicknesses away across the lattice planes, and of the cell at o <= -1, (u_a - o - 1); a
// cell is visited only if that gap stays below reach_a = (r_c^R + skin + margin) / thickness.
// The skipped candidates would all fail the distance test, so the lists (and their order)
// are those of the full (2R+1)^3 scan. pl: atom i's cell-local coordinates (pos4).
template <class F>
__device__ __forceinline__ void for_candidates(int i, const float4 &pi, const float4 &pl, int gid, const Grid &g,
                                               const int *start, const float4 *posA, F &&f) {
  const int id = gid - g.cell_off;
  const int cx = id / (g.nc[1] * g.nc[2]);
  const int cy = (id / g.nc[2]) % g.nc[1];
  const int cz = id % g.nc[2];
  int lo[3], hi[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float s = pl.x * g.Hinvf[0][a] + pl.y * g.Hinvf[1][a] + pl.z * g.Hinvf[2][a];
    const float u = fminf(fmaxf(s * (float)g.nc[a], 0.f), 1.f);
    hi[a] = min(g.R[a], (int)ceilf(u + g.reach[a]) - 1);
    lo[a] = max(-g.R[a], 1 - (int)ceilf(1.f - u + g.reach[a]));
  }
  for (int ox = lo[0]; ox <= hi[0]; ++ox) {
    const int kx = floor_div(cx + ox, g.nc[0]);
    const int xm = cx + ox - kx * g.nc[0];
    for (int oy = lo[1]; oy <= hi[1]; ++oy) {
      const int ky = floor_div(cy + oy, g.nc[1]);
      const int ym = cy + oy - ky * g.nc[1];
      const int col = g.cell_off + (xm * g.nc[1] + ym) * g.nc[2];
      const float sx = __fadd_rn(__fmul_rn((float)kx, g.Hf[0][0]), __fmul_rn((float)ky, g.Hf[1][0]));
      const float sy = __fadd_rn(__fmul_rn((float)kx, g.Hf[0][1]), __fmul_rn((float)ky, g.Hf[1][1]));
      const float sz = __fadd_rn(__fmul_rn((float)kx, g.Hf[0][2]), __fmul_rn((float)ky, g.Hf[1][2]));
      const unsigned code_xy = (unsigned)(ox + g.R[0]) | ((unsigned)(oy + g.R[1]) << g.obits);
      int z = cz + lo[2];
      while (z <= cz + hi[2]) {
        const int kz = floor_div(z, g.nc[2]);
        const int zm = z - kz * g.nc[2];
        const int run = min(cz + hi[2] - z, g.nc[2] - 1 - zm) + 1;  // cells of this image
        const float4 S = make_float4(__fadd_rn(sx, __fmul_rn((float)kz, g.Hf[2][0])),
                                     __fadd_rn(sy, __fmul_rn((float)kz, g.Hf[2][1])),
                                     __fadd_rn(sz, __fmul_rn((float)kz, g.Hf[2][2])), 0.f);
        for (int c = 0; c < run; ++c) {
          const int oz = z + c - cz;
          const unsigned code = code_xy | ((unsigned)(oz + g.R[2]) << (2 * g.obits));
          const bool self_image = (ox == 0 && oy == 0 && oz == 0);
          const int cell = col + zm + c;
          const int pe = start[cell + 1];
          for (int j = start[cell]; j < pe; ++j) {
            if (self_image && j == i) continue;
            const float4 pj = posA[j];
            f(j, (unsigned)j | (code << g.jbits), norm2(pair_vector(pi, pj, S)), type_of(pj));
          }
        }
        z += run;
      }
    }
  }
}

// Thread-per-atom form of the list build, for many atoms (the rule is in launch_rebuild). Two
// passes over the candidates: count, then write. The radial list is grouped by
// neighbour type; inside every group (and in the angular list) the pairs already inside
// r_c come before the skin pairs, so the warps of the pair loops stay convergent.
// count_only: record only the length statistics (used to size the lists). TT: the number of
// atom types (compile time, so the per-type counters of a candidate cost TT compares).
template <int TT>
__global__ void build_lists_kernel(int N, const float4 *posA, const float4 *pos4, const int *cell_of, const int *start,
                                   const Grid g0, const Batch B, float rlR2, float rlA2, float rcR2, float rcA2,
                                   ListBufs L, int count_only, BuildStatus *st) {
  if (!rebuild_pending(st)) return;
  const int i0 = blockIdx.x * blockDim.x + threadIdx.x;
  // lanes past the last atom (and atoms of structures this build keeps) stay until the
  // warp-level statistics below
  const bool active = i0 < N && !kept_by_build(B, st, i0);
  const int i = active ? i0 : 0;  // a valid index for the idle lanes (N >= 1)
  const Grid &g = grid_of(B, g0, i);
  const float4 pi = posA[i];
  const float4 pl = pos4[i];
  const int id = cell_of[i];
  // per-type counters stay in registers: every update is unrolled over the types
  int cr0[TT], cr1[TT];
#pragma unroll
  for (int t = 0; t < TT; ++t) cr0[t] = cr1[t] = 0;
  int ca0 = 0, ca1 = 0;
  // with a staging area the accepted candidates are kept in visiting order together with
  // their group (type, inside r_c or skin, angular or not), so the lists are written from
  // them instead of a second candidate scan
  const bool staged = !count_only && L.stage_e;
  int n_seen = 0;
  if (active && staged) {
    // the scan only stages the accepted candidates (angular pairs are a subset of the radial
    // ones, r_c^A <= r_c^R); their groups are counted afterwards from the staged bytes
    unsigned *se = L.stage_e + i;
    unsigned char *sg = L.stage_g + i;
    for_candidates(i, pi, pl, id, g, start, posA, [&](int, unsigned ent, float r2, int tj) {
      if (r2 < rlR2) {
        if (n_seen < L.cap_r) {
          const int ang = r2 < rlA2 ? (r2 < rcA2 ? 1 : 2) : 0;
          *se = ent;
          *sg = (unsigned char)(tj | (r2 < rcR2 ? 0 : 8) | (ang << 4));
          se += N;
          sg += N;
        }
        ++n_seen;
      }
    });
    const int ns = n_seen < L.cap_r ? n_seen : L.cap_r;
    for (int m = 0; m < ns; ++m) {
      const unsigned gb = L.stage_g[(size_t)m * N + i];
      const int tj = (int)(gb & 7u);
      const bool core = (gb & 8u) == 0;
#pragma unroll
      for (int t = 0; t < TT; ++t) {
        cr0[t] += (tj == t && core) ? 1 : 0;
        cr1[t] += (tj == t && !core) ? 1 : 0;
      }
      const unsigned ang = gb >> 4;
      ca0 += ang == 1u ? 1 : 0;
      ca1 += ang == 2u ? 1 : 0;
    }
    // past the staging capacity the groups are unknown: the build overflows and is redone
    // with lists sized from these counts (the unstaged pairs counted as skin pairs of type 0,
    // and as angular ones, an upper bound)
    cr1[0] += n_seen - ns;
    ca1 += n_seen - ns;
  } else if (active) {
    for_candidates(i, pi, pl, id, g, start, posA, [&](int, unsigned ent, float r2, int tj) {
      if (r2 < rlR2) {
        const bool core = r2 < rcR2;
#pragma unroll
        for (int t = 0; t < TT; ++t) {
          cr0[t] += (tj == t && core) ? 1 : 0;
          cr1[t] += (tj == t && !core) ? 1 : 0;
        }
        ++n_seen;
      }
      if (r2 < rlA2) {
        if (r2 < rcA2) ++ca0;
        else ++ca1;
      }
    });
  }
  int nr = 0, inr = 0;
#pragma unroll
  for (int t = 0; t < TT; ++t) {
    nr += cr0[t] + cr1[t];
    inr += cr0[t];
  }
  const int nA = ca0 + ca1;
  add_list_stats(nr, nA, inr, ca0, L.part, st);
  if (count_only || !active) return;
  if (nr > L.cap_r || nA > L.cap_a) {  // leave the lists empty; the host grows them and rebuilds
    atomicOr(&st->overflow, 1);
    for (int t = 0; t < TT; ++t) L.nn_r[t * N + i] = 0;
    L.nn_a[i] = 0;
    return;
  }
  int cur0[TT], cur1[TT];
  int off = 0;
#pragma unroll
  for (int t = 0; t < TT; ++t) {
    cur0[t] = off;
    cur1[t] = off + cr0[t];
    off += cr0[t] + cr1[t];
    L.nn_r[t * N + i] = cr0[t] + cr1[t];
  }
  int ka0 = 0, ka1 = ca0;
  if (staged) {
    for (int m = 0; m < nr; ++m) {
      const unsigned ent = L.stage_e[(size_t)m * N + i];
      const unsigned gb = L.stage_g[(size_t)m * N + i];
      const int tj = (int)(gb & 7u);
      const bool core = (gb & 8u) == 0;
      int slot = 0;
#pragma unroll
      for (int t = 0; t < TT; ++t) {
        if (tj == t) {
          slot = core ? cur0[t] : cur1[t];
          cur0[t] += core ? 1 : 0;
          cur1[t] += core ? 0 : 1;
        }
      }
      L.nl_r[(size_t)slot * N + i] = ent;
      const unsigned ang = gb >> 4;
      if (ang) L.nl_a[(size_t)(ang == 1u ? ka0++ : ka1++) * N + i] = ent;
    }
    L.nn_a[i] = nA;
    return;
  }
  for_candidates(i, pi, pl, id, g, start, posA, [&](int, unsigned ent, float r2, int tj) {
    if (r2 < rlR2) {
      const bool core = r2 < rcR2;
      int slot = 0;
#pragma unroll
      for (int t = 0; t < TT; ++t) {
        if (tj == t) {
          slot = core ? cur0[t] : cur1[t];
          cur0[t] += core ? 1 : 0;
          cur1[t] += core ? 0 : 1;
        }
      }
      L.nl_r[(size_t)slot * N + i] = ent;
    }
    if (r2 < rlA2) L.nl_a[(size_t)(r2 < rcA2 ? ka0++ : ka1++) * N + i] = ent;
  });
  L.nn_a[i] = nA;
}

// Warp-per-atom form of the list build, for few atoms: the same lists in the same order.
//
// Scan. Atoms are in cell order, and the z index of a cell runs fastest: the candidates in one
// (x, y) column of neighbouring cells that share a periodic image are one contiguous range of
// atoms. The lanes prepare the ranges side by side (first and last atom, shift vector S, image
// code), then the warp walks them in order, 32 candidates at a time (one coalesced load), and
// the accepted candidates are staged in shared memory at the places a ballot gives (with the
// image index kz in the place of the cell offset oz, which needs the candidate's cell). The
// distance and the pruned cells are those of for_candidates.
//
// Lists. Then the warp takes the staged entries 32 at a time: class counts, then places.
// COUNT: only the list lengths (used to size the lists).
//
// What bounds it: latency (start offsets, then positions, then the class ballots): a few atoms
// occupy few warps. 216 Si atoms (skin 1 A): 10 us against 118 us of the thread form; 4999
// atoms of a three-species cell: 17 us.
// List of atom i by a whole warp; se: cap_r entries of shared memory of the warp. The positions
// and cells were written by other blocks of the running kernel: no read-only (ld.global.nc) loads.
template <int TT, bool COUNT>
__device__ __forceinline__ void list_of_atom(int i, int N, const float4 *posA, const float4 *pos4, const int *cell_of,
                                             const int *start, const Grid &g, float rlR2, float rlA2, float rcR2,
                                             float rcA2, const ListBufs &L, uint2 *se, BuildStatus *st) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const int cap = COUNT ? 0 : L.cap_r;
  const int nc1 = g.nc[1], nc2 = g.nc[2];
  const int id = cell_of[i] - g.cell_off;
  const int cx = id / (nc1 * nc2), cy = (id / nc2) % nc1, cz = id % nc2;
  const float4 pi = posA[i], pl = pos4[i];
  int lo[3], hi[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float s = pl.x * g.Hinvf[0][a] + pl.y * g.Hinvf[1][a] + pl.z * g.Hinvf[2][a];
    const float u = fminf(fmaxf(s * (float)g.nc[a], 0.f), 1.f);
    hi[a] = min(g.R[a], (int)ceilf(u + g.reach[a]) - 1);
    lo[a] = max(-g.R[a], 1 - (int)ceilf(1.f - u + g.reach[a]));
  }
  // ranges (ox, oy, kz) in visiting order; kz numbers the images of the column's cells
  const int ny = hi[1] - lo[1] + 1;
  const int kz0 = floor_div(cz + lo[2], nc2), nk = floor_div(cz + hi[2], nc2) - kz0 + 1;
  const int nseg = (hi[0] - lo[0] + 1) * ny * nk;
  const int zsh = g.jbits + 2 * g.obits;  // the z field of an entry's image code
  int nr = 0, nA = 0;
  for (int s0 = 0; s0 < nseg; s0 += 32) {
    int jb = 0, je = 0;
    bool home = false;
    unsigned code = 0u;
    float Sx = 0.f, Sy = 0.f, Sz = 0.f;
    const int sg = s0 + lane;
    if (sg < nseg) {
      const int cxy = sg / nk, kz = kz0 + (sg - cxy * nk);
      const int oxi = cxy / ny;
      const int ox = lo[0] + oxi, oy = lo[1] + (cxy - oxi * ny);
      const int kx = floor_div(cx + ox, g.nc[0]), ky = floor_div(cy + oy, nc1);
      const int xm = cx + ox - kx * g.nc[0], ym = cy + oy - ky * nc1;
      const int z0 = max(cz + lo[2], kz * nc2), z1 = min(cz + hi[2], kz * nc2 + nc2 - 1);
      const int c0 = g.cell_off + (xm * nc1 + ym) * nc2 + (z0 - kz * nc2);
      jb = start[c0];
      je = start[c0 + (z1 - z0) + 1];
      code = ((unsigned)(ox + g.R[0]) | ((unsigned)(oy + g.R[1]) << g.obits)) << g.jbits |
             (unsigned)(kz + g.R[2]) << zsh;
      home = (kx | ky | kz) == 0;
      Sx = __fadd_rn(__fadd_rn(__fmul_rn((float)kx, g.Hf[0][0]), __fmul_rn((float)ky, g.Hf[1][0])),
                     __fmul_rn((float)kz, g.Hf[2][0]));
      Sy = __fadd_rn(__fadd_rn(__fmul_rn((float)kx, g.Hf[0][1]), __fmul_rn((float)ky, g.Hf[1][1])),
                     __fmul_rn((float)kz, g.Hf[2][1]));
      Sz = __fadd_rn(__fadd_rn(__fmul_rn((float)kx, g.Hf[0][2]), __fmul_rn((float)ky, g.Hf[1][2])),
                     __fmul_rn((float)kz, g.Hf[2][2]));
    }
    const unsigned mhome = __ballot_sync(kAll, home);
    const int ns = min(32, nseg - s0);
    for (int t = 0; t < ns; ++t) {
      const int b0 = __shfl_sync(kAll, jb, t), e0 = __shfl_sync(kAll, je, t);
      const float4 S = make_float4(__shfl_sync(kAll, Sx, t), __shfl_sync(kAll, Sy, t), __shfl_sync(kAll, Sz, t), 0.f);
      const unsigned ct = __shfl_sync(kAll, code, t);
      const int self = (mhome >> t) & 1 ? i : -1;  // an atom is no neighbour of itself (home image)
      for (int j0 = b0; j0 < e0; j0 += 32) {
        const int j = j0 + lane;
        bool ok = false;
        float r2 = 0.f;
        if (j < e0) {
          r2 = norm2(pair_vector(pi, posA[j], S));
          ok = r2 < rlR2 && j != self;
        }
        const unsigned m = __ballot_sync(kAll, ok);
        if constexpr (COUNT) {
          nA += __popc(__ballot_sync(kAll, ok && r2 < rlA2));
        } else {
          const int w = nr + __popc(m & lt);
          if (ok && w < cap) se[w] = make_uint2((unsigned)j | ct, __float_as_uint(r2));
        }
        nr += __popc(m);
      }
    }
  }
  int n_in = 0, n_ain = 0;
  if constexpr (!COUNT) {
    __syncwarp();
    const int nst = min(nr, cap);
    const unsigned om = (1u << g.obits) - 1u;
    // final entries and classes: 2 t for neighbours of type t inside r_c, 2 t + 1 for its skin
    // pairs; bits 4 and 5: angular pairs (inside r_c, skin)
    int c0[2 * TT];
#pragma unroll
    for (int c = 0; c < 2 * TT; ++c) c0[c] = 0;
    int nskA = 0;
    for (int m0 = 0; m0 < nst; m0 += 32) {
      const int m = m0 + lane;
      int cls = -1, ang = 0;
      if (m < nst) {
        const uint2 v = se[m];
        const unsigned j = v.x & g.jmask;
        const float r2 = __uint_as_float(v.y);
        const int kz = (int)((v.x >> zsh) & om) - g.R[2];
        const int oz = (cell_of[j] - g.cell_off) % nc2 + kz * nc2 - cz;
        cls = 2 * type_of(posA[j]) + (r2 < rcR2 ? 0 : 1);
        ang = r2 < rlA2 ? (r2 < rcA2 ? 1 : 2) : 0;
        se[m] = make_uint2((v.x & ~(om << zsh)) | ((unsigned)(oz + g.R[2]) << zsh), (unsigned)(cls | (ang << 4)));
      }
#pragma unroll
      for (int c = 0; c < 2 * TT; ++c) c0[c] += __popc(__ballot_sync(kAll, cls == c));
      n_ain += __popc(__ballot_sync(kAll, ang == 1));
      nskA += __popc(__ballot_sync(kAll, ang == 2));
    }
    nA = n_ain + nskA + (nr - nst);  // unstaged pairs counted as angular ones: an upper bound
    // an overflow leaves the lists empty; the host grows them and rebuilds
    const bool over = nr > cap || nA > L.cap_a;
    int off = 0;
#pragma unroll
    for (int t = 0; t < TT; ++t) {
      const int n0 = c0[2 * t], n1 = c0[2 * t + 1];
      n_in += n0;
      c0[2 * t] = off;
      c0[2 * t + 1] = off + n0;
      off += n0 + n1;
      if (lane == 0) L.nn_r[(size_t)t * N + i] = over ? 0 : n0 + n1;
    }
    if (lane == 0) {
      L.nn_a[i] = over ? 0 : nA;
      if (over) atomicOr(&st->overflow, 1);
    }
    if (!over) {
      int ka0 = 0, ka1 = n_ain;
      for (int m0 = 0; m0 < nst; m0 += 32) {
        const int m = m0 + lane;
        const uint2 v = m < nst ? se[m] : make_uint2(0u, 0u);  // this lane's own entry of the pass above
        const int cls = m < nst ? (int)(v.y & 15u) : -1, ang = (int)(v.y >> 4);
        int slot = 0;
#pragma unroll
        for (int c = 0; c < 2 * TT; ++c) {
          const unsigned mk = __ballot_sync(kAll, cls == c);
          if (cls == c) slot = c0[c] + __popc(mk & lt);
          c0[c] += __popc(mk);
        }
        const unsigned a1 = __ballot_sync(kAll, ang == 1), a2 = __ballot_sync(kAll, ang == 2);
        if (cls >= 0) L.nl_r[(size_t)slot * N + i] = v.x;
        if (ang) L.nl_a[(size_t)(ang == 1 ? ka0 + __popc(a1 & lt) : ka1 + __popc(a2 & lt)) * N + i] = v.x;
        ka0 += __popc(a1);
        ka1 += __popc(a2);
      }
    }
  }
  const bool l0 = lane == 0;
  add_list_stats(l0 ? nr : 0, l0 ? nA : 0, l0 ? n_in : 0, l0 ? n_ain : 0, L.part, st);
}

// Slot of the reverse pair of every angular pair. A block takes 32 consecutive atoms with 8
// threads each (entries m, m + 8, ...), so that the searches of an atom's pairs run side by
// side and every search keeps four list entries in flight (a thread per atom searched its
// pairs one after the other: 50 us for 216 atoms, 253 us for a 4096-structure batch; now 10 and
// 222 us).
__device__ __forceinline__ void reverse_pairs(int i, int first, int N, const ListBufs &L, const Grid &g,
                                              BuildStatus *st) {
  const unsigned om = (1u << g.obits) - 1u;
  const int na = L.nn_a[i];
  for (int m = first; m < na; m += 8) {
    const size_t slot = (size_t)m * N + i;
    const unsigned e = L.nl_a[slot];
    const int j = e & g.jmask;
    const unsigned code = e >> g.jbits;
    const unsigned cx = code & om, cy = (code >> g.obits) & om, cz = (code >> (2 * g.obits)) & om;
    const unsigned rc = (2u * g.R[0] - cx) | ((2u * g.R[1] - cy) << g.obits) | ((2u * g.R[2] - cz) << (2 * g.obits));
    const unsigned target = (unsigned)i | (rc << g.jbits);
    const int nj = L.nn_a[j];
    const unsigned *col = L.nl_a + j;
    int found = -1;
    for (int q = 0; q < nj && found < 0; q += 4) {
      unsigned v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = q + k < nj ? col[(size_t)(q + k) * N] : ~target;
#pragma unroll
      for (int k = 3; k >= 0; --k)
        if (v[k] == target) found = q + k;
    }
    if (found < 0) {
      atomicAdd(&st->rev_missing, 1);
      L.rev_a[slot] = (int)slot;  // a finite entry; the status reports the error
    } else {
      L.rev_a[slot] = (int)((size_t)found * N + j);
    }
  }
}

__global__ void __launch_bounds__(256) build_rev_kernel(int N, const ListBufs L, const Grid g0, const Batch B,
                                                        BuildStatus *st) {
  if (!rebuild_pending(st)) return;
  const int i = blockIdx.x * 32 + (threadIdx.x & 31);
  if (i >= N || kept_by_build(B, st, i)) return;
  reverse_pairs(i, threadIdx.x >> 5, N, L, grid_of(B, g0, i), st);
}

// The pending build is done, and the per-structure requests (sflag) are served; its list
// statistics are summed. One block of 256 threads.
__device__ __forceinline__ void finish_build(int n_struct, int *sflag, const unsigned long long *part,
                                             BuildStatus *st) {
  for (int s = threadIdx.x; s < n_struct; s += blockDim.x) sflag[s] = 0;
  static_assert(4 * kStatSlots == 256, "one partial sum per thread");
  __shared__ unsigned long long red[8][4];
  unsigned long long v = __ldcg(part + threadIdx.x);  // statistic threadIdx.x % 4
#pragma unroll
  for (int o = 16; o >= 4; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) < 4) red[threadIdx.x >> 5][threadIdx.x & 3] = v;
  __syncthreads();
  if (threadIdx.x < 4) {
    v = 0ull;
    for (int k = 0; k < 8; ++k) v += red[k][threadIdx.x];
    unsigned long long *out[4] = {&st->sum_r, &st->sum_a, &st->in_r, &st->in_a};
    *out[threadIdx.x] = v;
  }
  if (threadIdx.x == 0) {
    st->rebuild = 0;
    st->full = 0;
    st->n_rebuilds += 1;
  }
}

__global__ void finish_build_kernel(int n_struct, int *sflag, const unsigned long long *part, BuildStatus *st) {
  if (!rebuild_pending(st)) return;  // read before thread 0 clears it
  __syncthreads();
  finish_build(n_struct, sflag, part, st);
}

// The whole build of up to kWideBuildAtoms atoms in one cooperative launch: the steps above with
// barriers over the grid in place of kernel boundaries, and a warp per atom for the lists. Ten
// launches become one, and a step of a dynamics run that needs no build pays for one kernel that
// returns at once instead of a conditional graph node, which costs about 10 us. Bound by latency:
// six to eight phases of a few us. A dynamics step of 216 Si atoms 50 -> 44 us, of 13,824 atoms
// 69 -> 62 us; a serving iteration 153 -> 135 us; a build by itself about as before (20,000 atoms
// 102 us, with two blocks per SM 121, with one 163).
//
// Blocks that run at the same time by the cooperative launch wait at `bar` (L.bar[0], zero
// between launches). The wait is bounded: one that runs out sets tc_timeout and bit 2 of bad_input
// and ends the block; later builds return at once until the host has cleared both.
constexpr int kBuildBlock = kScanBlock;
constexpr int kBuildWarps = kBuildBlock / 32;
constexpr int kBuildPerSM = 3;           // blocks per SM at most (registers and shared memory hold that many)

struct GridBarrier {
  unsigned *bar;
  unsigned target = 0, polls;
  BuildStatus *st;
  __device__ __forceinline__ bool wait() {
    __shared__ int ok;
    __syncthreads();
    target += gridDim.x;
    if (threadIdx.x == 0) {
      __threadfence();
      atomicAdd(bar, 1u);
      unsigned seen, n = 0;
      do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
      } while (seen < target && ++n < polls);
      ok = seen >= target;
      if (!ok) {
        st->tc_timeout = 1;
        atomicOr(&st->bad_input, 4);
      }
      __threadfence();
    }
    __syncthreads();
    return ok != 0;
  }
};

struct BuildArgs {
  int N, T, ncell, move;
  LoadSrc src;
  AtomState a;
  ListBufs L;
  Grid g;
  Batch B;
  float rlR2, rlA2, rcR2, rcA2;
  BuildStatus *st;
};

template <int TT, bool COUNT>
__global__ void __launch_bounds__(kBuildBlock, kBuildPerSM) build_kernel(const BuildArgs p) {
  BuildStatus *const st = p.st;
  const bool load = p.src.pos != nullptr;
  // the whole block alike: a block of this launch may already have given up
  if (!load && __syncthreads_or(!rebuild_pending(st) || *(volatile const int *)&st->tc_timeout)) return;
  const int N = p.N, G = gridDim.x, tid = threadIdx.x, t0 = blockIdx.x * kBuildBlock + tid, nt = G * kBuildBlock;
  const AtomState &a = p.a;
  const ListBufs &L = p.L;
  const Batch &B = p.B;
  GridBarrier grid{L.bar, 0u, L.polls, st};
  extern __shared__ uint2 bl_stage[];  // [kBuildWarps][cap_r]
  __shared__ int wsum[kBuildWarps], carry_s;

  // a barrier that ran out: empty lists, whatever is queued behind
  auto give_up = [&]() {
    if (COUNT) return;
    for (int i = t0; i < N; i += nt) {
      for (int t = 0; t < p.T; ++t) L.nn_r[(size_t)t * N + i] = 0;
      L.nn_a[i] = 0;
    }
  };
  // the caller's shift table, cell counts and list statistics cleared
  if (load) {
    if (t0 == 0) arm_status(st);
    if (p.src.dtab)
      for (int c = t0; c < p.g.ncode; c += nt) p.src.dtab[c] = shift_vector(p.g, c);
  }
  for (int c = t0; c < p.ncell; c += nt) L.cell_count[c] = 0;
  for (int k = t0; k < 4 * kStatSlots; k += nt) L.part[k] = 0ull;
  if (!grid.wait()) return give_up();

  // bin: wrapped positions and everything that moves into the scratch arrays, atoms counted
  for (int i = t0; i < N; i += nt) {
    if (kept_by_build(B, st, i)) {  // counted in its old cell: its structure's order stays
      atomicAdd(L.cell_count + a.cell_of[i], 1);
      continue;
    }
    const size_t k = 3 * (size_t)i;
    const double *x = (load ? p.src.pos : a.x) + k;
    double r[3] = {x[0], x[1], x[2]};
    int ti = load ? p.src.types[i] : a.types[i];
    bool moved;
    const int id = bin_position(grid_of(B, p.g, i), p.T, r, &ti, &moved, st);
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      a.x2[k + b] = r[b];
      if (p.move & 1) a.v2[k + b] = a.v[k + b];
      if (p.move & 2) a.F2[k + b] = a.F[k + b];
    }
    a.types2[i] = ti;
    a.perm2[i] = load ? i : a.perm[i];
    a.cell2[i] = id;
    atomicAdd(L.cell_count + id, 1);
  }
  if (!grid.wait()) return give_up();

  // cell starts: block b scans the b-th part of the cells from the sum of the parts before
  const int part = (p.ncell + G - 1) / G, c0 = blockIdx.x * part, c1 = min(p.ncell, c0 + part);
  int before = 0;
  if (p.ncell > 8192) {  // the parts' sums by one block each
    int v = 0;
    for (int c = c0 + tid; c < c1; c += kBuildBlock) v += L.cell_count[c];
    v = block_sum(v, wsum);
    if (tid == 0) L.bar[1 + blockIdx.x] = (unsigned)v;
    if (!grid.wait()) return give_up();
    for (int b = tid; b < (int)blockIdx.x; b += kBuildBlock) before += (int)L.bar[1 + b];
  } else {  // every block adds the counts before its own part
    for (int c = tid; c < min(c0, p.ncell); c += kBuildBlock) before += L.cell_count[c];
  }
  before = block_sum(before, wsum);
  block_scan(L.cell_count, L.cell_start, c0, c1, before, wsum, &carry_s);
  if (t0 == 0) L.cell_start[p.ncell] = N;
  if (!grid.wait()) return give_up();

  // the atoms of every cell, in any order (the counts run down to zero)
  for (int i = t0; i < N; i += nt) {
    if (kept_by_build(B, st, i)) continue;
    const int c = a.cell2[i];
    L.cell_atoms[L.cell_start[c] + atomicSub(L.cell_count + c, 1) - 1] = i;
  }
  if (!grid.wait()) return give_up();

  // into their places: the cell's atoms in index order
  for (int q = t0; q < N; q += nt) {
    if (kept_by_build(B, st, q)) continue;
    const int o = L.cell_atoms[q], c = a.cell2[o], b0 = L.cell_start[c], b1 = L.cell_start[c + 1];
    int d = b0;
    for (int k = b0; k < b1; ++k) d += L.cell_atoms[k] < o ? 1 : 0;
    const size_t f = 3 * (size_t)o, k = 3 * (size_t)d;
    double r[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      r[b] = a.x2[f + b];
      if (p.move & 1) a.v[k + b] = a.v2[f + b];
      if (p.move & 2) a.F[k + b] = a.F2[f + b];
    }
    const int ti = a.types2[o];
    a.types[d] = ti;
    a.perm[d] = a.perm2[o];
    a.cell_of[d] = c;
    commit_position(grid_of(B, p.g, d), c, ti | ((B.grids ? B.sid[d] : 0) << 8), r, d, a);
  }
  if (!grid.wait()) return give_up();

  // lists: a warp per atom
  for (int i = blockIdx.x * kBuildWarps + (tid >> 5); i < N; i += G * kBuildWarps) {
    if (kept_by_build(B, st, i)) continue;  // uniform over the warp
    list_of_atom<TT, COUNT>(i, N, a.posA, a.pos4, a.cell_of, L.cell_start, grid_of(B, p.g, i), p.rlR2, p.rlA2, p.rcR2,
                            p.rcA2, L, bl_stage + (size_t)(tid >> 5) * (COUNT ? 0 : L.cap_r), st);
    __syncwarp();
  }
  if constexpr (!COUNT) {
    if (!grid.wait()) return give_up();
    for (int b = blockIdx.x * 32; b < N; b += G * 32) {
      const int i = b + (tid & 31);
      if (i < N && !kept_by_build(B, st, i)) reverse_pairs(i, tid >> 5, N, L, grid_of(B, p.g, i), st);
    }
  }
  // the last block to get here ends the build and leaves the barrier at zero
  __shared__ int last;
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    last = atomicAdd(L.bar, 1u) == grid.target + G - 1;
    __threadfence();
  }
  __syncthreads();
  if (!last) return;
  finish_build(B.sflag ? B.n : 0, B.sflag, L.part, st);
  if (tid == 0) L.bar[0] = 0u;
}

// Sets the condition of the graph's rebuild node from the drift kernel's request.
__global__ void rebuild_condition_kernel(cudaGraphConditionalHandle hc, const BuildStatus *st) {
  cudaGraphSetConditional(hc, *(volatile const int *)&st->rebuild != 0 ? 1u : 0u);
}

// Velocity Verlet, first half: v += dt/2 F/m; x += dt v; refresh cell-local coordinates;
// request a rebuild when an atom moved more than skin/2 since the last build.
// With a FIRE state, its time step is used and a converged relaxation stays where it is.
__global__ void md_drift_kernel(int N, AtomState a, const double *inv_mass_kappa, double dt, double half_skin2,
                                BuildStatus *st, const FireState *fire, int *step_ctl) {
  if (step_ctl && blockIdx.x == 0 && threadIdx.x == 0) step_ctl[0] += 1;  // the call's step number
  if (fire) {
    if (fire->converged) return;
    dt = fire->dt;
  }
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) st->md_steps += 1;
  if (i >= N) return;
  float4 p = a.pos4[i];
  const double s = 0.5 * dt * inv_mass_kappa[type_of(p)];
  double r[3], d2 = 0.0;
  for (int b = 0; b < 3; ++b) {
    const size_t k = 3 * (size_t)i + b;
    const double vb = a.v[k] + s * a.F[k];
    a.v[k] = vb;
    r[b] = a.x[k] + dt * vb;
    a.x[k] = r[b];
    const double dd = r[b] - a.x_ref[k];
    d2 += dd * dd;
  }
  p.x = (float)(r[0] - a.origin[3 * (size_t)i]);
  p.y = (float)(r[1] - a.origin[3 * (size_t)i + 1]);
  p.z = (float)(r[2] - a.origin[3 * (size_t)i + 2]);
  a.pos4[i] = p;
  if (!(d2 <= half_skin2)) st->rebuild = 1;  // also for a non-finite displacement, which the build reports
}

// Caller-order copies of the MD state: positions wrapped into the cell, velocities, forces.
__global__ void export_state_kernel(int N, const AtomState a, const Grid g0, const Batch B, double *pos, double *vel,
                                    double *force) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const Grid &g = grid_of(B, g0, i);
  const size_t u = 3 * (size_t)a.perm[i];
  if (pos) {
    const double r[3] = {a.x[3 * (size_t)i], a.x[3 * (size_t)i + 1], a.x[3 * (size_t)i + 2]};
    double s[3];
    for (int b = 0; b < 3; ++b) {
      s[b] = r[0] * g.Hinv[0][b] + r[1] * g.Hinv[1][b] + r[2] * g.Hinv[2][b];
      s[b] -= floor(s[b]);
    }
    for (int b = 0; b < 3; ++b) pos[u + b] = s[0] * g.H[0][b] + s[1] * g.H[1][b] + s[2] * g.H[2][b];
  }
  for (int b = 0; b < 3; ++b) {
    if (vel) vel[u + b] = a.v[3 * (size_t)i + b];
    if (force) force[u + b] = a.F[3 * (size_t)i + b];
  }
}

// Deterministic totals: E = sum U_i, W = sum W_i, kinetic energy, heat current J = sum J_i (the
// ones in `sums`); optional thermo row. Warp s of a block adds slot s over the block's rows
// (every lane a fixed stride, then a fixed tree); with several blocks the last one to finish
// adds the blocks' sums in block order (nothing waits: the others have left). In MD mode
// (thermo_ctl set) steps without a thermo row return at once. A thermo row holds E_pot, E_kin,
// T, P, J_x, J_y, J_z and the thermostat factor; with a thermostat (ts) the kinetic energy is
// that after the step's velocity rescaling. t_fac = 2 / ((3N - 3) k_B), p_fac: eV / (3 V) in GPa.
// One block of 256 threads with a tree of 15-slot FP64 additions took 18 us for any small system
// and 0.6 ms for 8,000,000 atoms; now 6 and 23 us.
constexpr int kThermoCols = 8;
constexpr int kFinalRows = 1024;  // rows of a block
constexpr int kFinalBlocks = 64;  // at most

__global__ void __launch_bounds__(32 * kReduceSlots)
    finalize_kernel(int nb_atom, const double *partial_atom, int nb_gather, const double *partial_gather, int sums,
                    double *energy_total, double *virial_total, double *heat_total, double *thermo_stage,
                    int *thermo_ctl /* [0] step-in-call, [1] rows written, [2] every */, double t_fac, double p_fac,
                    const ThermoState *ts, double *scratch, int *ticket, const BuildStatus *guard) {
  if (build_failed(guard)) return;
  if (thermo_ctl && thermo_ctl[0] % thermo_ctl[2] != 0) return;
  __shared__ double tot[kReduceSlots];
  __shared__ int last;
  const int s = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool mine = s == 0 ? (sums & kSumU) : s == 1 ? (sums & kSumKE)
                    : s <= 10 ? (sums & kSumW) || (s <= 4 && (sums & kSumP))
                    : s >= 12 && s <= 14 ? (sums & kSumJ) : 0;
  auto warp_sum = [&](const double *p, int stride, int n) -> double {
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = lane; b < n; b += 128)
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (b + 32 * k < n) acc[k] += p[(size_t)(b + 32 * k) * stride];
    double v = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
  };
  double v = 0.0;
  if (mine) {
    const int n = s == 0 ? nb_atom : nb_gather;
    const int per = (n + gridDim.x - 1) / gridDim.x, b0 = min(n, (int)blockIdx.x * per), b1 = min(n, b0 + per);
    v = s == 0 ? warp_sum(partial_atom + b0, 1, b1 - b0)
               : warp_sum(partial_gather + (size_t)b0 * kReduceSlots + s, kReduceSlots, b1 - b0);
  }
  if (gridDim.x > 1) {
    if (lane == 0) scratch[blockIdx.x * kReduceSlots + s] = v;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      last = atomicAdd(ticket, 1) == (int)gridDim.x - 1;
      if (last) *ticket = 0;  // for the next launch
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    v = mine ? warp_sum(scratch + s, kReduceSlots, gridDim.x) : 0.0;
  }
  if (lane == 0) tot[s] = v;
  __syncthreads();
  if (threadIdx.x != 0) return;
  if (energy_total) *energy_total = tot[0];
  if (virial_total)
    for (int c = 0; c < 9; ++c) virial_total[c] = tot[2 + c];
  if (heat_total)
    for (int c = 0; c < 3; ++c) heat_total[c] = tot[12 + c];
  if (thermo_ctl) {
    const int row = thermo_ctl[1]++;
    const double alpha = ts ? ts->alpha : 1.0;
    const double ke = tot[1] * alpha * alpha;
    double *o = thermo_stage + kThermoCols * (size_t)row;
    o[0] = tot[0];
    o[1] = ke;
    o[2] = ke * t_fac;
    o[3] = (2.0 * ke + tot[2] + tot[3] + tot[4]) * p_fac;
    // J with the rescaled velocities: J is linear in v
    for (int c = 0; c < 3; ++c) o[4 + c] = tot[12 + c] * alpha;
    o[7] = alpha;
  }
}

// Bussi-Donadio-Parrinello rescaling after a velocity-Verlet step: K from the gather
// kernel's block sums (fixed order), then with c = exp(-dt/tau), Kbar = N_f k_B T0 / 2 and
// this step's R1, S: alpha^2 = c + (1 - c)(S + R1^2) Kbar / (N_f K)
//                              + 2 R1 sqrt(c (1 - c) Kbar / (N_f K)),
// alpha taking the sign of R1 + sqrt(c N_f K / ((1 - c) Kbar)); then v <- alpha v.
__global__ void thermostat_factor_kernel(int nb_gather, const double *partial_gather, ThermoState *ts) {
  __shared__ double red[256];
  double k = 0.0;
  for (int b = threadIdx.x; b < nb_gather; b += blockDim.x) k += partial_gather[(size_t)b * kReduceSlots + 1];
  red[threadIdx.x] = k;
  __syncthreads();
  for (int off = blockDim.x / 2; off > 0; off >>= 1) {
    if (threadIdx.x < off) red[threadIdx.x] += red[threadIdx.x + off];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double K = red[0], c = ts->c, kbar = ts->kbar, nf = ts->nf;
    const double R1 = ts->rand[2 * ts->step], S = ts->rand[2 * ts->step + 1];
    double alpha = 1.0;
    if (K > 0.0) {
      const double q = kbar / (nf * K);
      const double a2 = c + (1.0 - c) * (S + R1 * R1) * q + 2.0 * R1 * sqrt(c * (1.0 - c) * q);
      alpha = sqrt(fmax(a2, 0.0));
      if (c < 1.0 && R1 + sqrt(c / ((1.0 - c) * q)) < 0.0) alpha = -alpha;
    }
    ts->alpha = alpha;
    ts->step += 1;
  }
}

__global__ void scale_velocities_kernel(int N, double *v, const ThermoState *ts) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const double a = ts->alpha;
  for (int b = 0; b < 3; ++b) v[3 * (size_t)i + b] *= a;
}

void launch_thermostat(int N, const AtomState &a, int nb_gather, const double *partial_gather, ThermoState *ts,
                       cudaStream_t s) {
  thermostat_factor_kernel<<<1, 256, 0, s>>>(nb_gather, partial_gather, ts);
  scale_velocities_kernel<<<(N + 255) / 256, 256, 0, s>>>(N, a.v, ts);
}

// ------------------------------------------------------------------ batches
// Structure s owns the atoms [offsets[s], offsets[s+1]) in the caller's order, and (the
// cells being numbered structure by structure) the same range in the internal order.
__global__ void struct_ids_kernel(int n_struct, const int *offsets, int *sid) {
  const int s = blockIdx.x;
  if (s >= n_struct) return;
  for (int i = offsets[s] + threadIdx.x; i < offsets[s + 1]; i += blockDim.x) sid[i] = s;
}

// Shift vector of every image code of every structure (zero for codes outside the range).
__global__ void shift_tables_kernel(int n_struct, const Grid *grids, int ncode, float4 *dtab) {
  const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= (long long)n_struct * ncode) return;
  const int s = (int)(v / ncode), code = (int)(v % ncode);
  dtab[grids[s].dtab_off + code] = shift_vector(grids[s], code);
}

// Per-structure sums E_s = sum U_i and W_s = sum W_i (FP64, fixed order). A structure of at
// most kWideSum atoms takes one warp (WIDE = false); a larger one one block of kSumThreads
// threads (WIDE = true), so its FP64 additions run on eight warps. Every thread adds a fixed
// stride of the structure's atoms into four partial sums by round (round mod 4: independent
// chains), combined in a fixed order, then a fixed shuffle tree (and, wide, the warp totals in
// warp order): the result depends only on the structure's atom range.
constexpr int kWideSum = 2048;
constexpr int kSumThreads = 256;
template <bool WIDE>
__global__ void struct_sums_kernel(int n_struct, int members, const int *offsets, int N, const double *e_atom,
                                   const double *w_atom, double *e_struct, double *w_struct,
                                   const BuildStatus *guard) {
  if (build_failed(guard)) return;
  const int lane = threadIdx.x & 31;
  const long long unit = WIDE ? (long long)blockIdx.x : ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (unit >= (long long)n_struct * members) return;  // uniform over the warp (block, WIDE)
  const int m = (int)(unit / n_struct), s = (int)(unit % n_struct);
  const int a0 = offsets[s], a1 = offsets[s + 1];
  if ((a1 - a0 > kWideSum) != WIDE) return;  // the other form takes this structure
  const size_t base = (size_t)m * N;
  const int t = WIDE ? (int)threadIdx.x : lane, nt = WIDE ? kSumThreads : 32;
  double acc[4][10];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 10; ++c) acc[r][c] = 0.0;
  auto add = [&](double *a, size_t k) {
    if (e_atom) a[0] += e_atom[k];
    if (w_atom)
#pragma unroll
      for (int c = 0; c < 9; ++c) a[1 + c] += w_atom[9 * k + c];
  };
  int i = a0 + t;
  for (; i + 3 * nt < a1; i += 4 * nt) {  // four rounds at a time
#pragma unroll
    for (int r = 0; r < 4; ++r) add(acc[r], base + i + (size_t)nt * r);
  }
#pragma unroll
  for (int r = 0; r < 3; ++r)  // at most three rounds left
    if (i < a1) {
      add(acc[r], base + i);
      i += nt;
    }
  double tot[10];
#pragma unroll
  for (int c = 0; c < 10; ++c) {
    tot[c] = (acc[0][c] + acc[1][c]) + (acc[2][c] + acc[3][c]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tot[c] += __shfl_down_sync(0xffffffffu, tot[c], o);
  }
  const size_t o = (size_t)m * n_struct + s;
  if constexpr (WIDE) {
    __shared__ double red[kSumThreads / 32][10];
    if (lane == 0)
#pragma unroll
      for (int c = 0; c < 10; ++c) red[threadIdx.x >> 5][c] = tot[c];
    __syncthreads();
    if (threadIdx.x < 10) {
      double v = 0.0;
      for (int w = 0; w < kSumThreads / 32; ++w) v += red[w][threadIdx.x];
      if (threadIdx.x == 0) {
        if (e_struct) e_struct[o] = v;
      } else if (w_struct) {
        w_struct[9 * o + threadIdx.x - 1] = v;
      }
    }
  } else if (lane == 0) {
    if (e_struct) e_struct[o] = tot[0];
    if (w_struct)
#pragma unroll
      for (int c = 0; c < 9; ++c) w_struct[9 * o + c] = tot[1 + c];
  }
}

// Marks a rebuild as pending and clears the per-build flags (the device form of the host
// reset before a forced rebuild, for captured graphs).
__global__ void arm_rebuild_kernel(BuildStatus *st, unsigned *bar) {
  arm_status(st);
  bar[0] = 0u;
}

// ------------------------------------------------------------------ population evaluation
// Candidate parameter vectors z [P][N_par], in the order c^R, c^A, w0, b0, w1, b1, become
// the FP32 model tables of the batched kernels (TableLayout; padding zeroed before);
// reg[m] = (sum |z|, sum z^2) for the regularisation terms of Eq. loss. One block per member.
__global__ void unpack_population_kernel(const double *z, int n_par, const TableLayout t, float *tab, double *reg) {
  const int m = blockIdx.x;
  const double *zm = z + (size_t)m * n_par;
  double s1 = 0.0, s2 = 0.0;
  for (int v = threadIdx.x; v < n_par; v += blockDim.x) {
    const double x = zm[v];
    s1 += fabs(x);
    s2 += x * x;
    tab[(size_t)m * t.total + table_place(t, v)] = (float)x;
  }
  __shared__ double r1[256], r2[256];
  r1[threadIdx.x] = s1;
  r2[threadIdx.x] = s2;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      r1[threadIdx.x] += r1[threadIdx.x + o];
      r2[threadIdx.x] += r2[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    reg[2 * m] = r1[0];
    reg[2 * m + 1] = r2[0];
  }
}

// BF16 operand tiles of every member's w0 in its model table (TableLayout).
__global__ void population_tiles_kernel(int n_pop, float *tab, const TableLayout t) {
  const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= (long long)n_pop * t.H * t.D) return;
  const int m = (int)(v / ((long long)t.H * t.D));
  const int r = (int)(v % ((long long)t.H * t.D));
  const int mu = r / t.D, nu = r % t.D;
  float *tm = tab + (size_t)m * t.total;
  float x = tm[mu * t.ndp + nu];
  __nv_bfloat16 *tile = reinterpret_cast<__nv_bfloat16 *>(tm + t.tc) + tile_place(t, mu, nu);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const __nv_bfloat16 b = __float2bfloat16_rn(x);
    tile[(size_t)k * t.np1 * t.kp1] = b;
    x -= __bfloat162float(b);
  }
}

// Eq. loss for `members` candidates (one block each, fixed-order sums): RMSE of the energy
// per atom over the non-empty structures, RMSE of the force components (from the gather
// kernel's per-block sums), RMSE of the six virial components per atom (symmetric part of
// W_s / N_s; skipped without targets), and the l1 / l2 regularisation of z.
// loss[m] = (L, RMSE_E, RMSE_F, RMSE_W, sum|z| / N_par, sqrt(sum z^2 / N_par)).
__global__ void population_loss_kernel(int n_struct, const int *offsets, const double *e_struct,
                                       const double *w_struct, const double *e_tar, const double *w_tar,
                                       const double *partial_gather, int nb_gather, int N, const double *reg,
                                       int n_par, double le, double lf, double lv, double l1, double l2,
                                       double *loss) {
  const int m = blockIdx.x;
  double se = 0.0, sv = 0.0, sf = 0.0, cnt = 0.0;
  for (int s = threadIdx.x; s < n_struct; s += blockDim.x) {
    const int n = offsets[s + 1] - offsets[s];
    if (n <= 0) continue;
    cnt += 1.0;
    const double inv = 1.0 / n;
    const double de = e_struct[(size_t)m * n_struct + s] * inv - e_tar[s];
    se += de * de;
    if (w_struct && w_tar) {
      const double *w = w_struct + 9 * ((size_t)m * n_struct + s);
      const double sym[6] = {w[0], w[1], w[2], 0.5 * (w[3] + w[6]), 0.5 * (w[5] + w[8]), 0.5 * (w[4] + w[7])};
      for (int c = 0; c < 6; ++c) {
        const double dw = sym[c] * inv - w_tar[6 * (size_t)s + c];
        sv += dw * dw;
      }
    }
  }
  for (int b = threadIdx.x; b < nb_gather; b += blockDim.x)
    sf += partial_gather[((size_t)m * nb_gather + b) * kReduceSlots + 11];
  __shared__ double red[4][256];
  red[0][threadIdx.x] = se;
  red[1][threadIdx.x] = sv;
  red[2][threadIdx.x] = sf;
  red[3][threadIdx.x] = cnt;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o)
      for (int c = 0; c < 4; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double ns = red[3][0];
    const double rmse_e = ns > 0 ? sqrt(red[0][0] / ns) : 0.0;
    const double rmse_w = (ns > 0 && w_struct && w_tar) ? sqrt(red[1][0] / (6.0 * ns)) : 0.0;
    const double rmse_f = N > 0 ? sqrt(red[2][0] / (3.0 * N)) : 0.0;
    const double r1 = reg[2 * m] / n_par, r2 = sqrt(reg[2 * m + 1] / n_par);
    double *o = loss + 6 * (size_t)m;
    o[0] = le * rmse_e + lf * rmse_f + lv * rmse_w + l1 * r1 + l2 * r2;
    o[1] = rmse_e;
    o[2] = rmse_f;
    o[3] = rmse_w;
    o[4] = r1;
    o[5] = r2;
  }
}

void launch_arm_rebuild(BuildStatus *st, unsigned *bar, cudaStream_t s) { arm_rebuild_kernel<<<1, 1, 0, s>>>(st, bar); }

void launch_unpack_population(int n_pop, const double *z, int n_par, const TableLayout &t, float *tab, double *reg,
                              cudaStream_t s) {
  if (n_pop > 0) unpack_population_kernel<<<n_pop, 256, 0, s>>>(z, n_par, t, tab, reg);
}

void launch_population_tiles(int n_pop, float *tab, const TableLayout &t, cudaStream_t s) {
  const long long n = (long long)n_pop * t.H * t.D;
  if (n > 0 && t.np1) population_tiles_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n_pop, tab, t);
}

void launch_population_loss(int members, int n_struct, const int *offsets, const double *e_struct,
                            const double *w_struct, const double *e_tar, const double *w_tar,
                            const double *partial_gather, int nb_gather, int N, const double *reg, int n_par,
                            const double *lambda, double *loss, cudaStream_t s) {
  if (members > 0)
    population_loss_kernel<<<members, 256, 0, s>>>(n_struct, offsets, e_struct, w_struct, e_tar, w_tar,
                                                    partial_gather, nb_gather, N, reg, n_par, lambda[0], lambda[1],
                                                    lambda[2], lambda[3], lambda[4], loss);
}

void launch_struct_ids(int n_struct, const int *offsets, int *sid, cudaStream_t s) {
  if (n_struct > 0) struct_ids_kernel<<<n_struct, 128, 0, s>>>(n_struct, offsets, sid);
}

void launch_shift_tables(int n_struct, const Grid *grids, int ncode, float4 *dtab, cudaStream_t s) {
  const long long n = (long long)n_struct * ncode;
  if (n > 0) shift_tables_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n_struct, grids, ncode, dtab);
}

void launch_struct_sums(int n_struct, int members, const int *offsets, int N, const double *e_atom,
                        const double *w_atom, double *e_struct, double *w_struct, int max_atoms,
                        const BuildStatus *guard, cudaStream_t s) {
  const long long units = (long long)n_struct * members;
  if (units > 0) {
    struct_sums_kernel<false><<<(unsigned)((units * 32 + 255) / 256), 256, 0, s>>>(n_struct, members, offsets, N,
                                                                                    e_atom, w_atom, e_struct, w_struct,
                                                                                    guard);
    if (max_atoms > kWideSum)
      struct_sums_kernel<true><<<(unsigned)units, kSumThreads, 0, s>>>(n_struct, members, offsets, N, e_atom, w_atom,
                                                                      e_struct, w_struct, guard);
  }
}

// ------------------------------------------------------------------ host launchers
template <bool COUNT>
cudaError_t launch_build(const BuildArgs &p, cudaStream_t s) {
  const size_t smem = COUNT ? 0 : sizeof(uint2) * kBuildWarps * (size_t)p.L.cap_r;
  static_assert(sizeof(uint2) * kBuildWarps * kListBuf <= 48 * 1024, "within the default shared memory limit");
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int want = (p.N + kBuildWarps - 1) / kBuildWarps, most = std::min(kBuildPerSM * sms, kBuildSums);
  auto go = [&](auto kern) -> cudaError_t {
    BuildArgs args = p;
    void *av[] = {&args};
    for (int grid = std::max(1, std::min(want, most));; grid = (grid + 1) / 2) {
      const cudaError_t r = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(kern), dim3(grid),
                                                        dim3(kBuildBlock), av, smem, s);
      // a stream that may use only part of the SMs holds fewer blocks at a time; any number works
      if (r != cudaErrorCooperativeLaunchTooLarge || grid == 1) return r;
      cudaGetLastError();
    }
  };
  if constexpr (COUNT) return go(build_kernel<1, true>);
  else
    switch (p.T) {
      case 1: return go(build_kernel<1, false>);
      case 2: return go(build_kernel<2, false>);
      case 3: return go(build_kernel<3, false>);
      case 4: return go(build_kernel<4, false>);
      case 5: return go(build_kernel<5, false>);
      case 6: return go(build_kernel<6, false>);
      case 7: return go(build_kernel<7, false>);
      default: return go(build_kernel<8, false>);
    }
}

cudaError_t launch_lists(int N, int T, const Grid &g, const Batch &B, float rlR2, float rlA2, float rcR2, float rcA2,
                         const AtomState &a, const ListBufs &L, int count_only, BuildStatus *st, cudaStream_t s) {
  auto lists = [&](auto kern) {
    kern<<<(N + 127) / 128, 128, 0, s>>>(N, a.posA, a.pos4, a.cell_of, L.cell_start, g, B, rlR2, rlA2, rcR2, rcA2, L,
                                         count_only, st);
    return cudaGetLastError();
  };
  switch (T) {
    case 1: return lists(build_lists_kernel<1>);
    case 2: return lists(build_lists_kernel<2>);
    case 3: return lists(build_lists_kernel<3>);
    case 4: return lists(build_lists_kernel<4>);
    case 5: return lists(build_lists_kernel<5>);
    case 6: return lists(build_lists_kernel<6>);
    case 7: return lists(build_lists_kernel<7>);
    default: return lists(build_lists_kernel<8>);
  }
}

cudaError_t launch_rebuild(int N, int T, const Grid &g, const Batch &B, float rlR2, float rlA2, float rcR2, float rcA2,
                           const AtomState &a, const ListBufs &L, int count_only, int move,
                           const LoadSrc &src, BuildStatus *st, cudaStream_t s) {
  const int tb = 256;
  const int nb = (N + tb - 1) / tb;
  const int cb = (g.ncell + tb - 1) / tb;
  // One cooperative kernel with a warp per atom up to kWideBuildAtoms atoms, separate kernels with a
  // thread per atom above: a small system leaves the thread form with a few long serial scans, a
  // large one makes the warp form pay for its idle lanes (ranges of ~20 candidates). Whole build of a
  // call, thread / warp form, us: 20,000 Si atoms 150 / 99, 66,000 182 / 184, 100,000 212 / 245, 131,072
  // 238 / 311, 262,144 PbTe atoms 404 / 482; batches of 15,384 atoms of three species 232 / 94, 67,259
  // 294 / 241, 128,755 378 / 402, 1.05 million 2056 / 2371. A single call would have the line at 66,000, a batch at
  // 120,000. It lies at 131,072 for dynamics, where the separate kernels need a conditional graph node
  // of about 10 us in every step: 20 steps with a build at the start, 30,000 Si atoms 2123 / 1860,
  // 100,000 4453 / 4401, 131,072 5424 / 5456; PbTe 100,000 3911 / 3775. (A run that builds in nearly
  // every step is better off with the threads from about 60,000 on: 120,000 atoms 12,131 / 15,268.)
  if (N <= kWideBuildAtoms) {
    const BuildArgs p{N, T, g.ncell, move, src, a, L, g, B, rlR2, rlA2, rcR2, rcA2, st};
    return count_only ? launch_build<true>(p, s) : launch_build<false>(p, s);
  }
  if (src.pos) {
    const int lb = (3LL * N + tb - 1) / tb < 8 * 152 ? (int)((3LL * N + tb - 1) / tb) : 8 * 152;
    load_kernel<<<lb, tb, 0, s>>>(N, src, a, g, st);
  }
  zero_cells_kernel<<<cb < 1024 ? cb : 1024, tb, 0, s>>>(g.ncell, L.cell_count, L.cell_cursor, L.part, st);
  bin_atoms_kernel<<<nb, tb, 0, s>>>(N, T, a, L.cell_count, g, B, st);
  const int scans = std::min(kBuildSums, (g.ncell + 1023) / 1024);
  sum_cells_kernel<<<scans, kScanBlock, 0, s>>>(g.ncell, L.cell_count, L.bar + 1, st);
  scan_cells_kernel<<<scans, kScanBlock, 0, s>>>(N, g.ncell, L.cell_count, L.cell_start, L.bar + 1, st);
  scatter_atoms_kernel<<<nb, tb, 0, s>>>(N, a.cell_of, L.cell_start, L.cell_cursor, L.cell_atoms, B, st);
  reorder_gather_kernel<<<nb, tb, 0, s>>>(N, L.cell_start, L.cell_atoms, a, move, B, st);
  reorder_commit_kernel<<<nb, tb, 0, s>>>(N, a, move, g, B, st);
  const cudaError_t e = launch_lists(N, T, g, B, rlR2, rlA2, rcR2, rcA2, a, L, count_only, st, s);
  if (e != cudaSuccess) return e;
  if (!count_only) build_rev_kernel<<<(N + 31) / 32, 256, 0, s>>>(N, L, g, B, st);
  finish_build_kernel<<<1, 256, 0, s>>>(B.sflag ? B.n : 0, B.sflag, L.part, st);
  return cudaGetLastError();
}

void launch_rebuild_condition(cudaGraphConditionalHandle hc, const BuildStatus *st, cudaStream_t s) {
  rebuild_condition_kernel<<<1, 1, 0, s>>>(hc, st);
}

void launch_drift(int N, const AtomState &a, const double *inv_mass_kappa, double dt, double half_skin2,
                  BuildStatus *st, cudaStream_t s, const FireState *fire, int *step_ctl) {
  md_drift_kernel<<<(N + 255) / 256, 256, 0, s>>>(N, a, inv_mass_kappa, dt, half_skin2, st, fire, step_ctl);
}

// FIRE velocity mixing after a velocity-Verlet step (Bitzek et al. 2006), FP64 sums in a fixed
// order: P = F . v, |F|, |v| over all atoms and max_i |F_i|^2. Converged when max_i |F_i| < fmax
// (then nothing moves again). Otherwise, for P > 0: v <- (1 - alpha) v + alpha |v| F / |F|, and
// after more than N_min such steps in a row the step grows (dt <- min(f_inc dt, dt_max)) and
// alpha shrinks (alpha <- f_alpha alpha); for P <= 0: v <- 0, dt <- f_dec dt, alpha <-
// alpha_start. check_only: only the convergence test (for the starting forces).
//
// One cluster of 8 CTAs takes the atoms [b0, b1) of one relaxation; the CTAs read each other's
// four sums from shared memory. Bound by the FP64 pipe (16 cycles of its SM per warp
// instruction), which is why one CTA is not enough: 1,001 atoms 17.5 us in one CTA of 1024 threads,
// now 5; the serving engine's jobs (up to 4,000 atoms) 21 us in one CTA each.
constexpr int kFireNmin = 5;
constexpr double kFireFinc = 1.1, kFireFdec = 0.5, kFireAlphaStart = 0.1, kFireFalpha = 0.99;
constexpr int kFireCluster = 8;

// Returns on thread 0 of the cluster's first CTA, and only there, the state after the step in
// `next` (the caller writes it, now that every CTA has read the old one); converged in *done.
__device__ __forceinline__ void fire_mix(int b0, int b1, const AtomState &a, const FireState &old, bool check_only,
                                         FireState *next) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ double red[32][4], tot[4];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int first = b0 + (int)cl.block_rank() * blockDim.x + tid, step = kFireCluster * blockDim.x;
  double sum[4] = {0.0, 0.0, 0.0, 0.0};  // P, |F|^2, |v|^2, max |F_i|^2
  double F0[3] = {0.0, 0.0, 0.0}, v0[3] = {0.0, 0.0, 0.0};  // of the thread's first atom, kept
  for (int i = first; i < b1; i += step) {
    double F[3], v[3];
    for (int b = 0; b < 3; ++b) F[b] = a.F[3 * (size_t)i + b], v[b] = a.v[3 * (size_t)i + b];
    const double f2 = F[0] * F[0] + F[1] * F[1] + F[2] * F[2];
    sum[0] += F[0] * v[0] + F[1] * v[1] + F[2] * v[2];
    sum[1] += f2;
    sum[2] += v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    sum[3] = fmax(sum[3], f2);
    if (i == first)
      for (int b = 0; b < 3; ++b) F0[b] = F[b], v0[b] = v[b];
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double y = __shfl_xor_sync(0xffffffffu, sum[k], o);
      sum[k] = k == 3 ? fmax(sum[k], y) : sum[k] + y;
    }
    if (lane == 0) red[warp][k] = sum[k];
  }
  __syncthreads();
  if (tid < 4) {
    double t = red[0][tid];
    for (int w = 1; w < (int)blockDim.x / 32; ++w) t = tid == 3 ? fmax(t, red[w][tid]) : t + red[w][tid];
    tot[tid] = t;
  }
  cl.sync();
  double all[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    all[k] = *cl.map_shared_rank(&tot[k], 0);
    for (int c = 1; c < kFireCluster; ++c) {
      const double t = *cl.map_shared_rank(&tot[k], c);
      all[k] = k == 3 ? fmax(all[k], t) : all[k] + t;
    }
  }
  cl.sync();  // every CTA has read the others' sums (and the old state)
  const double P = all[0], FF = all[1], VV = all[2];
  const bool converged = all[3] < old.fmax2, mix = !converged && !check_only, up = P > 0.0;
  const double c1 = up ? 1.0 - old.alpha : 0.0;
  const double c2 = (up && FF > 0.0) ? old.alpha * sqrt(VV / FF) : 0.0;
  if (mix)
    for (int i = first; i < b1; i += step)
      for (int b = 0; b < 3; ++b) {
        const double v = i == first ? v0[b] : a.v[3 * (size_t)i + b], F = i == first ? F0[b] : a.F[3 * (size_t)i + b];
        a.v[3 * (size_t)i + b] = c1 * v + c2 * F;
      }
  if (cl.block_rank() != 0 || tid != 0) return;
  *next = old;
  if (converged) next->converged = 1;
  if (!mix) return;
  if (up) {
    if (old.n_pos > kFireNmin) {
      next->dt = fmin(old.dt * kFireFinc, old.dt_max);
      next->alpha = old.alpha * kFireFalpha;
    }
    next->n_pos = old.n_pos + 1;
  } else {
    next->dt = old.dt * kFireFdec;
    next->alpha = kFireAlphaStart;
    next->n_pos = 0;
  }
}

__global__ void __cluster_dims__(kFireCluster, 1, 1) __launch_bounds__(512)
    fire_mix_kernel(int N, AtomState a, FireState *fire, int check_only) {
  const FireState old = *fire;  // read before the cluster's barriers, written after them
  if (old.converged) return;
  FireState next;
  fire_mix(0, N, a, old, check_only != 0, &next);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (!check_only) next.steps = old.steps + 1;  // velocity-Verlet steps taken
    *fire = next;
  }
}

void launch_fire_mix(int N, const AtomState &a, FireState *fire, int check_only, cudaStream_t s) {
  fire_mix_kernel<<<kFireCluster, N > kFireCluster * 128 ? 512 : 128, 0, s>>>(N, a, fire, check_only);
}

// ------------------------------------------------------------------ batched serving engine
// Every job is one structure of a batch; one iteration advances all of them together. The
// first iteration of a job only evaluates its forces (phase 0); each later one is a velocity-
// Verlet step (phase 1) of the job's own length (NVE) or FIRE step; finished jobs stay frozen.

// First half of the velocity-Verlet step of the stepping jobs: v += dt/2 F/m, x += dt v.
// A neighbour build is requested when an atom moved more than skin/2 since the last one.
__global__ void engine_drift_kernel(int N, AtomState a, const int *sid, const EngineSlot *slots,
                                    const double *inv_mass_kappa, double half_skin2, int *sflag, BuildStatus *st) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const EngineSlot &sl = slots[sid[i]];
  if (sl.phase != 1 || sl.kind == kJobSingle || (sl.kind == kJobFire && sl.fire.converged)) return;
  const double dt = sl.kind == kJobFire ? sl.fire.dt : sl.dt;
  const double s = 0.5 * dt * inv_mass_kappa[a.types[i]];
  double d2 = 0.0, r[3];
  for (int b = 0; b < 3; ++b) {
    const size_t k = 3 * (size_t)i + b;
    const double vb = a.v[k] + s * a.F[k];
    a.v[k] = vb;
    r[b] = a.x[k] + dt * vb;
    a.x[k] = r[b];
    const double dd = r[b] - a.x_ref[k];
    d2 += dd * dd;
  }
  // the force kernels read the cell-local FP32 coordinates
  float4 p = a.pos4[i];
  p.x = (float)(r[0] - a.origin[3 * (size_t)i]);
  p.y = (float)(r[1] - a.origin[3 * (size_t)i + 1]);
  p.z = (float)(r[2] - a.origin[3 * (size_t)i + 2]);
  a.pos4[i] = p;
  // a build of this structure (also for a non-finite displacement, which the build reports)
  if (!(d2 <= half_skin2)) {
    if (sflag) sflag[sid[i]] = 1;
    st->rebuild = 1;
  }
}

// Clears the error flags of a chunk of iterations and the barrier that a build which ran out may
// have left in mid-count (a build is not requested).
__global__ void clear_flags_kernel(BuildStatus *st, unsigned *bar) {
  bar[0] = 0u;
  st->overflow = 0;
  st->rev_missing = 0;
  st->bad_input = 0;
  st->tc_timeout = 0;
}

void launch_clear_flags(BuildStatus *st, unsigned *bar, cudaStream_t s) { clear_flags_kernel<<<1, 1, 0, s>>>(st, bar); }

// End of an engine iteration, one cluster per job: the FIRE update of a FIRE job after its step,
// then the phase and step bookkeeping.
__global__ void __cluster_dims__(kFireCluster, 1, 1) __launch_bounds__(128)
    engine_advance_kernel(const int *offsets, AtomState a, EngineSlot *slots) {
  EngineSlot &sl = slots[blockIdx.x / kFireCluster];
  const EngineSlot old = sl;  // read before the cluster's barriers, written after them
  if (old.phase == 2) return;
  const int s = blockIdx.x / kFireCluster;
  bool converged = old.kind == kJobFire && old.fire.converged;
  if (old.kind == kJobFire && !converged) {
    FireState next;
    fire_mix(offsets[s], offsets[s + 1], a, old.fire, old.phase == 0, &next);
    if (blockIdx.x % kFireCluster != 0 || threadIdx.x != 0) return;
    sl.fire = next;
    converged = next.converged;
  } else if (blockIdx.x % kFireCluster != 0 || threadIdx.x != 0) return;
  if (old.phase == 0) {
    sl.phase = (old.kind == kJobSingle || old.n_steps <= 0 || converged) ? 2 : 1;
  } else {
    sl.steps_done = old.steps_done + 1;
    if (sl.steps_done >= old.n_steps || converged) sl.phase = 2;
  }
}

// Move the atoms of the kept jobs to their new ranges: table[k] = (from, to, count, index
// shift of perm); one block per job.
__global__ void engine_relayout_kernel(const int4 *table, AtomState src, AtomState dst) {
  const int4 t = table[blockIdx.x];
  for (int k = threadIdx.x; k < t.z; k += blockDim.x) {
    const size_t i = (size_t)t.x + k, o = (size_t)t.y + k;
    for (int b = 0; b < 3; ++b) {
      dst.x[3 * o + b] = src.x[3 * i + b];
      dst.v[3 * o + b] = src.v[3 * i + b];
      dst.F[3 * o + b] = src.F[3 * i + b];
    }
    dst.types[o] = src.types[i];
    dst.perm[o] = src.perm[i] + t.w;
  }
}

void launch_engine_drift(int N, const AtomState &a, const int *sid, const EngineSlot *slots,
                         const double *inv_mass_kappa, double half_skin2, int *sflag, BuildStatus *st,
                         cudaStream_t s) {
  if (N > 0)
    engine_drift_kernel<<<(N + 255) / 256, 256, 0, s>>>(N, a, sid, slots, inv_mass_kappa, half_skin2, sflag, st);
}

void launch_engine_advance(int n_struct, const int *offsets, const AtomState &a, EngineSlot *slots, cudaStream_t s) {
  if (n_struct > 0) engine_advance_kernel<<<n_struct * kFireCluster, 128, 0, s>>>(offsets, a, slots);
}

// Arrays of a finished job (internal atoms o .. o + n - 1) in its own atom order, [3][n][3]: wrapped
// positions, forces, velocities. out may be host memory.
__global__ void engine_export_kernel(int o, int n, const AtomState a, const Grid g, double *out, int *bad) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int t = a.perm[o + i] - o;
  if (t < 0 || t >= n) {
    *bad = 1;
    return;
  }
  const size_t k = 3 * (size_t)(o + i), u = 3 * (size_t)t, m = 3 * (size_t)n;
  const double r[3] = {a.x[k], a.x[k + 1], a.x[k + 2]};
  double s[3];
  for (int b = 0; b < 3; ++b) {
    s[b] = r[0] * g.Hinv[0][b] + r[1] * g.Hinv[1][b] + r[2] * g.Hinv[2][b];
    s[b] -= floor(s[b]);
  }
  for (int b = 0; b < 3; ++b) {
    out[u + b] = s[0] * g.H[0][b] + s[1] * g.H[1][b] + s[2] * g.H[2][b];
    out[m + u + b] = a.F[k + b];
    out[2 * m + u + b] = a.v[k + b];
  }
}

void launch_engine_export(int o, int n, const AtomState &a, const Grid &g, double *out, int *bad, cudaStream_t s) {
  if (n > 0) engine_export_kernel<<<(n + 127) / 128, 128, 0, s>>>(o, n, a, g, out, bad);
}

void launch_engine_relayout(int n_keep, const int4 *table, const AtomState &src, AtomState dst, cudaStream_t s) {
  if (n_keep > 0) engine_relayout_kernel<<<n_keep, 256, 0, s>>>(table, src, dst);
}

// Neighbour lists of internal atom i written to row perm[i] (the caller's order): the caller
// index of every neighbour and the FP32 pair vector the kernels use (cell-local coordinates
// plus the image shift). Radial lists are the per-type groups in type order.
__global__ void export_lists_kernel(int N, int T, const float4 *pos4, const int *perm, const ListBufs L,
                                    const float4 *dtab, int ncode, int jbits, unsigned jmask, int cap,
                                    int *nn_r, int *j_r, float *d_r, int *nn_a, int *j_a, float *d_a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const float4 pi = pos4[i];
  const float4 *tab = dtab + (size_t)struct_of(pi) * ncode;  // structure 0 for a single structure
  const size_t row = (size_t)perm[i];
  int cnt = 0;
  for (int t = 0; t < T; ++t) cnt += L.nn_r[(size_t)t * N + i];
  nn_r[row] = cnt;
  for (int m = 0; m < cnt && m < cap && m < L.cap_r; ++m) {
    const unsigned e = L.nl_r[(size_t)m * N + i];
    const unsigned j = e & jmask;
    const float3 d = pair_vector(pi, pos4[j], tab[e >> jbits]);
    j_r[row * cap + m] = perm[j];
    d_r[(row * cap + m) * 3] = d.x;
    d_r[(row * cap + m) * 3 + 1] = d.y;
    d_r[(row * cap + m) * 3 + 2] = d.z;
  }
  const int na = L.nn_a[i];
  nn_a[row] = na;
  for (int m = 0; m < na && m < cap && m < L.cap_a; ++m) {
    const unsigned e = L.nl_a[(size_t)m * N + i];
    const unsigned j = e & jmask;
    const float3 d = pair_vector(pi, pos4[j], tab[e >> jbits]);
    j_a[row * cap + m] = perm[j];
    d_a[(row * cap + m) * 3] = d.x;
    d_a[(row * cap + m) * 3 + 1] = d.y;
    d_a[(row * cap + m) * 3 + 2] = d.z;
  }
}

void launch_export_lists(int N, int T, const float4 *pos4, const int *perm, const ListBufs &L, const float4 *dtab,
                         int ncode, int jbits, unsigned jmask, int cap, int *nn_r, int *j_r, float *d_r,
                         int *nn_a, int *j_a, float *d_a, cudaStream_t s) {
  export_lists_kernel<<<(N + 127) / 128, 128, 0, s>>>(N, T, pos4, perm, L, dtab, ncode, jbits, jmask, cap,
                                                       nn_r, j_r, d_r, nn_a, j_a, d_a);
}

void launch_export(int N, const AtomState &a, const Grid &g, const Batch &B, double *pos, double *vel, double *force,
                   cudaStream_t s) {
  export_state_kernel<<<(N + 255) / 256, 256, 0, s>>>(N, a, g, B, pos, vel, force);
}

void launch_finalize(int nb_atom, const double *partial_atom, int nb_gather, const double *partial_gather, int sums,
                     double *energy_total, double *virial_total, double *heat_total, double *thermo_stage,
                     int *thermo_ctl, int N, double volume, const ThermoState *ts, double *scratch, int *ticket,
                     const BuildStatus *guard, cudaStream_t s) {
  const double kb = 8.617333262e-5;
  const double t_fac = N > 1 ? 2.0 / ((3.0 * N - 3.0) * kb) : 0.0;
  const double p_fac = 160.21766208 / (3.0 * volume);  // eV/A^3 -> GPa
  const int nb = nb_atom > nb_gather ? nb_atom : nb_gather;
  int blocks = (nb + kFinalRows - 1) / kFinalRows;
  blocks = blocks < 1 ? 1 : blocks > kFinalBlocks ? kFinalBlocks : blocks;
  finalize_kernel<<<blocks, 32 * kReduceSlots, 0, s>>>(nb_atom, partial_atom, nb_gather, partial_gather, sums,
                                                       energy_total, virial_total, heat_total, thermo_stage, thermo_ctl,
                                                       t_fac, p_fac, ts, scratch, ticket, guard);
}

}  // namespace nep
