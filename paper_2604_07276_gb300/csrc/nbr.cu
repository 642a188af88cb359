// Stages a1-a2: cell binning and the full neighbour list (Sec. II-C: DP
// models need full lists; the O(N) cutoff search of Sec. II-A), plus the
// reverse list used by the deterministic force gather.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace dpa1 {

// The cell grid of a box, by one warp (a lane per axis).  Cell edges are >= rcut, so
// every neighbour of an atom lies in the 27 cells around it; an axis with fewer than 3
// cells is treated as a single cell (no cell would otherwise be visited twice).
__device__ void make_grid(const double* __restrict__ box, double rcut, int cap_dim, CellGrid* g, int* __restrict__ err) {
  const int lane = threadIdx.x & 31, a = min(lane, 2);
  const double L = box[4 * a];
  bool ok = L > 2.0 * rcut && isfinite(L);
  for (int b = 0; b < 3; ++b)
    if (a != b && box[3 * a + b] != 0.0) ok = false;
  int nc = ok ? (int)floor(L / (rcut * (1.0 + 1e-9))) : 1;
  if (nc < 3) nc = 1;
  if (nc > cap_dim) nc = cap_dim;
  ok = __all_sync(0xffffffffu, ok);
  if (!ok) nc = 1;
  if (lane < 3) {
    g->nc[a] = nc;
    g->L[a] = ok ? L : 1.0;
    g->scale[a] = ok ? (double)nc / L : 1.0;
  }
  const int ncells = nc * __shfl_sync(0xffffffffu, nc, 1) * __shfl_sync(0xffffffffu, nc, 2);
  if (lane == 0) {
    g->ncells = ncells;
    g->ok = ok ? 1 : 0;
    if (!ok) set_err(err, ERR_BOX);
  }
}

// Clears the cell counters, and one warp validates the box and derives the cell grid.
__global__ void k_cell_setup(const double* __restrict__ box, double rcut, int cap_dim,
                             CellGrid* __restrict__ cg, int* __restrict__ err, int* __restrict__ cell_count,
                             int cell_cap) {
  pdl_wait();
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < cell_cap; c += gridDim.x * blockDim.x) cell_count[c] = 0;
  if (threadIdx.x < 32 && blockIdx.x == 0) make_grid(box, rcut, cap_dim, cg, err);
}

// A coordinate's image inside the box: itself, without a division, if it is inside
// (0 <= x < L, compared by the bits: negative values and NaN have larger ones).
__device__ __forceinline__ double wrap_coord(double x, double L) {
  const bool inside = (unsigned long long)__double_as_longlong(x) < (unsigned long long)__double_as_longlong(L);
  return inside ? x : x - L * floor(x / L);
}

__device__ __forceinline__ int cell_coord(double x, double L, double scale, int nc) {
  int c = (int)(wrap_coord(x, L) * scale);
  return c < 0 ? 0 : (c >= nc ? nc - 1 : c);
}

// An atom's entry of the list by cells: FP32 coordinates for the candidate screen, of
// its image inside the box (far from the origin FP32 is too coarse), the index in w.
__device__ __forceinline__ float4 cell_entry(double x, double y, double z, const double* L, int i) {
  return make_float4((float)wrap_coord(x, L[0]), (float)wrap_coord(y, L[1]), (float)wrap_coord(z, L[2]),
                     __int_as_float(i));
}

// The cell of atom i, its type checked into atype_c.
__device__ __forceinline__ int atom_cell(double x, double y, double z, const CellGrid& g, int t, int ntypes, int* atype_c,
                                         int* err) {
  int c = 0;
  if (!isfinite(x) || !isfinite(y) || !isfinite(z)) {
    set_err(err, ERR_NAN);
  } else {
    int cx = cell_coord(x, g.L[0], g.scale[0], g.nc[0]);
    int cy = cell_coord(y, g.L[1], g.scale[1], g.nc[1]);
    int cz = cell_coord(z, g.L[2], g.scale[2], g.nc[2]);
    c = (cz * g.nc[1] + cy) * g.nc[0] + cx;
  }
  if (t < 0 || t >= ntypes) {
    set_err(err, ERR_TYPE);
    t = t < 0 ? 0 : ntypes - 1;  // every later table lookup stays in bounds
  }
  *atype_c = t;
  return c;
}

// frame non-null (packed batches): slot i belongs to frame frame[i] (-1:
// padding, no cell) with grid cgp[f] and cells from cell_base[f] - cb0 on.  An atom's
// rank in its cell is what the count was before it.
__global__ void k_cell_count(const double* __restrict__ coord, const int* __restrict__ atype, int n,
                             int ntypes, const CellGrid* __restrict__ cgp, int* __restrict__ cell_of,
                             int* __restrict__ cell_count, int* __restrict__ cell_rank, int* __restrict__ atype_c,
                             int* __restrict__ rev_cnt, int* __restrict__ err, const int* __restrict__ frame,
                             const int* __restrict__ cell_base, int cb0) {
  pdl_wait();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (rev_cnt) rev_cnt[i] = 0;
  int cbase = 0;
  const CellGrid* gp = cgp;
  if (frame) {
    const int f = frame[i];
    if (f < 0) {
      atype_c[i] = 0;
      cell_of[i] = -1;
      return;
    }
    gp = cgp + f;
    cbase = cell_base[f] - cb0;
  }
  const CellGrid& g = *gp;
  const int c = cbase + atom_cell(coord[3 * i], coord[3 * i + 1], coord[3 * i + 2], g, atype[i], ntypes, atype_c + i, err);
  cell_of[i] = c;
  cell_rank[i] = atomicAdd(&cell_count[c], 1);
}

// Exclusive scan of the cell counts (one block).
__global__ void k_cell_scan(const int* __restrict__ cell_count, int* __restrict__ cell_start,
                            const CellGrid* __restrict__ cgp, int ncells_given) {
  pdl_wait();
  __shared__ int part[1024];
  __shared__ int carry;
  const int ncells = ncells_given >= 0 ? ncells_given : cgp->ncells;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < ncells; base += 1024) {
    int i = base + threadIdx.x;
    int v = i < ncells ? cell_count[i] : 0;
    part[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
      int t = threadIdx.x >= o ? part[threadIdx.x - o] : 0;
      __syncthreads();
      part[threadIdx.x] += t;
      __syncthreads();
    }
    if (i < ncells) cell_start[i] = carry + part[threadIdx.x] - v;
    __syncthreads();
    if (threadIdx.x == 1023) carry += part[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) cell_start[ncells] = carry;
}

// The atoms cell by cell.
__global__ void k_cell_fill(const double* __restrict__ coord, const int* __restrict__ cell_of,
                            const int* __restrict__ cell_rank, int n, const int* __restrict__ cell_start,
                            const CellGrid* __restrict__ cgp, const int* __restrict__ frame,
                            float4* __restrict__ cell_pos) {
  pdl_wait();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int c = cell_of[i];
  if (c < 0) return;  // padding of a packed batch
  cell_pos[cell_start[c] + cell_rank[i]] =
      cell_entry(coord[3 * i], coord[3 * i + 1], coord[3 * i + 2], cgp[frame ? frame[i] : 0].L, i);
}

// The four kernels above in one block, for up to SMALL_ATOMS atoms: each of them is a
// launch and a chain of loads there (192 atoms: 14.9 us together; this takes 5.4, of
// 582 7.8).  Two atoms a thread; the counters of up to SMALL_CELLS cells stay in shared
// memory.
constexpr int SMALL_T = 1024, SMALL_ATOMS = 2 * SMALL_T, SMALL_CELLS = 4096;
__global__ void __launch_bounds__(SMALL_T) k_cells_small(const double* __restrict__ coord,
                                                         const double* __restrict__ box,
                                                         const int* __restrict__ atype, int n, int ntypes, double rcut,
                                                         int cap_dim, CellGrid* __restrict__ cg, int* __restrict__ cell_of,
                                                         int* cell_count, int* cell_start, float4* __restrict__ cell_pos,
                                                         int* __restrict__ atype_c, int* __restrict__ rev_cnt,
                                                         int* __restrict__ err) {
  pdl_wait();
  __shared__ CellGrid s_g;
  __shared__ int s_cnt[SMALL_CELLS], s_warp[SMALL_T / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int U = SMALL_ATOMS / SMALL_T;
  double x[U][3];
  int type[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = tid + u * SMALL_T;
    if (i < n) {
      x[u][0] = coord[3 * i]; x[u][1] = coord[3 * i + 1]; x[u][2] = coord[3 * i + 2];
      type[u] = atype[i];
      if (rev_cnt) rev_cnt[i] = 0;
    }
  }
  if (warp == 0) make_grid(box, rcut, cap_dim, &s_g, err);
  __syncthreads();
  if (tid == 0) *cg = s_g;
  const int ncells = s_g.ncells;
  const bool sh = ncells <= SMALL_CELLS;
  for (int c = tid; c < ncells; c += SMALL_T) (sh ? s_cnt : cell_count)[c] = 0;
  __syncthreads();
  int cell[U], rank[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = tid + u * SMALL_T;
    if (i < n) {
      cell[u] = atom_cell(x[u][0], x[u][1], x[u][2], s_g, type[u], ntypes, atype_c + i, err);
      cell_of[i] = cell[u];
      rank[u] = atomicAdd((sh ? s_cnt : cell_count) + cell[u], 1);
    }
  }
  __syncthreads();
  // exclusive scan, a run of cells per thread
  const int per = (ncells + SMALL_T - 1) / SMALL_T, c0 = min(tid * per, ncells), c1 = min(c0 + per, ncells);
  auto count = [&](int c) { return sh ? s_cnt[c] : __ldcg(cell_count + c); };
  int sum = 0;
  for (int c = c0; c < c1; ++c) sum += count(c);
  int run = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, run, d);
    if (lane >= d) run += y;
  }
  if (lane == 31) s_warp[warp] = run;
  __syncthreads();
  if (warp == 0) {
    int w = s_warp[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, d);
      if (lane >= d) w += y;
    }
    s_warp[lane] = w;
  }
  __syncthreads();
  run += (warp > 0 ? s_warp[warp - 1] : 0) - sum;
  for (int c = c0; c < c1; ++c) {
    const int v = count(c);
    cell_start[c] = run;
    if (sh) s_cnt[c] = run;
    run += v;
  }
  if (tid == SMALL_T - 1) cell_start[ncells] = run;
  __syncthreads();
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int i = tid + u * SMALL_T;
    if (i < n)
      cell_pos[(sh ? s_cnt[cell[u]] : __ldcg(cell_start + cell[u])) + rank[u]] =
          cell_entry(x[u][0], x[u][1], x[u][2], s_g.L, i);
  }
}

// Sort keys: the bit pattern of d^2 >= 0 (+0 or positive, never NaN) read as an
// unsigned integer orders like the value, so the sort needs no FP64 compare.
__device__ __forceinline__ bool key_gt(unsigned long long da, int ja, unsigned long long db, int jb) {
  return da > db || (da == db && ja > jb);
}

constexpr int NBR_WARPS = 4;
constexpr int NBR_SEGS = 18;  // 9 rows of 3 cells along x, each cut in two by the box edge at most

// One warp's buffers.
struct NbrShared {
  unsigned long long key[NBR_CAP];  // bits of d^2
  int idx[NBR_CAP];                 // candidate
  unsigned char order[NBR_CAP];     // candidates' places, sorted
  int2 seg[NBR_SEGS];               // running end of a segment's candidates, its offset in cell_pos
};

// The order of the cnt <= 32 R candidates by (d^2, j).  The registers sort 24 bits of
// d^2 - the value's exponent and 20 fraction bits below rc^2, everything under
// rc^2 / 65,536 alike - with the place in the low byte; pairs of neighbours that these
// bits leave undecided are put right by exchanges on the full key.
template <int R>
__device__ __forceinline__ void sort_candidates(NbrShared& sh, int cnt, int hi_rc2, int lane) {
  unsigned k[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int e = 32 * r + lane;
    k[r] = 0xffffffffu;
    if (e < cnt) {
      const int hi = (int)(sh.key[e] >> 32) - (hi_rc2 - 0xffffff);
      k[r] = (unsigned)max(hi, 0) << 8 | (unsigned)e;
    }
  }
  warp_sort<R>(k);
  const unsigned next = __shfl_down_sync(0xffffffffu, k[0], 1);
  bool tie = false;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int p = R * lane + r;  // the place after it: p + 1
    sh.order[p] = (unsigned char)(k[r] & 0xff);
    tie |= p + 1 < cnt && k[r] >> 8 == (r + 1 < R ? k[(r + 1) % R] : next) >> 8;
  }
  __syncwarp();
  if (!__any_sync(0xffffffffu, tie)) return;
  // odd-even transposition sorts cnt values in cnt rounds at most
  for (int round = 0; round < cnt; round += 2) {
    bool moved = false;
    for (int odd = 0; odd < 2; ++odd) {
      for (int p = 2 * lane + odd; p + 1 < cnt; p += 64) {
        const int x = sh.order[p], y = sh.order[p + 1];
        if (key_gt(sh.key[x], sh.idx[x], sh.key[y], sh.idx[y])) {
          sh.order[p] = (unsigned char)y;
          sh.order[p + 1] = (unsigned char)x;
          moved = true;
        }
      }
      __syncwarp();
    }
    if (!__any_sync(0xffffffffu, moved)) break;
  }
}

// One warp per centre atom: gather every candidate j != i with d^2 < rc^2 from
// the 27 surrounding cells (screened in FP32, decided in FP64 and
// bit-reproducible), then sort the candidates by (d^2, j) and keep the first sel; a
// kept pair also enters j's reverse list, as row i * NP + slot.  FP64 is slow on this
// part, so it is kept to the ~11 % of candidates that pass the screen.  A chain of
// dependent loads and of sort stages binds, so loads go out in groups of four, a row
// of cells is one stretch, and the sort stays in registers.  15,668 atoms: the
// search's kernels took 181 us, and 26 for the reverse list's own -> 87 together; 192
// atoms: 42 + 6 -> 32.  63 registers: held to 48 for two more blocks an SM, 183.
__global__ void __launch_bounds__(32 * NBR_WARPS, 8)
k_neighbors(const double* __restrict__ coord, int n, int n_out, int base, const CellGrid* __restrict__ cgp,
            const int* __restrict__ cell_of, const int* __restrict__ cell_start,
            const float4* __restrict__ cell_pos, double rc2, float rc, int sel, int* __restrict__ nlist,
            int* __restrict__ nnei, int* __restrict__ ncand, int* __restrict__ atype_c, int* __restrict__ err,
            const int* __restrict__ frame, const int* __restrict__ cell_base, int cb0, int* __restrict__ rev_cnt,
            int* __restrict__ rev_rows) {
  pdl_wait();
  __shared__ NbrShared s_sh[NBR_WARPS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * NBR_WARPS + warp;
  const int fi = frame && i < n ? frame[i] : 0;
  if (i >= n || fi < 0) {
    // padding atoms of a packed batch: no neighbours, a valid type
    if (i < n_out || (i < n && fi < 0)) {
      for (int s = lane; s < NP; s += 32) nlist[(size_t)i * NP + s] = -1;
      if (lane == 0) {
        nnei[i] = 0;
        ncand[i] = 0;
        atype_c[i] = 0;
        if (rev_cnt) rev_cnt[i] = 0;
      }
    }
    return;
  }
  NbrShared& sh = s_sh[warp];
  const CellGrid* g = cgp + (frame ? fi : 0);
  const double xi = coord[3 * i], yi = coord[3 * i + 1], zi = coord[3 * i + 2];
  const float4 fi4 = cell_entry(xi, yi, zi, g->L, i);
  const float Lx = (float)g->L[0], Ly = (float)g->L[1], Lz = (float)g->L[2];
  const float iLx = 1.0f / Lx, iLy = 1.0f / Ly, iLz = 1.0f / Lz;
  // The cells of a row along x follow each other in cell_pos: a lane finds one
  // contiguous stretch of candidates (part 1: what wraps around the box edge).
  int ns = 0, total;
  {
    const int cbase = frame ? cell_base[fi] - cb0 : 0;  // the frame's first cell
    const int nx = g->nc[0], ny = g->nc[1], nz = g->nc[2];
    const int ci = cell_of[i] - cbase;
    const int cx = ci % nx, cy = (ci / nx) % ny, cz = ci / (nx * ny);
    const int row = lane >> 1, dy = row % 3 - 1, dz = row / 3 - 1;
    int b = 0, cnt = 0;
    // an axis of fewer than 3 cells has one, visited once
    if (lane < NBR_SEGS && (ny >= 3 || dy == 0) && (nz >= 3 || dz == 0)) {
      auto wrap = [](int x, int nc) { return x < 0 ? x + nc : (x >= nc ? x - nc : x); };
      int lo = cx, hi = cx;
      if (nx >= 3) { lo = cx - 1; hi = cx + 1; }
      if (lane & 1) {
        if (lo < 0) lo = hi = nx - 1;
        else if (hi >= nx) lo = hi = 0;
        else lo = 0, hi = -1;
      } else {
        lo = max(lo, 0);
        hi = min(hi, nx - 1);
      }
      if (lo <= hi) {
        const int c = cbase + (wrap(cz + dz, nz) * ny + wrap(cy + dy, ny)) * nx;
        b = cell_start[c + lo];
        cnt = cell_start[c + hi + 1] - b;
      }
    }
    int end = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, end, d);
      if (lane >= d) end += y;
    }
    if (lane < NBR_SEGS) sh.seg[lane] = make_int2(end, b - (end - cnt));
    total = __shfl_sync(0xffffffffu, end, 31);
    __syncwarp();
  }
  // pass 1: FP32 screen of the candidates, all lanes busy and NBR_U loads under way;
  // survivors are compacted into idx[] so that the FP64 decision below runs on full
  // warps (this part's FP64 rate is low, and a divergent FP64 branch costs the whole
  // warp).  No neighbour may fail it.  With the coordinates in [0, L] and u = 2^-24,
  // the two roundings, those of the difference and the edge make a component of the
  // FP32 difference wrong by at most 4.5 u L, and, where the division by L tips to
  // the other image within 5 u L of half an edge, by 14.5 u L; e = 16 u L per
  // component lengthens a neighbour's distance to rc + sqrt(3) e at most.  The
  // fixed margin is wider for edges up to 180 A (rc = 6 A).
  constexpr int NBR_U = 4;
  const float far = rc + 1.7320509f * (16.f / 16777216.f) * fmaxf(Lx, fmaxf(Ly, Lz));
  const float rc2_screen = fmaxf((float)rc2 * 1.0001f + 1e-4f, far * far * 1.000002f);
  constexpr float RINT = 12582912.f;  // 1.5 * 2^23: x + RINT - RINT rounds x to an integer
  int cur = 0;
  int2 seg = sh.seg[0];
  for (int b = 0; b < total; b += 32 * NBR_U) {
    float4 p[NBR_U];
#pragma unroll
    for (int u = 0; u < NBR_U; ++u) {
      const int t = b + 32 * u + lane;
      p[u].w = __int_as_float(i);  // no candidate
      if (t < total) {
        while (t >= seg.x) seg = sh.seg[++cur];
        p[u] = cell_pos[t + seg.y];
      }
    }
#pragma unroll
    for (int u = 0; u < NBR_U; ++u) {
      const int j = __float_as_int(p[u].w);
      bool pass = false;
      if (j != i) {
        float fx = p[u].x - fi4.x, fy = p[u].y - fi4.y, fz = p[u].z - fi4.z;
        fx -= Lx * (__fmaf_rn(fx, iLx, RINT) - RINT);
        fy -= Ly * (__fmaf_rn(fy, iLy, RINT) - RINT);
        fz -= Lz * (__fmaf_rn(fz, iLz, RINT) - RINT);
        pass = fx * fx + fy * fy + fz * fz < rc2_screen;
      }
      const unsigned bal = __ballot_sync(0xffffffffu, pass);
      const int pos = ns + __popc(bal & ((1u << lane) - 1u));
      if (pass && pos < NBR_CAP) sh.idx[pos] = j;
      ns += __popc(bal);
    }
  }
  if (ns > NBR_CAP) {
    if (lane == 0) set_err(err, ERR_CAPACITY);
    ns = NBR_CAP;
  }
  __syncwarp();
  // pass 2: the exact FP64 decision on the survivors, compacted in place
  // (a write never reaches an entry that is still to be read)
  int cnt = 0;
  const unsigned long long rc2_bits = (unsigned long long)__double_as_longlong(rc2);
  for (int b = 0; b < ns; b += 32) {
    const int t = b + lane;
    bool hit = false;
    unsigned long long d2 = 0;
    int j = -1;
    if (t < ns) {
      j = sh.idx[t];
      const double ddx = mic_near(__dsub_rn(coord[3 * j], xi), g->L[0]);
      const double ddy = mic_near(__dsub_rn(coord[3 * j + 1], yi), g->L[1]);
      const double ddz = mic_near(__dsub_rn(coord[3 * j + 2], zi), g->L[2]);
      d2 = (unsigned long long)__double_as_longlong(sqdist(ddx, ddy, ddz));
      hit = d2 < rc2_bits;
    }
    const unsigned bal = __ballot_sync(0xffffffffu, hit);
    const int pos = cnt + __popc(bal & ((1u << lane) - 1u));
    if (hit) {
      sh.key[pos] = d2;
      sh.idx[pos] = j;
    }
    cnt += __popc(bal);
    __syncwarp();
  }
  if (lane == 0) ncand[i] = cnt;
  const int hi_rc2 = __double2hiint(rc2);
  if (cnt <= 32)
    sort_candidates<1>(sh, cnt, hi_rc2, lane);
  else if (cnt <= 64)
    sort_candidates<2>(sh, cnt, hi_rc2, lane);
  else if (cnt <= 128)
    sort_candidates<4>(sh, cnt, hi_rc2, lane);
  else
    sort_candidates<8>(sh, cnt, hi_rc2, lane);
  const int keep = cnt < sel ? cnt : sel;
  for (int s = lane; s < NP; s += 32) {
    const int j = s < keep ? sh.idx[sh.order[s]] : -1;
    nlist[(size_t)i * NP + s] = j >= 0 ? j + base : -1;
    if (rev_rows && j >= 0) {
      const int pos = atomicAdd(&rev_cnt[j], 1);
      if (pos < REV_CAP)
        rev_rows[(size_t)j * REV_CAP + pos] = (i + base) * NP + s;
      else
        set_err(err, ERR_CAPACITY);
    }
  }
  if (lane == 0) nnei[i] = keep;
}

void launch_neighbors(const NbrArgs& a, cudaStream_t st) {
  const int n_out = a.n_out > a.n ? a.n_out : a.n;
  const int tb = 256;
  if (a.n > 0 && a.n <= SMALL_ATOMS) {
    launch_pdl(k_cells_small, 1, SMALL_T, 0, st, a.coord, a.box, a.atype, a.n, a.ntypes, a.rcut, a.cap_dim, a.grid,
               a.cell_of, a.cell_count, a.cell_start, a.cell_pos, a.atype_c, a.rev_cnt, a.err);
    note_launch();
  } else {
    launch_pdl(k_cell_setup, std::min(152, (a.cell_cap + 255) / 256), 256, 0, st, a.box, a.rcut, a.cap_dim, a.grid,
               a.err, a.cell_count, a.cell_cap);
    note_launch();
  }
  if (n_out == 0) return;
  if (a.n > SMALL_ATOMS) {
    launch_pdl(k_cell_count, (a.n + tb - 1) / tb, tb, 0, st, a.coord, a.atype, a.n, a.ntypes, a.grid, a.cell_of,
               a.cell_count, a.cell_rank, a.atype_c, a.rev_cnt, a.err, nullptr, nullptr, 0);
    note_launch();
    launch_pdl(k_cell_scan, 1, 1024, 0, st, a.cell_count, a.cell_start, a.grid, -1);
    note_launch();
    launch_pdl(k_cell_fill, (a.n + tb - 1) / tb, tb, 0, st, a.coord, a.cell_of, a.cell_rank, a.n, a.cell_start,
               a.grid, nullptr, a.cell_pos);
    note_launch();
  }
  launch_pdl(k_neighbors, (n_out + NBR_WARPS - 1) / NBR_WARPS, 32 * NBR_WARPS, 0, st,
             a.coord, a.n, n_out, a.base, a.grid, a.cell_of, a.cell_start, a.cell_pos, a.rcut * a.rcut, (float)a.rcut, a.sel, a.nlist,
             a.nnei, a.ncand, a.atype_c, a.err, nullptr, nullptr, 0, a.rev_cnt, a.rev_rows);
  note_launch();
}

void launch_neighbors_packed(const NbrArgs& a, const int* frame, const int* cell_base, int cb0, int ncells_total,
                             cudaStream_t st) {
  if (a.n == 0) return;
  cudaMemsetAsync(a.cell_count, 0, sizeof(int) * (size_t)ncells_total, st);
  const int tb = 256;
  launch_pdl(k_cell_count, (a.n + tb - 1) / tb, tb, 0, st, a.coord, a.atype, a.n, a.ntypes, a.grid, a.cell_of,
             a.cell_count, a.cell_rank, a.atype_c, a.rev_cnt, a.err, frame, cell_base, cb0);
  note_launch();
  launch_pdl(k_cell_scan, 1, 1024, 0, st, a.cell_count, a.cell_start, a.grid, ncells_total);
  note_launch();
  launch_pdl(k_cell_fill, (a.n + tb - 1) / tb, tb, 0, st, a.coord, a.cell_of, a.cell_rank, a.n, a.cell_start,
             a.grid, frame, a.cell_pos);
  note_launch();
  launch_pdl(k_neighbors, (a.n + NBR_WARPS - 1) / NBR_WARPS, 32 * NBR_WARPS, 0, st,
             a.coord, a.n, a.n, 0, a.grid, a.cell_of, a.cell_start, a.cell_pos, a.rcut * a.rcut, (float)a.rcut, a.sel, a.nlist, a.nnei,
             a.ncand, a.atype_c, a.err, frame, cell_base, cb0, a.rev_cnt, a.rev_rows);
  note_launch();
}

// The list of live rows: a block of 256 threads takes ROWL_ATOMS atoms.  Its first
// place is the sum of the counts before it: those of whole ROW_SEG segments from
// seg (written by k_row_seg; a single segment needs none), the rest summed here.
constexpr int ROWL_ATOMS = 32, ROWL_T = 256;

__device__ __forceinline__ int block_sum(int v, int* s_red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
  __syncthreads();
  int t = 0;
#pragma unroll
  for (int w = 0; w < ROWL_T / 32; ++w) t += s_red[w];
  return t;
}

__global__ void __launch_bounds__(ROWL_T) k_row_seg(const int* __restrict__ nnei, int n, int* __restrict__ seg) {
  pdl_wait();
  __shared__ int s_red[ROWL_T / 32];
  int v = 0;
  for (int i = blockIdx.x * ROW_SEG + threadIdx.x; i < min(n, (int)(blockIdx.x + 1) * ROW_SEG); i += ROWL_T) v += nnei[i];
  v = block_sum(v, s_red);
  if (threadIdx.x == 0) seg[blockIdx.x] = v;
}

__global__ void __launch_bounds__(ROWL_T) k_row_list(const int* __restrict__ nnei, int n, const int* __restrict__ seg,
                                                     int* __restrict__ row_off, int* __restrict__ rowmap) {
  pdl_wait();
  __shared__ int s_red[ROWL_T / 32], s_off[ROWL_ATOMS];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int first = blockIdx.x * ROWL_ATOMS, s0 = first / ROW_SEG;
  int v = 0;
  for (int k = t; k < s0; k += ROWL_T) v += seg[k];
  for (int i = s0 * ROW_SEG + t; i < first; i += ROWL_T) v += nnei[i];
  const int base = block_sum(v, s_red);
  if (w == 0) {
    const int nn = first + lane < n ? nnei[first + lane] : 0;
    int x = nn;  // inclusive sum over the block's atoms
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, d);
      if (lane >= d) x += y;
    }
    s_off[lane] = base + x - nn;
    if (first + lane < n) row_off[first + lane] = base + x - nn;
    if (first + lane == n - 1) row_off[n] = base + x;
  }
  __syncthreads();
  for (int j = w; j < ROWL_ATOMS && first + j < n; j += ROWL_T / 32) {
    const int nj = nnei[first + j], oj = s_off[j];
    for (int s = lane; s < nj; s += 32) rowmap[oj + s] = (first + j) * NP + s;
  }
}

void launch_row_list(const int* nnei, int n, int* row_off, int* rowmap, int* seg, cudaStream_t st) {
  if (n == 0) return;
  if (n > ROW_SEG) {
    launch_pdl(k_row_seg, (n + ROW_SEG - 1) / ROW_SEG, ROWL_T, 0, st, nnei, n, seg);
    note_launch();
  }
  launch_pdl(k_row_list, (n + ROWL_ATOMS - 1) / ROWL_ATOMS, ROWL_T, 0, st, nnei, n, seg, row_off, rowmap);
  note_launch();
}

}  // namespace dpa1
