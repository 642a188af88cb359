// Stage a3 (smooth environment matrix), a14 (its adjoint: the per-pair
// gradient g_ij = dE/dr_ij) and a15 (forces and virial), plus the FP64
// energy reduction a9.
#include "common.cuh"
#include "kernels.h"

namespace dpa1 {

// Smooth environment matrix (Sec. II-B, DP-SE): s(r) = w(r)/r with the C2
// switch w, a row R_ij = (s, s x/r, s y/r, s z/r) normalised per centre type
// by (R - davg)/dstd.  Displacements come from the FP64 coordinates through
// the minimum image.  Real = double (the FP32 path) evaluates the row in FP64;
// Real = float (the 16-bit paths) rounds the FP64 displacement to FP32 and
// evaluates the rest in FP32, which keeps this part's error at ~1e-7
// relative, far below those paths' operand rounding.  Both store FP32.
template <typename Real>
__global__ void k_env(EnvArgs a) {
  pdl_wait();
  __shared__ double rec[sizeof(Real) == 8 ? 9 : 1];
  if constexpr (sizeof(Real) == 8) env_reciprocals(rec, a.dstd, a.atype, a.n, a.rcs, a.rc);
  long long row = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= (long long)a.n * NP) return;
  const int i = (int)(row / NP);
  const int j = a.nlist[row];
  float4 R = make_float4(0.f, 0.f, 0.f, 0.f), rw = R, rv = R;
  double w64 = 0.0;
  if (j >= 0) {
    const CellGrid& g = a.frame ? a.grid[a.frame[i]] : *a.grid;
    const double ex = a.coord[3 * j] - a.coord[3 * i];
    const double ey = a.coord[3 * j + 1] - a.coord[3 * i + 1];
    const double ez = a.coord[3 * j + 2] - a.coord[3 * i + 2];
    const Real dx = (Real)mic_near(ex, g.L[0]);
    const Real dy = (Real)mic_near(ey, g.L[1]);
    const Real dz = (Real)mic_near(ez, g.L[2]);
    const Real d = sqrt(dx * dx + dy * dy + dz * dz);
    const Real rcs = a.rcs, rc = a.rc;
    Real sw;
    if (d < rcs) {
      sw = 1;
    } else if (d < rc) {
      Real u;
      if constexpr (sizeof(Real) == 8) u = (d - rcs) * rec[8];
      else u = (d - rcs) / (rc - rcs);
      sw = u * u * u * ((Real)-6 * u * u + (Real)15 * u - (Real)10) + (Real)1;
    } else {
      sw = 0;
    }
    const Real inv_d = (Real)1 / d;
    const Real s = sw * inv_d;
    const Real hx = dx * inv_d, hy = dy * inv_d, hz = dz * inv_d;
    const int t = a.atype[i];
    const float* av = a.davg + 4 * t;
    const float* sv = a.dstd + 4 * t;
    if constexpr (sizeof(Real) == 8) {
      const double* iv = rec + 4 * (i & 1);
      R = make_float4((float)((s - av[0]) * iv[0]), (float)((s * hx - av[1]) * iv[1]), (float)((s * hy - av[2]) * iv[2]),
                      (float)((s * hz - av[3]) * iv[3]));
    } else {
      R = make_float4((s - av[0]) / sv[0], (s * hx - av[1]) / sv[1], (s * hy - av[2]) / sv[2], (s * hz - av[3]) / sv[3]);
    }
    rw = make_float4((float)hx, (float)hy, (float)hz, (float)sw);
    rv = make_float4((float)dx, (float)dy, (float)dz, (float)d);
    w64 = sw;
  }
  if (a.w64) a.w64[row] = w64;
  reinterpret_cast<float4*>(a.R)[row] = R;
  reinterpret_cast<float4*>(a.rw)[row] = rw;
  reinterpret_cast<float4*>(a.rv)[row] = rv;
  reinterpret_cast<float4*>(a.dgeo)[row] = make_float4(0.f, 0.f, 0.f, 0.f);
}

void launch_env(const EnvArgs& a, cudaStream_t st) {
  long long rows = (long long)a.n * NP;
  if (rows == 0) return;
  if (a.fp64)
    launch_pdl(k_env<double>, (unsigned)((rows + 2 * NP - 1) / (2 * NP)), 2 * NP, 0, st, a);
  else
    launch_pdl(k_env<float>, (unsigned)((rows + 2 * NP - 1) / (2 * NP)), 2 * NP, 0, st, a);
  note_launch();
}

// Chain rule from dE/dR (4 columns), dE/dw and dE/drhat back to r_ij:
//   R0 = s(d), R1..3 = q(d) r with q = s/d, w = sw(d), rhat = r/d.
// Real = double recomputes r_ij from the FP64 coordinates (the FP32 path);
// Real = float uses the stored FP32 displacement.
template <typename Real>
__global__ void k_env_bwd(EnvBwdArgs a) {
  pdl_wait();
  __shared__ double rec[sizeof(Real) == 8 ? 9 : 1];
  if constexpr (sizeof(Real) == 8) env_reciprocals(rec, a.dstd, a.atype, a.n, a.rcs, a.rc);
  long long row = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= (long long)a.n * NP) return;
  float4 out = make_float4(0.f, 0.f, 0.f, 0.f);
  const int j = a.nlist[row];
  if (j >= 0) {
    const int i = (int)(row / NP);
    Real rx, ry, rz;
    if (sizeof(Real) == 8) {
      const CellGrid g = a.frame ? a.grid[a.frame[i]] : *a.grid;
      rx = (Real)mic_near(a.coord[3 * j] - a.coord[3 * i], g.L[0]);
      ry = (Real)mic_near(a.coord[3 * j + 1] - a.coord[3 * i + 1], g.L[1]);
      rz = (Real)mic_near(a.coord[3 * j + 2] - a.coord[3 * i + 2], g.L[2]);
    } else {
      const float4 rv = reinterpret_cast<const float4*>(a.rv)[row];
      rx = rv.x; ry = rv.y; rz = rv.z;
    }
    const float4 dR = reinterpret_cast<const float4*>(a.dR)[row];
    const float4 dg = reinterpret_cast<const float4*>(a.dgeo)[row];
    const int t = a.atype[i];
    const Real d = sqrt(rx * rx + ry * ry + rz * rz);
    const Real inv = Real(1) / d;
    const Real hx = rx * inv, hy = ry * inv, hz = rz * inv;
    const Real rcs = a.rcs, rc = a.rc;
    Real sw, dsw;
    if (d < rcs) {
      sw = 1; dsw = 0;
    } else if (d < rc) {
      const Real wdt = rc - rcs;
      Real u;
      if constexpr (sizeof(Real) == 8) u = (d - rcs) * rec[8];
      else u = (d - rcs) / wdt;
      sw = u * u * u * (Real(-6) * u * u + Real(15) * u - Real(10)) + Real(1);
      dsw = Real(-30) * u * u * (u - Real(1)) * (u - Real(1));
      if constexpr (sizeof(Real) == 8) dsw *= rec[8];
      else dsw /= wdt;
    } else {
      sw = 0; dsw = 0;
    }
    const Real ds = dsw * inv - sw * inv * inv;  // d s / d d
    const Real q = sw * inv * inv;                // s / d
    const Real dq = dsw * inv * inv - Real(2) * sw * inv * inv * inv;
    const float* sv = a.dstd + 4 * t;
    Real r0, r1, r2, r3;
    if constexpr (sizeof(Real) == 8) {
      const double* iv = rec + 4 * (i & 1);
      r0 = dR.x * iv[0]; r1 = dR.y * iv[1]; r2 = dR.z * iv[2]; r3 = dR.w * iv[3];
    } else {
      r0 = dR.x / sv[0]; r1 = dR.y / sv[1]; r2 = dR.z / sv[2]; r3 = dR.w / sv[3];
    }
    const Real vdotr = r1 * rx + r2 * ry + r3 * rz;
    const Real radial = r0 * ds + dq * vdotr + (Real)dg.w * dsw;  // coefficient of rhat
    const Real hdot = (Real)dg.x * hx + (Real)dg.y * hy + (Real)dg.z * hz;
    out.x = (float)(radial * hx + q * r1 + ((Real)dg.x - hdot * hx) * inv);
    out.y = (float)(radial * hy + q * r2 + ((Real)dg.y - hdot * hy) * inv);
    out.z = (float)(radial * hz + q * r3 + ((Real)dg.z - hdot * hz) * inv);
  }
  reinterpret_cast<float4*>(a.g)[row] = out;
}

void launch_env_bwd(const EnvBwdArgs& a, cudaStream_t st) {
  long long rows = (long long)a.n * NP;
  if (rows == 0) return;
  if (a.fp64)
    launch_pdl(k_env_bwd<double>, (unsigned)((rows + 2 * NP - 1) / (2 * NP)), 2 * NP, 0, st, a);
  else
    launch_pdl(k_env_bwd<float>, (unsigned)((rows + 2 * NP - 1) / (2 * NP)), 2 * NP, 0, st, a);
  note_launch();
}

// Forces F_k = sum_j g_kj - sum_{i: k in N(i)} g_ik (Eq. eq_forceAtomicEnergy
// with e_i depending on r_ij = x_j - x_i) and virial W = -sum r_ij (x) g_ij.
// One warp per atom; the reverse rows are sorted so that every sum runs in a
// fixed order (bitwise reproducible, no atomics).  A lane adds its few terms
// and the warp its 32 lane sums in FP32 (a fixed tree; the FP64 pipe of this
// GPU is narrow), the per-block virial and energy in FP64.  Two chains of loads bind:
// the reverse rows are fetched before the atom's own pairs, all loads of either are
// issued at once and the sort (32 R places) stays in registers.  15,668 atoms: 58.6 ->
// 22.9 us, 192 atoms 15.7 -> 5.1, against the sort in shared memory before the loads.
constexpr int FWARPS = FORCE_BLOCK_ATOMS;

template <int R>
__device__ __forceinline__ void pair_sums(const ForceArgs& a, int k, int nn, int cnt, int* rows, int lane, float* f,
                                          float* v) {
  unsigned key[R];
#pragma unroll
  for (int r = 0; r < R; ++r)
    key[r] = 32 * r + lane < cnt ? (unsigned)a.rev_rows[(size_t)k * REV_CAP + 32 * r + lane] : 0x7fffffffu;
  const float4* gk = reinterpret_cast<const float4*>(a.g) + (size_t)k * NP;
  const float4* rk = reinterpret_cast<const float4*>(a.rv) + (size_t)k * NP;
  float4 g[NP / 32], x[NP / 32];
#pragma unroll
  for (int u = 0; u < NP / 32; ++u)
    if (32 * u + lane < nn) {
      g[u] = gk[32 * u + lane];
      x[u] = rk[32 * u + lane];
    }
  warp_sort<R>(key);
#pragma unroll
  for (int r = 0; r < R; ++r) rows[R * lane + r] = (int)key[r];
#pragma unroll
  for (int u = 0; u < NP / 32; ++u)
    if (32 * u + lane < nn) {
      f[0] += g[u].x; f[1] += g[u].y; f[2] += g[u].z;
      v[0] -= x[u].x * g[u].x; v[1] -= x[u].x * g[u].y; v[2] -= x[u].x * g[u].z;
      v[3] -= x[u].y * g[u].x; v[4] -= x[u].y * g[u].y; v[5] -= x[u].y * g[u].z;
      v[6] -= x[u].z * g[u].x; v[7] -= x[u].z * g[u].y; v[8] -= x[u].z * g[u].z;
    }
  __syncwarp();
  // rows of ghost centres (from row_end on) are not evaluated: their gradients are
  // zeros, taken without a load; they keep their places in the sums
  const int row_end = a.nlocal * NP;
  float4 h[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int row = rows[32 * r + lane];
    h[r] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (32 * r + lane < cnt && row < row_end) h[r] = reinterpret_cast<const float4*>(a.g)[row];
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    f[0] -= h[r].x; f[1] -= h[r].y; f[2] -= h[r].z;
  }
}

__global__ void __launch_bounds__(32 * FWARPS) k_force(ForceArgs a) {
  pdl_wait();
  __shared__ int srev[FWARPS][REV_CAP];
  __shared__ double sred[FWARPS][10];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int k = blockIdx.x * FWARPS + warp;
  float f[3] = {0.f, 0.f, 0.f};
  float v[9] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  double ek = 0;
  if (k < a.n) {
    const int nn = k < a.nlocal ? a.nnei[k] : 0;
    const int cnt = min(a.rev_cnt[k], REV_CAP);
    if (cnt <= 32)
      pair_sums<1>(a, k, nn, cnt, srev[warp], lane, f, v);
    else if (cnt <= 64)
      pair_sums<2>(a, k, nn, cnt, srev[warp], lane, f, v);
    else if (cnt <= 128)
      pair_sums<4>(a, k, nn, cnt, srev[warp], lane, f, v);
    else
      pair_sums<8>(a, k, nn, cnt, srev[warp], lane, f, v);
#pragma unroll
    for (int c = 0; c < 3; ++c) f[c] = warp_sum(f[c]);
    if (lane == 0) {
      a.force[3 * k] = f[0]; a.force[3 * k + 1] = f[1]; a.force[3 * k + 2] = f[2];
      // ghost atoms: m_k = 0 (Eq. eq_forcesLocalGhost); padding of a packed batch: no atom
      ek = k < a.nlocal && (!a.frame || a.frame[k] >= 0) ? (double)a.e[k] : 0.0;
      if (a.atom_energy) a.atom_energy[k] = ek;
    }
  }
#pragma unroll
  for (int c = 0; c < 9; ++c) v[c] = warp_sum(v[c]);
  if (lane == 0) {
    for (int c = 0; c < 9; ++c) sred[warp][c] = v[c];
    sred[warp][9] = ek;
  }
  __syncthreads();
  if (threadIdx.x < 10) {
    double s = 0;
    for (int w = 0; w < FWARPS; ++w) s += sred[w][threadIdx.x];
    a.partials[(size_t)blockIdx.x * 10 + threadIdx.x] = s;
  }
}

// Sums the block partials in a fixed order, a block per frame of a packed batch (x)
// and quantity (y; seg non-null: frame b owns partial rows [seg[b] - seg[0], seg[b+1] -
// seg[0]), else all of [0, nblocks)): thread 32 u + l adds the rows l + 32 u + 256 m,
// the rows that do not fill a group of 256 go to u = 0.  FP64 additions are slow on
// this part, so a quantity's 256 sums are spread over threads and the quantities over
// SMs: one warp a quantity took 16.6 us for 15,668 atoms, this 5.8.
constexpr int FIN_T = 256;
__global__ void __launch_bounds__(FIN_T) k_finalize(const double* __restrict__ partials, int nblocks,
                                                    const int* __restrict__ seg, double* __restrict__ energy,
                                                    double* __restrict__ virial) {
  pdl_wait();
  __shared__ double red[FIN_T / 32][32];
  const int lane = threadIdx.x & 31, u = threadIdx.x >> 5, c = blockIdx.y, fr = blockIdx.x;
  int b0 = 0, cnt = nblocks;
  if (seg) {
    b0 = seg[fr] - seg[0];
    cnt = seg[fr + 1] - seg[fr];
  }
  const double* p = partials + (size_t)b0 * 10 + c;
  double s = 0;
  int b = lane;
#pragma unroll 4
  for (; b + 7 * 32 < cnt; b += FIN_T) s += p[(size_t)(b + 32 * u) * 10];
  if (u == 0)
    for (; b < cnt; b += 32) s += p[(size_t)b * 10];
  red[u][lane] = s;
  __syncthreads();
  if (u != 0) return;
  s = ((red[0][lane] + red[1][lane]) + (red[2][lane] + red[3][lane])) +
      ((red[4][lane] + red[5][lane]) + (red[6][lane] + red[7][lane]));
  s = warp_sum_d(s);
  if (lane != 0) return;
  if (c < 9)
    virial[9 * fr + c] = s;
  else
    energy[fr] = s;
}

void launch_force_virial(const ForceArgs& a, cudaStream_t st) {
  const int nb = a.n > 0 ? (a.n + FWARPS - 1) / FWARPS : 0;
  if (nb > 0) {
    launch_pdl(k_force, nb, 32 * FWARPS, 0, st, a);
    note_launch();
  }
  if (a.seg) {
    if (a.nseg > 0) {
      launch_pdl(k_finalize, dim3(a.nseg, 10), FIN_T, 0, st, a.partials, nb, a.seg, a.energy, a.virial);
      note_launch();
    }
  } else {
    launch_pdl(k_finalize, dim3(1, 10), FIN_T, 0, st, a.partials, nb, nullptr, a.energy, a.virial);
    note_launch();
  }
}

// The gradient of E with respect to the cell h (rows = cell vectors) at fixed
// Cartesian coordinates, dE/dh = h^-T (sum_k x_k (x) F_k - W): per-block sums of the
// nine products, then one warp adds them in order and solves the 3 x 3 system by
// elimination with partial pivoting.  out: dE/dh [9], a flag (1: h singular), then
// the block sums.
constexpr int BG_T = 256;
__global__ void __launch_bounds__(BG_T) k_box_grad_sum(int n, const double* __restrict__ x, const double* __restrict__ f,
                                                       double* __restrict__ part) {
  pdl_wait();
  __shared__ double red[9][BG_T / 32];
  double s[9] = {};
  for (int k = blockIdx.x * BG_T + threadIdx.x; k < n; k += gridDim.x * BG_T) {
    const double a[3] = {x[3 * k], x[3 * k + 1], x[3 * k + 2]}, b[3] = {f[3 * k], f[3 * k + 1], f[3 * k + 2]};
#pragma unroll
    for (int i = 0; i < 9; ++i) s[i] = fma(a[i / 3], b[i % 3], s[i]);
  }
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    s[i] = warp_sum_d(s[i]);
    if ((threadIdx.x & 31) == 0) red[i][threadIdx.x >> 5] = s[i];
  }
  __syncthreads();
  if (threadIdx.x < 9) {
    double t = 0.0;
    for (int w = 0; w < BG_T / 32; ++w) t += red[threadIdx.x][w];
    part[9 * blockIdx.x + threadIdx.x] = t;
  }
}

__global__ void k_box_grad_solve(int nblocks, const double* __restrict__ part, const double* __restrict__ box,
                                 const double* __restrict__ virial, double* __restrict__ out) {
  pdl_wait();
  __shared__ double M[9];
  if (threadIdx.x < 9) {
    double t = 0.0;
    for (int b = 0; b < nblocks; ++b) t += part[9 * b + threadIdx.x];
    M[threadIdx.x] = t - virial[threadIdx.x];
  }
  __syncwarp();
  if (threadIdx.x != 0) return;
  double A[3][6];  // [h^T | M]
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      A[i][j] = box[3 * j + i];
      A[i][3 + j] = M[3 * i + j];
    }
  double flag = 0.0;
  for (int c = 0; c < 3; ++c) {
    int p = c;
    for (int r = c + 1; r < 3; ++r)
      if (fabs(A[r][c]) > fabs(A[p][c])) p = r;
    if (A[p][c] == 0.0) flag = 1.0;
    for (int j = 0; j < 6; ++j) {
      const double t = A[c][j];
      A[c][j] = A[p][j];
      A[p][j] = t;
    }
    for (int r = 0; r < 3; ++r) {
      if (r == c) continue;
      const double m = A[r][c] / A[c][c];
      for (int j = c; j < 6; ++j) A[r][j] -= m * A[c][j];
    }
  }
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) out[3 * i + j] = A[i][3 + j] / A[i][i];
  out[9] = flag;
}

int box_grad_blocks(int n) { return n < 1 ? 1 : (n + 4 * BG_T - 1) / (4 * BG_T) < 152 ? (n + 4 * BG_T - 1) / (4 * BG_T) : 152; }

void launch_box_grad(int n, const double* x, const double* box, const double* f, const double* virial, double* out,
                     cudaStream_t st) {
  const int nb = box_grad_blocks(n);
  launch_pdl(k_box_grad_sum, nb, BG_T, 0, st, n, x, f, out + 10);
  launch_pdl(k_box_grad_solve, 1, 32, 0, st, nb, out + 10, box, virial, out);
  note_launch(2);
}

}  // namespace dpa1
