// Training kernels of the distilled student potential (stage a17): weight
// gradients of the energy, the per-frame energy / force loss, Adam, and the
// refresh of the derived weight copies the forward kernels read.
//
// Loss of one frame (N atoms): L = pe ((E - E_ref) / N)^2 + pf mean |F - F_ref|^2.
// dL/dtheta = 2 pe (E - E_ref) / N^2 dE/dtheta
//           - (2 pf / 3N) d/dtheta [ sum_k (F - F_ref)_k . dE/dx_k ],
// and the bracket's theta-gradient is the derivative of dE/dtheta along the
// fixed displacement field v = F - F_ref: d/de dE/dtheta(x + e v) at e = 0.
// It is evaluated exactly in forward mode over the adjoint: every quantity q
// of the energy evaluation and of its adjoint gets its tangent q' = dq/de,
// and the weight gradients (sums over rows of input (x) adjoint) get theirs by
// the product rule.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace dpa1 {

// Gradient of a fitting layer, both loss terms at once: with s1, s2 the energy and
// force terms' scales, M = s2 dZ' + s1 dZ and D = s2 dZ,
//   C[i][o] += sum_n A'[n][i] D[n][o] + A[n][i] M[n][o],  c[o] += sum_n M[n][o]
// (A the layer's input, ' the tangents).  The n range is split over grid.z slices that
// add their parts atomically.  A frame of some hundred atoms is a chain of launches and
// load latencies, hence one launch a layer, and 32 rows of all four operands fetched at
// once.  A launch for each of the three products and two sums of a layer took 34 us a
// layer of a 582-atom frame (and one more to add the energy term up), this 11.
constexpr int WG_ROWS = 32;
__global__ void __launch_bounds__(256) k_fit_grad(const float* __restrict__ A, const float* __restrict__ Ad,
                                                  const float* __restrict__ dZ, const float* __restrict__ dZd,
                                                  float* __restrict__ C, float* __restrict__ c, int I, int O, int N,
                                                  int chunk, const float* __restrict__ scales) {
  pdl_wait();
  __shared__ float As[WG_ROWS][64 + 4], Ads[WG_ROWS][64 + 4], Ms[WG_ROWS][64 + 4], Ds[WG_ROWS][64 + 4];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int i0 = blockIdx.x * 64, o0 = blockIdx.y * 64;
  const int n_begin = blockIdx.z * chunk;
  const int n_end = min(N, n_begin + chunk);
  const float s1 = scales[0], s2 = scales[1];
  float acc[4][4] = {}, bias = 0.f;
  for (int n0 = n_begin; n0 < n_end; n0 += WG_ROWS) {
#pragma unroll
    for (int q = 0; q < WG_ROWS * 64 / 256; ++q) {
      const int t = threadIdx.x + 256 * q, k = t / 64, j = t % 64, n = n0 + k;
      const bool ai = n < n_end && i0 + j < I, bo = n < n_end && o0 + j < O;
      const size_t ia = (size_t)n * I + i0 + j, ib = (size_t)n * O + o0 + j;
      As[k][j] = ai ? A[ia] : 0.f;
      Ads[k][j] = ai ? Ad[ia] : 0.f;
      const float z = bo ? dZ[ib] : 0.f, zd = bo ? dZd[ib] : 0.f;
      Ms[k][j] = fmaf(s2, zd, s1 * z);
      Ds[k][j] = s2 * z;
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < WG_ROWS; ++k) {
      float a[4], ad[4], m[4], d[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        a[q] = As[k][ty * 4 + q]; ad[q] = Ads[k][ty * 4 + q];
        m[q] = Ms[k][tx * 4 + q]; d[q] = Ds[k][tx * 4 + q];
      }
#pragma unroll
      for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(a[p], m[q], fmaf(ad[p], d[q], acc[p][q]));
    }
    if (blockIdx.x == 0 && threadIdx.x < 64) {
#pragma unroll 8
      for (int k = 0; k < WG_ROWS; ++k) bias += Ms[k][threadIdx.x];
    }
    __syncthreads();
  }
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = i0 + ty * 4 + p, o = o0 + tx * 4 + q;
      if (i < I && o < O) atomicAdd(&C[(size_t)i * O + o], acc[p][q]);
    }
  if (blockIdx.x == 0 && threadIdx.x < 64 && o0 + (int)threadIdx.x < O) atomicAdd(&c[o0 + threadIdx.x], bias);
}

// Gradient of the energy head, e_i = out_scale (H_i . w_out + b_out) + ebias[t_i]:
// w_out[o] += out_scale sum_n s1 H[n][o] + s2 H'[n][o], over grid.y - 2 slices of the
// rows; the biases, constant in the forces, are two blocks of their own: ebias[t] += s1
// times the type's atoms (counted, so exact), b_out += s1 times out_scale added up atom
// by atom in FP32.  That sum is 4e-6 off at 582 atoms and 1e-4 at 8,000 (out_scale 537);
// out_scale N, rounded once, is not, but moves the whole gradient of frames above 6,400
// atoms by 2.0 - 2.6e-5 of its norm, more than results are to move between versions.
__global__ void k_head_grad(const float* __restrict__ H, const float* __restrict__ Hd, const int* __restrict__ atype,
                            float* __restrict__ g_wout, float* __restrict__ g_bout, float* __restrict__ g_ebias, int O,
                            int N, int ntypes, int chunk, const float* __restrict__ scales, float out_scale) {
  pdl_wait();
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  const float s1 = scales[0], s2 = scales[1];
  if (blockIdx.y >= gridDim.y - 2) {
    if (blockIdx.x > 0) return;
    if (blockIdx.y == gridDim.y - 1) {
      for (int t = 0; t < ntypes; ++t) {
        int count = 0;
        for (int n = threadIdx.x; n - (int)threadIdx.x < N; n += blockDim.x)
          count += __syncthreads_count(n < N && atype[n] == t);
        if (threadIdx.x == 0) g_ebias[t] += s1 * (float)count;
      }
    } else if (threadIdx.x == 0) {
      float b = 0.f;
#pragma unroll 8
      for (int n = 0; n < N; ++n) b += out_scale;
      *g_bout += s1 * b;
    }
    return;
  }
  const int n_begin = blockIdx.y * chunk, n_end = min(N, n_begin + chunk);
  if (o >= O) return;
  float s = 0.f, sd = 0.f;
#pragma unroll 8
  for (int n = n_begin; n < n_end; ++n) {
    s += H[(size_t)n * O + o];
    sd += Hd[(size_t)n * O + o];
  }
  atomicAdd(&g_wout[o], out_scale * fmaf(s2, sd, s1 * s));
}

// One block: loss of the frame, the gradient scales and the direction
// v = F - F_ref.
__global__ void k_train_prep(int n, const double* __restrict__ energy, double e_ref,
                             const double* __restrict__ force, const double* __restrict__ force_ref, double pe,
                             double pf, double* __restrict__ v, double* __restrict__ loss,
                             float* __restrict__ scales) {
  pdl_wait();
  __shared__ double red_s[32];
  double ss = 0.0;
  for (int k = threadIdx.x; k < 3 * n; k += blockDim.x) {
    const double d = force[k] - force_ref[k];
    v[k] = d;
    ss += d * d;
  }
  ss = warp_sum_d(ss);
  if ((threadIdx.x & 31) == 0) red_s[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (threadIdx.x == 0) {
    double S = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) S += red_s[w];
    const double nn = n > 0 ? (double)n : 1.0;
    const double de = *energy - e_ref;
    const double lE = pe * (de / nn) * (de / nn);
    const double lF = pf * S / (3.0 * nn);
    loss[0] = lE + lF;
    loss[1] = lE;
    loss[2] = lF;
    scales[0] = (float)(2.0 * pe * de / (nn * nn));
    scales[1] = (float)(-2.0 * pf / (3.0 * nn));
  }
}

// ------------------------------------------------------------------ tangents
// R'_ij = dR_ij/dr_ij . (v_j - v_i), in FP64 like the FP32 path's environment
// rows: with d = |r|, s = sw(d)/d, q = s/d, R = ((s - avg0)/std0,
// (q r_a - avg_a)/std_a): s' = s_d d', (q r_a)' = q_d d' r_a + q r_a',
// d' = r.r'/d.  (The image shift of r is constant.)
__global__ void k_env_jvp(JvpArgs a) {
  pdl_wait();
  __shared__ double rec[9];
  env_reciprocals(rec, a.dstd, a.atype, a.n, a.rcs, a.rc);
  const long long row = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= (long long)a.n * NP) return;
  float4 out = make_float4(0.f, 0.f, 0.f, 0.f);
  const int j = a.nlist[row];
  if (j >= 0) {
    const int i = (int)(row / NP);
    const CellGrid& g = *a.grid;
    const double rx = mic_near(a.coord[3 * j] - a.coord[3 * i], g.L[0]);
    const double ry = mic_near(a.coord[3 * j + 1] - a.coord[3 * i + 1], g.L[1]);
    const double rz = mic_near(a.coord[3 * j + 2] - a.coord[3 * i + 2], g.L[2]);
    const double vx = a.v[3 * j] - a.v[3 * i], vy = a.v[3 * j + 1] - a.v[3 * i + 1], vz = a.v[3 * j + 2] - a.v[3 * i + 2];
    const double d = sqrt(rx * rx + ry * ry + rz * rz), inv = 1.0 / d;
    const double dd = (rx * vx + ry * vy + rz * vz) * inv;
    const double rcs = a.rcs, rc = a.rc;
    double sw, dsw;
    if (d < rcs) {
      sw = 1.0; dsw = 0.0;
    } else if (d < rc) {
      const double u = (d - rcs) * rec[8];
      sw = u * u * u * (-6.0 * u * u + 15.0 * u - 10.0) + 1.0;
      dsw = -30.0 * u * u * (u - 1.0) * (u - 1.0) * rec[8];
    } else {
      sw = 0.0; dsw = 0.0;
    }
    const double s_d = dsw * inv - sw * inv * inv;
    const double q = sw * inv * inv, q_d = dsw * inv * inv - 2.0 * sw * inv * inv * inv;
    const double* iv = rec + 4 * (i & 1);
    out.x = (float)(s_d * dd * iv[0]);
    out.y = (float)((q_d * dd * rx + q * vx) * iv[1]);
    out.z = (float)((q_d * dd * ry + q * vy) * iv[2]);
    out.w = (float)((q_d * dd * rz + q * vz) * iv[3]);
  }
  reinterpret_cast<float4*>(a.Rd)[row] = out;
}

// The embedding net G = net(s) (1 + Gt[t_i][t_j]), net: 1 -> E0 -> E1 -> E2,
// tanh layers with the residual rule (same width: x + f; double: [x, x] + f),
// input s = R_ij,0, over the packed live rows.  A CTA takes JROWS rows and
// evaluates the activations and their tangents (s' = R'_ij,0).  Mode 0 writes
// G'.  Mode 1 also runs the adjoint from dE/dG and (dE/dG)' and adds the weight
// gradients of both loss terms to grad: with s1, s2 the scales of the energy and
// force terms, the tangents are seeded with s2 s' and s2 (dE/dG)' + s1 dE/dG,
// which (everything being linear in them) makes sum_r in' (x) dz + in (x) dz' the
// sum of s2 times the tangent of the energy's weight gradient and s1 times that
// gradient itself: no pass of its own for the latter.
//
// Activations lie in shared memory as [unit][row]; a thread owns 4 rows x 1 - 4
// units of a layer, its value and tangent sums sharing the weight loads (3
// 16-byte loads for 32 FMAs in the widest layer), and fixed elements of the weight
// gradients, 2 x 4 of W2, whose sums stay in registers until the last block, as do its
// rows' parts of the bias gradients.  Shared-memory wavefronts and scattered loads bind:
// per 582-atom frame 136 us with neighbouring units in one thread (8-way bank conflicts
// in W2's gradient), dE/dG read once more for the skip's adjoint and the bias sums taken
// from shared memory by a few warps; 84 us now.
constexpr int JROWS = 64;
constexpr int JTHREADS = 256;
constexpr int JLD = JROWS + 4;   // row stride of a unit's rows (16-byte aligned)
constexpr int JQ = JROWS / 4;    // row quads

template <int E0, int E1, int E2>
struct JvpEmbedSmem {
  static constexpr int pad4(int x) { return (x + 3) / 4 * 4; }
  static constexpr int L1 = pad4(E1), L2 = pad4(E2), L0 = pad4(E0);
  // packed weights in the parameter vector
  static constexpr int gB0 = E0, gW1 = 2 * E0, gB1 = gW1 + E0 * E1, gW2 = gB1 + E1, gB2 = gW2 + E1 * E2;
  // shared memory (floats)
  static constexpr int W1 = 0, W2 = W1 + E0 * L1, W0 = W2 + E1 * L2, B0 = W0 + L0, B1 = B0 + L0, B2 = B1 + L1,
                       X = B2 + L2, XD = X + JROWS, TP = XD + JROWS;  // TP: the rows' type pairs (int)
  static constexpr int H1 = TP + JROWS, H1D = H1 + E0 * JLD, H2 = H1D + E0 * JLD, H2D = H2 + E1 * JLD;
  static constexpr int FWD_TOTAL = H2D + E1 * JLD;
  // mode 1: the transposes W2^T [E2][L1], W1^T [E1][L0], dz3 and dz3'; once those
  // are used up, dH2, dH2', dz2, dz2' lie over them
  static constexpr int W2T = FWD_TOTAL, W1T = W2T + E2 * L1, Z3 = W1T + E1 * L0, Z3D = Z3 + E2 * JLD;
  static constexpr int DH2 = Z3, DH2D = DH2 + E1 * JLD, DZ2 = DH2D + E1 * JLD, DZ2D = DZ2 + E1 * JLD;
  static constexpr int TOTAL = Z3 + (2 * E2 > 4 * E1 ? 2 * E2 : 4 * E1) * JLD;
  static_assert(TOTAL * 4 <= 227 * 1024, "shared memory");
};

template <int IN, int OUT>
__device__ __forceinline__ int jskip(int o) {  // the skip input of output o, or -1
  return OUT == IN ? o : (OUT == 2 * IN ? (o < IN ? o : o - IN) : -1);
}

__device__ __forceinline__ float4 jld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void jst4(float* p, const float* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}

// z[u][o] += sum_k in[k][r + u] W[k][unit o], u < 4, o < OC, and likewise zd from ind.
// The units are c + o, or with HALF c, c + 1, c + HALF, c + HALF + 1.
template <int K, int OC, int LDW, int HALF = 0>
__device__ __forceinline__ void jtile(const float* in, const float* ind, const float* W, int r, int c, float (&z)[4][OC],
                                      float (&zd)[4][OC]) {
#pragma unroll 4
  for (int k = 0; k < K; ++k) {
    const float4 h4 = jld4(in + k * JLD + r), d4 = jld4(ind + k * JLD + r);
    const float h[4] = {h4.x, h4.y, h4.z, h4.w}, d[4] = {d4.x, d4.y, d4.z, d4.w};
    float w[OC];
    if constexpr (HALF > 0) {
      const float2 x = *reinterpret_cast<const float2*>(W + k * LDW + c);
      const float2 y = *reinterpret_cast<const float2*>(W + k * LDW + c + HALF);
      w[0] = x.x; w[1] = x.y; w[2] = y.x; w[3] = y.y;
    } else if constexpr (OC == 4) {
      const float4 w4 = jld4(W + k * LDW + c);
      w[0] = w4.x; w[1] = w4.y; w[2] = w4.z; w[3] = w4.w;
    } else {
#pragma unroll
      for (int o = 0; o < OC; ++o) w[o] = W[k * LDW + c + o];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int o = 0; o < OC; ++o) {
        z[u][o] = fmaf(h[u], w[o], z[u][o]);
        zd[u][o] = fmaf(d[u], w[o], zd[u][o]);
      }
  }
}

// acc[i][j] += sum over the block's rows of a'[i] b[j] + a[i] b'[j] (units a0 + i,
// b0 + j BS of the [unit][row] arrays; neighbouring threads take neighbouring b0, whose
// rows are JLD apart: 16-byte loads without bank conflicts).
template <int I, int J, int BS>
__device__ __forceinline__ void jouter(const float* A, const float* AD, const float* B, const float* BD, int a0, int b0,
                                       float (&acc)[I][J]) {
#pragma unroll 2
  for (int r = 0; r < JROWS; r += 4) {
    float a[I][4], ad[I][4];
#pragma unroll
    for (int i = 0; i < I; ++i) {
      const float4 x = jld4(A + (a0 + i) * JLD + r), y = jld4(AD + (a0 + i) * JLD + r);
      a[i][0] = x.x; a[i][1] = x.y; a[i][2] = x.z; a[i][3] = x.w;
      ad[i][0] = y.x; ad[i][1] = y.y; ad[i][2] = y.z; ad[i][3] = y.w;
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const float4 x = jld4(B + (b0 + j * BS) * JLD + r), y = jld4(BD + (b0 + j * BS) * JLD + r);
      const float b[4] = {x.x, x.y, x.z, x.w}, bd[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
      for (int i = 0; i < I; ++i)
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[i][j] = fmaf(ad[i][u], b[u], fmaf(a[i][u], bd[u], acc[i][j]));
    }
  }
}

template <int E0, int E1, int E2, int MODE>
__global__ void __launch_bounds__(JTHREADS) k_embed_jvp(JvpArgs a, float* __restrict__ grad,
                                                         const float* __restrict__ scales) {
  pdl_wait();
  using S = JvpEmbedSmem<E0, E1, E2>;
  static_assert(E1 % 2 == 0 && E1 == 2 * E0 && E2 == 2 * E1, "register tiles");
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x;
  for (int t = tid; t < E0 * E1; t += JTHREADS) sm[S::W1 + (t / E1) * S::L1 + t % E1] = a.w[S::gW1 + t];
  for (int t = tid; t < E1 * E2; t += JTHREADS) sm[S::W2 + (t / E2) * S::L2 + t % E2] = a.w[S::gW2 + t];
  for (int t = tid; t < E0; t += JTHREADS) {
    sm[S::W0 + t] = a.w[t];
    sm[S::B0 + t] = a.w[S::gB0 + t];
  }
  for (int t = tid; t < E1; t += JTHREADS) sm[S::B1 + t] = a.w[S::gB1 + t];
  for (int t = tid; t < E2; t += JTHREADS) sm[S::B2 + t] = a.w[S::gB2 + t];
  float s1 = 0.f, s2 = 1.f;
  if (MODE == 1) {
    s1 = scales[0];
    s2 = scales[1];
    for (int t = tid; t < E1 * E2; t += JTHREADS) sm[S::W2T + (t % E2) * S::L1 + t / E2] = a.w[S::gW2 + t];
    for (int t = tid; t < E0 * E1; t += JTHREADS) sm[S::W1T + (t % E1) * S::L0 + t / E1] = a.w[S::gW1 + t];
  }
  // this thread's elements of the weight gradients: N2 tasks of 2 x 4 of W2, N1 of
  // 1 x 2 of W1; and its rows' part of the others (NH tasks of 4 rows x 2 units of
  // layers 2 and 3: b2, b1; N0 of 4 rows x 1 unit of layer 1: W0, b0)
  constexpr int T2 = (E1 / 2) * (E2 / 4), T1 = E0 * (E1 / 2), TH = JQ * (E1 / 2), T0 = JQ * E0;
  constexpr int N2 = (T2 + JTHREADS - 1) / JTHREADS, N1 = (T1 + JTHREADS - 1) / JTHREADS,
                NH = (TH + JTHREADS - 1) / JTHREADS, N0 = (T0 + JTHREADS - 1) / JTHREADS;
  float g2[N2][2][4] = {}, g1[N1][1][2] = {}, gb2[NH][4] = {}, gb1[NH][2] = {}, g0[N0][2] = {};
  const int* pair = reinterpret_cast<const int*>(sm + S::TP);
  const int nrows = a.row_off[a.n];
  for (int p0 = blockIdx.x * JROWS; p0 < nrows; p0 += gridDim.x * JROWS) {
    const int cnt = min(JROWS, nrows - p0);
    __syncthreads();  // the previous block is done with the activations
    for (int r = tid; r < JROWS; r += JTHREADS) {
      const int rg = r < cnt ? a.rowmap[p0 + r] : 0;
      sm[S::X + r] = r < cnt ? a.R[(size_t)rg * 4] : 0.f;
      sm[S::XD + r] = r < cnt ? (MODE == 1 ? s2 : 1.f) * a.Rd[(size_t)rg * 4] : 0.f;
      reinterpret_cast<int*>(sm + S::TP)[r] = r < cnt ? a.atype[rg / NP] * a.ntypes + a.atype[a.nlist[rg]] : 0;
    }
    __syncthreads();
    // layer 1: h1 = tanh(s W0 + b0), h1' = (1 - h1^2) s' W0
    for (int idx = tid; idx < JROWS * E0; idx += JTHREADS) {
      const int r = idx % JROWS, p = idx / JROWS;
      const float b0 = a.b0t ? a.b0t[(size_t)pair[r] * E0 + p] : sm[S::B0 + p];
      const float h = tanhf(fmaf(sm[S::X + r], sm[S::W0 + p], b0));
      sm[S::H1 + p * JLD + r] = h;
      sm[S::H1D + p * JLD + r] = (1.f - h * h) * sm[S::XD + r] * sm[S::W0 + p];
    }
    __syncthreads();
    // layer 2: H2 = skip(h1) + tanh(h1 W1 + b1), and its tangent
    for (int task = tid; task < JQ * (E1 / 2); task += JTHREADS) {
      const int r = (task % JQ) * 4, c = (task / JQ) * 2;
      float z[4][2], zd[4][2] = {};
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int o = 0; o < 2; ++o) z[u][o] = sm[S::B1 + c + o];
      jtile<E0, 2, S::L1>(sm + S::H1, sm + S::H1D, sm + S::W1, r, c, z, zd);
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        const int sk = jskip<E0, E1>(c + o);
        float h[4], hd[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float t = tanhf(z[u][o]);
          h[u] = (sk >= 0 ? sm[S::H1 + sk * JLD + r + u] : 0.f) + t;
          hd[u] = (sk >= 0 ? sm[S::H1D + sk * JLD + r + u] : 0.f) + (1.f - t * t) * zd[u][o];
        }
        jst4(sm + S::H2 + (c + o) * JLD + r, h);
        jst4(sm + S::H2D + (c + o) * JLD + r, hd);
      }
    }
    __syncthreads();
    // layer 3: t3 = tanh(H2 W2 + b2), t3'; mode 0: G' out; mode 1: its adjoint with
    // g = dE/dG (1 + Gt): dz3 = g (1 - t3^2), dz3' = g' (1 - t3^2) - 2 g t3 t3'.  There a
    // thread's units are c, c + 1 and those E1 further, so that it holds skip^T(g) for
    // its 4 rows x 2 units of dH2, the start of the sums dh
    float dh[NH][4][2], dhd[NH][4][2];
#pragma unroll
    for (int k = 0; k < NH; ++k) {
      const int task = tid + k * JTHREADS;
      if (task >= TH) continue;
      const int r = (task % JQ) * 4, c = (task / JQ) * (MODE == 0 ? 4 : 2);
      float z[4][4], zd[4][4] = {};
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int o = 0; o < 4; ++o) z[u][o] = sm[S::B2 + c + (MODE == 0 || o < 2 ? o : E1 + o - 2)];
      jtile<E1, 4, S::L2, MODE == 0 ? 0 : E1>(sm + S::H2, sm + S::H2D, sm + S::W2, r, c, z, zd);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool live = r + u < cnt;
        const size_t at = (size_t)(p0 + r + u) * a.m1 + c;
        if (MODE == 0) {
          const float4 f4 = jld4(a.Gt + (size_t)pair[r + u] * E2 + c);
          const float f[4] = {1.f + f4.x, 1.f + f4.y, 1.f + f4.z, 1.f + f4.w};
          float gd[4];
#pragma unroll
          for (int o = 0; o < 4; ++o) {
            const int sk = jskip<E1, E2>(c + o);
            const float t = tanhf(z[u][o]);
            gd[o] = ((sk >= 0 ? sm[S::H2D + sk * JLD + r + u] : 0.f) + (1.f - t * t) * zd[u][o]) * f[o];
          }
          if (live) jst4(a.Gd + at, gd);
        } else {
          float q[4] = {}, qd[4] = {}, f[4];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float2 x = *reinterpret_cast<const float2*>(a.Gt + (size_t)pair[r + u] * E2 + c + h * E1);
            f[2 * h] = 1.f + x.x; f[2 * h + 1] = 1.f + x.y;
            if (live) {
              const float2 y = *reinterpret_cast<const float2*>(a.dG + at + h * E1);
              const float2 yd = *reinterpret_cast<const float2*>(a.dGd + at + h * E1);
              q[2 * h] = y.x; q[2 * h + 1] = y.y;
              qd[2 * h] = yd.x; qd[2 * h + 1] = yd.y;
            }
          }
          dh[k][u][0] = dh[k][u][1] = dhd[k][u][0] = dhd[k][u][1] = 0.f;
#pragma unroll
          for (int o = 0; o < 4; ++o) {
            const float g = q[o] * f[o], gd = fmaf(s2, qd[o], s1 * q[o]) * f[o];
            const float t = tanhf(z[u][o]), td = (1.f - t * t) * zd[u][o];
            z[u][o] = g * (1.f - t * t);
            zd[u][o] = gd * (1.f - t * t) - 2.f * g * t * td;
            gb2[k][o] += zd[u][o];
            dh[k][u][o & 1] += g;
            dhd[k][u][o & 1] += gd;
          }
        }
      }
      if (MODE == 1) {
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          const float v[4] = {z[0][o], z[1][o], z[2][o], z[3][o]}, vd[4] = {zd[0][o], zd[1][o], zd[2][o], zd[3][o]};
          const int cu = c + (o & 1) + (o >> 1) * E1;
          jst4(sm + S::Z3 + cu * JLD + r, v);
          jst4(sm + S::Z3D + cu * JLD + r, vd);
        }
      }
    }
    if (MODE == 0) continue;
    __syncthreads();
    // dH2 = skip^T(g) + W2 dz3 and its tangent, kept in registers until W2's
    // gradient has read dz3
#pragma unroll
    for (int k = 0; k < NH; ++k) {
      const int task = tid + k * JTHREADS;
      if (task >= TH) continue;
      const int r = (task % JQ) * 4, b = (task / JQ) * 2;
      jtile<E2, 2, S::L1>(sm + S::Z3, sm + S::Z3D, sm + S::W2T, r, b, dh[k], dhd[k]);
    }
#pragma unroll
    for (int k = 0; k < N2; ++k) {
      const int task = tid + k * JTHREADS;
      if (task < T2) jouter<2, 4, E2 / 4>(sm + S::H2, sm + S::H2D, sm + S::Z3, sm + S::Z3D, 2 * (task / (E2 / 4)), task % (E2 / 4), g2[k]);
    }
    __syncthreads();
    // dz2 = dH2 (1 - t2^2) with t2 = H2 - skip(h1), over dz3's place
#pragma unroll
    for (int k = 0; k < NH; ++k) {
      const int task = tid + k * JTHREADS;
      if (task >= TH) continue;
      const int r = (task % JQ) * 4, b = (task / JQ) * 2;
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        const int sk = jskip<E0, E1>(b + o);
        float d[4], dd[4], e[4], ed[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float t = sm[S::H2 + (b + o) * JLD + r + u] - (sk >= 0 ? sm[S::H1 + sk * JLD + r + u] : 0.f);
          const float td = sm[S::H2D + (b + o) * JLD + r + u] - (sk >= 0 ? sm[S::H1D + sk * JLD + r + u] : 0.f);
          d[u] = dh[k][u][o];
          dd[u] = dhd[k][u][o];
          e[u] = d[u] * (1.f - t * t);
          ed[u] = dd[u] * (1.f - t * t) - 2.f * d[u] * t * td;
          gb1[k][o] += ed[u];
        }
        jst4(sm + S::DH2 + (b + o) * JLD + r, d);
        jst4(sm + S::DH2D + (b + o) * JLD + r, dd);
        jst4(sm + S::DZ2 + (b + o) * JLD + r, e);
        jst4(sm + S::DZ2D + (b + o) * JLD + r, ed);
      }
    }
    __syncthreads();
    // dh1 = W1 dz2 + skip^T(dH2), dz1 = dh1 (1 - h1^2)
#pragma unroll
    for (int k = 0; k < N0; ++k) {
      const int task = tid + k * JTHREADS;
      if (task >= T0) continue;
      const int r = (task % JQ) * 4, p = task / JQ;
      float d1[4][1] = {}, d1d[4][1] = {};
      jtile<E1, 1, S::L0>(sm + S::DZ2, sm + S::DZ2D, sm + S::W1T, r, p, d1, d1d);
      float e[4], ed[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float d = d1[u][0], dd = d1d[u][0];
#pragma unroll
        for (int b = p; b < E1; b += E0) {
          d += sm[S::DH2 + b * JLD + r + u];
          dd += sm[S::DH2D + b * JLD + r + u];
        }
        const float h = sm[S::H1 + p * JLD + r + u], hd = sm[S::H1D + p * JLD + r + u];
        e[u] = d * (1.f - h * h);
        ed[u] = dd * (1.f - h * h) - 2.f * d * h * hd;
        g0[k][0] += sm[S::XD + r + u] * e[u] + sm[S::X + r + u] * ed[u];
        g0[k][1] += ed[u];
      }
    }
    // W1's gradient (dz2) does not wait for dz1
#pragma unroll
    for (int k = 0; k < N1; ++k) {
      const int task = tid + k * JTHREADS;
      if (task < T1) jouter<1, 2, E1 / 2>(sm + S::H1, sm + S::H1D, sm + S::DZ2, sm + S::DZ2D, task / (E1 / 2), task % (E1 / 2), g1[k]);
    }
  }
  if (MODE == 0) return;
#pragma unroll
  for (int k = 0; k < N2; ++k) {
    const int task = tid + k * JTHREADS;
    if (task < T2)
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          atomicAdd(grad + S::gW2 + (2 * (task / (E2 / 4)) + i) * E2 + task % (E2 / 4) + j * (E2 / 4), g2[k][i][j]);
  }
#pragma unroll
  for (int k = 0; k < N1; ++k) {
    const int task = tid + k * JTHREADS;
    if (task < T1)
#pragma unroll
      for (int j = 0; j < 2; ++j) atomicAdd(grad + S::gW1 + (task / (E1 / 2)) * E1 + task % (E1 / 2) + j * (E1 / 2), g1[k][0][j]);
  }
  // the JQ threads of a unit are neighbouring lanes
  static_assert(JQ == 16 && JTHREADS % 32 == 0, "half warps");
  auto unit_sum = [&](float v, bool live, int at) {
#pragma unroll
    for (int o = JQ / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (live && tid % JQ == 0) atomicAdd(grad + at, v);
  };
#pragma unroll
  for (int k = 0; k < NH; ++k) {
    const int task = tid + k * JTHREADS, c = (task / JQ) * 2;
#pragma unroll
    for (int o = 0; o < 4; ++o) unit_sum(gb2[k][o], task < TH, S::gB2 + c + (o & 1) + (o >> 1) * E1);
#pragma unroll
    for (int o = 0; o < 2; ++o) unit_sum(gb1[k][o], task < TH, S::gB1 + c + o);
  }
#pragma unroll
  for (int k = 0; k < N0; ++k) {
    const int task = tid + k * JTHREADS;
    unit_sum(g0[k][0], task < T0, task / JQ);
    unit_sum(g0[k][1], task < T0, E0 + task / JQ);
  }
}

// T' = (R'^T G + R^T G') / sel and D' = T'^T T_< + T^T T'_< (the type row of
// X is constant).  One CTA per atom; a thread takes a column of G and G' and every
// (JDESC_T / m1)-th row, for all four columns of R: 582 atoms 30.5 -> 12.5 us against a
// thread per element of T', which read G four times over.
constexpr int JDESC_T = 256;
__global__ void __launch_bounds__(JDESC_T) k_desc_jvp_fwd(JvpArgs a) {
  pdl_wait();
  extern __shared__ float sm[];
  const int m1 = a.m1, ax = a.axis;
  float* Ts = sm;            // [4][m1]
  float* Tds = Ts + 4 * m1;  // [4][m1]
  float* part = Tds + 4 * m1;  // [parts][4][m1]
  const int atom = blockIdx.x, parts = JDESC_T / m1;
  const int nn = a.nnei[atom];
  const size_t base = (size_t)atom * NP, gbase = a.row_off[atom];
  const float inv_sel = 1.0f / (float)a.sel;
  const int p = threadIdx.x % m1, h = threadIdx.x / m1;
  if (h < parts) {
    const float4* R = reinterpret_cast<const float4*>(a.R) + base;
    const float4* Rd = reinterpret_cast<const float4*>(a.Rd) + base;
    float v[4] = {};
#pragma unroll 8
    for (int s = h; s < nn; s += parts) {
      const float4 r = R[s], rd = Rd[s];
      const float g = a.G[(gbase + s) * m1 + p], gd = a.Gd[(gbase + s) * m1 + p];
      v[0] = fmaf(r.x, gd, fmaf(rd.x, g, v[0]));
      v[1] = fmaf(r.y, gd, fmaf(rd.y, g, v[1]));
      v[2] = fmaf(r.z, gd, fmaf(rd.z, g, v[2]));
      v[3] = fmaf(r.w, gd, fmaf(rd.w, g, v[3]));
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) part[(4 * h + c) * m1 + p] = v[c];
  }
  for (int t = threadIdx.x; t < 4 * m1; t += JDESC_T) Ts[t] = a.T[(size_t)atom * 4 * m1 + t];
  __syncthreads();
  for (int t = threadIdx.x; t < 4 * m1; t += JDESC_T) {
    float v = 0.f;
    for (int k = 0; k < parts; ++k) v += part[4 * k * m1 + t];
    Tds[t] = v * inv_sel;
    a.Td[(size_t)atom * 4 * m1 + t] = v * inv_sel;
  }
  __syncthreads();
  float* xd = a.Xd + (size_t)atom * a.fit_in;
  for (int idx = threadIdx.x; idx < m1 * ax; idx += JDESC_T) {
    const int q = idx / ax, b = idx % ax;
    float d = 0.f;
#pragma unroll
    for (int c = 0; c < 4; ++c) d += Tds[c * m1 + q] * Ts[c * m1 + b] + Ts[c * m1 + q] * Tds[c * m1 + b];
    xd[idx] = d;
  }
  for (int t = m1 * ax + threadIdx.x; t < a.fit_in; t += JDESC_T) xd[t] = 0.f;
}

// dT = (dD T_< + [p < axis] dD^T T) / sel as in the descriptor adjoint, its
// tangent by the product rule, and (dE/dG)' = R' dT + R dT'.  The sums over all columns
// of the first axis ones are spread over the block, and a thread keeps its column of dT
// and dT' in registers over its rows: 582 atoms 21.4 -> 14.4 us.
__global__ void __launch_bounds__(JDESC_T) k_desc_jvp_bwd(JvpArgs a) {
  pdl_wait();
  extern __shared__ float sm[];
  const int m1 = a.m1, ax = a.axis;
  float* Ts = sm;
  float* Tds = Ts + 4 * m1;
  float* dTs = Tds + 4 * m1;
  float* dTds = dTs + 4 * m1;
  float* dD = dTds + 4 * m1;  // [m1][axis]
  float* dDd = dD + m1 * ax;
  float* part = dDd + m1 * ax;  // [2][JDESC_T]
  const int atom = blockIdx.x;
  const int nn = a.nnei[atom];
  const size_t base = (size_t)atom * NP, gbase = a.row_off[atom];
  const float inv_sel = 1.0f / (float)a.sel;
  for (int t = threadIdx.x; t < 4 * m1; t += JDESC_T) {
    Ts[t] = a.T[(size_t)atom * 4 * m1 + t];
    Tds[t] = a.Td[(size_t)atom * 4 * m1 + t];
  }
  for (int t = threadIdx.x; t < m1 * ax; t += JDESC_T) {
    dD[t] = a.dX[(size_t)atom * a.fit_in + t];
    dDd[t] = a.dXd[(size_t)atom * a.fit_in + t];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 4 * m1; t += JDESC_T) {
    const int c = t / m1, p = t % m1;
    float v = 0.f, vd = 0.f;
    for (int b = 0; b < ax; ++b) {
      v = fmaf(dD[p * ax + b], Ts[c * m1 + b], v);
      vd += dDd[p * ax + b] * Ts[c * m1 + b] + dD[p * ax + b] * Tds[c * m1 + b];
    }
    dTs[t] = v;
    dTds[t] = vd;
  }
  // the axis columns' other term: element e = (c, p < axis), pieces of its sum over q
  for (int e0 = 0; e0 < 4 * ax; e0 += JDESC_T) {
    const int ne = min(4 * ax - e0, JDESC_T), pieces = JDESC_T / ne;
    const int e = e0 + threadIdx.x % ne, k = threadIdx.x / ne, c = e / ax, p = e % ax;
    float v = 0.f, vd = 0.f;
    if (k < pieces)
      for (int q = k; q < m1; q += pieces) {
        v = fmaf(dD[q * ax + p], Ts[c * m1 + q], v);
        vd += dDd[q * ax + p] * Ts[c * m1 + q] + dD[q * ax + p] * Tds[c * m1 + q];
      }
    part[threadIdx.x] = v;
    part[JDESC_T + threadIdx.x] = vd;
    __syncthreads();
    if (threadIdx.x < ne) {
      for (int i = 1; i < pieces; ++i) {
        v += part[i * ne + threadIdx.x];
        vd += part[JDESC_T + i * ne + threadIdx.x];
      }
      dTs[c * m1 + p] += v;
      dTds[c * m1 + p] += vd;
    }
    __syncthreads();
  }
  const int parts = JDESC_T / m1, p = threadIdx.x % m1, h = threadIdx.x / m1;
  if (h >= parts) return;
  float d[4], dd[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    d[c] = dTs[c * m1 + p] * inv_sel;
    dd[c] = dTds[c * m1 + p] * inv_sel;
  }
  const float4* R = reinterpret_cast<const float4*>(a.R) + base;
  const float4* Rd = reinterpret_cast<const float4*>(a.Rd) + base;
#pragma unroll 4
  for (int s = h; s < nn; s += parts) {
    const float4 r = R[s], rd = Rd[s];
    float v = rd.x * d[0] + r.x * dd[0];
    v += rd.y * d[1] + r.y * dd[1];
    v += rd.z * d[2] + r.z * dd[2];
    v += rd.w * d[3] + r.w * dd[3];
    a.dGd[(gbase + s) * m1 + p] = v;
  }
}

__global__ void k_tanh_jvp(const float* __restrict__ Zd, const float* __restrict__ H, const float* __restrict__ Hprev,
                           const float* __restrict__ Hprevd, float* __restrict__ Hd, long long count) {
  pdl_wait();
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= count) return;
  const float t = Hprev ? H[k] - Hprev[k] : H[k];
  Hd[k] = (1.f - t * t) * Zd[k] + (Hprevd ? Hprevd[k] : 0.f);
}

__global__ void k_tanh_bwd_jvp(const float* __restrict__ dH, const float* __restrict__ dHd, const float* __restrict__ H,
                               const float* __restrict__ Hprev, const float* __restrict__ Hd,
                               const float* __restrict__ Hprevd, float* __restrict__ dZd, long long count) {
  pdl_wait();
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= count) return;
  const float t = Hprev ? H[k] - Hprev[k] : H[k];
  const float td = Hprevd ? Hd[k] - Hprevd[k] : Hd[k];
  const float d = dH[k];
  dZd[k] = (dHd ? dHd[k] * (1.f - t * t) : 0.f) - 2.f * d * t * td;
}

__global__ void k_adam(float* __restrict__ theta, float* __restrict__ g, float* __restrict__ m1, float* __restrict__ m2,
                       int n, float lr, float b1, float b2, float eps, float bc1, float bc2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float a = b1 * m1[i] + (1.f - b1) * gi;
  const float b = b2 * m2[i] + (1.f - b2) * gi * gi;
  m1[i] = a;
  m2[i] = b;
  theta[i] -= lr * (a / bc1) / (sqrtf(b / bc2) + eps);
  g[i] = 0.f;
}

__global__ void k_transpose(const float* __restrict__ W, int R, int C, float* __restrict__ WT) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= R * C) return;
  const int r = t / C, c = t % C;
  WT[(size_t)c * R + r] = W[t];
}

__global__ void k_scale_copy(const float* __restrict__ src, float* __restrict__ dst, int n, float s) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) dst[t] = s * src[t];
}

__global__ void k_add_rows(const float* __restrict__ rows, const float* __restrict__ vec, int nrows, int width,
                           float* __restrict__ out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < nrows * width) out[t] = rows[t] + vec[t % width];
}

static int blocks(long long n, int t) { return (int)((n + t - 1) / t); }

void launch_fit_grad(const float* A, const float* Ad, const float* dZ, const float* dZd, float* C, float* c, int I,
                     int O, int N, const float* scales, cudaStream_t st) {
  if (N <= 0 || I <= 0 || O <= 0) return;
  // slices of the rows: 256 rows or more each in large frames; in small ones down
  // to 32, until the grid holds two blocks per SM (582 atoms: 2 slices -> 17, 53 -> 11 us
  // for one product)
  const int tiles = blocks(I, 64) * blocks(O, 64);
  const int splits = std::min(64, std::max({1, N / 256, std::min(N / 32, 304 / tiles)}));
  // whole groups of WG_ROWS
  const int chunk = blocks(blocks(N, splits), WG_ROWS) * WG_ROWS;
  launch_pdl(k_fit_grad, dim3(blocks(I, 64), blocks(O, 64), blocks(N, chunk)), 256, 0, st, A, Ad, dZ, dZd, C, c, I, O,
             N, chunk, scales);
  note_launch();
}

void launch_head_grad(const float* H, const float* Hd, const int* atype, float* g_wout, float* g_bout, float* g_ebias,
                      int O, int N, int ntypes, const float* scales, float out_scale, cudaStream_t st) {
  if (N <= 0 || O <= 0) return;
  const int splits = std::min(128, std::max(1, N / 32));
  const int chunk = (N + splits - 1) / splits;
  launch_pdl(k_head_grad, dim3(blocks(O, 128), splits + 2), 128, 0, st, H, Hd, atype, g_wout, g_bout, g_ebias, O, N,
             ntypes, chunk, scales, out_scale);
  note_launch();
}

void launch_train_prep(int n, const double* energy, double e_ref, const double* force, const double* force_ref,
                       double pe, double pf, double* v, double* loss, float* scales, cudaStream_t st) {
  launch_pdl(k_train_prep, 1, 1024, 0, st, n, energy, e_ref, force, force_ref, pe, pf, v, loss, scales);
  note_launch();
}

void launch_env_jvp(const JvpArgs& a, cudaStream_t st) {
  const long long rows = (long long)a.n * NP;
  if (rows == 0) return;
  launch_pdl(k_env_jvp, (unsigned)((rows + 2 * NP - 1) / (2 * NP)), 2 * NP, 0, st, a);
  note_launch();
}

template <int E0, int E1, int E2, int MODE>
static void embed_jvp_launch(const JvpArgs& a, float* grad, const float* scales, cudaStream_t st) {
  using S = JvpEmbedSmem<E0, E1, E2>;
  const size_t smem = sizeof(float) * (MODE == 1 ? S::TOTAL : S::FWD_TOTAL);
  cudaFuncSetAttribute(k_embed_jvp<E0, E1, E2, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int sms = 0, dev = 0, per_sm = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_embed_jvp<E0, E1, E2, MODE>, JTHREADS, smem);
  // at most n * NP rows
  const int grid = std::min(a.n * (NP / JROWS), std::max(1, per_sm) * std::max(1, sms));
  launch_pdl(k_embed_jvp<E0, E1, E2, MODE>, grid, JTHREADS, smem, st, a, grad, scales);
  note_launch();
}

template <int MODE>
static bool embed_jvp_dispatch(const JvpArgs& a, const int* w, float* grad, const float* scales, cudaStream_t st) {
  if (a.n == 0) return true;
  if (w[0] == 16 && w[1] == 32 && w[2] == 64) { embed_jvp_launch<16, 32, 64, MODE>(a, grad, scales, st); return true; }
  if (w[0] == 25 && w[1] == 50 && w[2] == 100) { embed_jvp_launch<25, 50, 100, MODE>(a, grad, scales, st); return true; }
  if (w[0] == 32 && w[1] == 64 && w[2] == 128) { embed_jvp_launch<32, 64, 128, MODE>(a, grad, scales, st); return true; }
  return false;
}

bool launch_embed_jvp(const JvpArgs& a, const int* w, cudaStream_t st) {
  return embed_jvp_dispatch<0>(a, w, nullptr, nullptr, st);
}

bool launch_embed_grad(const JvpArgs& a, const int* w, float* grad, const float* scales, cudaStream_t st) {
  return embed_jvp_dispatch<1>(a, w, grad, scales, st);
}

void launch_desc_jvp_fwd(const JvpArgs& a, cudaStream_t st) {
  if (a.n == 0) return;
  const size_t smem = sizeof(float) * (8 * a.m1 + 4 * JDESC_T);
  launch_pdl(k_desc_jvp_fwd, a.n, JDESC_T, smem, st, a);
  note_launch();
}

void launch_desc_jvp_bwd(const JvpArgs& a, cudaStream_t st) {
  if (a.n == 0) return;
  const size_t smem = sizeof(float) * (16 * a.m1 + 2 * a.m1 * a.axis + 2 * JDESC_T);
  if (smem > 48 * 1024) cudaFuncSetAttribute(k_desc_jvp_bwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  launch_pdl(k_desc_jvp_bwd, a.n, JDESC_T, smem, st, a);
  note_launch();
}

void launch_tanh_jvp(const float* Zd, const float* H, const float* Hprev, const float* Hprevd, float* Hd,
                     long long count, cudaStream_t st) {
  if (count <= 0) return;
  launch_pdl(k_tanh_jvp, (unsigned)((count + 255) / 256), 256, 0, st, Zd, H, Hprev, Hprevd, Hd, count);
  note_launch();
}

void launch_tanh_bwd_jvp(const float* dH, const float* dHd, const float* H, const float* Hprev, const float* Hd,
                         const float* Hprevd, float* dZd, long long count, cudaStream_t st) {
  if (count <= 0) return;
  launch_pdl(k_tanh_bwd_jvp, (unsigned)((count + 255) / 256), 256, 0, st, dH, dHd, H, Hprev, Hd, Hprevd, dZd, count);
  note_launch();
}

void launch_adam(float* theta, float* g, float* m1, float* m2, int n, float lr, float b1, float b2, float eps,
                 float bc1, float bc2, cudaStream_t st) {
  if (n <= 0) return;
  k_adam<<<blocks(n, 256), 256, 0, st>>>(theta, g, m1, m2, n, lr, b1, b2, eps, bc1, bc2);
  note_launch();
}

void launch_transpose(const float* W, int R, int C, float* WT, cudaStream_t st) {
  if (R * C <= 0) return;
  k_transpose<<<blocks((long long)R * C, 256), 256, 0, st>>>(W, R, C, WT);
  note_launch();
}

void launch_scale_copy(const float* src, float* dst, int n, float s, cudaStream_t st) {
  if (n <= 0) return;
  k_scale_copy<<<blocks(n, 256), 256, 0, st>>>(src, dst, n, s);
  note_launch();
}

void launch_add_rows(const float* rows, const float* vec, int nrows, int width, float* out, cudaStream_t st) {
  if (nrows * width <= 0) return;
  k_add_rows<<<blocks((long long)nrows * width, 256), 256, 0, st>>>(rows, vec, nrows, width, out);
  note_launch();
}

}  // namespace dpa1
