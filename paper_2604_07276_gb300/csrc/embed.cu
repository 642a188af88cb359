// The FP32 SIMT embedding net (stages a5, a13) over live neighbour rows:
// net_s = 1 -> E0 -> E1 -> E2 (tanh, residual rule), G0 = net_s * (1 + Gt),
// and its adjoint dR[:, 0] += d net_s / dx . (dG0 * (1 + Gt)).
//
// A thread owns one live row; the rows come from the list of all atoms' live
// rows, so no lane works on padding.  The row's layer-1 and layer-2 units stay
// in its registers (and, where an index runs, in its own shared-memory column),
// the weights are read from shared memory as 16-byte broadcasts.  The products
// run on pairs of outputs (fma.rn.f32x2: two FP32 FMAs, each rounded as fmaf):
// the bound is shared memory's data path (two wavefronts for 16 bytes to every lane,
// 80 - 87 % busy), then the issue of FMAs and tanhf (E0 + E1 + E2 per row and
// direction).  Two rows per thread, which halve the weight loads, leave 12 warps on an
// SM: 272 us against 283 forward, the adjoint spills.  Every product sums in the order
// of a plain loop over its inputs.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace dpa1 {

namespace {

constexpr int ER_T = 128;  // threads (rows) per tile
constexpr int ER_B = 8;    // outputs per weight pass

// A pair of FP32 values in one 64-bit register, and its FMA.
using f2 = unsigned long long;
__device__ __forceinline__ f2 f2_pack(float x, float y) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void f2_unpack(f2 v, float& x, float& y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v)); }
__device__ __forceinline__ void f2_fma(f2& acc, f2 a, f2 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b)); }
// four consecutive floats of shared memory as two pairs
__device__ __forceinline__ ulonglong2 f2_ld4(const float* p) { return *reinterpret_cast<const ulonglong2*>(p); }

template <int E0, int E1, int E2>
struct RowNet {
  static constexpr int P1 = (E1 + ER_B - 1) / ER_B * ER_B, P2 = (E2 + ER_B - 1) / ER_B * ER_B;  // padded row strides
  // packed global weights
  static constexpr int gB0 = E0, gW1 = 2 * E0, gB1 = gW1 + E0 * E1, gW2 = gB1 + E1, gB2 = gW2 + E1 * E2;
  // shared memory (floats)
  static constexpr int W1 = 0, W2 = W1 + E0 * P1, B1 = W2 + E1 * P2, B2 = B1 + P1, W0 = B2 + P2, B0 = W0 + E0,
                       H1 = (B0 + E0 + 3) / 4 * 4, H2 = H1 + E0 * ER_T, FWD = H2 + E1 * ER_T;
  // the adjoint also holds the transposes, rows padded to 4: W2^T [E2][Q1], W1^T [E1][Q0]
  static constexpr int Q1 = (E1 + 3) / 4 * 4, Q0 = (E0 + 3) / 4 * 4;
  static constexpr int W2T = FWD, W1T = W2T + P2 * Q1, BWD = W1T + E1 * Q0;
  // CTAs per SM that registers and shared memory (228 KB) allow
  static constexpr int F_CTAS = E1 <= 32 ? 4 : (E1 <= 50 ? 3 : 2), B_CTAS = E1 <= 32 ? 3 : (E1 <= 50 ? 2 : 1);
  static_assert(F_CTAS * (FWD * 4 + 1024) <= 228 * 1024 && B_CTAS * (BWD * 4 + 1024) <= 228 * 1024, "shared memory");
};

template <int IN, int OUT>
__host__ __device__ constexpr bool doubles() {
  return OUT == 2 * IN;
}

template <int E0, int E1, int E2>
__device__ __forceinline__ void row_weights(float* sm, const float* __restrict__ w) {
  using N = RowNet<E0, E1, E2>;
  for (int t = threadIdx.x; t < E0 * N::P1; t += ER_T) {
    const int p = t / N::P1, b = t % N::P1;
    sm[N::W1 + t] = b < E1 ? w[N::gW1 + p * E1 + b] : 0.f;
  }
  for (int t = threadIdx.x; t < E1 * N::P2; t += ER_T) {
    const int b = t / N::P2, c = t % N::P2;
    sm[N::W2 + t] = c < E2 ? w[N::gW2 + b * E2 + c] : 0.f;
  }
  for (int t = threadIdx.x; t < N::P1; t += ER_T) sm[N::B1 + t] = t < E1 ? w[N::gB1 + t] : 0.f;
  for (int t = threadIdx.x; t < N::P2; t += ER_T) sm[N::B2 + t] = t < E2 ? w[N::gB2 + t] : 0.f;
  for (int t = threadIdx.x; t < E0; t += ER_T) {
    sm[N::W0 + t] = w[t];
    sm[N::B0 + t] = w[N::gB0 + t];
  }
  __syncthreads();
}

// z[u] = bias[c + u] + sum_k in[k] W[k][c + u], u < 8 (W with row stride LD).  The
// pair (in[k], in[k]) is made here: held as pairs the inputs take twice the registers,
// and the adjoint spilled (16-32-64, 1.36 M rows: 578 -> 508 us).
template <int K, int LD>
__device__ __forceinline__ void row_block(const float* in, const float* W, const float* bias, int c, float* z) {
  const ulonglong2 b0 = f2_ld4(bias + c), b1 = f2_ld4(bias + c + 4);
  f2 acc[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const ulonglong2 w0 = f2_ld4(W + k * LD + c), w1 = f2_ld4(W + k * LD + c + 4);
    const f2 h = f2_pack(in[k], in[k]);
    f2_fma(acc[0], h, w0.x);
    f2_fma(acc[1], h, w0.y);
    f2_fma(acc[2], h, w1.x);
    f2_fma(acc[3], h, w1.y);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) f2_unpack(acc[q], z[2 * q], z[2 * q + 1]);
}

// Layers 1 and 2 of this thread's row: its shared columns H1 and H2 and the
// layer-2 units in h2.
template <int E0, int E1, int E2>
__device__ __forceinline__ void row_front(float* sm, float x, const float* b0t, float* h2) {
  using N = RowNet<E0, E1, E2>;
  float* c1 = sm + N::H1 + threadIdx.x;
  float* c2 = sm + N::H2 + threadIdx.x;
  float h1[E0];
#pragma unroll
  for (int p = 0; p < E0; ++p) {
    const float h = tanhf(fmaf(x, sm[N::W0 + p], b0t ? b0t[p] : sm[N::B0 + p]));
    h1[p] = h;
    c1[p * ER_T] = h;
  }
#pragma unroll 1
  for (int b = 0; b < E1; b += ER_B) {
    float z[ER_B];
    row_block<E0, N::P1>(h1, sm + N::W1, sm + N::B1, b, z);
#pragma unroll
    for (int u = 0; u < ER_B; ++u)
      if (b + u < E1) {
        const int s = b + u < E0 ? b + u : b + u - E0;  // the skip input of a doubling layer
        c2[(b + u) * ER_T] = (doubles<E0, E1>() ? c1[s * ER_T] : 0.f) + tanhf(z[u]);
      }
  }
#pragma unroll
  for (int b = 0; b < E1; ++b) h2[b] = c2[b * ER_T];
}

// Where a list row's data lie: row rg = atom * NP + slot of the per-row
// arrays, and G0 / dE/dG0 as stored (four columns c .. c + 3, c % 4 == 0).
struct RowPos {
  int rg, ti, tj;
  size_t g0;  // of column 0
  int gs;     // distance of consecutive column quads
  __device__ RowPos(const EmbedArgs& a, int p, int nrows) : rg(-1), ti(0), tj(0), g0(0), gs(4) {
    if (p >= nrows) return;
    rg = a.rowmap[p];
    const int atom = rg / NP;
    ti = a.atype[atom];
    tj = a.atype[a.nlist[rg]];
    g0 = a.packed ? (size_t)p * a.m1 : (size_t)atom * NP * a.m1 + (size_t)(rg % NP) * 4;
    gs = a.packed ? 4 : NP * 4;
  }
  __device__ size_t quad(int c) const { return g0 + (size_t)(c >> 2) * gs; }
};

template <int E0, int E1, int E2>
__global__ void __launch_bounds__(ER_T, RowNet<E0, E1, E2>::F_CTAS) k_embed_rows_fwd(EmbedArgs a) {
  pdl_wait();
  using N = RowNet<E0, E1, E2>;
  extern __shared__ __align__(16) float sm[];
  row_weights<E0, E1, E2>(sm, a.w);
  const int nrows = *a.nrows;
  for (int p0 = blockIdx.x * ER_T; p0 < nrows; p0 += gridDim.x * ER_T) {
    const RowPos r(a, p0 + threadIdx.x, nrows);
    const size_t pair = (size_t)r.ti * a.ntypes + r.tj;
    float h2[E1];
    row_front<E0, E1, E2>(sm, r.rg >= 0 ? a.R[(size_t)r.rg * 4] : 0.f, a.b0t ? a.b0t + pair * E0 : nullptr, h2);
    const float4* gt4 = reinterpret_cast<const float4*>(a.Gt + pair * E2);
    const float* c2 = sm + N::H2 + threadIdx.x;
#pragma unroll 1
    for (int c = 0; c < E2; c += ER_B) {
      float z[ER_B];
      row_block<E1, N::P2>(h2, sm + N::W2, sm + N::B2, c, z);
#pragma unroll
      for (int q = 0; q < ER_B; q += 4) {
        if (c + q >= E2) continue;
        const float4 gt = gt4[(c + q) >> 2];
        const float gg[4] = {gt.x, gt.y, gt.z, gt.w};
        float o[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int k = c + q + u;
          const float h3 = (doubles<E1, E2>() ? c2[(k < E1 ? k : k - E1) * ER_T] : 0.f) + tanhf(z[q + u]);
          o[u] = h3 * (1.f + gg[u]);
        }
        if (r.rg >= 0) *reinterpret_cast<float4*>(a.G0 + r.quad(c + q)) = make_float4(o[0], o[1], o[2], o[3]);
      }
    }
  }
}

// dE/dG0 of four columns of a row: read, or with FOLD formed from the row of R and the
// atom's dT as the descriptor's adjoint forms it.
template <bool FOLD>
__device__ __forceinline__ float4 row_dg(const EmbedArgs& a, const RowPos& r, float4 R, const float* dT, int c,
                                         float4 (&t)[4]) {
  if (!FOLD) return *reinterpret_cast<const float4*>(a.dG0 + r.quad(c));
#pragma unroll
  for (int k = 0; k < 4; ++k) t[k] = *reinterpret_cast<const float4*>(dT + k * a.m1 + c);
  float4 v;
  float* vp = &v.x;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float t0 = (&t[0].x)[k], t1 = (&t[1].x)[k], t2 = (&t[2].x)[k], t3 = (&t[3].x)[k];
    vp[k] = R.x * t0 + R.y * t1 + R.z * t2 + R.w * t3;
  }
  return v;
}

// FOLD: no layer lies between the net and the descriptor, so the descriptor's adjoint
// of the row, dG0 = R dT and dR = G0 dT^T, is formed here, G0 from the net's own
// recomputed output: its kernel's pass over G0, and dE/dG0 in memory, fall away
// (16-32-64, 15,668 atoms: 508 us and 182 for the descriptor's adjoint -> 586 and 47 for
// dT alone).  Interleaved layout only, whose descriptor adjoint sums dR over a row's
// columns in this order.
template <int E0, int E1, int E2, bool FOLD>
__global__ void __launch_bounds__(ER_T, RowNet<E0, E1, E2>::B_CTAS) k_embed_rows_bwd(EmbedArgs a) {
  pdl_wait();
  using N = RowNet<E0, E1, E2>;
  extern __shared__ __align__(16) float sm[];
  row_weights<E0, E1, E2>(sm, a.w);
  for (int t = threadIdx.x; t < N::P2 * N::Q1; t += ER_T) {
    const int c = t / N::Q1, b = t % N::Q1;
    sm[N::W2T + t] = b < E1 ? sm[N::W2 + b * N::P2 + c] : 0.f;
  }
  for (int t = threadIdx.x; t < E1 * N::Q0; t += ER_T) {
    const int b = t / N::Q0, p = t % N::Q0;
    sm[N::W1T + t] = p < E0 ? sm[N::W1 + p * N::P1 + b] : 0.f;
  }
  __syncthreads();
  const int nrows = *a.nrows;
  for (int p0 = blockIdx.x * ER_T; p0 < nrows; p0 += gridDim.x * ER_T) {
    const RowPos r(a, p0 + threadIdx.x, nrows);
    const bool live = r.rg >= 0;
    const size_t pair = (size_t)r.ti * a.ntypes + r.tj;
    float4 R = make_float4(0.f, 0.f, 0.f, 0.f);
    if (FOLD) {
      if (live) R = reinterpret_cast<const float4*>(a.R)[r.rg];
    } else if (live) {
      R.x = a.R[(size_t)r.rg * 4];
    }
    const float* dT = FOLD ? a.dT + (size_t)(live ? r.rg / NP : 0) * 4 * a.m1 : nullptr;
    float dr[4] = {0.f, 0.f, 0.f, 0.f};
    float h2[E1];
    row_front<E0, E1, E2>(sm, R.x, a.b0t ? a.b0t + pair * E0 : nullptr, h2);
    const float* c2 = sm + N::H2 + threadIdx.x;
    const float4* gt4 = reinterpret_cast<const float4*>(a.Gt + pair * E2);
    // dH2[b] = sum_c W2[b][c] dZ3[c], dZ3 = g (1 - t3^2), g = dG0 (1 + Gt)
    f2 s2[N::Q1 / 2];
#pragma unroll
    for (int b = 0; b < N::Q1 / 2; ++b) s2[b] = 0ull;
#pragma unroll 1
    for (int c = 0; c < E2; c += ER_B) {
      float z[ER_B];
      row_block<E1, N::P2>(h2, sm + N::W2, sm + N::B2, c, z);
#pragma unroll
      for (int q = 0; q < ER_B; q += 4) {
        float4 dg = make_float4(0.f, 0.f, 0.f, 0.f), gt = dg, td[4] = {dg, dg, dg, dg};
        if (c + q < E2) {
          gt = gt4[(c + q) >> 2];
          if (live) dg = row_dg<FOLD>(a, r, R, dT, c + q, td);
        }
        const float dd[4] = {dg.x, dg.y, dg.z, dg.w}, gg[4] = {gt.x, gt.y, gt.z, gt.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float g = dd[u] * (1.f + gg[u]);
          const float t = tanhf(z[q + u]);
          if (FOLD && c + q < E2) {
            const int k = c + q + u;
            const float h3 = (doubles<E1, E2>() ? c2[(k < E1 ? k : k - E1) * ER_T] : 0.f) + t;
            const float g0 = h3 * (1.f + gg[u]);
#pragma unroll
            for (int w = 0; w < 4; ++w) dr[w] = fmaf(g0, (&td[w].x)[u], dr[w]);
          }
          z[q + u] = g * (1.f - t * t);
        }
      }
#pragma unroll
      for (int u = 0; u < ER_B; ++u) {
        const f2 zz = f2_pack(z[u], z[u]);
        const float* wt = sm + N::W2T + (c + u) * N::Q1;
#pragma unroll
        for (int b = 0; b < N::Q1; b += 4) {
          const ulonglong2 w = f2_ld4(wt + b);
          f2_fma(s2[b / 2], w.x, zz);
          f2_fma(s2[b / 2 + 1], w.y, zz);
        }
      }
    }
    float s[N::Q1];
#pragma unroll
    for (int b = 0; b < N::Q1 / 2; ++b) f2_unpack(s2[b], s[2 * b], s[2 * b + 1]);
    // the skip part of dH2 (a doubling layer: columns b and b + E1), then
    // dZ2 = dH2 (1 - t2^2) with t2 = H2 - skip(H1)
    const float* c1 = sm + N::H1 + threadIdx.x;
    if (doubles<E1, E2>()) {
#pragma unroll
      for (int c = 0; c < E2; c += 4) {
        const float4 g4 = gt4[c >> 2];
        float4 dg = make_float4(0.f, 0.f, 0.f, 0.f), td[4];
        if (live) dg = row_dg<FOLD>(a, r, R, dT, c, td);
        s[c % E1] += dg.x * (1.f + g4.x);
        s[(c + 1) % E1] += dg.y * (1.f + g4.y);
        s[(c + 2) % E1] += dg.z * (1.f + g4.z);
        s[(c + 3) % E1] += dg.w * (1.f + g4.w);
      }
    }
    // dH1[p] = skip^T(dH2)[p] + sum_b W1[p][b] dZ2[b]; dx = sum_p W0[p] dH1 (1 - H1^2)
    f2 v2[N::Q0 / 2];
#pragma unroll
    for (int p = 0; p < N::Q0 / 2; ++p) v2[p] = 0ull;
#pragma unroll
    for (int b = 0; b < E1; ++b) {
      const float t = c2[b * ER_T] - (doubles<E0, E1>() ? c1[(b % E0) * ER_T] : 0.f);
      const float dz = s[b] * (1.f - t * t);
      const f2 zz = f2_pack(dz, dz);
#pragma unroll
      for (int p = 0; p < N::Q0; p += 4) {
        const ulonglong2 w = f2_ld4(sm + N::W1T + b * N::Q0 + p);
        f2_fma(v2[p / 2], w.x, zz);
        f2_fma(v2[p / 2 + 1], w.y, zz);
      }
    }
    float v[N::Q0], dx = 0.f;
#pragma unroll
    for (int p = 0; p < N::Q0 / 2; ++p) f2_unpack(v2[p], v[2 * p], v[2 * p + 1]);
#pragma unroll
    for (int p = 0; p < E0; ++p) {
      if (doubles<E0, E1>()) {
        v[p] += s[p];
        v[p] += s[p + E0 < E1 ? p + E0 : 0];
      }
      const float h1 = c1[p * ER_T];
      dx = __fadd_rn(dx, __fmul_rn(v[p] * (1.f - h1 * h1), sm[N::W0 + p]));
    }
    if (FOLD) {
      if (live) reinterpret_cast<float4*>(a.dR)[r.rg] = make_float4(dr[0] + dx, dr[1], dr[2], dr[3]);
    } else if (live) {
      a.dR[(size_t)r.rg * 4] += dx;
    }
  }
}

template <int E0, int E1, int E2>
void rows_launch(const EmbedArgs& a, bool bwd, cudaStream_t st) {
  using N = RowNet<E0, E1, E2>;
  const size_t smem = sizeof(float) * (bwd ? N::BWD : N::FWD);
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // at most n * NP rows in tiles of ER_T = NP
  const int grid = std::min(a.n, (bwd ? N::B_CTAS : N::F_CTAS) * std::max(1, sms));
  if (!bwd) {
    cudaFuncSetAttribute(k_embed_rows_fwd<E0, E1, E2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_pdl(k_embed_rows_fwd<E0, E1, E2>, grid, ER_T, smem, st, a);
  } else {
    auto* k = a.dT ? k_embed_rows_bwd<E0, E1, E2, true> : k_embed_rows_bwd<E0, E1, E2, false>;
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_pdl(k, grid, ER_T, smem, st, a);
  }
  note_launch();
}

}  // namespace

bool launch_embed_rows(const EmbedArgs& a, const int* w, bool bwd, cudaStream_t st) {
  static_assert(ER_T == NP, "n tiles hold every live row");
  if (a.n == 0) return true;
  if (w[0] == 25 && w[1] == 50 && w[2] == 100) { rows_launch<25, 50, 100>(a, bwd, st); return true; }
  if (w[0] == 16 && w[1] == 32 && w[2] == 64) { rows_launch<16, 32, 64>(a, bwd, st); return true; }
  if (w[0] == 32 && w[1] == 64 && w[2] == 128) { rows_launch<32, 64, 128>(a, bwd, st); return true; }
  return false;
}

}  // namespace dpa1
