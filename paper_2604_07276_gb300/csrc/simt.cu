// FP32 SIMT kernels of the network stages a5-a13: embedding net, gated
// attention (forward and adjoint), LayerNorm, descriptor, fitting helpers
// and a general FP32 GEMM.  These form the FP32 path and provide the
// stages the tensor-core path shares with it.
#include "common.cuh"
#include "kernels.h"

namespace dpa1 {

static int sm_count();

// ----------------------------------------------------------------- FP32 GEMM
// C = epi(A B + bias (+R)), A [M][K], B [K][N] row-major.  128x128 tile, K
// step 16, 256 threads with 8x8 outputs each (two 4x4 quadrants 64 apart, so
// that the 16 threads of a half warp read 16 consecutive float4 of a shared
// row), shared-memory double buffering with the next tile held in registers.
// VEC: 16-byte global loads and stores (every leading dimension, K and N
// multiples of 4, the arrays 16-byte aligned); otherwise 4-byte ones.
constexpr int GBK = 16, GLD = 128 + 4;

template <int EPI, bool VEC>
__global__ void __launch_bounds__(256, 2)
k_sgemm128(const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb,
           const float* __restrict__ bias, const float* __restrict__ R, int ldr, float* __restrict__ C, int ldc,
           int M, int N, int K, const int* __restrict__ m_dev) {
  pdl_wait();
  if (m_dev) M = *m_dev;
  if ((long long)blockIdx.x * 128 >= M) return;
  __shared__ __align__(16) float As[2][GBK][GLD];  // k-major: As[k][row]
  __shared__ __align__(16) float Bs[2][GBK][GLD];  // Bs[k][column]
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const long long m0 = (long long)blockIdx.x * 128;
  const int n0 = blockIdx.y * 128;
  const int ar = tid >> 1, ak = (tid & 1) * 8;   // A: row, first of its 8 k
  const int bk = tid >> 4, bc = (tid & 15) * 8;  // B: k, first of its 8 columns
  float ra[8], rb[8];
  auto load = [&](int k0) {
    const long long gm = m0 + ar;
    const int gka = k0 + ak, gkb = k0 + bk;
    if (VEC) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        if (gm < M && gka + 4 * h < K) x = *reinterpret_cast<const float4*>(A + gm * lda + gka + 4 * h);
        ra[4 * h] = x.x; ra[4 * h + 1] = x.y; ra[4 * h + 2] = x.z; ra[4 * h + 3] = x.w;
        float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
        const int gn = n0 + bc + 4 * h;
        if (gkb < K && gn < N) y = *reinterpret_cast<const float4*>(B + (long long)gkb * ldb + gn);
        rb[4 * h] = y.x; rb[4 * h + 1] = y.y; rb[4 * h + 2] = y.z; rb[4 * h + 3] = y.w;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int gk = gka + q, gn = n0 + bc + q;
        ra[q] = (gm < M && gk < K) ? A[gm * lda + gk] : 0.f;
        rb[q] = (gkb < K && gn < N) ? B[(long long)gkb * ldb + gn] : 0.f;
      }
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int q = 0; q < 8; ++q) As[buf][ak + q][ar] = ra[q];
    *reinterpret_cast<float4*>(&Bs[buf][bk][bc]) = make_float4(rb[0], rb[1], rb[2], rb[3]);
    *reinterpret_cast<float4*>(&Bs[buf][bk][bc + 4]) = make_float4(rb[4], rb[5], rb[6], rb[7]);
  };
  float acc[8][8];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
  load(0);
  store(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += GBK) {
    const bool more = k0 + GBK < K;
    if (more) load(k0 + GBK);
#pragma unroll
    for (int k = 0; k < GBK; ++k) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][k][ty * 4]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][k][64 + ty * 4]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[buf][k][tx * 4]);
      const float4 b1 = *reinterpret_cast<const float4*>(&Bs[buf][k][64 + tx * 4]);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) {
      store(buf ^ 1);
      __syncthreads();
      buf ^= 1;
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const long long m = m0 + (i < 4 ? ty * 4 + i : 64 + ty * 4 + i - 4);
    if (m >= M) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int nq = n0 + h * 64 + tx * 4;  // first of this thread's 4 columns
      float v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int n = nq + j;
        float x = acc[i][4 * h + j];
        if (n < N) {
          if (EPI == EPI_BIAS || EPI == EPI_TANH || EPI == EPI_RES_TANH) x += bias ? bias[n] : 0.f;
          if (EPI == EPI_TANH || EPI == EPI_RES_TANH) x = tanhf(x);
        }
        v[j] = x;
      }
      if (VEC) {
        if (nq < N) {  // N % 4 == 0: the 4 columns are all in range
          float4 o = make_float4(v[0], v[1], v[2], v[3]);
          if (EPI == EPI_RES_TANH || EPI == EPI_RES) {
            const float4 r = *reinterpret_cast<const float4*>(R + m * ldr + nq);
            o.x += r.x; o.y += r.y; o.z += r.z; o.w += r.w;
          }
          float4* c = reinterpret_cast<float4*>(C + m * ldc + nq);
          if (EPI == EPI_ACCUM) {
            const float4 cc = *c;
            o.x += cc.x; o.y += cc.y; o.z += cc.z; o.w += cc.w;
          }
          *c = o;
        }
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int n = nq + j;
          if (n >= N) continue;
          float* c = C + m * ldc + n;
          if (EPI == EPI_RES_TANH || EPI == EPI_RES) *c = R[m * ldr + n] + v[j];
          else if (EPI == EPI_ACCUM) *c = *c + v[j];
          else *c = v[j];
        }
      }
    }
  }
}

template <int EPI>
static void sgemm_launch(dim3 grid, bool vec, const float* A, int lda, const float* B, int ldb, const float* bias,
                         const float* R, int ldr, float* C, int ldc, int M, int N, int K, const int* m_dev,
                         cudaStream_t st) {
  if (vec)
    launch_pdl(k_sgemm128<EPI, true>, grid, 256, 0, st, A, lda, B, ldb, bias, R, ldr, C, ldc, M, N, K, m_dev);
  else
    launch_pdl(k_sgemm128<EPI, false>, grid, 256, 0, st, A, lda, B, ldb, bias, R, ldr, C, ldc, M, N, K, m_dev);
}

void gemm_f32(const float* A, int lda, const float* B, int ldb, const float* bias, const float* R, int ldr,
              float* C, int ldc, int M, int N, int K, int epi, cudaStream_t st, const int* m_dev) {
  if (M <= 0 || N <= 0) return;
  dim3 grid((unsigned)((M + 127) / 128), (unsigned)((N + 127) / 128));
  const bool res = epi == EPI_RES || epi == EPI_RES_TANH;
  const uintptr_t addr = reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B) |
                         reinterpret_cast<uintptr_t>(C) | (res ? reinterpret_cast<uintptr_t>(R) : 0);
  const bool vec = (addr & 15) == 0 && lda % 4 == 0 && ldb % 4 == 0 && ldc % 4 == 0 && (!res || ldr % 4 == 0) &&
                   N % 4 == 0 && K % 4 == 0;
  switch (epi) {
    case EPI_BIAS: sgemm_launch<EPI_BIAS>(grid, vec, A, lda, B, ldb, bias, R, ldr, C, ldc, M, N, K, m_dev, st); break;
    case EPI_TANH: sgemm_launch<EPI_TANH>(grid, vec, A, lda, B, ldb, bias, R, ldr, C, ldc, M, N, K, m_dev, st); break;
    case EPI_RES_TANH: sgemm_launch<EPI_RES_TANH>(grid, vec, A, lda, B, ldb, bias, R, ldr, C, ldc, M, N, K, m_dev, st); break;
    case EPI_ACCUM: sgemm_launch<EPI_ACCUM>(grid, vec, A, lda, B, ldb, bias, R, ldr, C, ldc, M, N, K, m_dev, st); break;
    default: sgemm_launch<EPI_RES>(grid, vec, A, lda, B, ldb, bias, R, ldr, C, ldc, M, N, K, m_dev, st); break;
  }
  note_launch();
}

// ---------------------------------------------------------------- LayerNorm
// G_out = G_in + LN(Y), row by row.
__global__ void k_ln_res_fwd(const float* __restrict__ Y, const float* __restrict__ Gin, const int* __restrict__ nrows,
                             const float* __restrict__ gamma, const float* __restrict__ beta, float eps,
                             float* __restrict__ Gout, float* __restrict__ stats, int m1) {
  pdl_wait();
  const long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (row >= *nrows) return;
  const float* y = Y + row * m1;
  float v[4];
  float s = 0.f;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = lane + 32 * q;
    v[q] = c < m1 ? y[c] : 0.f;
    s += v[q];
  }
  const float mean = warp_sum(s) / (float)m1;
  float s2 = 0.f;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = lane + 32 * q;
    const float d = c < m1 ? v[q] - mean : 0.f;
    s2 += d * d;
  }
  const float var = warp_sum(s2) / (float)m1;
  const float rstd = 1.0f / sqrtf(var + eps);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = lane + 32 * q;
    if (c < m1) {
      const float gin = Gin[row * m1 + c];
      Gout[row * m1 + c] = gin + (v[q] - mean) * rstd * gamma[c] + beta[c];
    }
  }
  if (lane == 0) {
    stats[2 * row] = mean;
    stats[2 * row + 1] = rstd;
  }
}

__global__ void k_ln_bwd(const float* __restrict__ dZ, const float* __restrict__ Y, const float* __restrict__ stats,
                         const int* __restrict__ nrows, const float* __restrict__ gamma, float* __restrict__ dY,
                         int m1) {
  pdl_wait();
  const long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (row >= *nrows) return;
  const float mean = stats[2 * row], rstd = stats[2 * row + 1];
  float gz[4], yh[4];
  float s1 = 0.f, s2 = 0.f;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = lane + 32 * q;
    if (c < m1) {
      gz[q] = gamma[c] * dZ[row * m1 + c];
      yh[q] = (Y[row * m1 + c] - mean) * rstd;
    } else {
      gz[q] = 0.f; yh[q] = 0.f;
    }
    s1 += gz[q];
    s2 += gz[q] * yh[q];
  }
  s1 = warp_sum(s1) / (float)m1;
  s2 = warp_sum(s2) / (float)m1;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = lane + 32 * q;
    if (c < m1) dY[row * m1 + c] = rstd * (gz[q] - s1 - yh[q] * s2);
  }
}

void launch_ln_res_fwd(const float* Y, const float* Gin, const int* nrows, const float* gamma, const float* beta,
                       float eps, float* Gout, float* stats, int rows_i, int m1, cudaStream_t st) {
  long long rows = rows_i;
  if (rows == 0) return;
  launch_pdl(k_ln_res_fwd, (unsigned)((rows * 32 + 255) / 256), 256, 0, st, Y, Gin, nrows, gamma, beta, eps, Gout, stats, m1);
  note_launch();
}
void launch_ln_bwd(const float* dZ, const float* Y, const float* stats, const int* nrows, const float* gamma,
                   float* dY, int rows_i, int m1, cudaStream_t st) {
  long long rows = rows_i;
  if (rows == 0) return;
  launch_pdl(k_ln_bwd, (unsigned)((rows * 32 + 255) / 256), 256, 0, st, dZ, Y, stats, nrows, gamma, dY, m1);
  note_launch();
}

// ------------------------------------------------- gated attention (FP32)
// Per centre atom, over its valid neighbour slots j, k < n_i:
//   l_jk = Q_j.K_k / sqrt(A);  l'_jk = (l_jk + S) w_j w_k - S
//   A_jk = softmax_k(l'_jk);   P_jk = A_jk w_j w_k (rhat_j . rhat_k);  O = P V
// (the forward evaluates O Wo through P G, see k_attn_fwd_f32)

// Smooth logits l'_jk = (l_jk + S) w_j w_k carry the shift S = 20, whose
// FP32 spacing (2e-6) is far coarser than the logit differences that matter.
// They are evaluated as unevaluated float pairs (h + l): l + S exactly by a
// two-sum, the product of the switch weights (FP64, held as float pairs) and
// the final product with their rounding errors by FMA; ~44 bits, without the
// FP64 pipe (narrow on this GPU).  Only differences to the row maximum are
// used, as floats.
__device__ __forceinline__ float2 split_pair(double w) {
  const float h = (float)w;
  return make_float2(h, (float)(w - (double)h));
}

__device__ __forceinline__ float2 smooth_logit(float t, float S, float2 wj, float2 wk) {
  const float uh = t + S;
  const float bb = uh - t;
  const float ul = (t - (uh - bb)) + (S - bb);
  const float ph = wj.x * wk.x;
  float pl = fmaf(wj.x, wk.x, -ph);
  pl = fmaf(wj.x, wk.y, pl);
  pl = fmaf(wj.y, wk.x, pl);
  const float hh = uh * ph;
  float hl = fmaf(uh, ph, -hh);
  hl = fmaf(uh, pl, hl);
  hl = fmaf(ul, ph, hl);
  return make_float2(hh, hl);
}

__device__ __forceinline__ float pair_diff(float2 a, float2 b) { return (a.x - b.x) + (a.y - b.y); }

// Forward, register-tiled, 512 threads.  The products (S, then each 128-column
// part of PG) give a warp 16 rows x 64 columns and a thread 4 x 8 of them (PTile):
// per step a warp then reads 64 bytes of A and 2 x 128 of B, three 16-byte loads for
// 32 FMAs with one wavefront each (8 x 128 a warp: five), and a warp whose rows, or a
// half of it whose columns, are past the last neighbour has nothing to do.  The live
// warps are spread over the four schedulers, and the loops unrolled eight times so
// that loads run ahead of the FMAs: latency binds, not the shared-memory pipe (the
// same tiles, one scheduler with twice the FMAs of another: 8 % slower; not unrolled:
// 8 % more).  The softmax works on
// rows 4 ty + i (i < 4) and keys t_rc(tx, jj) (jj < 8) of a 32 x 16 thread grid, S
// passing through shared memory.  Q and K pass through shared memory
// feature-major, 128 features at a time; P stays row-major and [G 1] comes in
// 128-column parts, key-major.  S sums over the features and PG over the keys in
// order, as a plain loop would.  3,001 atoms, width 128: 654 -> 593 us a layer (the
// adjoint 1,385 -> 1,226).
//
// The kernel writes PG = [P G, rowsum(P)] instead of O = P V: with V = G Wv +
// bv, O Wo + bo = [P G, rowsum(P)] [Wv Wo; bv Wo] + bo, which a GEMM with the
// FP64-formed [Wv Wo; bv Wo] then evaluates.  The two are equal in exact
// arithmetic, but the gate (rhat_j . rhat_k of both signs) makes sum_k P_jk
// V_k cancel, and the accumulation errors of each computed V_k (a 100-term
// FP32 sum) survive that cancellation; the LayerNorm of weakly attended rows
// (variance << eps) then turns them into force errors up to ~5e-4 eV/A on
// a few atoms.  Summing the exact layer input G instead leaves only the
// rounding of the cancelling sum itself (a CPU emulation of both forms on the
// 15,668-atom box: force RMSE 7.5e-6 -> 2.4e-6 eV/A).
constexpr int FTF = 512;       // threads of the forward and the adjoint (4 x 8 tiles)
static_assert(4 * (FTF / 16) == NP, "32 thread rows of 4 rows each cover the 128 rows of an atom");
static_assert((FTF / 16) * NP * 4 <= 128 * (NP + 4), "the adjoint's column parts fit one shared tile");
constexpr int TLD = NP + 4;    // row stride of their shared tiles (16-byte rows)

// Row (or column) i < 8 of thread coordinate t < 16: the quarter tiles
// 4 t .. 4 t + 3 and 64 + 4 t .. 64 + 4 t + 3, so that the 16 threads of a
// half warp read 16 consecutive float4 of a shared row (no bank conflicts).
__device__ __forceinline__ int t_rc(int t, int i) { return i < 4 ? 4 * t + i : 60 + 4 * t + i; }

// Feature-major staging of a 128-row chunk: element idx (0 .. 4095) of the
// CTA's accesses takes row j and features f .. f + 3, 16 rows x 32 bytes per
// warp access (full sectors), and its transposed stores (feature f + u, row
// j) fall on distinct banks.
__device__ __forceinline__ void fm_pos(int idx, int& j, int& f) {
  const int w = idx >> 5, l = idx & 31;
  j = 16 * (w & 7) + (l >> 1);
  f = 4 * ((l & 1) + 2 * (w >> 3));
}

__device__ __forceinline__ void fm_store(float* T, int j, int f, float4 v) {
  T[(f + 0) * TLD + j] = v.x; T[(f + 1) * TLD + j] = v.y;
  T[(f + 2) * TLD + j] = v.z; T[(f + 3) * TLD + j] = v.w;
}

// A thread's part of a 128 x 128 product: rows r .. r + 3, columns c .. c + 3
// and c + 32 .. c + 35.
struct PTile {
  int r, c;
  __device__ PTile(int tid) {
    const int warp = tid >> 5, lane = tid & 31;
    // live rows come first: consecutive row blocks over the SM's four schedulers
    // (warp % 4), the column halves alternating
    r = 16 * (warp >> 1) + 4 * (lane >> 3);
    c = 64 * ((warp ^ (warp >> 2)) & 1) + 4 * (lane & 7);
  }
  // of the warp: rows below nrows, columns of its first and second half below ncols
  __device__ int halves(int nrows, int ncols) const {
    if ((r & ~15) >= nrows) return 0;
    const int c0 = c & ~63;
    return c0 + 32 < ncols ? 2 : (c0 < ncols ? 1 : 0);
  }
};

// acc[i][j] += a[i] b[j] with a = A[ra .. ra + 3], b = (B[rb .. rb + 3], B[rb + 32
// .. rb + 35] for H = 2).
template <int H>
__device__ __forceinline__ void tile_fma(float (&acc)[4][8], const float* A, int ra, const float* B, int rb) {
  const float4 a0 = *reinterpret_cast<const float4*>(A + ra);
  const float av[4] = {a0.x, a0.y, a0.z, a0.w};
#pragma unroll
  for (int h = 0; h < H; ++h) {
    const float4 b0 = *reinterpret_cast<const float4*>(B + rb + 32 * h);
    const float bv[4] = {b0.x, b0.y, b0.z, b0.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][4 * h + j] = fmaf(av[i], bv[j], acc[i][4 * h + j]);
  }
}

// acc[i][j] += sum over k0 .. k0 + 3 of A[r + i][k] B[k][c ..] (A row-major, B
// key-major, both with row stride TLD).
template <int H>
__device__ __forceinline__ void tile_fma4(float (&acc)[4][8], const float* A, const float* B, int k0, const PTile& t) {
  float4 pa[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) pa[i] = *reinterpret_cast<const float4*>(A + (t.r + i) * TLD + k0);
#pragma unroll
  for (int u = 0; u < 4; ++u) {
#pragma unroll
    for (int h = 0; h < H; ++h) {
      const float4 v = *reinterpret_cast<const float4*>(B + (k0 + u) * TLD + t.c + 32 * h);
      const float vb[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float p = u == 0 ? pa[i].x : u == 1 ? pa[i].y : u == 2 ? pa[i].z : pa[i].w;
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][4 * h + j] = fmaf(p, vb[j], acc[i][4 * h + j]);
      }
    }
  }
}

// acc = sum over k < n of the outer products of A[k][r ..] and B[k][c ..] (both
// k-major with row stride TLD).
__device__ __forceinline__ void tile_outer(float (&acc)[4][8], const float* A, const float* B, int n, const PTile& t,
                                           int halves) {
  if (halves == 2) {
#pragma unroll 8
    for (int k = 0; k < n; ++k) tile_fma<2>(acc, A, k * TLD + t.r, B, k * TLD + t.c);
  } else if (halves == 1) {
#pragma unroll 8
    for (int k = 0; k < n; ++k) tile_fma<1>(acc, A, k * TLD + t.r, B, k * TLD + t.c);
  }
}

// acc = sum over k < n (n % 4 == 0) of A[r ..][k] B[k][c ..].
__device__ __forceinline__ void tile_inner(float (&acc)[4][8], const float* A, const float* B, int n, const PTile& t,
                                           int halves) {
  if (halves == 2) {
#pragma unroll 4
    for (int k = 0; k < n; k += 4) tile_fma4<2>(acc, A, B, k, t);
  } else if (halves == 1) {
#pragma unroll 4
    for (int k = 0; k < n; k += 4) tile_fma4<1>(acc, A, B, k, t);
  }
}

__device__ __forceinline__ void tile_zero(float (&acc)[4][8]) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
}

// The tile's rows below nrows -> dst (row stride ld, column 0 of the product at dst),
// each float4 only below ncols.
__device__ __forceinline__ void tile_store(float* dst, size_t ld, const float (&acc)[4][8], const PTile& t, int nrows,
                                           int ncols) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (t.r + i >= nrows) continue;
    float* p = dst + (size_t)(t.r + i) * ld + t.c;
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (t.c + 32 * h < ncols)
        *reinterpret_cast<float4*>(p + 32 * h) =
            make_float4(acc[i][4 * h], acc[i][4 * h + 1], acc[i][4 * h + 2], acc[i][4 * h + 3]);
  }
}

// One row of the softmax's thread grid -> dst row (columns 4 tx .. and 64 + 4 tx ..).
__device__ __forceinline__ void grid_store_row(float* dst, const float* v, int tx) {
  *reinterpret_cast<float4*>(dst + 4 * tx) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(dst + 64 + 4 * tx) = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void grid_load_row(const float* src, float* v, int tx) {
  const float4 a = *reinterpret_cast<const float4*>(src + 4 * tx), b = *reinterpret_cast<const float4*>(src + 64 + 4 * tx);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

// The next atom's rows into L2, a row per thread.
__device__ __forceinline__ void prefetch_rows(const float* p, int row_floats, int row0, int rows) {
  const int t = threadIdx.x;
  if (t < rows)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p + (size_t)(row0 + t) * row_floats),
                 "r"((uint32_t)(row_floats * sizeof(float)))
                 : "memory");
}

template <int A>
__global__ void __launch_bounds__(FTF, 1) k_attn_fwd_f32(AttnArgs a, float scale) {
  pdl_wait();
  extern __shared__ float sm[];
  float* X = sm;                 // [128][TLD]: Q chunk (feature-major), then P (row-major)
  float* Y = X + 128 * TLD;      // [128][TLD]: K chunk (feature-major), then a part of [G 1] (key-major)
  float4* rws = reinterpret_cast<float4*>(Y + 128 * TLD);  // [NP]
  float2* w2s = reinterpret_cast<float2*>(rws + NP);       // [NP] switch weights as float pairs
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int ld = a.ldq;  // Q | K
  const PTile pt(tid);
  for (int atom = blockIdx.x; atom < a.n; atom += gridDim.x) {
    const int nn = a.nnei[atom];
    const size_t base = a.row_off[atom], gbase = (size_t)atom * NP;
    if (atom + (int)gridDim.x < a.n) {
      const int r0 = a.row_off[atom + gridDim.x], rows = a.row_off[atom + gridDim.x + 1] - r0;
      prefetch_rows(a.QK, ld, r0, rows);
      prefetch_rows(a.G, a.m1, r0, rows);
    }
    __syncthreads();  // the previous atom is done with every shared array
    for (int r = tid; r < NP; r += FTF) {
      rws[r] = r < nn ? reinterpret_cast<const float4*>(a.rw)[gbase + r] : make_float4(0.f, 0.f, 0.f, 0.f);
      w2s[r] = split_pair(r < nn ? a.w64[gbase + r] : 0.0);
    }
    float acc[4][8];
    tile_zero(acc);
    const int live = pt.halves(nn, nn);
    for (int c0 = 0; c0 < A; c0 += 128) {
      if (c0 > 0) __syncthreads();  // the previous chunk's products are done
      for (int idx = tid; idx < NP * 32; idx += FTF) {
        int j, f;
        fm_pos(idx, j, f);
        float4 qv = make_float4(0.f, 0.f, 0.f, 0.f), kv = qv;
        if (j < nn) {
          qv = *reinterpret_cast<const float4*>(a.QK + (base + j) * ld + c0 + f);
          kv = *reinterpret_cast<const float4*>(a.QK + (base + j) * ld + A + c0 + f);
        }
        fm_store(X, j, f, qv);
        fm_store(Y, j, f, kv);
      }
      __syncthreads();
      tile_outer(acc, X, Y, 128, pt, live);
    }
    __syncthreads();  // X and Y are free: S passes through X to the softmax's threads
    if (live) tile_store(X, TLD, acc, pt, 128, 128);
    __syncthreads();
    float s[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i) grid_load_row(X + (4 * ty + i) * TLD, s[i], tx);
    // (a thread reads the entries of S that it overwrites with P)
    // softmax per row over the 16 threads of a half warp (every lane takes
    // part in the shuffles; rows and keys past nnei come out zero)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int j = 4 * ty + i;
      const float4 rj = rws[j];
      const float2 wj = w2s[j];
      float2 lp[8], mx = make_float2(-3.0e38f, 0.f);
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const int k = t_rc(tx, jj);
        lp[jj] = make_float2(-3.0e38f, 0.f);
        if (k < nn) {
          lp[jj] = smooth_logit(s[i][jj] * scale, a.shift, wj, w2s[k]);
          if (lp[jj].x > mx.x || (lp[jj].x == mx.x && lp[jj].y > mx.y)) mx = lp[jj];
        }
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, mx.x, o);
        const float ol = __shfl_xor_sync(0xffffffffu, mx.y, o);
        if (oh > mx.x || (oh == mx.x && ol > mx.y)) mx = make_float2(oh, ol);
      }
      float e[8], sum = 0.f;
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        e[jj] = t_rc(tx, jj) < nn ? expf(pair_diff(lp[jj], mx)) : 0.f;
        sum += e[jj];
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      const float inv = sum > 0.f ? 1.0f / sum : 0.f;
      float pv[8];
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const int k = t_rc(tx, jj);
        pv[jj] = 0.f;
        if (j < nn && k < nn) {
          const float4 rk = rws[k];
          pv[jj] = e[jj] * inv * (rj.w * rk.w) * (rj.x * rk.x + rj.y * rk.y + rj.z * rk.z);
        }
      }
      grid_store_row(X + j * TLD, pv, tx);
    }
    // PG = P [G 1], 128 columns at a time (column m1 of [G 1] is 1, later
    // ones 0; m1 % 4 == 0)
    const int nn4 = (nn + 3) & ~3;
    for (int c0 = 0; c0 < a.ldpg; c0 += 128) {
      if (c0 > 0) __syncthreads();  // the previous part's products are done
      for (int idx = tid; idx < NP * 32; idx += FTF) {
        const int k = idx >> 5, f = c0 + 4 * (idx & 31);
        float4 vv = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k < nn) {
          if (f < a.m1) vv = *reinterpret_cast<const float4*>(a.G + (base + k) * a.m1 + f);
          else if (f == a.m1) vv.x = 1.f;
        }
        *reinterpret_cast<float4*>(Y + k * TLD + f - c0) = vv;
      }
      __syncthreads();  // P (first part) and this part of [G 1] are in place
      tile_zero(acc);
      const int ncols = min(128, a.ldpg - c0);
      tile_inner(acc, X, Y, nn4, pt, pt.halves(nn, ncols));
      tile_store(a.PG + base * a.ldpg + c0, a.ldpg, acc, pt, nn, ncols);
    }
  }
}

// Adjoint of one attention layer for one centre, register-tiled like the
// forward, in the form of its output Y = [P G, rowsum P] [Wv Wo; bv Wo] + bo: with
// dPG = dE/d[P G, rowsum P] (a GEMM of dY with [Wv Wo; bv Wo]^T),
//   dP_jk = sum_c dPG_jc G_kc + dPG_j,m1        (the values V never appear)
//   softmax adjoint: dS, and the row / column parts of dE/dw and dE/drhat
//   dQ = dS K,  dK = dS^T Q,  dE/dG += P^T dPG (columns below m1).
// S and dP pass through shared memory to the threads of the softmax adjoint; dS
// and P go back there (row-major), where the three last products read them.  The
// column parts are summed over the 32 row groups in a fixed order.
template <int A>
__global__ void __launch_bounds__(FTF, 1) k_attn_bwd_f32(AttnArgs a, float scale) {
  pdl_wait();
  extern __shared__ float sm[];
  float* B0 = sm;               // [128][TLD] operand chunks
  float* B1 = B0 + 128 * TLD;   // [128][TLD] K / G chunk, then dS (row-major)
  float* B2 = B1 + 128 * TLD;   // [128][TLD] P (row-major)
  float4* rws = reinterpret_cast<float4*>(B2 + 128 * TLD);  // [NP]
  float2* w2s = reinterpret_cast<float2*>(rws + NP);         // [NP] switch weights as float pairs
  float4* rowg = reinterpret_cast<float4*>(w2s + NP);        // [NP] row parts of (d rhat, d w)
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int ld = a.ldq;  // Q | K, and dQ | dK
  const PTile pt(tid);
  for (int atom = blockIdx.x; atom < a.n; atom += gridDim.x) {
    const int nn = a.nnei[atom];
    const size_t base = a.row_off[atom], gbase = (size_t)atom * NP;
    if (atom + (int)gridDim.x < a.n) {
      const int r0 = a.row_off[atom + gridDim.x], rows = a.row_off[atom + gridDim.x + 1] - r0;
      prefetch_rows(a.QK, ld, r0, rows);
      prefetch_rows(a.G, a.m1, r0, rows);
      prefetch_rows(a.dPG, a.ldpg, r0, rows);
    }
    __syncthreads();  // the previous atom is done with every shared array
    for (int r = tid; r < NP; r += FTF) {
      rws[r] = r < nn ? reinterpret_cast<const float4*>(a.rw)[gbase + r] : make_float4(0.f, 0.f, 0.f, 0.f);
      w2s[r] = split_pair(r < nn ? a.w64[gbase + r] : 0.0);
    }
    const int live = pt.halves(nn, nn);
    float ps[4][8], pd[4][8];  // this thread's tiles of S and dP
    tile_zero(ps);
    tile_zero(pd);
    // S = Q K^T over feature chunks of 128 (feature-major in B0, B1)
    for (int c0 = 0; c0 < A; c0 += 128) {
      if (c0 > 0) __syncthreads();
      for (int idx = tid; idx < NP * 32; idx += FTF) {
        int j, f;
        fm_pos(idx, j, f);
        float4 qv = make_float4(0.f, 0.f, 0.f, 0.f), kv = qv;
        if (j < nn) {
          qv = *reinterpret_cast<const float4*>(a.QK + (base + j) * ld + c0 + f);
          kv = *reinterpret_cast<const float4*>(a.QK + (base + j) * ld + A + c0 + f);
        }
        fm_store(B0, j, f, qv);
        fm_store(B1, j, f, kv);
      }
      __syncthreads();
      tile_outer(ps, B0, B1, 128, pt, live);
    }
    __syncthreads();
    // dP = dPG G^T over the m1 columns (feature-major: dPG in B0, G in B1;
    // m1 % 4 == 0)
    for (int idx = tid; idx < NP * 32; idx += FTF) {
      int j, f;
      fm_pos(idx, j, f);
      float4 dv = make_float4(0.f, 0.f, 0.f, 0.f), gv = dv;
      if (j < nn && f < a.m1) {
        dv = *reinterpret_cast<const float4*>(a.dPG + (base + j) * a.ldpg + f);
        gv = *reinterpret_cast<const float4*>(a.G + (base + j) * a.m1 + f);
      }
      fm_store(B0, j, f, dv);
      fm_store(B1, j, f, gv);
    }
    __syncthreads();
    tile_outer(pd, B0, B1, a.m1, pt, live);
    __syncthreads();  // B0 and B1 are free: S passes through B1, dP through B2
    if (live) {
      tile_store(B1, TLD, ps, pt, 128, 128);
      tile_store(B2, TLD, pd, pt, 128, 128);
    }
    __syncthreads();
    float s[4][8], dp[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      grid_load_row(B1 + (4 * ty + i) * TLD, s[i], tx);
      grid_load_row(B2 + (4 * ty + i) * TLD, dp[i], tx);
    }
    // (a thread reads the entries that it overwrites: dS goes to B1, P to B2,
    // column parts to B0)
    // softmax adjoint per row over the 16 threads of a half warp (every lane
    // takes part in the shuffles; rows and keys past nnei come out zero)
    float cw[8], cx[8], cy[8], cz[8];
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) { cw[jj] = 0.f; cx[jj] = 0.f; cy[jj] = 0.f; cz[jj] = 0.f; }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int j = 4 * ty + i;
      const float4 rj = rws[j];
      const float2 wj = w2s[j];
      const float dpg1 = j < nn ? a.dPG[(base + j) * a.ldpg + a.m1] : 0.f;  // adjoint of rowsum P
      float2 lp[8], mx = make_float2(-3.0e38f, 0.f);
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const int k = t_rc(tx, jj);
        lp[jj] = make_float2(-3.0e38f, 0.f);
        if (k < nn) {
          lp[jj] = smooth_logit(s[i][jj] * scale, a.shift, wj, w2s[k]);  // as in the forward kernel
          if (lp[jj].x > mx.x || (lp[jj].x == mx.x && lp[jj].y > mx.y)) mx = lp[jj];
        }
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, mx.x, o);
        const float ol = __shfl_xor_sync(0xffffffffu, mx.y, o);
        if (oh > mx.x || (oh == mx.x && ol > mx.y)) mx = make_float2(oh, ol);
      }
      float e[8], sum = 0.f;
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        e[jj] = t_rc(tx, jj) < nn ? expf(pair_diff(lp[jj], mx)) : 0.f;
        sum += e[jj];
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      const float inv = sum > 0.f ? 1.0f / sum : 0.f;
      float At[8], dA[8], tsum = 0.f;
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const int k = t_rc(tx, jj);
        const float4 rk = rws[k];
        At[jj] = e[jj] * inv;
        dA[jj] = k < nn ? (dp[i][jj] + dpg1) * (rj.w * rk.w) * (rj.x * rk.x + rj.y * rk.y + rj.z * rk.z) : 0.f;
        tsum += At[jj] * dA[jj];
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) tsum += __shfl_xor_sync(0xffffffffu, tsum, o);
      float rw_ = 0.f, rx = 0.f, ry = 0.f, rz = 0.f, ds[8], pv[8];
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) {
        const int k = t_rc(tx, jj);
        ds[jj] = 0.f;
        pv[jj] = 0.f;
        if (j < nn && k < nn) {
          const float4 rk = rws[k];
          const float ww = rj.w * rk.w;
          const float c = rj.x * rk.x + rj.y * rk.y + rj.z * rk.z;
          const float dpv = dp[i][jj] + dpg1;
          const float dLp = At[jj] * (dA[jj] - tsum);
          ds[jj] = dLp * ww * scale;
          pv[jj] = At[jj] * ww * c;
          const float H = dpv * At[jj] * c + dLp * (s[i][jj] * scale + a.shift);  // dE/d(w_j w_k)
          const float dc = dpv * At[jj] * ww;                                      // dE/dc_jk
          rw_ += H * rk.w;
          rx += dc * rk.x; ry += dc * rk.y; rz += dc * rk.z;
          cw[jj] += H * rj.w;
          cx[jj] += dc * rj.x; cy[jj] += dc * rj.y; cz[jj] += dc * rj.z;
        }
      }
      grid_store_row(B1 + j * TLD, ds, tx);
      grid_store_row(B2 + j * TLD, pv, tx);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
        rw_ += __shfl_xor_sync(0xffffffffu, rw_, o);
        rx += __shfl_xor_sync(0xffffffffu, rx, o);
        ry += __shfl_xor_sync(0xffffffffu, ry, o);
        rz += __shfl_xor_sync(0xffffffffu, rz, o);
      }
      if (tx == 0) rowg[j] = make_float4(rx, ry, rz, rw_);
    }
    // column parts of this thread's 4 rows -> B0 as [ty][key] (32 x 128 float4)
    float4* colp = reinterpret_cast<float4*>(B0);
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) colp[ty * NP + t_rc(tx, jj)] = make_float4(cx[jj], cy[jj], cz[jj], cw[jj]);
    __syncthreads();
    if (tid < nn) {
      float4 acc = rowg[tid];
      for (int q = 0; q < 32; ++q) {
        const float4 c = colp[q * NP + tid];
        acc.x += c.x; acc.y += c.y; acc.z += c.z; acc.w += c.w;
      }
      // one writer per row in a launch: a reduction without a return
      atomicAdd(reinterpret_cast<float4*>(a.dgeo) + gbase + tid, acc);
    }
    const int nn4 = (nn + 3) & ~3;
    for (int c0 = 0; c0 < A; c0 += 128) {
      // dQ = dS K: K key-major in B0
      __syncthreads();
      for (int idx = tid; idx < NP * 32; idx += FTF) {
        const int k = idx >> 5, f = 4 * (idx & 31);
        *reinterpret_cast<float4*>(B0 + k * TLD + f) =
            k < nn ? *reinterpret_cast<const float4*>(a.QK + (base + k) * ld + A + c0 + f) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      __syncthreads();
      float acc[4][8];
      const int lv = pt.halves(nn, 128);
      tile_zero(acc);
      tile_inner(acc, B1, B0, nn4, pt, lv);
      tile_store(a.dQK + base * ld + c0, ld, acc, pt, nn, 128);
      // dK = dS^T Q: Q row-major in B0
      __syncthreads();
      for (int idx = tid; idx < NP * 32; idx += FTF) {
        const int j = idx >> 5, f = 4 * (idx & 31);
        *reinterpret_cast<float4*>(B0 + j * TLD + f) =
            j < nn ? *reinterpret_cast<const float4*>(a.QK + (base + j) * ld + c0 + f) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      __syncthreads();
      tile_zero(acc);
      tile_outer(acc, B1, B0, nn, pt, lv);
      tile_store(a.dQK + base * ld + A + c0, ld, acc, pt, nn, 128);
    }
    // dE/dG += P^T dPG: dPG row-major in B0 (columns below m1; m1 <= 128)
    __syncthreads();
    for (int idx = tid; idx < NP * 32; idx += FTF) {
      const int j = idx >> 5, f = 4 * (idx & 31);
      *reinterpret_cast<float4*>(B0 + j * TLD + f) = j < nn && f < a.m1
                                                         ? *reinterpret_cast<const float4*>(a.dPG + (base + j) * a.ldpg + f)
                                                         : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    if (const int lv = pt.halves(nn, a.m1)) {
      float acc[4][8];
      tile_zero(acc);
      tile_outer(acc, B2, B0, nn, pt, lv);
      // one writer per element: reductions without a return
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (pt.r + i >= nn) continue;
        float* p = a.dG + (base + pt.r + i) * a.m1 + pt.c;
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (pt.c + 32 * h < a.m1)
            atomicAdd(reinterpret_cast<float4*>(p + 32 * h),
                      make_float4(acc[i][4 * h], acc[i][4 * h + 1], acc[i][4 * h + 2], acc[i][4 * h + 3]));
      }
    }
  }
}

static int sm_count() {
  static int count = 0;
  if (count == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&count, cudaDevAttrMultiProcessorCount, dev);
    if (count <= 0) count = 1;
  }
  return count;
}

template <int A>
static void attn_f32_launch(const AttnArgs& a, bool bwd, cudaStream_t st) {
  const float scale = (float)(1.0 / sqrt((double)A));
  const int grid = a.n < sm_count() ? a.n : sm_count();
  if (!bwd) {
    const size_t smem = sizeof(float) * (2 * 128 * TLD + 4 * NP) + sizeof(float2) * NP;
    cudaFuncSetAttribute(k_attn_fwd_f32<A>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_pdl(k_attn_fwd_f32<A>, grid, FTF, smem, st, a, scale);
  } else {
    const size_t smem = sizeof(float) * (3 * 128 * TLD + 8 * NP) + sizeof(float2) * NP;
    cudaFuncSetAttribute(k_attn_bwd_f32<A>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_pdl(k_attn_bwd_f32<A>, grid, FTF, smem, st, a, scale);
  }
  note_launch();
}

// Attention widths with a kernel instance: 128 (the measured model) and 256
// (the paper's own model size).
void launch_attn_fwd_f32(const AttnArgs& a, cudaStream_t st) {
  if (a.n == 0) return;
  if (a.A == 256) attn_f32_launch<256>(a, false, st);
  else attn_f32_launch<128>(a, false, st);
}

void launch_attn_bwd_f32(const AttnArgs& a, cudaStream_t st) {
  if (a.n == 0) return;
  if (a.A == 256) attn_f32_launch<256>(a, true, st);
  else attn_f32_launch<128>(a, true, st);
}

// ------------------------------------------------------------- descriptor
// T = R^T G / sel (4 x m1); D = T^T T[:, :axis]; X = [D (row-major), Z[t_i]].
// A block of 128 threads per atom, 10 blocks per SM (48 registers): the kernel
// waits on its loads, and more resident warps hide more of them.  CQ: G and dG
// interleaved per atom (the fused paths), else packed rows.
template <bool CQ>
__global__ void __launch_bounds__(128, CQ ? 10 : 6) k_desc_fwd(DescArgs a) {
  pdl_wait();
  extern __shared__ float sm[];
  float* Ts = sm;  // [4][m1]
  const int atom = blockIdx.x;
  const int nn = a.nnei[atom];
  const size_t base = (size_t)atom * NP;
  const float inv_sel = 1.0f / (float)a.sel;
  if (CQ) {
    // a warp per column quad, its lanes over the rows
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const float4* G4 = reinterpret_cast<const float4*>(a.G + base * a.m1);
    const float4* R4 = reinterpret_cast<const float4*>(a.R) + base;
    for (int q = warp; q < a.m1 / 4; q += nw) {
      float t[4][4] = {};
      // the lane's (at most NP / 32) rows, their loads issued together
      float4 rq[NP / 32], gq[NP / 32];
#pragma unroll
      for (int it = 0; it < NP / 32; ++it) {
        const int s = lane + 32 * it;
        rq[it] = s < nn ? R4[s] : make_float4(0.f, 0.f, 0.f, 0.f);
        gq[it] = s < nn ? G4[(size_t)q * NP + s] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int it = 0; it < NP / 32; ++it) {
        const float rr[4] = {rq[it].x, rq[it].y, rq[it].z, rq[it].w};
        const float gg[4] = {gq[it].x, gq[it].y, gq[it].z, gq[it].w};
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
          for (int k = 0; k < 4; ++k) t[c][k] = fmaf(rr[c], gg[k], t[c][k]);
      }
      float tv[16];
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int k = 0; k < 4; ++k) tv[4 * c + k] = t[c][k];
      const float v = warp_reduce_scatter16(tv);  // lane l: entry l % 16 = (c, k) = (l / 4, l % 4)
      if (lane < 16) Ts[(lane >> 2) * a.m1 + 4 * q + (lane & 3)] = v * inv_sel;
    }
  } else {
    const size_t gbase = a.row_off[atom];
    for (int c = threadIdx.x; c < a.m1; c += blockDim.x) {
      float t0 = 0.f, t1 = 0.f, t2 = 0.f, t3 = 0.f;
#pragma unroll 8  // eight rows' loads in flight ahead of the FMA chains
      for (int s = 0; s < nn; ++s) {
        const float4 r = reinterpret_cast<const float4*>(a.R)[base + s];
        const float gv = a.G[(gbase + s) * a.m1 + c];
        t0 = fmaf(r.x, gv, t0); t1 = fmaf(r.y, gv, t1); t2 = fmaf(r.z, gv, t2); t3 = fmaf(r.w, gv, t3);
      }
      Ts[c] = t0 * inv_sel; Ts[a.m1 + c] = t1 * inv_sel; Ts[2 * a.m1 + c] = t2 * inv_sel; Ts[3 * a.m1 + c] = t3 * inv_sel;
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 4 * a.m1; t += blockDim.x) a.T[(size_t)atom * 4 * a.m1 + t] = Ts[t];
  float* x = a.X + (size_t)atom * a.fit_in;
  // D, element p * axis + b: (p, b) advance without a division
  const int dp = blockDim.x / a.axis, db = blockDim.x % a.axis;
  int p = threadIdx.x / a.axis, b = threadIdx.x % a.axis;
  for (int idx = threadIdx.x; idx < a.m1 * a.axis; idx += blockDim.x) {
    float d = 0.f;
#pragma unroll
    for (int c = 0; c < 4; ++c) d = fmaf(Ts[c * a.m1 + p], Ts[c * a.m1 + b], d);
    x[idx] = d;
    p += dp;
    b += db;
    if (b >= a.axis) {
      b -= a.axis;
      ++p;
    }
  }
  const int ti = a.atype[atom];
  for (int t = threadIdx.x; t < a.tebd_dim; t += blockDim.x) x[a.m1 * a.axis + t] = a.tebd[ti * a.tebd_dim + t];
}

// dT[c][p] = sum_b<axis dD[p][b] T[c][b] + (p < axis) sum_q dD[q][p] T[c][q];
// dG_s = R_s dT / sel; dR_s = G_s dT^T / sel.
// The adjoint's first part, a block per atom: dT [4][m1] in shared memory.
__device__ __forceinline__ float* desc_dt(const DescArgs& a, float* sm, int atom) {
  const int m1 = a.m1, ax = a.axis;
  float* Ts = sm;              // [4][m1]
  float* dTs = Ts + 4 * m1;    // [4][m1]
  float* dD = dTs + 4 * m1;    // [m1][axis]
  float* dDt = dD + m1 * ax;   // [axis][m1]: dD transposed, so that threads with consecutive p read consecutive words
  const float inv_sel = 1.0f / (float)a.sel;
  for (int t = threadIdx.x; t < 4 * m1; t += blockDim.x) Ts[t] = a.T[(size_t)atom * 4 * m1 + t];
  {
    const float* dX = a.dX + (size_t)atom * a.fit_in;
    const int dp = blockDim.x / ax, db = blockDim.x % ax;
    int p = threadIdx.x / ax, b = threadIdx.x % ax;
#pragma unroll 4
    for (int t = threadIdx.x; t < m1 * ax; t += blockDim.x) {
      const float v = dX[t];
      dD[t] = v;
      dDt[b * m1 + p] = v;
      p += dp;
      b += db;
      if (b >= ax) {
        b -= ax;
        ++p;
      }
    }
  }
  __syncthreads();
  for (int p = threadIdx.x; p < m1; p += blockDim.x) {
    float v[4] = {};
    for (int b = 0; b < ax; ++b) {
      const float d = dDt[b * m1 + p];
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = fmaf(d, Ts[c * m1 + b], v[c]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) dTs[c * m1 + p] = p < ax ? v[c] : v[c] * inv_sel;
  }
  __syncthreads();
  // the axis columns' other term: all four rows of T at once, in as few warps
  for (int t = threadIdx.x; t < 4 * ax; t += blockDim.x) {
    const int c = t / ax, p = t % ax;
    float v = dTs[c * m1 + p];
#pragma unroll 8
    for (int q = 0; q < m1; ++q) v = fmaf(dD[q * ax + p], Ts[c * m1 + q], v);
    dTs[c * m1 + p] = v * inv_sel;
  }
  __syncthreads();
  return dTs;
}

__global__ void __launch_bounds__(128, 10) k_desc_dt(DescArgs a) {
  pdl_wait();
  extern __shared__ float sm[];
  const int atom = blockIdx.x, m1 = a.m1;
  const float* dTs = desc_dt(a, sm, atom);
  for (int t = threadIdx.x; t < 4 * m1; t += blockDim.x) a.dG[(size_t)atom * 4 * m1 + t] = dTs[t];
}

template <bool CQ>
__global__ void __launch_bounds__(128, 10) k_desc_bwd(DescArgs a) {
  pdl_wait();
  extern __shared__ float sm[];
  const int m1 = a.m1;
  const int atom = blockIdx.x;
  const int nn = a.nnei[atom];
  const size_t base = (size_t)atom * NP;
  const float* dTs = desc_dt(a, sm, atom);
  if constexpr (CQ) {
    // A thread per row: its dG row in column quads (consecutive threads ->
    // consecutive rows; live rows only: the fused layer kernels and the
    // embedding adjoint read no others) and its dR row, with the columns of
    // dT read as float4 broadcasts (m1 % 4 == 0)
    const int q4 = m1 / 4;
    float4* dG4 = reinterpret_cast<float4*>(a.dG + base * m1);
    const float4* G4 = reinterpret_cast<const float4*>(a.G + base * m1);
    const float4* dT4 = reinterpret_cast<const float4*>(dTs);
    for (int s = threadIdx.x; s < NP; s += blockDim.x) {
      float d0 = 0.f, d1 = 0.f, d2 = 0.f, d3 = 0.f;
      if (s < nn) {
        const float4 r = reinterpret_cast<const float4*>(a.R)[base + s];
#pragma unroll 1  // at 48 registers 10 blocks fit per SM (unrolled: 66 and 7, 30 % slower)
        for (int q = 0; q < q4; ++q) {
          const float4 g = G4[(size_t)q * NP + s];
          const float4 t[4] = {dT4[q], dT4[q4 + q], dT4[2 * q4 + q], dT4[3 * q4 + q]};
          const float gg[4] = {g.x, g.y, g.z, g.w};
          float4 v;
          float* vp = &v.x;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float t0 = (&t[0].x)[k], t1 = (&t[1].x)[k], t2 = (&t[2].x)[k], t3 = (&t[3].x)[k];
            vp[k] = r.x * t0 + r.y * t1 + r.z * t2 + r.w * t3;
            d0 = fmaf(gg[k], t0, d0); d1 = fmaf(gg[k], t1, d1);
            d2 = fmaf(gg[k], t2, d2); d3 = fmaf(gg[k], t3, d3);
          }
          dG4[(size_t)q * NP + s] = v;
        }
      }
      reinterpret_cast<float4*>(a.dR)[base + s] = make_float4(d0, d1, d2, d3);
    }
    return;
  }
  // Packed rows: a warp per row, a column quad per lane (m1 / 4 <= 32), whose four
  // rows of dT stay in registers: dG = R dT, dR = G dT^T.  Two rows at a time, so
  // that their loads and reductions overlap (four spill at 10 blocks per SM).
  // 15,668 atoms in bf16x: 651 us with a thread per dG element and a second pass
  // over G for dR, 332 so, 311 without the integer divisions of the first part.
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int q4 = m1 / 4;
  const size_t gbase = a.row_off[atom];
  const float4* G4 = reinterpret_cast<const float4*>(a.G + gbase * m1);
  float4* dG4 = reinterpret_cast<float4*>(a.dG + gbase * m1);
  const float4* R4 = reinterpret_cast<const float4*>(a.R) + base;
  float4* dR4 = reinterpret_cast<float4*>(a.dR) + base;
  const bool on = lane < q4;
  float t[4][4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float4 x = on ? reinterpret_cast<const float4*>(dTs + c * m1)[lane] : make_float4(0.f, 0.f, 0.f, 0.f);
    t[c][0] = x.x; t[c][1] = x.y; t[c][2] = x.z; t[c][3] = x.w;
  }
  constexpr int RB = 2;
  for (int s0 = warp; s0 < nn; s0 += nw * RB) {
    float4 g[RB], r[RB];
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const int s = s0 + i * nw;
      g[i] = on && s < nn ? G4[(size_t)s * q4 + lane] : make_float4(0.f, 0.f, 0.f, 0.f);
      r[i] = s < nn ? R4[s] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float d[RB][4];
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const int s = s0 + i * nw;
      const float gg[4] = {g[i].x, g[i].y, g[i].z, g[i].w};
      float4 v;
      float* vp = &v.x;
#pragma unroll
      for (int c = 0; c < 4; ++c) d[i][c] = 0.f;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        vp[k] = r[i].x * t[0][k] + r[i].y * t[1][k] + r[i].z * t[2][k] + r[i].w * t[3][k];
#pragma unroll
        for (int c = 0; c < 4; ++c) d[i][c] = fmaf(gg[k], t[c][k], d[i][c]);
      }
      if (on && s < nn) dG4[(size_t)s * q4 + lane] = v;
    }
#pragma unroll
    for (int i = 0; i < RB; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) d[i][c] = warp_sum(d[i][c]);
#pragma unroll
    for (int i = 0; i < RB; ++i) {
      const int s = s0 + i * nw;
      if (lane == 0 && s < nn) dR4[s] = make_float4(d[i][0], d[i][1], d[i][2], d[i][3]);
    }
  }
  for (int s = nn + threadIdx.x; s < NP; s += blockDim.x) dR4[s] = make_float4(0.f, 0.f, 0.f, 0.f);
}

void launch_desc_fwd(const DescArgs& a, cudaStream_t st) {
  if (a.n == 0) return;
  launch_pdl(a.cq ? k_desc_fwd<true> : k_desc_fwd<false>, a.n, 128, sizeof(float) * 4 * a.m1, st, a);
  note_launch();
}
void launch_desc_bwd(const DescArgs& a, cudaStream_t st) {
  if (a.n == 0) return;
  size_t sm = sizeof(float) * (8 * a.m1 + 2 * a.m1 * a.axis);
  launch_pdl(a.cq ? k_desc_bwd<true> : k_desc_bwd<false>, a.n, 128, sm, st, a);
  note_launch();
}
void launch_desc_dt(const DescArgs& a, cudaStream_t st) {
  if (a.n == 0) return;
  launch_pdl(k_desc_dt, a.n, 128, sizeof(float) * (8 * a.m1 + 2 * a.m1 * a.axis), st, a);
  note_launch();
}

// ------------------------------------------------------------ fitting head
__global__ void k_energy_head(const float* __restrict__ H, const float* __restrict__ Hp, int n, int nlocal, int width,
                              const float* __restrict__ w, const float* __restrict__ bptr,
                              const float* __restrict__ ebias, const int* __restrict__ atype, float* __restrict__ e,
                              float* __restrict__ dH, float* __restrict__ dZ) {
  pdl_wait();
  const int atom = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (atom >= n) return;
  float s = 0.f;
  for (int c = lane; c < width; c += 32) {
    const size_t i = (size_t)atom * width + c;
    const float h = H[i], wc = w[c];
    s = fmaf(h, wc, s);
    const float t = Hp ? h - Hp[i] : h;
    const float d = atom < nlocal ? wc : 0.f;
    dH[i] = d;
    dZ[i] = d * (1.f - t * t);
  }
  s = warp_sum(s);
  if (lane == 0) e[atom] = (s + *bptr) + ebias[atype[atom]];
}

void launch_energy_head(const float* H, const float* Hprev, int n, int nlocal, int width, const float* w_out,
                        const float* b_out, const float* ebias, const int* atype, float* e, float* dH, float* dZ,
                        cudaStream_t st) {
  if (n == 0) return;
  launch_pdl(k_energy_head, (unsigned)(((long long)n * 32 + 255) / 256), 256, 0, st, H, Hprev, n, nlocal, width, w_out, b_out,
                                                                          ebias, atype, e, dH, dZ);
  note_launch();
}

__global__ void k_tanh_bwd(const float* __restrict__ dH, const float* __restrict__ Hc, const float* __restrict__ Hp,
                           float* __restrict__ dZ, long long count) {
  pdl_wait();
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const float t = Hp ? Hc[i] - Hp[i] : Hc[i];
  dZ[i] = dH[i] * (1.f - t * t);
}

void launch_tanh_bwd(const float* dH, const float* Hcur, const float* Hprev, float* dZ, long long count,
                     cudaStream_t st) {
  if (count == 0) return;
  launch_pdl(k_tanh_bwd, (unsigned)((count + 255) / 256), 256, 0, st, dH, Hcur, Hprev, dZ, count);
  note_launch();
}

}  // namespace dpa1
