// Shared definitions of the DPA-1 CUDA path (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <cstdint>
#include <utility>

namespace dpa1 {

// Programmatic dependent launch.  A small evaluation is some thirty kernels of
// 3 - 30 us, and a plain launch starts only once its predecessor has drained.
// Kernels of the evaluation are launched with launch_pdl: the next kernel is
// launched, and runs up to its pdl_wait, as this one's last blocks exit.  pdl_wait
// waits until the preceding kernel of the stream has finished and its writes are
// visible.  A kernel launched with launch_pdl calls it, in every thread that goes
// on, before it reads or writes anything that another kernel of the stream writes
// or reads (before it: barriers, TMEM, weights, which are written by ordinary launches
// ahead of the evaluation's first kernel only).  192 atoms: 484
// -> 426 us, 16 training frames of 582 atoms 14.3 -> 12.5 ms, 15,668 atoms 6.82 ->
// 6.75 ms.  An explicit early trigger (griddepcontrol.launch_dependents after the
// wait) made the waiting blocks compete with the running kernel: 15.6 ms for those
// frames, 6.82 ms.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... KArgs, class... Args>
void launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, KArgs(std::forward<Args>(args))...);
}

// Rows reserved per centre atom: the neighbour cap sel (<= 128) padded to one
// 128-row tile, so that every per-atom matrix has a fixed 128-row shape.
constexpr int NP = 128;
// Per-atom [NP][W] FP32 matrices of the tensor-core path (the layer inputs
// G_l and dE/dG) are stored column-quad interleaved: the 4 columns
// 4q..4q+3 of a row are contiguous and the NP rows of one column quad follow
// each other, so that one thread per row reading or writing 16 bytes makes a
// warp access 512 contiguous bytes.  The atom block keeps the size NP * W.
__host__ __device__ __forceinline__ size_t cq_off(int r, int c) {
  return ((size_t)(c >> 2) * NP + (size_t)r) * 4 + (size_t)(c & 3);
}

// Candidate capacity of the neighbour search per centre (before the sel cap).
constexpr int NBR_CAP = 256;
// Capacity of the reverse neighbour list per atom (centres that list it).
constexpr int REV_CAP = 256;

// Bits of the device status flag.
enum ErrBits : int {
  ERR_BOX = 1,       // box not orthorhombic or an edge <= 2 rcut
  ERR_CAPACITY = 2,  // candidate / reverse-list / workspace overflow
  ERR_NAN = 4,       // non-finite coordinate
  ERR_TIMEOUT = 8,   // a bounded wait gave up
  ERR_TYPE = 16,     // atom type out of range
};

// Cell grid derived on the device from the (device) box.
struct CellGrid {
  double L[3];
  double scale[3];  // nc / L
  int nc[3];
  int ncells;
  int ok;
};

__device__ __forceinline__ void set_err(int* err, int bits) { atomicOr(err, bits); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the 32 lanes of a warp of 16 values per lane; lanes l and l + 16
// return the sum of value l % 16 (butterfly reduce-scatter, fixed order;
// 16 shuffles instead of 16 full reductions).
__device__ __forceinline__ float warp_reduce_scatter16(float* v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int w = 8; w >= 1; w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const float send = up ? v[i] : v[i + w];
      const float keep = up ? v[i + w] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 16);
}

// Minimum-image displacement component d - L * rint(d / L), every operation
// rounded separately (no FMA contraction) so that the host can reproduce it
// bit for bit.
__device__ __forceinline__ double mic(double d, double L) {
  return __dsub_rn(d, __dmul_rn(L, rint(__ddiv_rn(d, L))));
}

// mic() without its division when no image shift is possible: for |d| < L/2 the
// rounded d / L lies in [-0.5, 0.5], rint gives 0 and mic returns d up to the sign of
// a zero.  The test compares the high words (strictly less there: less in value; NaN
// is not), since an FP64 instruction takes as long as some 70 of FP32 here (0.53 T
// FMA/s against 38.3).
__device__ __forceinline__ double mic_near(double d, double L) {
  return (__double2hiint(d) & 0x7fffffff) < __double2hiint(L) - 0x100000 ? d : mic(d, L);
}

// For the FP64 environment kernels, whose blocks of 2 NP threads hold the rows of two
// atoms: rec[4 a + c] = 1 / dstd[t_a][c], rec[8] = 1 / (rc - rcs).  An FP64 division is
// some twenty instructions at that rate, and with one a row for each of
// these the divisions bound the kernels: rows of the FP32 path, 3,001 atoms, 64 -> 45 us
// and 86 -> 63 (adjoint), tangents of 582 atoms 21 -> 15.
__device__ __forceinline__ void env_reciprocals(double* rec, const float* dstd, const int* atype, int n, double rcs,
                                                double rc) {
  const int t = threadIdx.x, i = 2 * blockIdx.x + (t >> 2);
  if (t < 8 && i < n) rec[t] = 1.0 / (double)dstd[4 * atype[i] + (t & 3)];
  if (t == 8) rec[8] = 1.0 / (rc - rcs);
  __syncthreads();
}

// Sorts 32 R unsigned values over a warp in ascending order: a bitonic network in
// registers, lane l ending up with places R l to R l + R - 1.  Strides below R need
// no exchange, the others one shuffle per value; in shared memory each of the
// network's stages waited for its loads and stores (128 values: 28 stages).
template <int R>
__device__ __forceinline__ void warp_sort(unsigned (&k)[R]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int kk = 2; kk <= 32 * R; kk <<= 1)
#pragma unroll
    for (int jj = kk >> 1; jj > 0; jj >>= 1) {
      if (jj >= R) {
        const bool up = kk == 32 * R || (lane & (kk / R)) == 0, low = (lane & (jj / R)) == 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const unsigned o = __shfl_xor_sync(0xffffffffu, k[r], jj / R);
          k[r] = up == low ? min(k[r], o) : max(k[r], o);
        }
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r)
          if ((r & jj) == 0) {
            const bool up = kk < R ? (r & kk) == 0 : kk == 32 * R || (lane & (kk / R)) == 0;
            const unsigned a = k[r], b = k[r | jj], lo = min(a, b), hi = max(a, b);
            k[r] = up ? lo : hi;
            k[r | jj] = up ? hi : lo;
          }
      }
    }
}

// (dx*dx + dy*dy) + dz*dz without contraction.
__device__ __forceinline__ double sqdist(double dx, double dy, double dz) {
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

}  // namespace dpa1
