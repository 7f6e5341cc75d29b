// Parts shared by the transform passes: lines of a shared-memory tile, the
// tile's header and the divisors of its copies.
#pragma once

#include "lgf_internal.h"

namespace lgf {

// Line l starts at (l / inner) * outer_stride + (l % inner) * inner_stride and
// its elements are es apart.
struct Lines {
  int nlines, inner, inner_stride, outer_stride, es;
  FastDiv dn, di;  // divisors by nlines and inner
};

static Lines make_lines(int nlines, int inner, int inner_stride, int outer_stride, int es) {
  return Lines{nlines, inner, inner_stride, outer_stride, es, FastDiv::make(nlines), FastDiv::make(inner)};
}

// Shared memory of a pass: twiddles of two directions, position tables of two
// directions, then the tile.  Returns the tile pointer.
template <typename R>
__device__ __forceinline__ C2<R>* setup_smem(unsigned char* raw, const C2<R>* __restrict__ twg,
                                             const short* __restrict__ posg, int n0, int n1, C2<R>** tw,
                                             short** pos) {
  *tw = reinterpret_cast<C2<R>*>(raw);
  const int twn = (n0 + n1 + 1) & ~1;
  *pos = reinterpret_cast<short*>(*tw + twn);
  const int posn = (n0 + n1 + 7) & ~7;  // keeps the tile 16-byte aligned
  for (int i = threadIdx.x; i < n0 + n1; i += blockDim.x) {
    (*tw)[i] = __ldg(&twg[i]);
    (*pos)[i] = __ldg(&posg[i]);
  }
  return reinterpret_cast<C2<R>*>(*pos + posn);
}

template <typename R> __host__ __device__ inline size_t smem_header_bytes(int n0, int n1) {
  return (size_t)((n0 + n1 + 1) & ~1) * sizeof(C2<R>) + (size_t)((n0 + n1 + 7) & ~7) * sizeof(short);
}

// Header of a plane pass: twiddles and position tables and, for FP64 fields,
// the block exponents of its planes (FxPlanes of lgf_fft_fx.cu).
constexpr size_t FX_PLANE_BYTES = 256;
constexpr int FX_MAX_THREADS = 384;  // CTA size limit of the FP64 plane passes
constexpr int FX_C_THREADS = 768;    // and of the one with g(x): threads per SM at 80 registers
constexpr int PAIR_MAX_THREADS = 384;  // and of the FP32 passes on pairs,
constexpr int PAIR_ZT_THREADS = 768;   // of the (z, t) pass where a tile fills an SM
inline size_t plane_header_bytes(int n0, int n1, int real_bytes) {
  return real_bytes == 8 ? smem_header_bytes<double>(n0, n1) + FX_PLANE_BYTES : smem_header_bytes<float>(n0, n1);
}

// Divisors of the global <-> shared copies of a pass.
struct CopyDiv {
  FastDiv a, b;
};

template <typename K> static cudaError_t allow_smem(K kernel, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace lgf
