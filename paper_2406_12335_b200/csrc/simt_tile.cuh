// Register-tiled fp32 products of two sets of rows (fp32 inputs, and bf16 ones without tensor cores): shared by the scoring
// passes and the history rebuild.  256 threads as 16 x 16, M x M results each; both operands transposed in shared memory.
#pragma once
#include "vatp_internal.cuh"

namespace vatp {
namespace {

constexpr int NTHREADS = 256;   // 16 x 16 threads, M x M results each

template <typename T> __device__ __forceinline__ float4 load4(const T* p);
template <> __device__ __forceinline__ float4 load4<float>(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
template <> __device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16* p) {
  const uint2 r = __ldg(reinterpret_cast<const uint2*>(p));
  return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16), __uint_as_float(r.y & 0xffff0000u));
}

// A tile of 16 M rows x D channels, transposed: element (row, c) at [c][row], leading dimension LD (a multiple of four).
// Neighbouring lanes take neighbouring rows, so that the stores are free of bank conflicts.
template <int M, int D>
struct Tile {
  static constexpr int ROWS = 16 * M, LD = ROWS + 4, NV = ROWS * (D / 4) / NTHREADS;
  template <typename T>
  static __device__ __forceinline__ void fetch(float4 (&r)[NV], const T* src, int64_t row_stride, int row0, int rows_valid, int first_valid = 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int idx = threadIdx.x + i * NTHREADS, row = idx % ROWS, c4 = idx / ROWS;
      r[i] = row < rows_valid && row >= first_valid ? load4(src + (int64_t)(row0 + row) * row_stride + c4 * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  static __device__ __forceinline__ void store(float* dst, const float4 (&r)[NV]) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int idx = threadIdx.x + i * NTHREADS, row = idx % ROWS, c4 = idx / ROWS;
      float* o = dst + c4 * 4 * LD + row;
      o[0] = r[i].x; o[LD] = r[i].y; o[2 * LD] = r[i].z; o[3 * LD] = r[i].w;
    }
  }
};

// row (or column) of element i of the thread's t-th group: four consecutive ones, the second four half a tile on
template <int M> __device__ __forceinline__ int micro_at(int t, int i) { return (i >> 2) * 64 + t * 4 + (i & 3); }

// s[i][j] = <A row micro_at(ty, i), B row micro_at(tx, j)>, channels in ascending order
template <int M, int D>
__device__ __forceinline__ void micro_gemm(const float* As, const float* Bs, int ty, int tx, float (&s)[M][M]) {
  constexpr int LD = Tile<M, D>::LD;
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int j = 0; j < M; ++j) s[i][j] = 0.f;
#pragma unroll 4
  for (int c = 0; c < D; ++c) {
    float a[M], b[M];
#pragma unroll
    for (int h = 0; h < M / 4; ++h) {
      *reinterpret_cast<float4*>(&a[4 * h]) = *reinterpret_cast<const float4*>(As + c * LD + h * 64 + ty * 4);
      *reinterpret_cast<float4*>(&b[4 * h]) = *reinterpret_cast<const float4*>(Bs + c * LD + h * 64 + tx * 4);
    }
#pragma unroll
    for (int i = 0; i < M; ++i)
#pragma unroll
      for (int j = 0; j < M; ++j) s[i][j] = fmaf(a[i], b[j], s[i][j]);
  }
}

// launch configuration: programmatic dependent, clusters of cs CTAs along x
struct ClusterLaunch {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  ClusterLaunch(dim3 grid, size_t smem, cudaStream_t st, int cs) : cfg{} {
    cfg.gridDim = grid;
    cfg.blockDim = dim3(NTHREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cs;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
  }
};

}  // namespace
}  // namespace vatp
