// Register-tiled fp32 products of two sets of rows (fp32 inputs, and bf16 ones of very large histories): shared by the scoring
// passes and the history rebuild.  256 threads as 16 x 16, M x M results each; both operands transposed in shared memory.
#pragma once
#include "vatp_internal.cuh"

namespace vatp {
namespace {

constexpr int NTHREADS = 256;   // 16 x 16 threads, M x M results each

template <typename T> __device__ __forceinline__ float4 load4(const T* p);
template <> __device__ __forceinline__ float4 load4<float>(const float* p) { return *reinterpret_cast<const float4*>(p); }
template <> __device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16* p) {
  const uint2 r = *reinterpret_cast<const uint2*>(p);
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

// Packed fp32 pairs: one instruction for two FMAs (same rounding), which leaves issue slots for the loads.
typedef unsigned long long f32x2_t;
__device__ __forceinline__ f32x2_t pack_f32x2(float lo, float hi) {
  f32x2_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void fma_f32x2(f32x2_t& d, f32x2_t a, f32x2_t b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }

// s[i][j] += <A row micro_at(ty, i), B row micro_at(tx, j)> over NC channels in ascending order, as pairs along j
template <int M, int NC, int LD>
__device__ __forceinline__ void micro_gemm_add(const float* As, const float* Bs, int ty, int tx, f32x2_t (&s)[M][M / 2]) {
#pragma unroll 4
  for (int c = 0; c < NC; ++c) {
    float a[M];
    f32x2_t b[M / 2];
#pragma unroll
    for (int h = 0; h < M / 4; ++h) {
      *reinterpret_cast<float4*>(&a[4 * h]) = *reinterpret_cast<const float4*>(As + c * LD + h * 64 + ty * 4);
      const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(Bs + c * LD + h * 64 + tx * 4);
      b[2 * h] = x.x;
      b[2 * h + 1] = x.y;
    }
#pragma unroll
    for (int i = 0; i < M; ++i) {
      const f32x2_t aa = pack_f32x2(a[i], a[i]);
#pragma unroll
      for (int j = 0; j < M / 2; ++j) fma_f32x2(s[i][j], aa, b[j]);
    }
  }
}
template <int M>
__device__ __forceinline__ void unpack_products(const f32x2_t (&s2)[M][M / 2], float (&s)[M][M]) {
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int j = 0; j < M / 2; ++j) asm("mov.b64 {%0, %1}, %2;" : "=f"(s[i][2 * j]), "=f"(s[i][2 * j + 1]) : "l"(s2[i][j]));
}
template <int M, int D>
__device__ __forceinline__ void micro_gemm(const float* As, const float* Bs, int ty, int tx, float (&s)[M][M]) {
  f32x2_t s2[M][M / 2];
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int j = 0; j < M / 2; ++j) s2[i][j] = 0ull;
  micro_gemm_add<M, D, Tile<M, D>::LD>(As, Bs, ty, tx, s2);
  unpack_products<M>(s2, s);
}
// The same with B brought into shared memory here, 64 channels at a time (M = 8: A whole and half of B are 101 KB at 128
// channels, so that two CTAs fit on an SM and hide one another's loads).  Ends with every thread past its last read but one
// barrier short of letting B be overwritten.
template <typename T, int M, int D>
__device__ __forceinline__ void stream_gemm(const float* As, float* Bs, const T* src, int64_t row_stride, int row0, int rows_valid, int ty, int tx,
                                            float (&s)[M][M]) {
  f32x2_t s2[M][M / 2];
#pragma unroll
  for (int i = 0; i < M; ++i)
#pragma unroll
    for (int j = 0; j < M / 2; ++j) s2[i][j] = 0ull;
#pragma unroll 1
  for (int c0 = 0; c0 < D; c0 += 64) {
    float4 r[Tile<M, 64>::NV];
    Tile<M, 64>::fetch(r, src + c0, row_stride, row0, rows_valid);
    __syncthreads();
    Tile<M, 64>::store(Bs, r);
    __syncthreads();
    micro_gemm_add<M, 64, Tile<M, 64>::LD>(As + c0 * Tile<M, D>::LD, Bs, ty, tx, s2);
  }
  unpack_products<M>(s2, s);
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
