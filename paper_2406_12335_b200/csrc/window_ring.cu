// History-window state of the decode step (Eq. 3) rebuilt from Q and the compacted keys.
//
// The windowed indicator needs, per kept token, its probability under each of the last w prompt queries:
// ring[u][j mod w][slot] = a_slot^j for j = T - w .. T - 1, and the exact fixed-point sum of those w values
// (the indicator itself).  Rather than have the scoring pass write all w x T probabilities of a unit and
// gather B + 1 of their columns afterwards, this kernel recomputes the w x cap block that is kept:
//   p[j][slot] = exp(scale * <q_j, k_slot> - lse_j)   for pos[slot] <= j (causal), else 0
// a w x cap x d contraction per unit (tiny next to the T x T scoring passes), written straight into the ring's
// layout.  With grouped queries the history holds the MEAN over the KV group's query heads of their probabilities (the
// group-mean indicator's rows).  bf16 runs on the tensor cores (window_ring_tc_kernel, beside the scoring kernel whose
// machinery it shares); this file holds the dispatch and the FMA kernel for fp32 and for histories of 2^31 elements and more
// per unit, which the tensor-core kernel's 32-bit ring offsets do not reach.  The sums are integers (2^52 fixed
// point), so they do not depend on the order in which rows are added.
#include <cooperative_groups.h>

#include "simt_tile.cuh"

namespace cg = cooperative_groups;

namespace vatp {
namespace {

// One cluster per (tile of 64 slots, unit); its CTAs take every cs-th tile of 64 window rows.  A thread holds 4 rows x 4
// neighbouring slots; per head of the group one 64 x 64 x D product, the probabilities summed in ascending head order.
// The slots' window sums are integers: added up over a CTA's rows in shared memory and over the cluster by rank 0.
// (One thread per slot walking the window's rows in turn, its key row re-read from L2 for each: 24 units x 68 slots x 400
// rows x 64 channels took 1.1 ms, the whole compaction with it now 18 us.)
constexpr int RW_MAX_CLUSTER = 8;
template <typename T, int D>
__global__ void __launch_bounds__(NTHREADS)
window_ring_fma_kernel(Shape sh, int G, int B, int cap, const T* q, int64_t q_head, const float* lse,
                       vatp_cache c, int cs) {
  using Tl = Tile<4, D>;
  constexpr int ROWS = Tl::ROWS, LD = Tl::LD, NV = Tl::NV;
  extern __shared__ __align__(16) float smem[];
  float* Qs = smem;
  float* Ks = smem + D * LD;
  __shared__ float lse_s[ROWS];
  __shared__ long long fx_s[ROWS];
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = cs > 1 ? (int)cluster.block_rank() : 0;
  const int u = blockIdx.y, slot0 = (int)(blockIdx.x / cs) * ROWS;
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
  const int w = sh.window, len = min(sh.T, B);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const T* qu = q + unit_offset_q(sh, u);
  const float* lu = lse + unit_offset_lse(sh, u);
  const T* ku = static_cast<const T*>(c.k_cache) + (int64_t)u * cap * D;
  const bool wide = (reinterpret_cast<uintptr_t>(c.ring) & 15) == 0;      // (cap is a multiple of eight)
  {
    float4 r[NV];
    Tl::fetch(r, ku, D, slot0, min(ROWS, cap - slot0));
    Tl::store(Ks, r);
  }
  int ps[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int slot = slot0 + tx * 4 + j;
    ps[j] = slot < len ? c.pos[(int64_t)u * cap + slot] : -1;
  }
  long long fx[4] = {0, 0, 0, 0};
  const float invG = 1.f / (float)G;
  for (int r0 = rank * ROWS; r0 < w; r0 += cs * ROWS) {
    const int j0 = sh.T - w + r0;               // query of the tile's first row (negative: before the prompt)
    const int first = max(-j0, 0), rows = min(ROWS, w - r0);
    float p[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) p[i][j] = 0.f;
    for (int g = 0; g < G; ++g) {
      float4 next[NV];
      Tl::fetch(next, qu + (int64_t)g * q_head, sh.st, j0, rows, first);
      const float l = tid < rows && tid >= first ? lu[(int64_t)g * sh.T + j0 + tid] : 0.f;
      __syncthreads();
      Tl::store(Qs, next);
      if (tid < ROWS) lse_s[tid] = l;
      __syncthreads();
      float s[4][4];
      micro_gemm<4, D>(Qs, Ks, ty, tx, s);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int row = ty * 4 + i;
        const float lr = lse_s[row];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (row >= first && row < rows && ps[j] >= 0 && ps[j] <= j0 + row) p[i][j] += expf(s[i][j] * sh.scale - lr);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int row = ty * 4 + i, slot = slot0 + tx * 4;
      if (row < rows && slot < cap) {
        const int jj = j0 + row, rr = jj >= 0 ? jj % w : jj + w;
        float* dst = c.ring + ((int64_t)u * w + rr) * cap + slot;
        if (G > 1) {
#pragma unroll
          for (int j = 0; j < 4; ++j) p[i][j] *= invG;
        }
        if (wide) {
          *reinterpret_cast<float4*>(dst) = make_float4(p[i][0], p[i][1], p[i][2], p[i][3]);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) dst[j] = p[i][j];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) fx[j] += prob_to_fixed(p[i][j]);
      }
    }
  }
  __syncthreads();                              // every thread is past its last read of Qs: the sums land there
  long long* red = reinterpret_cast<long long*>(Qs);      // [16][ROWS]
#pragma unroll
  for (int j = 0; j < 4; ++j) red[ty * ROWS + tx * 4 + j] = fx[j];
  __syncthreads();
  if (tid < ROWS) {
    long long tot = 0;
#pragma unroll
    for (int t = 0; t < 16; ++t) tot += red[t * ROWS + tid];
    fx_s[tid] = tot;
  }
  if (cs > 1) cluster.sync(); else __syncthreads();
  if (rank == 0 && tid < ROWS && slot0 + tid < cap) {
    long long tot = 0;
    for (int r = 0; r < cs; ++r) tot += cs > 1 ? cluster.map_shared_rank(fx_s, r)[tid] : fx_s[tid];
    c.acc_fixed[(int64_t)u * cap + slot0 + tid] = tot;
    c.acc[(int64_t)u * cap + slot0 + tid] = fixed_to_prob(tot);
  }
  if (cs > 1) cluster.sync();                   // nobody leaves while rank 0 reads
}

template <typename T, int D>
cudaError_t launch_fma(const Shape& s, int G, int B, const void* q, const float* lse, const vatp_cache& c, cudaStream_t st) {
  const int cap = cache_capacity(B);
  const int tiles = (cap + Tile<4, D>::ROWS - 1) / Tile<4, D>::ROWS, row_tiles = (s.window + Tile<4, D>::ROWS - 1) / Tile<4, D>::ROWS;
  // window rows go to a cluster while the grid leaves SMs idle
  int cs = 1;
  while (cs < RW_MAX_CLUSTER && (int64_t)tiles * s.units * cs * 2 <= 4 * device_sm_count() && cs < row_tiles) cs *= 2;
  const size_t smem = sizeof(float) * 2 * D * Tile<4, D>::LD;
  cudaError_t e = cudaFuncSetAttribute(window_ring_fma_kernel<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  ClusterLaunch cl(dim3(tiles * cs, s.units), smem, st, cs);
  return cudaLaunchKernelEx(&cl.cfg, window_ring_fma_kernel<T, D>, s, G, B, cap, static_cast<const T*>(q), s.qsh / G, lse, c, cs);
}

}  // namespace

cudaError_t launch_window_ring(const Shape& s, int G, int dtype, int B, const void* q, const float* lse, const vatp_cache& c,
                               int32_t* dev_status, cudaStream_t st) {
  if (dtype == VATP_BF16 && vatp_tc_available() && (int64_t)s.window * cache_capacity(B) < ((int64_t)1 << 31))
    return launch_window_ring_tc(s, G, B, q, lse, c, dev_status, st);
  if (dtype == VATP_F32)
    return s.d == 64 ? launch_fma<float, 64>(s, G, B, q, lse, c, st) : launch_fma<float, 128>(s, G, B, q, lse, c, st);
  return s.d == 64 ? launch_fma<__nv_bfloat16, 64>(s, G, B, q, lse, c, st) : launch_fma<__nv_bfloat16, 128>(s, G, B, q, lse, c, st);
}

}  // namespace vatp
