// fp32 FMA prefill scoring: exact-product two-pass column sums of the causal softmax matrix.
//
// Pass 1 gives every query row its log-sum-exp (the normaliser of Eq. 1); pass 2 recomputes the
// logits tile by tile and adds exp(s - lse) into per-key sums (Eq. 2, or Eq. 3 when only the last
// w query rows count), fused with the value norm and the Eq. 4 product.  This is the path for
// fp32 inputs (tensor cores would round the operands).
// No float atomics: the CTAs of a cluster own a tile of rows (pass 1) or of keys (pass 2).
//
// Bound by the FMA pipes when there are many tiles, by latency when there are few.  So
//   * a thread holds M x M logits (M = 4 or 8) of a 16 M x 16 M tile; both operands sit in shared memory transposed, so
//     that M elements of a channel are one or two 16-byte loads: 2 (4) loads per 16 (64) FMAs - issued as packed pairs -
//     where one element per load made it 8 per 16.  The next tile's rows are on their way to registers under the products (M = 4);
//   * few tiles are shared out over a cluster of up to eight CTAs along the other dimension, which combine their row
//     statistics or column sums through distributed shared memory;
//   * both passes are programmatic dependents: they are resident when the launch before them ends, and by then pass 2 has its
//     key tile and, with 64-row tiles, its first query tile and the value norms, which depend on nothing that pass 1 writes;
//   * the CTAs of a cluster push their partial results to rank 0 and meet once: with rank 0 reading them from its partners
//     there were two meetings and a round trip between them.  (Rank 0's shared memory must have been claimed by then: every
//     CTA announces itself at once and waits for the others only when it sends, long after.)  The 16 threads of a row agree on
//     its maximum before they exponentiate.
// The scoring call, us: pass 2 starting late / two meetings a cluster / the rows merged pair by pair / all three / as it is:
// 2 heads x 512 tokens x 64 channels 18.3 / 17.2 / 17.0 / 20.4 / 16.0; 12 heads of 128, 512 tokens, a window of 256
// 53.2 / 54.2 / 52.4 / 58.5 / 50.8; 8 heads x 700 x 64 66.0 / 65.1 / 64.9 / 67.9 / 64.2.  128-row tiles (no clusters): 50 heads x
// 700 x 64 203.1 / - / 203.9 / 204.4 / 202.1; the row merge is worth more there than the 36 bytes of registers that it spills.
#include <cooperative_groups.h>

#include <type_traits>

#include "simt_tile.cuh"

namespace cg = cooperative_groups;

namespace vatp {
namespace {

constexpr int MAX_CLUSTER = 8;

// Pass 1: one cluster per (query tile, unit), its CTAs take every cs-th key tile.  lse[j] over keys i <= j.
template <typename T, int M, int D>
__global__ void __launch_bounds__(NTHREADS, M == 8 ? 2 : 1) rowstats_kernel(Shape sh, const T* q, const T* k,
                                                            float* __restrict__ lse, int first_row, int cs) {
  constexpr int ROWS = Tile<M, D>::ROWS, LD = Tile<M, D>::LD, NV = Tile<M, D>::NV;
  extern __shared__ __align__(16) float smem[];
  float* Qs = smem;
  float* Ks = smem + D * LD;
  __shared__ float2 part[M == 4 ? MAX_CLUSTER : 1][ROWS];      // (M = 8 has tiles enough without clusters)
  if (cs > 1) cluster_arrive_relaxed();
  // nothing is read before all earlier work has completed; pass 2 may set up from then on
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (threadIdx.x == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = cs > 1 ? (int)cluster.block_rank() : 0;
  // the longest rows of all units first: with the units one after the other the last ones left half the SMs idle
  const int item = blockIdx.x / cs, u = item % sh.units;
  const int ntile = (sh.T - first_row + ROWS - 1) / ROWS;
  const int q0 = first_row + (ntile - 1 - item / sh.units) * ROWS;
  const T* qu = q + unit_offset_q(sh, u);
  const T* ku = k + unit_offset(sh, u);
  const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
  const int last_key = min(q0 + ROWS, sh.T);  // exclusive

  float m[M], l[M];
#pragma unroll
  for (int i = 0; i < M; ++i) { m[i] = -INFINITY; l[i] = 0.f; }
  [[maybe_unused]] float4 next[M == 4 ? NV : 1];
  {
    float4 r[NV];
    Tile<M, D>::fetch(r, qu, sh.st, q0, min(ROWS, sh.T - q0));
    Tile<M, D>::store(Qs, r);
    if constexpr (M == 4)
      if (rank * ROWS < last_key) Tile<M, D>::fetch(next, ku, sh.st, rank * ROWS, min(ROWS, sh.T - rank * ROWS));
  }
  for (int k0 = rank * ROWS; k0 < last_key; k0 += cs * ROWS) {
    float s[M][M];
    if constexpr (M == 4) {
      __syncthreads();
      Tile<M, D>::store(Ks, next);
      __syncthreads();
      if (k0 + cs * ROWS < last_key) Tile<M, D>::fetch(next, ku, sh.st, k0 + cs * ROWS, min(ROWS, sh.T - k0 - cs * ROWS));
      micro_gemm<M, D>(Qs, Ks, ty, tx, s);
    } else {
      stream_gemm<T, M, D>(Qs, Ks, ku, sh.st, k0, min(ROWS, sh.T - k0), ty, tx, s);
    }
#pragma unroll
    for (int i = 0; i < M; ++i) {
      const int row = q0 + micro_at<M>(ty, i);
      float tile_max = -INFINITY;
#pragma unroll
      for (int j = 0; j < M; ++j) {
        const int col = k0 + micro_at<M>(tx, j);
        s[i][j] = (col <= row) ? s[i][j] * sh.scale : -INFINITY;
        tile_max = fmaxf(tile_max, s[i][j]);
      }
      if (tile_max > -INFINITY) {
        const float m_new = fmaxf(m[i], tile_max);
        float add = 0.f;
#pragma unroll
        for (int j = 0; j < M; ++j) add += expf(s[i][j] - m_new);
        l[i] = l[i] * expf(m[i] - m_new) + add;
        m[i] = m_new;
      }
    }
  }
  // merge the 16 threads (same ty, consecutive lanes) that share each row: the maximum first, then one factor a thread
  if (cs > 1) cluster_wait_acquire();
#pragma unroll
  for (int i = 0; i < M; ++i) {
    float mx = m[i];
#pragma unroll
    for (int off = 8; off >= 1; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    float sum = m[i] > -INFINITY ? l[i] * expf(m[i] - mx) : 0.f;
#pragma unroll
    for (int off = 8; off >= 1; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
    const int at = micro_at<M>(ty, i);
    if (tx == 0) {
      if (cs > 1) cluster.map_shared_rank(&part[0][0], 0)[(M == 4 ? rank : 0) * ROWS + at] = make_float2(mx, sum);
      else if (q0 + at < sh.T) lse[unit_offset_lse(sh, u) + q0 + at] = mx + logf(sum);
    }
  }
  if (cs > 1) {
    cluster.sync();       // (nobody reads another CTA's shared memory after it)
    if (rank == 0 && (int)threadIdx.x < ROWS && q0 + (int)threadIdx.x < sh.T) {
      float2 p[MAX_CLUSTER];
      float mx = -INFINITY, sum = 0.f;
#pragma unroll
      for (int r = 0; r < MAX_CLUSTER; ++r) {
        p[r] = r < cs ? part[M == 4 ? r : 0][threadIdx.x] : make_float2(-INFINITY, 0.f);
        mx = fmaxf(mx, p[r].x);
      }
#pragma unroll
      for (int r = 0; r < MAX_CLUSTER; ++r)
        if (p[r].x > -INFINITY) sum += p[r].y * expf(p[r].x - mx);
      lse[unit_offset_lse(sh, u) + q0 + threadIdx.x] = mx + logf(sum);
    }
  }
}

// Queries, keys and values of pass 2.  128-row tiles read them by the read-only path (32 heads x 2048 x 128 971 us, 1004 with
// ordinary loads): they are complete before the kernel starts, see launch_m.
template <typename T, int M> using Input = std::conditional_t<M == 8, const T* __restrict__, const T*>;

// Pass 2: one cluster per (key tile, unit), its CTAs take every cs-th query tile.  Column sums over query rows
// j >= max(first_row, k).
template <typename T, int M, int D>
__global__ void __launch_bounds__(NTHREADS, M == 8 ? 2 : 1)
colsum_kernel(Shape sh, Input<T, M> q, Input<T, M> k, Input<T, M> v, const float* lse, float* __restrict__ attn_acc,
              float* __restrict__ vnorm, float* __restrict__ score, float* __restrict__ win_rows, int first_row, int cs, bool after_pass1) {
  constexpr int ROWS = Tile<M, D>::ROWS, LD = Tile<M, D>::LD, NV = Tile<M, D>::NV;
  extern __shared__ __align__(16) float smem[];
  constexpr int DS = M == 4 ? D : 64;   // channels of the streamed tile in shared memory at a time
  float* Ks = smem;
  float* Qs = smem + D * LD;
  float* lse_s = Qs + DS * LD;          // [ROWS]
  float* red = Qs;                      // [16][ROWS], once the products are done (DS >= 16)
  __shared__ float vn_s[ROWS], part[M == 4 ? MAX_CLUSTER : 1][ROWS];
  if (cs > 1) cluster_arrive_relaxed();
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = cs > 1 ? (int)cluster.block_rank() : 0;
  const int item = blockIdx.x / cs, u = item % sh.units;      // the longest columns of all units first
  const int k0 = item / sh.units * ROWS;
  const T* qu = q + unit_offset_q(sh, u);
  const T* ku = k + unit_offset(sh, u);
  const T* vu = v + unit_offset(sh, u);
  const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
  const int keys_valid = min(ROWS, sh.T - k0);
  if (threadIdx.x == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // Everything this pass reads but the normalisers was complete before pass 1, which waits itself, released it: the first
  // tiles do not wait for pass 1, nor with 64-row tiles the value norms.  Without a pass 1 before it (normalisers given) it
  // waits first.  The normalisers are written while this kernel is resident: see DependentLaunch for how they may be loaded.
  if (!after_pass1) asm volatile("griddepcontrol.wait;" ::: "memory");

  // query tiles are aligned to first_row so that window rows map to whole tiles
  int qstart = first_row;
  if (k0 > first_row) qstart = first_row + ((k0 - first_row) / ROWS) * ROWS;
  const int qfirst = qstart + rank * ROWS;
  [[maybe_unused]] float4 next[M == 4 ? NV : 1];
  {
    float4 r[NV];
    Tile<M, D>::fetch(r, ku, sh.st, k0, keys_valid);
    Tile<M, D>::store(Ks, r);
    if constexpr (M == 4)
      if (qfirst < sh.T) Tile<M, D>::fetch(next, qu, sh.st, qfirst, min(ROWS, sh.T - qfirst));
  }
  // value norms (Eq. 4): four threads per row, by the last CTA of the cluster, which has the fewest query tiles
  auto value_norms = [&]() {
    if (rank != cs - 1) return;
    for (int r = threadIdx.x / 4; r < ROWS; r += NTHREADS / 4) {
      const int part4 = threadIdx.x % 4;
      float acc = 0.f;
      if (r < keys_valid) {
        const T* p = vu + (int64_t)(k0 + r) * sh.st;
#pragma unroll 4
        for (int c = part4 * 4; c < D; c += 16) {
          const float4 x = load4(p + c);
          acc = norm_fold(sh.norm, norm_fold(sh.norm, norm_fold(sh.norm, norm_fold(sh.norm, acc, x.x), x.y), x.z), x.w);
        }
      }
      acc = norm_merge(sh.norm, acc, __shfl_xor_sync(0xffffffffu, acc, 1));
      acc = norm_merge(sh.norm, acc, __shfl_xor_sync(0xffffffffu, acc, 2));
      if (part4 == 0) vn_s[r] = norm_finish(sh.norm, acc);
    }
  };
  if constexpr (M == 4) value_norms();      // (M = 8, whose launches fill the machine anyway: behind the products)
  float cs_sum[M];
#pragma unroll
  for (int j = 0; j < M; ++j) cs_sum[j] = 0.f;
  if (after_pass1) asm volatile("griddepcontrol.wait;" ::: "memory");

  const int wrow0 = sh.T - sh.window;   // query position of win_rows row 0 (may be negative)
  float* wr = win_rows ? win_rows + (int64_t)u * sh.window * sh.T : nullptr;

  if (wr && rank == 0) {
    // rows of the window that lie entirely above this key tile (j < k0): zeros
    for (int j = max(first_row, 0); j < min(qstart, sh.T); ++j)
      for (int c = threadIdx.x; c < keys_valid; c += NTHREADS) wr[(int64_t)(j - wrow0) * sh.T + k0 + c] = 0.f;
    // rows before the first token (T < w)
    for (int r = 0; r < -wrow0; ++r)
      for (int c = threadIdx.x; c < keys_valid; c += NTHREADS) wr[(int64_t)r * sh.T + k0 + c] = 0.f;
  }

  for (int q0 = qfirst; q0 < sh.T; q0 += cs * ROWS) {
    const int rows_valid = min(ROWS, sh.T - q0);
    // (s[i][j]: key k0 + micro_at(ty, i), query q0 + micro_at(tx, j))
    float s[M][M];
    const float l = (int)threadIdx.x < rows_valid ? lse[unit_offset_lse(sh, u) + q0 + threadIdx.x] : 0.f;
    if constexpr (M == 4) {
      __syncthreads();
      Tile<M, D>::store(Qs, next);
      if ((int)threadIdx.x < ROWS) lse_s[threadIdx.x] = l;
      __syncthreads();
      if (q0 + cs * ROWS < sh.T) Tile<M, D>::fetch(next, qu, sh.st, q0 + cs * ROWS, min(ROWS, sh.T - q0 - cs * ROWS));
      micro_gemm<M, D>(Ks, Qs, ty, tx, s);
    } else {
      __syncthreads();                  // (every thread is past its last read of lse_s)
      if ((int)threadIdx.x < ROWS) lse_s[threadIdx.x] = l;
      stream_gemm<T, M, D>(Ks, Qs, qu, sh.st, q0, rows_valid, ty, tx, s);
    }
#pragma unroll
    for (int j = 0; j < M; ++j) {
      const int row = q0 + micro_at<M>(tx, j);
      const float lr = lse_s[micro_at<M>(tx, j)];
#pragma unroll
      for (int i = 0; i < M; ++i) {
        const int col = k0 + micro_at<M>(ty, i);
        float p = 0.f;
        if (row < sh.T && col <= row && col < sh.T) p = expf(s[i][j] * sh.scale - lr);
        cs_sum[i] += p;
        if (wr && row < sh.T && col < sh.T) wr[(int64_t)(row - wrow0) * sh.T + col] = p;
      }
    }
  }
  if constexpr (M == 8) value_norms();
  __syncthreads();
#pragma unroll
  for (int i = 0; i < M; ++i) red[tx * ROWS + micro_at<M>(ty, i)] = cs_sum[i];
  __syncthreads();
  float tot = 0.f;
  if ((int)threadIdx.x < ROWS) {
#pragma unroll
    for (int t = 0; t < 16; ++t) tot += red[t * ROWS + threadIdx.x];
  }
  if (cs > 1) {
    cluster_wait_acquire();
    if ((int)threadIdx.x < ROWS) {
      cluster.map_shared_rank(&part[0][0], 0)[(M == 4 ? rank : 0) * ROWS + threadIdx.x] = tot;
      if (rank == cs - 1) cluster.map_shared_rank(vn_s, 0)[threadIdx.x] = vn_s[threadIdx.x];
    }
    cluster.sync();       // (nobody reads another CTA's shared memory after it)
  }
  if (rank == 0 && (int)threadIdx.x < keys_valid) {
    if (cs > 1) {
      tot = 0.f;
#pragma unroll
      for (int r = 0; r < MAX_CLUSTER; ++r)
        if (r < cs) tot += part[M == 4 ? r : 0][threadIdx.x];
    }
    const float n1 = vn_s[threadIdx.x];
    const int64_t o = (int64_t)u * sh.T + k0 + threadIdx.x;
    attn_acc[o] = tot;
    vnorm[o] = n1;
    score[o] = tot * n1;
  }
}

template <typename T, int M, int D>
cudaError_t launch_m(const Shape& s, const T* q, const T* k, const T* v, float* lse, float* attn_acc, float* vnorm,
                     float* score, float* win_rows, cudaStream_t st, bool lse_given) {
  using Tl = Tile<M, D>;
  const size_t smem1 = sizeof(float) * (D + (M == 4 ? D : 64)) * Tl::LD, smem2 = smem1 + sizeof(float) * Tl::ROWS;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(rowstats_kernel<T, M, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem1)) != cudaSuccess) return e;
  if ((e = cudaFuncSetAttribute(colsum_kernel<T, M, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2)) != cudaSuccess) return e;
  const int first_row = s.window > 0 ? (s.T > s.window ? s.T - s.window : 0) : 0;
  const int qtiles = (s.T - first_row + Tl::ROWS - 1) / Tl::ROWS, ktiles = (s.T + Tl::ROWS - 1) / Tl::ROWS;
  // Clusters while the grid leaves SMs idle and there are tiles to share: the longest row of tiles bounds the pass.
  auto cluster_for = [&](int tiles, int most) {
    int cs = 1;
    while (cs < MAX_CLUSTER && (int64_t)tiles * s.units * cs * 2 <= 2 * device_sm_count() && cs < most) cs *= 2;
    return cs;
  };
  if (!lse_given) {
    const int cs = cluster_for(qtiles, ktiles);
    ClusterLaunch c1(dim3((unsigned)(qtiles * s.units * cs)), smem1, st, cs);
    if ((e = cudaLaunchKernelEx(&c1.cfg, rowstats_kernel<T, M, D>, s, q, k, lse, first_row, cs)) != cudaSuccess) return e;
  }
  const int cs = cluster_for(ktiles, qtiles);
  ClusterLaunch c2(dim3((unsigned)(ktiles * s.units * cs)), smem2, st, cs);
  // Large tiles with the normalisers given, i.e. no pass 1 that has waited for what came before: an ordinary launch, when
  // everything is complete.  32 heads x 2048 x 128 506 -> 486 us, 50 x 700 x 64 106 -> 89 (as a dependent the next such call
  // takes SMs from this one), 32 x 2048 x 64 284 -> 288.  Short calls would lose the launch's latency (2 x 512 x 64 9.4 -> 10.7)
  // and stay dependents, with ordinary loads.
  if (M == 8 && lse_given) c2.attr[0].val.programmaticStreamSerializationAllowed = 0;
  return cudaLaunchKernelEx(&c2.cfg, colsum_kernel<T, M, D>, s, q, k, v, (const float*)lse, attn_acc, vnorm, score,
                            s.window > 0 ? win_rows : nullptr, first_row, cs, !lse_given);
}

template <typename T, int D>
cudaError_t launch_t(const Shape& s, const T* q, const T* k, const T* v, float* lse, float* attn_acc, float* vnorm,
                     float* score, float* win_rows, cudaStream_t st, bool lse_given) {
  // 128 x 128 tiles (half the shared-memory loads per FMA) once they fill the machine twice over in both passes
  const int rows = s.window > 0 && s.window < s.T ? s.window : s.T;
  const int64_t tiles = (int64_t)s.units * ((rows + 127) / 128);
  return tiles >= 2 * device_sm_count()
             ? launch_m<T, 8, D>(s, q, k, v, lse, attn_acc, vnorm, score, win_rows, st, lse_given)
             : launch_m<T, 4, D>(s, q, k, v, lse, attn_acc, vnorm, score, win_rows, st, lse_given);
}

template <typename T>
cudaError_t launch_d(const Shape& s, const T* q, const T* k, const T* v, float* lse, float* attn_acc, float* vnorm,
                     float* score, float* win_rows, cudaStream_t st, bool lse_given) {
  return s.d == 64 ? launch_t<T, 64>(s, q, k, v, lse, attn_acc, vnorm, score, win_rows, st, lse_given)
                   : launch_t<T, 128>(s, q, k, v, lse, attn_acc, vnorm, score, win_rows, st, lse_given);
}

}  // namespace

cudaError_t launch_prefill_simt(const Shape& s, int dtype, const void* q, const void* k, const void* v, float* lse,
                                float* attn_acc, float* vnorm, float* score, float* win_rows, cudaStream_t st,
                                bool lse_given) {
  if (dtype != VATP_F32) return cudaErrorNotSupported;      // (bf16: launch_prefill_tc)
  return launch_d<float>(s, (const float*)q, (const float*)k, (const float*)v, lse, attn_acc, vnorm, score, win_rows, st, lse_given);
}

}  // namespace vatp
