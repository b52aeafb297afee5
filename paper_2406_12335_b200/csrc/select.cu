// Budgeted selection: per unit, the top (B - F - R) scores of the middle range [F, T - R) by a
// block-wide radix select on the fp32 bit pattern, ties resolved towards the lower index, and
// the kept indices written in ascending order (first F, selected middle, last R).
// One CTA per unit; the unit's scores are staged in shared memory once when they fit and read
// from global memory (L2-resident) otherwise; for long prompts and few units a cluster of four or two CTAs shares a
// unit (select_cluster_kernel below).  Pure integer work after the key transform.
// The warps count into one to eight histograms that are summed per bin.  The scores
// of a head share a few exponents, so in the first passes nearly all keys of a warp fall into one bin:
// the lanes that agree with the warp's first candidate are counted by one addition (a ballot), the
// others by shared-memory atomics, which rarely collide once the digits spread.  (Grouping all equal
// digits with match.any cost more than everything else in the kernel: it takes time in proportion to
// the number of distinct values in the warp.)  As soon as at most 32 keys share the boundary's digits - after two passes
// for most units - one warp ranks those instead of two more passes.
// Lanes take four keys at a time: the passes were bound by issue slots (178 warp instructions per 32 keys).
// (256 units x 7936 keys with the compaction behind it 103.7 -> 98 us; 8 units x 7806 20.9 -> 19.6.)
#include <cooperative_groups.h>

#include "select_staging.h"
#include "vatp_internal.cuh"

namespace cg = cooperative_groups;

namespace vatp {
namespace {

constexpr int SEL_THREADS = 1024;
constexpr int SEL_WARPS = SEL_THREADS / 32;
constexpr size_t SEL_MAX = 168 * 1024, SEL_CLUSTER_MAX = 185 * 1024;      // dynamic shared memory of a CTA (beside 1 and 42 KB)

// order-preserving map float -> uint32 (larger float = larger key), valid for any sign
__device__ __forceinline__ uint32_t order_key(float x) {
  uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// THREADS: 1024 for one CTA per SM at a time, 512 when more units than SMs are to share the machine (the passes are chains
// of short phases; two or more CTAs per SM fill one another's).  copies: histograms the warps share out among them - one
// for short ranges, where clearing and summing 32 of them took longer than the counting.
template <bool STAGED, int THREADS>
__global__ void __launch_bounds__(THREADS) select_kernel(int copies, int T, int B, int F, int R, const float* score,
                                                             int32_t* __restrict__ kept, int32_t* dev_status) {
  constexpr int WARPS = THREADS / 32;
  extern __shared__ __align__(16) uint32_t sel_smem[];
  uint32_t* hist_c = sel_smem;                     // [copies][256] counts of the current pass
  uint32_t* keys_s = sel_smem + copies * 256;      // STAGED: keys of the middle range (from index `pad` on)
  __shared__ uint32_t hist[256];
  __shared__ uint32_t sh_prefix, sh_need, sh_in_bin, n_cand, cand[32];
  __shared__ uint32_t warp_keep[WARPS], warp_eq[WARPS];

  // Launched as a programmatic dependent: the next launch (the compaction) may set up now, and the
  // scores are read only once the launch that produced them has completed.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int u = blockIdx.x;
  const float* sc = score + (int64_t)u * T;
  int32_t* out = kept + (int64_t)u * B;
  const int tid = threadIdx.x;

  if (T <= B) {  // everything survives
    for (int i = tid; i < B; i += THREADS) out[i] = i < T ? i : -1;
    return;
  }
  const int n = T - R - F;   // middle range length (> 0 here because T > B >= F + R)
  const int ksel = B - F - R;  // how many of the middle range survive
  for (int i = tid; i < F; i += THREADS) out[i] = i;
  for (int i = tid; i < R; i += THREADS) out[B - R + i] = T - R + i;
  if (ksel == 0) return;

  // Staging: key i sits at keys_s[pad + i], pad chosen so that 16-byte loads from global memory pair with
  // 16-byte stores to shared memory.  Several loads per thread are in flight at once: one CTA has to pull the
  // whole unit through one SM, and with one 4-byte load per thread in flight that took longer than all the
  // rest of the kernel.
  int pad = 0;
  if (STAGED) {
    const float* mid = sc + F;
    const int a0 = min((int)(((16u - (uint32_t)(reinterpret_cast<uintptr_t>(mid) & 15u)) & 15u) >> 2), n);   // scalars before alignment
    pad = (4 - a0) & 3;
    const int nvec = (n - a0) >> 2;
    const float4* src4 = reinterpret_cast<const float4*>(mid + a0);
    uint4* dst4 = reinterpret_cast<uint4*>(keys_s + pad + a0);
    for (int v0 = 0; v0 < nvec; v0 += 4 * THREADS) {
      float4 x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int v = v0 + j * THREADS + tid;
        if (v < nvec) x[j] = load_behind_wait(src4 + v);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int v = v0 + j * THREADS + tid;
        if (v < nvec && VATP_INB(pad + a0 + 4 * v + 3, staged_words(n), dev_status)) dst4[v] = make_uint4(order_key(x[j].x), order_key(x[j].y), order_key(x[j].z), order_key(x[j].w));
      }
    }
    if (tid < a0) keys_s[pad + tid] = order_key(mid[tid]);
    const int tail0 = a0 + 4 * nvec;
    if (tid < n - tail0) keys_s[pad + tail0 + tid] = order_key(mid[tail0 + tid]);
    __syncthreads();
  }
  // Four keys at a time: group v holds keys 4 v - pad .. 4 v - pad + 3 of the middle range.
  const int nv = staged_groups(pad, n);
  struct Keys4 { uint32_t k[4]; };
  auto keys_of = [&](int v) -> Keys4 {
    Keys4 r;
    if (STAGED) {
      uint4 x = make_uint4(0u, 0u, 0u, 0u);
      if (VATP_INB(4 * v + 3, staged_words(n), dev_status)) x = reinterpret_cast<const uint4*>(keys_s)[v];
      r.k[0] = x.x; r.k[1] = x.y; r.k[2] = x.z; r.k[3] = x.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) r.k[e] = 4 * v + e < n ? order_key(sc[F + 4 * v + e]) : 0u;
    }
    return r;
  };
  auto in_range = [&](int v, int e) { return (unsigned)(4 * v + e - pad) < (unsigned)n; };

  // radix select, most significant byte first: find the key value tau of rank ksel (descending).
  uint32_t prefix = 0, mask = 0, need = (uint32_t)ksel, ties = 0xffffffffu;     // ties: keys equal to tau, when known
  const int lane = tid & 31, wid = tid >> 5;
  uint32_t* my_hist = hist_c + (wid % copies) * 256;
  for (int shift = 24; shift >= 0; shift -= 8) {
    for (int i = tid; i < copies * 256; i += THREADS) hist_c[i] = 0;
    if (tid == 0) n_cand = 0;
    __syncthreads();
    if (shift == 24) {
      // the top digit is a sign and seven exponent bits: most keys of a warp share the first lane's, which are counted
      // with ballots and added once; the others add one each
      for (int v0 = 0; v0 < nv; v0 += THREADS) {
        const int v = v0 + tid;
        Keys4 x;
        if (v < nv) x = keys_of(v);
        uint32_t d[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) d[e] = v < nv && in_range(v, e) ? x.k[e] >> 24 : 256u;
        const uint32_t d0 = __shfl_sync(0xffffffffu, d[3], 0);      // (256 where a warp begins in the padding: counts nothing)
        uint32_t same = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          same += __popc(__ballot_sync(0xffffffffu, d[e] == d0));
          if (d[e] != d0 && d[e] < 256u) atomicAdd(&my_hist[d[e]], 1u);
        }
        if (lane == 0 && d0 < 256u) atomicAdd(&my_hist[d0], same);
      }
    } else {
      // mantissa digits spread over the bins
      for (int v = tid; v < nv; v += THREADS) {
        const Keys4 x = keys_of(v);
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if ((x.k[e] & mask) == prefix && in_range(v, e)) atomicAdd(&my_hist[(x.k[e] >> shift) & 255u], 1u);
      }
    }
    __syncthreads();
    const uint32_t* totals = hist_c;
    if (copies > 1) {
      if (tid < 256) {
        uint32_t tot = 0;
#pragma unroll 8
        for (int w = 0; w < copies; ++w) tot += hist_c[w * 256 + tid];
        hist[tid] = tot;
      }
      __syncthreads();
      totals = hist;
    }
    if (tid < 32) {
      // walk the 256 bins from the top: 8 bins per lane, suffix sums by shuffles
      uint32_t c[8], tot = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) { c[j] = totals[255 - (tid * 8 + j)]; tot += c[j]; }
      uint32_t incl = tot;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
        if (tid >= off) incl += y;
      }
      uint32_t before = incl - tot;  // keys in strictly higher bins than this lane's first bin
      if (before < need && need <= incl) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (need <= before + c[j]) {
            sh_prefix = prefix | ((uint32_t)(255 - (tid * 8 + j)) << shift);
            sh_need = need - before;
            sh_in_bin = c[j];
            break;
          }
          before += c[j];
        }
      }
    }
    __syncthreads();
    prefix = sh_prefix;
    need = sh_need;
    ties = sh_in_bin;
    mask |= 255u << shift;
    if (shift > 0 && ties <= 32u) {
      // A warp's worth of keys share the digits so far (two passes are enough for most units): they are collected and
      // ranked against one another by one warp, in place of the remaining passes.
      for (int v = tid; v < nv; v += THREADS) {
        const Keys4 x = keys_of(v);
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if ((x.k[e] & mask) == prefix && in_range(v, e)) cand[atomicAdd(&n_cand, 1u)] = x.k[e];
      }
      __syncthreads();
      if (tid < 32) {
        const bool have = tid < (int)n_cand;
        const uint32_t key = have ? cand[tid] : 0u;
        uint32_t larger = 0, equal = 0;
        for (int j = 0; j < (int)n_cand; ++j) {
          const uint32_t other = __shfl_sync(0xffffffffu, key, j);
          larger += other > key;
          equal += other == key;
        }
        if (have && larger < need && need <= larger + equal) {    // lanes with equal keys write the same
          sh_prefix = key;
          sh_need = need - larger;
          sh_in_bin = equal;
        }
      }
      __syncthreads();
      prefix = sh_prefix;
      need = sh_need;
      ties = sh_in_bin;
      break;
    }
  }
  const uint32_t tau = prefix;     // the ksel-th largest key; `need` of the `ties` keys equal to tau survive
  const uint32_t need_eq = need;

  // Ordered compaction: keep key > tau, and the first need_eq (lowest index) keys equal to tau.
  // Warp w owns a contiguous range of key groups and walks it 32 groups at a time, a lane per group.
  // First the warps count their kept and tied keys, one scan over the warp totals gives every warp its
  // output offset and the rank of its first tie, then the warps write.
  const bool all_ties = ties == need_eq;             // the usual case: key >= tau decides
  const int per_w = (nv + WARPS - 1) / WARPS;
  const int lo = min(wid * per_w, nv), hi_v = min(lo + per_w, nv);
  const uint32_t lt_mask = (1u << lane) - 1u;
  uint32_t n_gt = 0, n_eq = 0;
  for (int v = lo + lane; v < hi_v; v += 32) {
    const Keys4 x = keys_of(v);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const bool in = in_range(v, e);
      n_gt += in && x.k[e] > tau;
      n_eq += in && x.k[e] == tau;
    }
  }
  n_gt = __reduce_add_sync(0xffffffffu, n_gt);
  n_eq = __reduce_add_sync(0xffffffffu, n_eq);
  if (lane == 0) { warp_keep[wid] = n_gt; warp_eq[wid] = n_eq; }
  __syncthreads();
  // exclusive prefix over the warps, computed by every warp for itself
  const uint32_t a = __reduce_add_sync(0xffffffffu, lane < wid ? warp_keep[lane] : 0u);
  uint32_t eq_rank = __reduce_add_sync(0xffffffffu, lane < wid ? warp_eq[lane] : 0u);     // ties before this warp's range
  uint32_t o = a + min(eq_rank, need_eq);           // output offset of this warp's first kept key
  for (int v0 = lo; v0 < hi_v; v0 += 32) {
    const int v = v0 + lane;
    Keys4 x;
    if (v < hi_v) x = keys_of(v);
    bool keep[4];
    uint32_t eq_before = eq_rank, eq_here = 0;
    if (!all_ties) {
#pragma unroll
      for (int e = 0; e < 4; ++e) eq_here += v < hi_v && in_range(v, e) && x.k[e] == tau;
      // ties of the lanes before this one
      uint32_t incl = eq_here;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
      }
      eq_before += incl - eq_here;
      eq_rank += __shfl_sync(0xffffffffu, incl, 31);
    }
    uint32_t at = o, step = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const bool in = v < hi_v && in_range(v, e);
      keep[e] = in && (x.k[e] > tau || (x.k[e] == tau && (all_ties || eq_before < need_eq)));
      if (!all_ties && in && x.k[e] == tau) ++eq_before;
      const uint32_t b = __ballot_sync(0xffffffffu, keep[e]);
      at += __popc(b & lt_mask);                     // kept keys of the lanes before this one
      step += __popc(b);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (keep[e]) {
        if (VATP_INB(F + at, B - R, dev_status)) out[F + at] = F + 4 * v + e - pad;
        ++at;
      }
    o += step;
  }
}


// ---- the same selection with a unit's middle range split over a cluster of CTAs -------------------------------
// For long prompts and few units one CTA per unit leaves most of the machine idle and counts 32 keys per thread and
// pass.  Here SPLIT CTAs take a contiguous quarter (or half) of the range each: a CTA counts its own keys, pushes its
// 256 bin totals into every partner's shared memory, and after one cluster barrier per pass all CTAs walk the same summed
// histogram to the same digit.  For the ordered write the CTAs exchange how many larger and how many equal keys they hold.
constexpr int SEL_MAXSPLIT = 4;
struct SelExchange {
  uint32_t hist[2][SEL_MAXSPLIT][256];     // per pass parity and rank: that CTA's bin totals
  uint32_t n_gt[SEL_MAXSPLIT], n_eq[SEL_MAXSPLIT];
};

__global__ void __launch_bounds__(SEL_THREADS) select_cluster_kernel(int T, int B, int F, int R, int split, int per,
                                                                     const float* score, int32_t* __restrict__ kept,
                                                                     int32_t* dev_status) {
  extern __shared__ __align__(16) uint32_t keys_s[];  // keys of this CTA's part of the middle range
  __shared__ uint32_t hist[256];
  __shared__ uint32_t hist_w[SEL_WARPS][256];
  __shared__ uint32_t sh_prefix, sh_need;
  __shared__ uint32_t warp_keep[SEL_WARPS], warp_eq[SEL_WARPS];
  __shared__ SelExchange xch;

  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int u = blockIdx.x / split;
  const float* sc = score + (int64_t)u * T;
  int32_t* out = kept + (int64_t)u * B;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  // (the host uses this kernel only when T > B and B - F - R > 0: every CTA passes every cluster barrier below)
  const int n = T - R - F;     // middle range length
  const int ksel = B - F - R;  // how many of the middle range survive
  // Remote shared memory may only be touched once its CTA runs: everyone arrives here and waits before the first remote store.
  cluster_arrive_release();
  if (rank == 0) {
    for (int i = tid; i < F; i += SEL_THREADS) out[i] = i;
    for (int i = tid; i < R; i += SEL_THREADS) out[B - R + i] = T - R + i;
  }
  const int lo_c = min(rank * per, n), hi_c = min(lo_c + per, n), n_c = hi_c - lo_c;    // this CTA's keys [lo_c, hi_c)
  for (int i = tid; i < n_c; i += SEL_THREADS) keys_s[i] = order_key(load_behind_wait(sc + F + lo_c + i));
  __syncthreads();
  cluster_wait_acquire();

  uint32_t prefix = 0, mask = 0, need = (uint32_t)ksel;
  int pass = 0;
  for (int shift = 24; shift >= 0; shift -= 8, ++pass) {
#pragma unroll
    for (int i = lane; i < 256; i += 32) hist_w[wid][i] = 0;
    __syncwarp();
    for (int base = 0; base < n_c; base += SEL_THREADS) {
      const int i = base + tid;
      uint32_t digit = 256u;                       // lanes without a candidate share a dummy digit
      if (i < n_c) {
        const uint32_t key = keys_s[i];
        if ((key & mask) == prefix) digit = (key >> shift) & 255u;
      }
      const uint32_t cand = __ballot_sync(0xffffffffu, digit < 256u);
      if (cand) {
        const int first = __ffs(cand) - 1;
        const uint32_t d0 = __shfl_sync(0xffffffffu, digit, first);
        const uint32_t same = __ballot_sync(0xffffffffu, digit == d0);
        if (lane == first) atomicAdd(&hist_w[wid][d0], (uint32_t)__popc(same));
        else if (digit < 256u && digit != d0) atomicAdd(&hist_w[wid][digit], 1u);
      }
    }
    __syncthreads();
    if (tid < 256) {
      uint32_t tot = 0;
#pragma unroll 8
      for (int w = 0; w < SEL_WARPS; ++w) tot += hist_w[w][tid];
      for (int r = 0; r < split; ++r) cluster.map_shared_rank(&xch, r)->hist[pass & 1][rank][tid] = tot;
    }
    cluster_arrive_release();
    cluster_wait_acquire();
    if (tid < 256) {
      uint32_t tot = 0;
      for (int r = 0; r < split; ++r) tot += xch.hist[pass & 1][r][tid];
      hist[tid] = tot;
    }
    __syncthreads();
    if (tid < 32) {
      // walk the 256 bins from the top: 8 bins per lane, suffix sums by shuffles
      uint32_t c[8], tot = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) { c[j] = hist[255 - (tid * 8 + j)]; tot += c[j]; }
      uint32_t incl = tot;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
        if (tid >= off) incl += y;
      }
      uint32_t before = incl - tot;  // keys in strictly higher bins than this lane's first bin
      if (before < need && need <= incl) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (need <= before + c[j]) {
            sh_prefix = prefix | ((uint32_t)(255 - (tid * 8 + j)) << shift);
            sh_need = need - before;
            break;
          }
          before += c[j];
        }
      }
    }
    __syncthreads();
    prefix = sh_prefix;
    need = sh_need;
    mask |= 255u << shift;
  }
  const uint32_t tau = prefix;     // the ksel-th largest key; `need` of the keys equal to tau survive
  const uint32_t need_eq = need;

  // Ordered compaction as in the single-CTA kernel, over this CTA's part; the CTAs before it in the range tell it how
  // many larger and how many equal keys precede its first one.
  const int per_w = ((n_c + SEL_WARPS - 1) / SEL_WARPS + 31) & ~31;
  const int lo = min(wid * per_w, n_c), hi_i = min(lo + per_w, n_c);
  const uint32_t lt_mask = (1u << lane) - 1u;
  uint32_t n_gt = 0, n_eq = 0;                      // warp-uniform
  for (int i0 = lo; i0 < hi_i; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t key = i < hi_i ? keys_s[i] : 0u;
    n_gt += __popc(__ballot_sync(0xffffffffu, i < hi_i && key > tau));
    n_eq += __popc(__ballot_sync(0xffffffffu, i < hi_i && key == tau));
  }
  if (lane == 0) { warp_keep[wid] = n_gt; warp_eq[wid] = n_eq; }
  __syncthreads();
  if (tid == 0) {
    uint32_t g = 0, e = 0;
    for (int w = 0; w < SEL_WARPS; ++w) { g += warp_keep[w]; e += warp_eq[w]; }
    for (int r = 0; r < split; ++r) {
      SelExchange* x = cluster.map_shared_rank(&xch, r);
      x->n_gt[rank] = g;
      x->n_eq[rank] = e;
    }
  }
  cluster_arrive_release();
  cluster_wait_acquire();
  uint32_t base_gt = 0, base_eq = 0;
  for (int r = 0; r < rank; ++r) { base_gt += xch.n_gt[r]; base_eq += xch.n_eq[r]; }
  // exclusive prefix over the warps, computed by every warp for itself
  uint32_t a = lane < wid ? warp_keep[lane] : 0u, b = lane < wid ? warp_eq[lane] : 0u;
#pragma unroll
  for (int off = 16; off; off >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, off);
    b += __shfl_xor_sync(0xffffffffu, b, off);
  }
  uint32_t eq_rank = base_eq + b;                   // ties before this warp's range
  uint32_t o = base_gt + a + min(eq_rank, need_eq); // output offset of this warp's first kept key
  for (int i0 = lo; i0 < hi_i; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t key = i < hi_i ? keys_s[i] : 0u;
    const bool is_eq = i < hi_i && key == tau;
    const uint32_t eq_b = __ballot_sync(0xffffffffu, is_eq);
    const bool keep = i < hi_i && (key > tau || (is_eq && eq_rank + __popc(eq_b & lt_mask) < need_eq));
    const uint32_t keep_b = __ballot_sync(0xffffffffu, keep);
    if (keep && VATP_INB(F + o + __popc(keep_b & lt_mask), B - R, dev_status)) out[F + o + __popc(keep_b & lt_mask)] = F + lo_c + i;
    o += __popc(keep_b);
    eq_rank += __popc(eq_b);
  }
  // nobody's shared memory is touched after the last barrier above: the CTAs may retire independently
}

}  // namespace

cudaError_t launch_select(int units, int T, int B, int F, int R, const float* score, int32_t* kept, int32_t* dev_status,
                          cudaStream_t st) {
  const int n = T > B ? T - R - F : 0;
  // long prompts, few units: the middle range of a unit goes to a cluster of four or two CTAs
  const int sms = device_sm_count();
  const int split = n >= 8192 && B - F - R > 0 ? (units * 4 <= sms ? 4 : (units * 2 <= sms ? 2 : 1)) : 1;
  const int per = ((n + split - 1) / split + 31) / 32 * 32;
  const size_t cbytes = (size_t)per * sizeof(uint32_t);
  // (a kernel's limit is always the same: another thread's call may be about to launch with a larger size than this one's)
  if (split > 1 && cbytes <= SEL_CLUSTER_MAX) {
    cudaError_t e = cudaFuncSetAttribute(select_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SEL_CLUSTER_MAX);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(units * split);
    cfg.blockDim = dim3(SEL_THREADS);
    cfg.dynamicSmemBytes = cbytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = split;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, select_cluster_kernel, T, B, F, R, split, per, score, kept, dev_status);
  }
  const int copies = n <= 2048 ? 1 : (n <= 16384 ? 4 : 8);
  const size_t hist_bytes = (size_t)copies * 256 * sizeof(uint32_t);
  const size_t bytes = hist_bytes + (size_t)staged_words(n) * sizeof(uint32_t);
  const bool staged = bytes <= SEL_MAX;
  // more units than SMs: CTAs of 512 threads, several to an SM
  const bool half = units > sms;
  auto kern = staged ? (half ? select_kernel<true, 512> : select_kernel<true, 1024>)
                     : (half ? select_kernel<false, 512> : select_kernel<false, 1024>);
  const size_t dyn = staged ? bytes : hist_bytes;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SEL_MAX);
  if (e != cudaSuccess) return e;
  DependentLaunch dl(dim3(units), dim3(half ? 512 : 1024), dyn, st);
  return cudaLaunchKernelEx(&dl.cfg, kern, copies, T, B, F, R, score, kept, dev_status);
}

}  // namespace vatp
