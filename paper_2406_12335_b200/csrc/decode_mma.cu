// Decode step for bf16, head_dim 64 or 128: append, attend (Eq. 1), indicator
// update (Eq. 2 / Eq. 3), importance (Eq. 4), release of the lowest-importance unprotected slot.
//
// The step is HBM-bound (every cached K and V row is read once) but so short - tens of megabytes -
// that fixed latencies decide its duration.  Hence:
//   * every warp has a ring of units - the K rows or the V rows of a 16-row group, one tiled TMA load each,
//     128-byte swizzled so that ldmatrix is conflict-free; the first units are requested before anything else happens;
//   * q.K^T and p.V run on the warp-level tensor-core path (mma.sync m16n8k16, bf16 in, fp32
//     accumulate) with the cached rows as the A operand, of which every row counts: S = K q^T with the queries in the eight
//     columns, O^T = V^T p with V^T out of ldmatrix.trans: sixteen rows or channels per instruction.  (With the queries as
//     A, half of the first phase's products were padding: 512 units x 1025 slots 57 against 55 us.)  p is split into two
//     bf16 halves (in columns of their own with up to four heads, as two products with more): the product keeps ~16 bits
//     of p;
//   * two phases, all K rows and then all V rows: no group of rows depends on another, and exponentials are taken once
//     per slot.  (One sweep with an online softmax was a chain of ~2300 cycles per 16-row group - fragments, products,
//     maximum, exponentials, fragments, products - of which eight warps per CTA hid too little: with the data already in
//     L2 it took 4 of a waiting step's 12.5 us.  tcgen05 with the rows as M and 16 columns was no faster than mma.sync:
//     its instructions issue 65 cycles apart for 4 KB of rows each.)
//   * eight warps and at most half of an SM's shared memory: two CTAs fit on an SM, so the
//     CTAs of the next launch are resident while this one runs.  A launch that has to wait for its predecessor has then
//     already filled its rings (its K and V rows are the one thing it may read early).  (Asking for the rest of its rows in
//     L2 as well, by bulk prefetch or line by line, made a step of 32 units x 2049 slots 0.1 to 2 us longer.);
//   * more units than CTAs fit on the machine: a CTA takes several, and a producer warp streams the next one's rows while
//     the tail of this one runs;
//   * a unit (sequence, head) is split over a thread-block cluster when units are few.  Every CTA pushes its
//     max and sum to all CTAs of the unit, and each of them the channels of its partial output that this one is to
//     sum up, with st.async: the receiver waits on an mbarrier of its own that counts the bytes (a cluster barrier
//     makes every CTA wait for a round trip of all).  Each CTA then knows the softmax normaliser, updates the indicators
//     of its own slots and sends its eviction candidate to rank 0, which picks.  No global scratch, one launch;
//   * consecutive steps overlap (programmatic dependent launch).  By default a step requests
//     K/V tiles early and reads everything else only after all earlier work in the stream has
//     completed; it releases the next launch after that wait (at once with a producer warp, else when its K rows are
//     in), so at most one unfinished predecessor exists while a step sets up, and the one cache row that predecessor
//     may have written - the row of its incoming token, recorded in last_slot - is re-read after
//     the wait and patched in.  A caller that steps several independent caches on one stream may
//     opt in (VATP_FLAG_DECODE_OVERLAP) to more: the host keeps, per stream, the buffers of the
//     last launches, and a launch that shares no buffer with any launch that can still be in
//     flight (another layer's or another sequence's cache) never waits: it releases
//     the next launch at once and only stays until the previous launch has completed, so
//     launches still complete in order and the number in flight is bounded by what fits on the
//     machine;
//   * grouped-query attention (several query heads share one cache; the paper leaves the case open and points at
//     a group-wise score, read here as the MEAN of the heads' probabilities): up to eight heads of a group ride
//     in the columns of the products (template parameter GT), so a K or V row is still read once per step.
// Measured (us per step, first and latest version): 32 units x 2049 slots, every launch waiting 12.5 -> 9.15; 256 units x
// 1639, launches overlapping 37 -> 32.5 (221 MB: 6.8 TB/s; a copy reaches 6.5); 512 units x 1025 with a history window
// 73 -> 55; 8 units x 2049, four heads each 11.0 -> 8.9.
#include <cooperative_groups.h>

#include <mutex>

#include "vatp_internal.cuh"

namespace cg = cooperative_groups;

namespace vatp {
namespace {

// Eight warps; the 16-row group g of a CTA goes to warp g mod 8, which takes its groups in ascending order
// (the logits of all of them, then their share of the output); the eight partial outputs are summed in warp order.
// Nothing of this depends on how a launch is scheduled or how much shared memory it takes: results are bit-identical
// either way.
constexpr int MW = 8;
constexpr int WT = MW * 32;           // consumer threads; a producer warp follows
constexpr int DM_THREADS = WT + 32;
// (the kernels' template parameter HD: head_dim, 64 or 128)
constexpr int GROUP = 16;             // rows per MMA group
template <int HD> constexpr int unit_bytes = GROUP * HD * 2;   // K rows (or V rows) of a group: [64-column half][16 rows][128 bytes]
constexpr int TILE_BYTES = GROUP * 128;    // 16 rows x 64 bf16, 128-byte swizzled
constexpr int MAX_SLOTS = 8;          // units a warp keeps in flight at most
constexpr int MAX_SPLIT = 8;
constexpr int GQ_HEADS = 8;           // grouped queries: query heads per cache this kernel takes (columns of the MMA tiles)
constexpr float LOG2E = 1.4426950408889634f;
constexpr unsigned long long NO_KEY = ~0ull;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// the same without suspending the warp (its other lanes have barriers of their own to look at)
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait (about one second): false when the copy never signalled.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  while (!mbar_try_wait(bar, parity))
    if (global_ns() - t0 > 1000000000ull) return false;
  return true;
}
// global -> shared bulk copy; dst, src and bytes are multiples of 16
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
__device__ __forceinline__ void st_shared16(uint32_t addr, const uint4& v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// address of `addr` (this CTA's shared memory) in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// asynchronous stores into another CTA's shared memory; its mbarrier counts the bytes when they have landed
__device__ __forceinline__ void st_async(uint32_t addr, float v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];"
               ::"r"(addr), "r"(__float_as_uint(v)), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async2(uint32_t addr, float a, float b, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];"
               ::"r"(addr), "r"(__float_as_uint(a)), "r"(__float_as_uint(b)), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d), "r"(bar) : "memory");
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
// D (16x8, fp32) += A (16x16, bf16, row) * B (16x8, bf16, col)
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// two floats -> packed bf16 pair (lo in the low half), round to nearest
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float warp_max(float x) {
  float y;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(x));
  return y;
}

// barrier over the consumer warps only
__device__ __forceinline__ void workers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(WT) : "memory"); }

struct __align__(16) Candidate {      // eviction candidate of a CTA, sent to rank 0 (key NO_KEY: none)
  unsigned long long key;
  int slot, pos;
};

// eviction order as one integer: lower importance first, among equals the higher position first
__device__ __forceinline__ unsigned long long evict_key(float I, int pos) {
  return ((unsigned long long)__float_as_uint(I) << 32) | (unsigned)(0x7fffffff - pos);
}
// minimum of a 64-bit key over the warp, in two 32-bit steps
__device__ __forceinline__ unsigned long long warp_min_key(unsigned long long key) {
  const unsigned h = (unsigned)(key >> 32);
  const unsigned mh = __reduce_min_sync(0xffffffffu, h);
  const unsigned ml = __reduce_min_sync(0xffffffffu, h == mh ? (unsigned)key : 0xffffffffu);
  return ((unsigned long long)mh << 32) | ml;
}

// GT = 1: one query head per cache (multi-head attention).  GT = GQ_HEADS: grouped queries - up to GQ_HEADS query
// heads (G of them, a run-time argument) share the cache of unit u: column g of the products carries head g, so every K and V row
// is read once for the whole group; the maxima, sums and partial outputs exist per head, and the indicator advances by
// the MEAN of the heads' probabilities.
// FEED: a producer warp keeps the rings full, for CTAs with several units.  Otherwise
// every warp requests its own rows: one warp less at 128 instead of 96 registers, and a shorter way from a freed slot to
// the next request, which is what a launch that has the machine to itself is bound by.
template <int HD, bool WINDOWED, int GT, bool FEED>
__global__ void __launch_bounds__(FEED ? DM_THREADS : WT, 2)
decode_mma_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v, int independent, int G,
                  int units, int state_in_smem, int part_in_ring, int split, int chunk, int ld, int nslot, int B, int cap, int F, int R, int w, int norm,
                  float scale_log2, vatp_cache c,
                  const __nv_bfloat16* q_new, const __nv_bfloat16* k_new,
                  const __nv_bfloat16* v_new, __nv_bfloat16* __restrict__ out,
                  int32_t* __restrict__ evicted, int32_t* __restrict__ dev_status) {
  constexpr int UNIT = unit_bytes<HD>, ROW_CHUNKS = HD / 8;   // 16-byte chunks of a row
  static_assert(WT >= HD, "one thread per output channel");
  extern __shared__ unsigned char dyn_raw[];
  unsigned char* dyn = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(dyn_raw) + 1023) & ~uintptr_t(1023));
  // [MW][nslot] units | partial outputs of the warps [MW][G][HD] (part_in_ring: in the warps' own rings instead) |
  // slices of partial outputs received [split][G][HD / split] | logits[G][ld] | per-slot state of this CTA's own
  // slots: acc (with a history window the ring row that leaves it), vnorm, pos, with a window the fixed-point sums.
  // Where the state does not fit beside the rings it is copied into the rings' memory once the streaming is over
  // (state_in_smem == 2; a CTA with one unit only) or read from global memory in the tail (state_in_smem == 0).
  unsigned char* ring_base = dyn;
  const int g_rows = GT > 1 ? G : 1;
  const int ring_bytes = MW * nslot * UNIT;
  float* part_o = reinterpret_cast<float*>(part_in_ring ? ring_base : dyn + ring_bytes);
  const int part_ld = part_in_ring ? nslot * (UNIT / 4) : g_rows * HD;       // floats from one warp's partial to the next
  float* xo = reinterpret_cast<float*>(dyn + ring_bytes + (part_in_ring ? 0 : MW * g_rows * HD * 4));
  float* logit_s = xo + g_rows * HD;
  float* acc_s = state_in_smem == 2 ? reinterpret_cast<float*>(ring_base) : logit_s + g_rows * ld;
  float* vn_s = acc_s + ld;
  int* pos_s = reinterpret_cast<int*>(vn_s + ld);
  long long* fx_s = reinterpret_cast<long long*>(pos_s + ld);

  __shared__ __align__(8) uint64_t full[MW * MAX_SLOTS], empty[MW * MAX_SLOTS], misc_bars[4];
  __shared__ float part_m[MW][GT], part_l[MW][GT];
  __shared__ float2 ex_ml[MAX_SPLIT][GT];          // per rank and head: max of its logits (log2 domain), sum of exp2(s - m)
  __shared__ float gq_fr[GT > 1 ? MAX_SPLIT : 1][GT], gq_f[GT], gq_invl[GT];
  __shared__ Candidate cand[MAX_SPLIT];            // in rank 0: every rank's eviction candidate
  __shared__ unsigned long long warp_key[MW];

  cg::cluster_group cluster = cg::this_cluster();
  const int rank = split > 1 ? (int)cluster.block_rank() : 0;
  const int tid = threadIdx.x, lane = tid & 31, wid = __shfl_sync(0xffffffffu, tid >> 5, 0);    // (wid: the same in every lane)
  const int j4 = lane & 3;
  uint64_t* state_full = &misc_bars[0];
  uint64_t* state_empty = &misc_bars[1];
  uint64_t* ex_bar = &misc_bars[2];                // the exchange of maxima, sums and partial outputs
  uint64_t* cand_bar = &misc_bars[3];              // rank 0: the candidates
  // This CTA's units: u0, u0 + u_step, ... (more than one only when no unit is split).
  const int u0 = blockIdx.x / split, u_step = gridDim.x / split;
  // its slot range inside a unit's allocation
  const int s0 = min(rank * chunk, cap);
  const int tile_alloc = min(chunk, cap - s0);
  // ld > chunk: the unit's last CTA takes a few slots more than its tiles hold, see tail_row
  const bool tail_cta = !FEED && ld > chunk && rank == split - 1;
  const int rows_alloc = tail_cta ? cap - s0 : tile_alloc;
  // Warp x's groups are x, x + MW, ...: as many as groups_of(x, rows) among the first `rows` rows.  Its units in order: the
  // K rows of its groups, then their V rows.  A launch requests the first units of its first unit (sequence, head) before
  // it may read how many rows are live; when fewer are than the allocation holds, those are dropped and the live ones
  // requested anew.
  auto groups_of = [](int x, int rows) { return x * GROUP < rows ? (rows - x * GROUP + MW * GROUP - 1) / (MW * GROUP) : 0; };
  auto copy_state = [&](int u, int t) {            // one thread: the per-slot state of this CTA's slots
    const int64_t o = (int64_t)u * cap + s0;
    mbar_expect_tx(smem_u32(state_full), (WINDOWED ? 20u : 12u) * rows_alloc);
    bulk_g2s(acc_s, WINDOWED ? c.ring + ((int64_t)u * w + (t % w)) * cap + s0 : c.acc + o, rows_alloc * 4, state_full);
    bulk_g2s(vn_s, c.vnorm + o, rows_alloc * 4, state_full);
    bulk_g2s(pos_s, c.pos + o, rows_alloc * 4, state_full);
    if (WINDOWED) bulk_g2s(fx_s, c.acc_fixed + o, rows_alloc * 8, state_full);
  };

  // Another CTA's shared memory may only be written once that CTA runs and its exchange barriers are armed: everyone
  // arrives here and waits (long since satisfied) just before the first remote store.
  // (A launch that waits for nobody lets its successor start first of all; with the barriers initialised by a thread each,
  // not one after the other, 16 units x 301 slots 2.7 -> 1.8 us per overlapping step.)
  if (independent && tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (tid < MW * MAX_SLOTS && tid % MAX_SLOTS < nslot) {
    mbar_init(&full[tid], 1);
    if (FEED) mbar_init(&empty[tid], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid == MW * MAX_SLOTS) {
    mbar_init(state_full, 1);
    mbar_init(state_empty, WT);
    mbar_init(ex_bar, 1);
    mbar_init(cand_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (split > 1) {
      mbar_expect_tx(smem_u32(ex_bar), (uint32_t)(8 * g_rows * split + 4 * g_rows * HD));
      if (rank == 0) mbar_expect_tx(smem_u32(cand_bar), (uint32_t)(split * sizeof(Candidate)));
    }
  }
  __syncthreads();
  if (split > 1) asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");

  auto issue = [&](int x, int u, int j, int n, int slot) {    // one lane: unit j of n groups into ring slot `slot` of warp x
    const uint32_t bar = smem_u32(&full[x * MAX_SLOTS + slot]);
    mbar_expect_tx(bar, UNIT);
    const bool is_v = j >= n;
    tma_load_3d(smem_u32(ring_base) + (x * nslot + slot) * UNIT, is_v ? &tm_v : &tm_k, bar, 0,
                u * cap + s0 + (x + MW * (is_v ? j - n : j)) * GROUP, 0);
  };
  auto bring_state = [&](int u) {            // one lane: the per-slot state into shared memory, or on its way to L2
    const int t = WINDOWED ? c.next_pos[u] : 0;
    if (state_in_smem == 1) {
      copy_state(u, t);
    } else {
      const int64_t o = (int64_t)u * cap + s0;
      if (WINDOWED) {
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"((const void*)((uintptr_t)(c.ring + ((int64_t)u * w + (t % w)) * cap + s0) & ~(uintptr_t)15)), "r"(rows_alloc * 4) : "memory");
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"((const void*)((uintptr_t)(c.acc_fixed + o) & ~(uintptr_t)15)), "r"(rows_alloc * 8) : "memory");
      } else {
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(c.acc + o), "r"(rows_alloc * 4) : "memory");
      }
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(c.vnorm + o), "r"(rows_alloc * 4) : "memory");
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(c.pos + o), "r"(rows_alloc * 4) : "memory");
    }
  };

  if (FEED && wid == MW) {
    // ---- the producer warp: lane x < MW feeds warp x, lane MW brings the per-slot state.  (A warp that issued its own
    // copies spent a quarter of its time on that.)
    const int na = lane < MW ? groups_of(lane, rows_alloc) : 0;
    const int early = min(nslot, 2 * na);
    // An independent launch has let its successor start at once, and stays until the launch before it has completed, so
    // that launches complete in order.  A launch that waits for its predecessor releases its successor
    // only after that wait: the successor's early tile requests then race with this launch alone, never with launches
    // before it.
    for (int j = 0; j < early; ++j) issue(lane, u0, j, na, j);
    __syncwarp();
    if (!independent) {
      __syncwarp();
      // Nothing but K and V rows is read before the previous launch has completed and its writes are visible.
      asm volatile("griddepcontrol.wait;" ::: "memory");
      if (lane == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    int u = u0, j = early, base = 0, n = na, total = 2 * na;     // next unit j of `total`; those below base were dropped
    int slot = early == nslot ? 0 : early, use = early == nslot ? 1 : 0;
    bool done = rows_alloc <= 0 || lane > MW || (lane == MW && state_in_smem == 2);
    auto live_groups = [&]() { return groups_of(lane, min(c.len[u] + 1 - s0, rows_alloc)); };
    if (lane < MW && !done) {
      n = live_groups();
      if (n != na) { base = early; total = early + 2 * n; }
    }
    __syncwarp();
    asm volatile("bar.arrive 2, %0;" ::"n"(WT + 32) : "memory");      // the live range has been read, see below
    uint64_t t0 = 0;
    for (uint32_t spins = 1; __any_sync(0xffffffffu, !done); ++spins) {
      if (!done && lane < MW) {
        if (j >= total) {
          u += u_step;
          done = u >= units;
          if (!done) { n = live_groups(); j = base = 0; total = 2 * n; }
        } else if (use == 0 || mbar_test(&empty[lane * MAX_SLOTS + slot], (use - 1) & 1)) {
          issue(lane, u, j - base, n, slot);
          ++j;
          if (++slot == nslot) { slot = 0; ++use; }
          spins = 0;
        }
      } else if (!done) {
        if (use == 0 || mbar_test(state_empty, (use - 1) & 1)) {
          bring_state(u);
          ++use;
          u += u_step;
          done = u >= units;
          spins = 0;
        }
      }
      if ((spins & 1023u) == 1023u) {      // nothing moved for a while: a bounded wait (lanes vote, so that all leave together)
        const uint64_t now = global_ns();
        if (t0 == 0) t0 = now;
        if (now - t0 > 1000000000ull) {
          if (!done && dev_status) atomicExch(dev_status, (int)VATP_ERR_TIMEOUT);
          done = true;
        }
      } else if (spins == 0) {
        t0 = 0;
      }
    }
    if (split > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (independent && lane == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
    return;
  }

  const int na_mine = groups_of(wid, tile_alloc), early_mine = min(nslot, 2 * na_mine);
  if (!FEED) {
    if (lane == 0)
      for (int j = 0; j < early_mine; ++j) issue(wid, u0, j, na_mine, j);
    __syncwarp();
  }
  // (their values are read after the wait; on their way to L2 meanwhile, since a layer's words have long left it)
  if (!FEED && !independent && tid < 4) {
    const int32_t* words = tid == 0 ? c.len : tid == 1 ? c.free_slot : tid == 2 ? c.next_pos : c.last_slot;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(words + u0));
  }
  if (!independent) asm volatile("griddepcontrol.wait;" ::: "memory");
  if (!FEED && tid == 32 && rows_alloc > 0 && state_in_smem != 2) bring_state(u0);
  const uint32_t full_a = smem_u32(&full[wid * MAX_SLOTS]), empty_a = smem_u32(&empty[wid * MAX_SLOTS]);
  const uint32_t ring_a = smem_u32(ring_base + (size_t)wid * nslot * UNIT);
  uint32_t slot = 0, unit_a = ring_a, par = 0;     // ring position of the next unit this warp consumes
  int n = na_mine;                        // live groups
  // !FEED: the units still to be requested, those of K among them, the next one's row
  const int row0 = u0 * cap + s0 + wid * GROUP;
  int to_request = 2 * na_mine - early_mine, k_left = max(na_mine - early_mine, 0);
  int next_row = row0 + (early_mine < na_mine ? early_mine : early_mine - na_mine) * (MW * GROUP);
  bool bad = false;                       // this lane's wait ran out: it no longer waits, the results are void
  // ldmatrix lane addressing: matrix i = lane / 8, row r = lane % 8.  A tile row is 128 bytes and its
  // 16-byte chunk c sits at position c ^ (row % 8).
  //   K (plain):  matrices (rows 0-7, k lo), (rows 0-7, k hi), (rows 8-15, k lo), (rows 8-15, k hi)
  //   V (trans):  matrices (rows 0-7, ch lo), (rows 0-7, ch hi), (rows 8-15, ch lo), (rows 8-15, ch hi): the A operand V^T
  const uint32_t row_off = (uint32_t)(((lane >> 4) * 8 + (lane & 7)) * 128), lm_x = (uint32_t)(((lane >> 3) & 1) ^ (lane & 7));
  auto arrived = [&]() {                  // the next unit is complete
    const uint32_t bar = full_a + 8 * slot;
    if (!mbar_try_wait(bar, par) && !bad && !mbar_wait(bar, par)) bad = true;
    __syncwarp();
  };
  auto request = [&](uint32_t bar, uint32_t dst) {       // the next unit of this warp
    if (lane == 0 && !bad) {
      mbar_expect_tx(bar, UNIT);
      tma_load_3d(dst, k_left > 0 ? &tm_k : &tm_v, bar, 0, next_row, 0);
    }
    --to_request;
    next_row = --k_left == 0 ? row0 : next_row + MW * GROUP;
  };
  auto release = [&](bool wrote) {        // this warp has read it: its slot may be filled again
    // generic-proxy stores into the slot must be ordered before the next bulk copy into it
    if (wrote) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (FEED) {
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty_a + 8 * slot) : "memory");
    } else {
      if (to_request > 0) request(full_a + 8 * slot, unit_a);
    }
    unit_a += UNIT;
    if (++slot == nslot) { slot = 0; unit_a = ring_a; par ^= 1; }
  };
  const bool has_chunk = (lane & 15) < ROW_CHUNKS;
  auto patch_row = [&](uint32_t tile, int rr, const uint4& raw, bool v_half) {
    const int ch = lane & 15;
    if (has_chunk && (lane >= 16) == v_half)
      st_shared16(tile + (ch >> 3) * TILE_BYTES + rr * 128 + (((ch & 7) ^ (rr & 7)) << 4), raw);
  };
  uint32_t state_par = 0;

  for (int u = u0; u < units; u += u_step) {
  // everything the step needs of the unit is requested at once
  const int len_m = c.len[u];
  const int fs_m = c.free_slot[u];
  const int t = c.next_pos[u];
  const int ls_m = c.last_slot[u];
  uint4 new_raw = make_uint4(0u, 0u, 0u, 0u), last_raw = make_uint4(0u, 0u, 0u, 0u);
  if (!FEED && has_chunk) new_raw = load_behind_wait(reinterpret_cast<const uint4*>((lane < 16 ? k_new : v_new) + (int64_t)u * HD) + (lane & 15));
  // B operand of K q^T: q in every column (grouped queries: column g carries head g of the unit's group, columns beyond the
  // group repeat its last head)
  const __nv_bfloat16* qn = GT > 1 ? q_new + ((int64_t)u * G + min(lane >> 2, G - 1)) * HD : q_new + (int64_t)u * HD;
  uint32_t qb[HD / 16][2];
#pragma unroll
  for (int ks = 0; ks < HD / 16; ++ks) {
    qb[ks][0] = load_behind_wait(reinterpret_cast<const uint32_t*>(qn + ks * 16 + 2 * j4));
    qb[ks][1] = load_behind_wait(reinterpret_cast<const uint32_t*>(qn + ks * 16 + 8 + 2 * j4));
  }
#ifdef VATP_DEBUG_BOUNDS
  // the state words come from memory: out of range they are clamped and reported (every access below stays inside)
  (void)(VATP_INB(len_m, cap, dev_status) && VATP_INB(fs_m, cap, dev_status) && VATP_INB(ls_m + 1, cap + 1, dev_status));
  const int len = min(max(len_m, 0), cap - 1), fs = min(max(fs_m, 0), cap - 1), ls = min(max(ls_m, -1), cap - 1);
#else
  const int len = len_m, fs = fs_m, ls = ls_m;
#endif
  const int hi = len + 1;                // slots [0, hi) are live once the new token is in
  const int cnt = max(min(hi - s0, rows_alloc), 0);
  const int fs_local = fs - s0;          // row of the incoming token inside this CTA's range (if owned)
  const bool owns_new = fs_local >= 0 && fs_local < cnt;
  const int ls_local = ls - s0;          // row the previous step appended (its tile may predate that store)
  const bool owns_last = !independent && ls >= 0 && ls != fs && ls_local >= 0 && ls_local < cnt;

  // ---- the group that holds the incoming token's row: its warp stores the row and its norm (Eq. 4) and patches the
  // row into the tiles it streams; the group that holds the row of the previous step's token likewise re-reads that row.
  // Lanes 0-15 take 16 bytes of the K row each, lanes 16-31 of the V row (with head_dim 64 the first eight of each).
  const int new_warp = owns_new ? (fs_local / GROUP) % MW : -1, last_warp = owns_last ? (ls_local / GROUP) % MW : -1;
  // the new row's norm is needed by the thread that updates its slot
  const int norm_warp = owns_new ? (fs_local % WT) / 32 : -1;
  if (FEED && has_chunk && (wid == new_warp || wid == norm_warp))
    new_raw = load_behind_wait(reinterpret_cast<const uint4*>((lane < 16 ? k_new : v_new) + (int64_t)u * HD) + (lane & 15));
  if (has_chunk && wid == last_warp)
    last_raw = *(reinterpret_cast<const uint4*>((const __nv_bfloat16*)(lane < 16 ? c.k_cache : c.v_cache) +
                                                ((int64_t)u * cap + ls) * HD) + (lane & 15));
  // ---- the slots beyond the tiles (a budget that fills whole tiles leaves the incoming token's): warp x takes row x / G for
  // head x mod G, a lane HD / 32 channels, with plain loads.  (As one more group of one warp, a single row made every
  // CTA of the unit wait for its two steps.)
  constexpr int TC = HD / 32;             // channels of a lane
  const int tail_row = GT > 1 ? wid / G : wid, tail_head = GT > 1 ? wid - tail_row * G : 0;
  const bool has_tail = tail_cta && chunk + tail_row < cnt;
  uint32_t tail_q[TC / 2], tail_k[TC / 2], tail_v[TC / 2];
#pragma unroll
  for (int x = 0; x < TC / 2; ++x) tail_q[x] = tail_k[x] = tail_v[x] = 0u;
  if (has_tail) {
    const int slot_u = s0 + chunk + tail_row;
    const int64_t o = ((int64_t)u * cap + slot_u) * HD + lane * TC, o_new = (int64_t)u * HD + lane * TC;
    const bool is_new = slot_u == fs;
    const __nv_bfloat16* kp = is_new ? k_new + o_new : (const __nv_bfloat16*)c.k_cache + o;
    const __nv_bfloat16* vp = is_new ? v_new + o_new : (const __nv_bfloat16*)c.v_cache + o;
    const __nv_bfloat16* qp = q_new + ((int64_t)u * g_rows + tail_head) * HD + lane * TC;
#pragma unroll
    for (int x = 0; x < TC / 2; ++x) {
      tail_q[x] = reinterpret_cast<const uint32_t*>(qp)[x];
      tail_k[x] = reinterpret_cast<const uint32_t*>(kp)[x];
      tail_v[x] = reinterpret_cast<const uint32_t*>(vp)[x];
    }
  }
  float new_norm = 0.f;
  auto incoming = [&]() {
    if (wid == new_warp || wid == norm_warp) {
      const uint32_t wv[4] = {new_raw.x, new_raw.y, new_raw.z, new_raw.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
        new_norm = norm_fold(norm, norm_fold(norm, new_norm, __uint_as_float(wv[i] << 16)), __uint_as_float(wv[i] & 0xffff0000u));
#pragma unroll
      for (int o = 8; o; o >>= 1) new_norm = norm_merge(norm, new_norm, __shfl_xor_sync(0xffffffffu, new_norm, o));
      new_norm = norm_finish(norm, __shfl_sync(0xffffffffu, new_norm, 16));      // the V half's partial
      if (wid == new_warp) {
        __nv_bfloat16* dst = (__nv_bfloat16*)(lane < 16 ? c.k_cache : c.v_cache) + ((int64_t)u * cap + fs) * HD;
        if (has_chunk) reinterpret_cast<uint4*>(dst)[lane & 15] = new_raw;
        if (lane == 0) {
          c.vnorm[(int64_t)u * cap + fs] = new_norm;
          c.pos[(int64_t)u * cap + fs] = t;
        }
      }
    }
  };
  if (FEED) incoming();                   // (otherwise while the unit's CTAs exchange)

  // ---- stream the rows: first all K rows (logits), then, with the CTA's maximum known, all V rows.  In one sweep with an
  // online softmax every 16-row group was a chain of ~2300 cycles (fragments, products, maximum, exponentials, fragments,
  // products) that eight warps walked through five times; here the groups of a warp depend on nothing, and exponentials
  // are taken once per slot instead of once per lane of an MMA tile.
  const int cnt_t = FEED ? cnt : min(cnt, chunk);     // live rows in tiles
  n = groups_of(wid, cnt_t);              // this warp's live groups
  if (u == u0 && n != na_mine) {          // rows requested before the live range was known: dropped (see the producer)
    if (!FEED) {
      to_request = 2 * n;
      k_left = n;
      next_row = row0;
      for (int j = early_mine; j < nslot && to_request > 0; ++j) request(full_a + 8 * j, ring_a + j * UNIT);     // (slots left free)
    }
    for (int i = early_mine; i > 0; --i) { arrived(); release(false); }
  }
  // The loops of both phases are software pipelined: a warp waits for its next group and requests its fragments while the
  // products of this one are under way.  (One group after the other was 950 cycles each of waits, fragments, products and
  // requests in turn; two groups at a
  // time found the rings, three units deep, empty.  What counts is the number of instructions: ring addresses and requests
  // kept as counters, edge cases behind one test per group: 32 units x 2049 slots 10.1 -> 9.7 us per step.)
  constexpr int RSTEP = MW * GROUP;       // rows from one group of a warp to its next
  const int r_end = n * RSTEP;
  float m_run[2] = {-INFINITY, -INFINITY};       // of heads 2 j4 and 2 j4 + 1 (one head: the same in every lane)
  uint32_t frag[HD / 16][4];              // a group's rows as the A operand
  bool wrote = false;
  const bool patches = wid == new_warp || wid == last_warp;
  // S = K q^T: the rows are the A operand, as in the second phase (as the B operand they took two products of which half
  // was padding)
  auto k_fetch = [&](int r0) {
    arrived();
    wrote = false;
    if (patches) {                        // the incoming token's row is not in the cache yet: patch it in
      const bool has_new = wid == new_warp && fs_local >= r0 && fs_local < r0 + GROUP;
      const bool has_last = wid == last_warp && ls_local >= r0 && ls_local < r0 + GROUP;
      if (has_new) patch_row(unit_a, fs_local - r0, new_raw, false);
      if (has_last) patch_row(unit_a, ls_local - r0, last_raw, false);
      wrote = has_new || has_last;
      __syncwarp();
    }
    const uint32_t kaddr = unit_a + row_off;
#pragma unroll
    for (int kk = 0; kk < HD / 16; ++kk) ldsm_x4(kaddr + (kk >> 2) * TILE_BYTES + ((lm_x ^ ((2 * kk) & 7)) << 4), frag[kk]);
  };
  if (!FEED && n > 0) k_fetch(wid * GROUP);
  for (int r0 = wid * GROUP; r0 < r_end; r0 += RSTEP) {
    if (FEED) k_fetch(r0);
    float sa[2][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) sa[0][i] = sa[1][i] = 0.f;
#pragma unroll
    for (int kk = 0; kk < HD / 16; ++kk)
      mma_bf16(sa[kk & 1], frag[kk][0], frag[kk][2], frag[kk][1], frag[kk][3], qb[kk][0], qb[kk][1]);
    release(wrote);
    if (!FEED && r0 + RSTEP < r_end) k_fetch(r0 + RSTEP);
    // this lane: rows lane / 4 and lane / 4 + 8, heads 2 j4 and 2 j4 + 1 (one head: the same value in every column)
    const int ra = r0 + (lane >> 2), rb = ra + 8;
    const bool ragged = r0 + GROUP > cnt_t;      // (chunk is a multiple of 16: dead rows of the last group have logits too, -inf)
#pragma unroll
    for (int x = 0; x < (GT > 1 ? 2 : 1); ++x) {
      float a = (sa[0][x] + sa[1][x]) * scale_log2, b = (sa[0][2 + x] + sa[1][2 + x]) * scale_log2;
      if (ragged) {
        if (ra >= cnt_t) a = -INFINITY;
        if (rb >= cnt_t) b = -INFINITY;
      }
      if (GT > 1 ? 2 * j4 + x < G : j4 == 0) {
        float* lg = logit_s + (GT > 1 ? (2 * j4 + x) * ld : 0);
        lg[ra] = a;
        lg[rb] = b;
      }
      m_run[x] = fmaxf(m_run[x], fmaxf(a, b));
    }
  }
  if (!FEED && has_tail) {
    float s = 0.f;
#pragma unroll
    for (int x = 0; x < TC / 2; ++x) {
      s = fmaf(__uint_as_float(tail_q[x] << 16), __uint_as_float(tail_k[x] << 16), s);
      s = fmaf(__uint_as_float(tail_q[x] & 0xffff0000u), __uint_as_float(tail_k[x] & 0xffff0000u), s);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    s *= scale_log2;
    if (lane == 0) logit_s[tail_head * ld + chunk + tail_row] = s;
#pragma unroll
    for (int x = 0; x < (GT > 1 ? 2 : 1); ++x)
      if (GT == 1 || 2 * j4 + x == tail_head) m_run[x] = fmaxf(m_run[x], s);
  }
#pragma unroll
  for (int x = 0; x < (GT > 1 ? 2 : 1); ++x) {
    if (GT == 1) {
      m_run[x] = warp_max(m_run[x]);
    } else {
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) m_run[x] = fmaxf(m_run[x], __shfl_xor_sync(0xffffffffu, m_run[x], o));
    }
    if (GT > 1 ? lane < 4 && 2 * j4 + x < G : lane == 0) part_m[wid][GT > 1 ? 2 * j4 + x : 0] = m_run[x];
  }
  // (The first time together with the producer warp: whoever finishes the step rewrites `len`, which every producer of the
  // unit must have read by then.)
  if (FEED && u == u0) asm volatile("bar.sync 2, %0;" ::"n"(WT + 32) : "memory");
  else workers_sync();
  // The next launch may start: its early requests queue behind this one's (released right after the wait they delayed this
  // launch's own rows by more than they gained).
  if (!FEED && !independent && tid == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // ---- exp2(s - m) of the CTA's slots, in place, and their sum (m: the CTA's maximum, finite when it has a live row)
  const int exp_rows = cnt > cnt_t ? cnt : (cnt + GROUP - 1) / GROUP * GROUP;
  if constexpr (GT == 1) {
    float m_c = -INFINITY, l = 0.f;
#pragma unroll
    for (int k = 0; k < MW; ++k) m_c = fmaxf(m_c, part_m[k][0]);
    for (int i = tid; i < exp_rows; i += WT) {
      const float e = ex2(logit_s[i] - m_c);
      logit_s[i] = e;
      l += e;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) part_l[wid][0] = l;
  } else {
    // warp x takes heads x, x + MW, ...; a lane every 32nd slot, four at a time
    for (int h = wid; h < G; h += MW) {
      float m_c = -INFINITY, l = 0.f;
#pragma unroll
      for (int k = 0; k < MW; ++k) m_c = fmaxf(m_c, part_m[k][h]);
      float* lg = logit_s + h * ld;
#pragma unroll 4
      for (int i = lane; i < exp_rows; i += 32) {
        const float e = ex2(lg[i] - m_c);
        lg[i] = e;
        l += e;
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
      if (lane == 0) { part_l[0][h] = l; part_m[0][h] = m_c; }      // (the CTA's: nobody else reads this head's maxima)
    }
  }
  workers_sync();
  // ---- O^T += V^T p
  float o_acc[HD / 16][4];                // channels 16 i + lane / 4 (+ 8) x columns 2 j4, 2 j4 + 1 of O^T
#pragma unroll
  for (int i = 0; i < HD / 16; ++i) { o_acc[i][0] = o_acc[i][1] = o_acc[i][2] = o_acc[i][3] = 0.f; }
  // columns of the B operand: with up to four heads the high bf16 halves of p of head 0, 1, ... and then the remainders; with
  // more a column per head, and two products
  const bool two_halves = GT == 1 || G <= GT / 2;
  const bool low_col = two_halves && (lane >> 2 & (GT == 1 ? 1 : GT / 2));
  const int my_head = GT == 1 ? 0 : min(two_halves ? lane >> 2 & (GT / 2 - 1) : lane >> 2, G - 1);
  const float* p_s = logit_s + my_head * ld + 2 * j4;
  uint32_t b0, b1, lo0, lo1;
  auto v_fetch = [&](int r0) {
    const float2 pa = *reinterpret_cast<const float2*>(p_s + r0), pb = *reinterpret_cast<const float2*>(p_s + r0 + 8);
    arrived();
    const bool ragged = cnt_t < r0 + GROUP;
    wrote = ragged;
    if (patches || ragged) {
      const bool has_new = wid == new_warp && fs_local >= r0 && fs_local < r0 + GROUP;
      const bool has_last = wid == last_warp && ls_local >= r0 && ls_local < r0 + GROUP;
      if (has_new) patch_row(unit_a, fs_local - r0, new_raw, true);
      if (has_last) patch_row(unit_a, ls_local - r0, last_raw, true);
      // rows beyond the live range must not reach the product (their probability is 0, but 0 * garbage need not be 0)
      if (ragged)
        for (int rr = cnt_t - r0 + (lane >> 4); rr < GROUP && has_chunk; rr += 2)
          st_shared16(unit_a + ((lane >> 3) & 1) * TILE_BYTES + rr * 128 + ((lane & 7) << 4), make_uint4(0u, 0u, 0u, 0u));
      wrote = has_new || has_last || ragged;
      __syncwarp();
    }
    const uint32_t vaddr = unit_a + row_off;
#pragma unroll
    for (int nn = 0; nn < HD / 16; ++nn) ldsm_x4_t(vaddr + (nn >> 2) * TILE_BYTES + ((lm_x ^ ((2 * nn) & 7)) << 4), frag[nn]);
    // B operand of V^T p: the high bf16 half of p and the remainder
    const uint32_t hi0 = pack_bf16(pa.x, pa.y), hi1 = pack_bf16(pb.x, pb.y);
    lo0 = pack_bf16(pa.x - __uint_as_float(hi0 << 16), pa.y - __uint_as_float(hi0 & 0xffff0000u));
    lo1 = pack_bf16(pb.x - __uint_as_float(hi1 << 16), pb.y - __uint_as_float(hi1 & 0xffff0000u));
    b0 = low_col ? lo0 : hi0;
    b1 = low_col ? lo1 : hi1;
  };
  if (!FEED && n > 0) v_fetch(wid * GROUP);
  for (int r0 = wid * GROUP; r0 < r_end; r0 += RSTEP) {
    if (FEED) v_fetch(r0);
#pragma unroll
    for (int nn = 0; nn < HD / 16; ++nn) {
      mma_bf16(o_acc[nn], frag[nn][0], frag[nn][1], frag[nn][2], frag[nn][3], b0, b1);
      if (!two_halves) mma_bf16(o_acc[nn], frag[nn][0], frag[nn][1], frag[nn][2], frag[nn][3], lo0, lo1);
    }
    release(wrote);
    if (!FEED && r0 + RSTEP < r_end) v_fetch(r0 + RSTEP);
  }
  // ---- the warp's partial
  {
    float* po = part_o + (size_t)wid * part_ld;
    const int row = lane >> 2;
    __syncwarp();                         // (part_in_ring: every lane is past its last read of the ring)
    if constexpr (GT > 1) {
      if (two_halves)
#pragma unroll
        for (int i = 0; i < HD / 16; ++i)
#pragma unroll
          for (int x = 0; x < 4; ++x) o_acc[i][x] += __shfl_xor_sync(0xffffffffu, o_acc[i][x], 2);
#pragma unroll
      for (int i = 0; i < HD / 16; ++i) {
        if (2 * j4 < G) { po[2 * j4 * HD + 16 * i + row] = o_acc[i][0]; po[2 * j4 * HD + 16 * i + 8 + row] = o_acc[i][2]; }
        if (2 * j4 + 1 < G) { po[(2 * j4 + 1) * HD + 16 * i + row] = o_acc[i][1]; po[(2 * j4 + 1) * HD + 16 * i + 8 + row] = o_acc[i][3]; }
      }
    } else {
      // every column pair holds the same two halves: lane j4 writes two of the eight tiles
#pragma unroll
      for (int i = 0; i < HD / 16; ++i)
        if ((i & 3) == j4) { po[16 * i + row] = o_acc[i][0] + o_acc[i][1]; po[16 * i + 8 + row] = o_acc[i][2] + o_acc[i][3]; }
    }
  }
  if (!FEED && has_tail) {
    const float p = logit_s[tail_head * ld + chunk + tail_row];
    float* po = part_o + (size_t)wid * part_ld + tail_head * HD + lane * TC;
    __syncwarp();
#pragma unroll
    for (int x = 0; x < TC / 2; ++x) {
      po[2 * x] = fmaf(p, __uint_as_float(tail_v[x] << 16), po[2 * x]);
      po[2 * x + 1] = fmaf(p, __uint_as_float(tail_v[x] & 0xffff0000u), po[2 * x + 1]);
    }
  }
  workers_sync();
  if (split > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  // every unit of this CTA has been consumed: the per-slot state of its slots lands in the rings while the CTAs of
  // the unit exchange (they were last written by bulk copies and read by ldmatrix; warps that stored into them have
  // fenced)
  if (!part_in_ring && state_in_smem == 2 && tid == 32 && rows_alloc > 0) copy_state(u, t);

  // ---- CTA partial: max and sum to every CTA of the unit, channel slice r of the partial output to rank r ----
  const int slice = HD / split;           // channels a CTA of the unit sums up and writes (a power of two)
  const int slice_log2 = 31 - __clz(slice);
  if (tid < split * g_rows) {
    const int h = GT > 1 ? tid / split : 0, dst = GT > 1 ? tid - h * split : tid;
    float m = part_m[0][h], l = part_l[0][h];
    if (GT == 1) {
#pragma unroll
      for (int k = 1; k < MW; ++k) { m = fmaxf(m, part_m[k][0]); l += part_l[k][0]; }
    }
    if (split > 1) st_async2(map_rank(smem_u32(&ex_ml[rank][h]), dst), m, l, map_rank(smem_u32(ex_bar), dst));
    else ex_ml[0][h] = make_float2(m, l);
  }
  for (int i = tid; i < g_rows * HD; i += WT) {
    const int h = GT > 1 ? i / HD : 0, ch = GT > 1 ? i - h * HD : i;
    float a = 0.f;
#pragma unroll
    for (int k = 0; k < MW; ++k) a += part_o[(size_t)k * part_ld + h * HD + ch];
    const int dst = ch >> slice_log2, off = (rank * g_rows + h) * slice + (ch & (slice - 1));
    if (split > 1) st_async(map_rank(smem_u32(&xo[off]), dst), a, map_rank(smem_u32(ex_bar), dst));
    else xo[off] = a;
  }
  if (!FEED) incoming();
  // ---- the state of this thread's slots tid, tid + WT, ...: SB of them in registers at a time, the first ones (where their
  // state has landed by now) read while the exchange is under way
  constexpr int SB = FEED ? 2 : 4;
  float old_r[SB], norm_r[SB], exp_r[SB];
  int pos_r[SB];
  long long fx_r[WINDOWED ? SB : 1];
  const float* old_g = WINDOWED ? c.ring + ((int64_t)u * w + (t % w)) * cap + s0 : c.acc + (int64_t)u * cap + s0;
  auto fetch = [&](int i0) {
#pragma unroll
    for (int k = 0; k < SB; ++k) {
      const int i = i0 + k * WT;
      exp_r[k] = old_r[k] = norm_r[k] = 0.f;
      pos_r[k] = 0;
      if (WINDOWED) fx_r[k] = 0;
      if (i < cnt) {
        const int64_t o = (int64_t)u * cap + s0 + i;
        if (GT == 1) exp_r[k] = logit_s[i];
        old_r[k] = state_in_smem ? acc_s[i] : old_g[i];
        norm_r[k] = state_in_smem ? vn_s[i] : c.vnorm[o];
        pos_r[k] = state_in_smem ? pos_s[i] : c.pos[o];
        if (WINDOWED) fx_r[k] = state_in_smem ? fx_s[i] : c.acc_fixed[o];
      }
    }
  };
  const bool fetch_early = !FEED && state_in_smem == 1 && rows_alloc > 0;
  if (fetch_early) {
    if (!mbar_wait(smem_u32(state_full), state_par)) bad = true;
    fetch(tid);
  }
  if (split > 1) {
    if (!mbar_wait(smem_u32(ex_bar), 0)) bad = true;
  } else {
    workers_sync();
  }

  // ---- every CTA: the unit's softmax normaliser (all data is local now) and its slice of the output ----
  float own_f = 0.f;       // own_f: this CTA's exp2(s - m) -> probability
  if constexpr (GT > 1) {
    if (tid < G) {         // one thread per head
      float2 ml[MAX_SPLIT];
      float m_h = -INFINITY, L_h = 0.f, own = 0.f;
#pragma unroll
      for (int r = 0; r < MAX_SPLIT; ++r) {
        ml[r] = r < split ? ex_ml[r][tid] : make_float2(-INFINITY, 0.f);
        m_h = fmaxf(m_h, ml[r].x);
      }
#pragma unroll
      for (int r = 0; r < MAX_SPLIT; ++r) {
        const float f = ml[r].x > -INFINITY ? ex2(ml[r].x - m_h) : 0.f;
        gq_fr[r][tid] = f;
        L_h += ml[r].y * f;
        if (r == rank) own = f;
      }
      const float inv = 1.f / L_h;
      gq_invl[tid] = inv;
      gq_f[tid] = own * inv;                             // this CTA's exp2(s - m) -> probability
    }
    workers_sync();
    for (int i = tid; i < G * slice; i += WT) {
      const int h = i >> slice_log2, ch = i & (slice - 1);
      float a = 0.f;
#pragma unroll
      for (int r = 0; r < MAX_SPLIT; ++r)
        if (r < split) a = fmaf(xo[(r * G + h) * slice + ch], gq_fr[r][h], a);
      out[((int64_t)u * G + h) * HD + rank * slice + ch] = __float2bfloat16(a * gq_invl[h]);
    }
  } else {
    float2 ml[MAX_SPLIT];
    float m_all = -INFINITY, L = 0.f, a = 0.f, part[MAX_SPLIT];
#pragma unroll
    for (int r = 0; r < MAX_SPLIT; ++r) {
      ml[r] = r < split ? ex_ml[r][0] : make_float2(-INFINITY, 0.f);
      part[r] = r < split && tid < slice ? xo[r * slice + tid] : 0.f;
      m_all = fmaxf(m_all, ml[r].x);
    }
#pragma unroll
    for (int r = 0; r < MAX_SPLIT; ++r) {
      const float f = ml[r].x > -INFINITY ? ex2(ml[r].x - m_all) : 0.f;
      L += ml[r].y * f;
      a = fmaf(part[r], f, a);
      if (r == rank) own_f = f;
    }
    const float invL = 1.f / L;
    own_f *= invL;
    if (tid < slice) out[(int64_t)u * HD + rank * slice + tid] = __float2bfloat16(a * invL);
  }

  // ---- indicator update (Eq. 2 / Eq. 3) and importance (Eq. 4) of this CTA's slots, its arg-min ----
  if (!fetch_early) {
    if (state_in_smem && rows_alloc > 0 && !mbar_wait(smem_u32(state_full), state_par)) bad = true;
    fetch(tid);
  }
  const bool evicting = hi > B;
  unsigned long long my_key = NO_KEY;
  int my_slot = -1, my_pos = -1;
  for (int i0 = tid; i0 < cnt;) {
#pragma unroll
    for (int k = 0; k < SB; ++k) {
      const int i = i0 + k * WT;
      if (i >= cnt) continue;
      const int slot_u = s0 + i;
      const int64_t o = (int64_t)u * cap + slot_u;
      float p;
      if constexpr (GT > 1) {      // the mean of the heads' probabilities
        float a = 0.f;
#pragma unroll
        for (int h = 0; h < GT; ++h)
          if (h < G) a = fmaf(logit_s[h * ld + i], gq_f[h], a);
        p = a / (float)G;
      } else {
        p = exp_r[k] * own_f;
      }
      const bool is_new = slot_u == fs;
      float S;
      if (WINDOWED) {
        // (a recycled slot's ring column is cleared below)
        const long long fx = is_new ? prob_to_fixed(p) : fx_r[k] + prob_to_fixed(p) - prob_to_fixed(old_r[k]);
        c.ring[((int64_t)u * w + (t % w)) * cap + slot_u] = p;
        c.acc_fixed[o] = fx;
        S = fixed_to_prob(fx);
      } else {
        S = is_new ? p : old_r[k] + p;
      }
      if (VATP_INB(o, (int64_t)units * cap, dev_status)) c.acc[o] = S;
      if (evicting) {
        const int ps = is_new ? t : pos_r[k];
        const float I = S * (is_new ? new_norm : norm_r[k]);
        if (ps >= F && ps <= t - R) {
          const unsigned long long key = evict_key(I, ps);
          if (key < my_key) { my_key = key; my_slot = slot_u; my_pos = ps; }
        }
      }
    }
    i0 += SB * WT;
    if (i0 < cnt) fetch(i0);
  }
  if (WINDOWED) {
    // recycled slot: the other rows of its ring column belong to the previous occupant (shared out over the unit's CTAs)
    for (int rr = rank * WT + tid; rr < w; rr += split * WT)
      if (rr != t % w && VATP_INB(((int64_t)u * w + rr) * cap + fs, (int64_t)units * w * cap, dev_status))
        c.ring[((int64_t)u * w + rr) * cap + fs] = 0.f;
  }
  // (units of one CTA one after the other: the next one's logits, partials and state may replace this one's)
  const bool more = u + u_step < units;
  if (more) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(state_empty)) : "memory");
  if (state_in_smem == 1) state_par ^= 1;
  if (evicting) {
    // this CTA's candidate (positions are unique: exactly one thread holds the winning key), sent to rank 0
    const unsigned long long wkey = warp_min_key(my_key);
    if (lane == 0) warp_key[wid] = wkey;
    workers_sync();
    const unsigned long long win = warp_min_key(lane < MW ? warp_key[lane] : NO_KEY);
    if (win == NO_KEY ? tid == 0 : my_key == win) {
      if (split > 1)
        st_async4(map_rank(smem_u32(&cand[rank]), 0), (uint32_t)win, (uint32_t)(win >> 32), (uint32_t)my_slot, (uint32_t)my_pos,
                  map_rank(smem_u32(cand_bar), 0));
      else
        cand[0] = Candidate{win, my_slot, my_pos};
    }
  }
  if (split == 1) workers_sync();
  if (rank == 0 && tid == 0) {            // nothing of the other CTAs' shared memory is read or written by anyone any more
    int out_slot = hi, left = hi, ev = -1;                         // not evicting: the cache grows
    if (evicting) {
      if (split > 1 && !mbar_wait(smem_u32(cand_bar), 0)) bad = true;
      unsigned long long best = NO_KEY;
      int br = -1;
      int best_slot = -1, best_pos = -1;
#pragma unroll
      for (int r = 0; r < MAX_SPLIT; ++r)
        if (r < split) {
          const Candidate x = cand[r];
          if (x.key < best) { best = x.key; best_slot = x.slot; best_pos = x.pos; br = r; }
        }
      if (br >= 0) {
        out_slot = best_slot;
        ev = best_pos;
        left = hi - 1;
        if (VATP_INB(out_slot, cap, dev_status)) c.pos[(int64_t)u * cap + out_slot] = -1;
      } else {   // nothing eligible (cannot happen when F + R <= B): keep the state consistent
        out_slot = min(hi, cap - 1);
      }
    }
    c.len[u] = left;
    c.free_slot[u] = out_slot;
    c.next_pos[u] = t + 1;
    c.last_slot[u] = fs;
    if (evicted) evicted[u] = ev;
  }
  if (!FEED) break;     // (one unit a CTA)
  }   // next unit of this CTA
  if (!FEED && independent && tid == WT - 1) asm volatile("griddepcontrol.wait;" ::: "memory");     // (launches complete in order)
  if (bad) {
    // Something never completed: flag it, give copies that may still be in flight time to land, and stay until the unit's
    // other CTAs have sent what they send here (threads that exit count as arrived).
    if (dev_status) atomicExch(dev_status, (int)VATP_ERR_TIMEOUT);
    for (int i = 0; i < 200; ++i) __nanosleep(1000);
    if (split > 1) {
      asm volatile("barrier.cluster.arrive.release;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    }
  }
}


// Host-side record, per stream, of the buffers the last launches write and read and of the share of the
// machine each occupies.  Every CTA of a launch stays resident until the previous launch has
// completed, so launch M - j can still be running when M starts only if the launches between them fit
// on the machine together: M may skip all waiting when it touches nothing that those launches write and writes
// nothing that they read.
struct Range {
  const char* p;
  size_t n;
};
constexpr int HIST = 8, NRANGE = 13, NTOUCHED = 16;   // of the ranges a launch touches the first NRANGE are written
struct LaunchRecord {
  Range r[NTOUCHED];
  double share;        // CTAs / (resident CTAs the machine holds of this launch's kind)
};
struct StreamHistory {
  cudaStream_t stream;
  unsigned long long capture;   // 0: launches issued for execution; else the id of the stream capture that recorded them
  bool valid;
  int count, head;     // records held, index of the newest
  LaunchRecord rec[HIST];
};
std::mutex g_hist_mutex;
StreamHistory g_hist[8];
int g_hist_next = 0;

inline bool overlaps(const Range& a, const Range& b) {
  return a.p && b.p && a.n && b.n && a.p < b.p + b.n && b.p < a.p + a.n;
}

// Id of the capture `st` is recording into, 0 when it is not capturing.  Launches recorded into a graph
// keep a history of their own: what was issued for execution before the capture says nothing about what
// precedes a node when the graph is replayed, and the recorded launches are not in flight afterwards.
unsigned long long capture_of(cudaStream_t st) {
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  unsigned long long id = 0;
  if (cudaStreamGetCaptureInfo(st, &status, &id) != cudaSuccess) { cudaGetLastError(); return 0; }
  return status == cudaStreamCaptureStatusActive ? (id ? id : ~0ull) : 0;
}

StreamHistory* history_of(cudaStream_t st, unsigned long long capture, bool create) {
  for (auto& x : g_hist)
    if (x.valid && x.stream == st && x.capture == capture) return &x;
  if (!create) return nullptr;
  StreamHistory* h = &g_hist[g_hist_next];
  g_hist_next = (g_hist_next + 1) % 8;
  h->stream = st;
  h->capture = capture;
  h->valid = true;
  h->count = 0;
  h->head = -1;
  return h;
}

// True when `touched` overlaps nothing that a launch possibly still in flight on `st` writes, nor its written part anything
// that such a launch reads; records this launch.  may_overlap false (the caller did not opt in): records it and answers false.
// share: of the machine, if as many of its CTAs share an SM as fit; share_alone: if each has an SM to itself, which *alone
// asks the caller to arrange (and which is recorded then).
bool independent_of_in_flight(cudaStream_t st, unsigned long long capture, bool may_overlap, const Range (&touched)[NTOUCHED],
                              double share, double share_alone, bool* alone) {
  std::lock_guard<std::mutex> lock(g_hist_mutex);
  StreamHistory* h = history_of(st, capture, true);
  // Launches too few CTAs wide for the ones between two steps of a cache to fill the machine would have to wait.  Alone on
  // their SMs (half as many fit) they may not: 8 units x 301 slots, eight caches in turn, 3.7 us per step waiting and 2.3 so;
  // 48 x 2001, four caches, 13.3 and 9.3.
  int apart = h->count == HIST ? HIST : 0;       // launches since the last one on this cache
  for (int j = 0; j < h->count; ++j)
    if (overlaps(touched[0], h->rec[(h->head - j + HIST) % HIST].r[0])) { apart = j; break; }
  *alone = may_overlap && apart * share < 1.0 && apart * share_alone >= 1.0;
  // The first recorded launch follows work this table knows nothing about (another kernel, the start of a
  // graph): it waits, and by the time it lets its successor start everything before it has completed.
  bool indep = may_overlap && h->count > 0;
  double between = 0.0;      // machine share of the launches between the candidate and this one
  for (int j = 0; indep && j < h->count && between < 1.0; ++j) {
    const LaunchRecord& r = h->rec[(h->head - j + HIST) % HIST];
    for (int i = 0; i < NTOUCHED && indep; ++i)
      for (int k = 0; k < (i < NRANGE ? NTOUCHED : NRANGE); ++k)      // (two launches may read the same)
        if (overlaps(touched[i], r.r[k])) { indep = false; break; }
    between += r.share;
    if (j == HIST - 1 && between < 1.0 && h->count == HIST) indep = false;   // history too short to tell
  }
  h->head = (h->head + 1) % HIST;
  if (h->count < HIST) ++h->count;
  LaunchRecord& r = h->rec[h->head];
  for (int k = 0; k < NTOUCHED; ++k) r.r[k] = touched[k];
  r.share = *alone ? share_alone : share;
  return indep;
}

}  // namespace

// Host-only probe of the overlap policy (no device work): feeds one pretend launch that touches and
// writes the first NRANGE of the `n` byte ranges [begin[i], begin[i] + bytes[i]) and only reads the others, on `stream`, and
// occupies `share` of the machine; returns whether it would have been allowed to run beside the launches before it.
bool decode_overlap_policy_probe(void* stream, const uint64_t* begin, const uint64_t* bytes, int n, double share) {
  Range r[NTOUCHED] = {};
  for (int i = 0; i < n && i < NTOUCHED; ++i) r[i] = Range{reinterpret_cast<const char*>(begin[i]), (size_t)bytes[i]};
  bool alone;
  return independent_of_in_flight(static_cast<cudaStream_t>(stream), 0, true, r, share, share, &alone);
}

// Any other work this library enqueues on `st` (prefill, selection, compaction, the general decode kernel)
// ends the record: the decode launch after it waits for everything before it.
void decode_history_forget(cudaStream_t st, bool probe_only) {
  const unsigned long long capture = probe_only ? 0 : capture_of(st);
  std::lock_guard<std::mutex> lock(g_hist_mutex);
  if (StreamHistory* h = history_of(st, capture, false)) {
    h->count = 0;
    h->head = -1;
  }
}

namespace {

template <int HD>
cudaError_t launch_hd(const Shape& s, int B, int F, int R, const vatp_cache& c, const void* q, const void* k,
                      const void* v, void* out, int32_t* evicted, int32_t* dev_status, cudaStream_t st,
                      bool may_overlap, int G) {
  constexpr int UNIT = unit_bytes<HD>, ROW_BYTES = HD * 2;
  const int cap = cache_capacity(B);
  const bool grouped = G > 1;           // s.units counts caches (KV heads); q and out hold G rows per unit
  const int sms = device_sm_count();
  // split a unit over a cluster while the grid still fits on the SMs once (a second launch can then be resident too)
  int split = 1;
  while (split < MAX_SPLIT && s.units * split * 2 <= sms && cap / (split * 2) >= 4 * GROUP) split *= 2;
  // Long units on a machine that they leave half idle: two CTAs per SM have twice the rows in flight (96 units x 1536 slots
  // 18.5 -> 15.3 us per waiting step and 19.9 -> 12.0 overlapping; 60 x 3501 22.3 -> 19.9).  Shorter ranges gain while
  // launches wait for one another (96 x 1025 13.6 -> 11.8) and lose a little of what overlapping gives (8.3 -> 9.1, 9.6 in
  // the first version); clusters of four do not fill every
  // SM twice (68 x 3501 23.8 -> 22.3, 72 x 3501 24.9 -> 31.9), of eight still less.  (The split decides in which order sums are
  // taken: it depends on the shape alone.)
  while (split < 4 && s.units * split * 2 <= (split == 1 ? 2 * sms : sms * 9 / 5) && s.units * split * 2 > sms &&
         cap / (split * 2) >= (split == 1 ? 28 : 40) * GROUP)
    split *= 2;
  int chunk = (cap + split - 1) / split;
  chunk = (chunk + GROUP - 1) / GROUP * GROUP;
  int ld = chunk;        // slots a CTA has room for
  // A few slots more than whole rounds of the warps (a group each) hold: the last CTA takes them with plain loads, at most
  // one row and head a warp.  (32 units x 2049 slots, four CTAs each: 9.6 us per step with them in one more group, 9.15 so;
  // 16 units x 1025 6.55 and 5.95.)  Only with one unit a CTA.
  const int rounds = (B + 1) / (MW * GROUP * split), extra = B + 1 - rounds * MW * GROUP * split;
  if (s.units * split <= 2 * sms && rounds > 0 && extra > 0 && extra * G <= MW) {
    chunk = rounds * MW * GROUP;
    ld = chunk + GROUP;  // (the capacity is the slots' number rounded up to eight)
  }
  // Two CTAs per SM at most; beyond that a CTA takes several units, one after the other (its producer warp then fills the
  // rings with the next unit's rows while the tail of this one runs).
  const int resident = 2;
  const int grid = s.units * split <= resident * sms ? s.units * split : resident * sms;
  const bool one_unit = grid == s.units * split;
  // Shared-memory plan.  Half an SM (two CTAs per SM, so that the next launch is resident while this one runs) with as
  // many units in flight per warp as fit there, at least two; the per-slot state beside them (1), in the rings' memory
  // after the streaming (2) or in global memory (0).  Only when not even that fits, a whole SM.
  const bool win = s.window > 0;
  // Dynamic bytes, 1 KB of it alignment slack.  (Two CTAs share 228 KB with 1 KB each for the system and their static arrays: 1376
  // bytes at most, 2592 with grouped queries, which leaves 113,120 there.  512 caches of 1337 slots, two heads each, w 40, whose
  // plan came to 113,408: 97.3 us per step with one CTA per SM, 70.2 so.)
  const size_t third_sm = 77 * 1024, half_sm = (grouped ? 110 : 111) * 1024, whole_sm = 222 * 1024;
  const int groups_per_warp = ((chunk / GROUP) + MW - 1) / MW;
  const bool part_in_ring = grouped && one_unit;                // a warp's partial outputs land in its ring
  const size_t fixed = 1024 + (part_in_ring ? 0 : (size_t)MW * G * HD * 4) + (size_t)G * HD * 4 + (size_t)G * ld * 4;
  const size_t state = (size_t)(win ? 20 : 12) * ld;
  const bool copyable = !win || (((uintptr_t)c.ring | (uintptr_t)c.acc_fixed) & 15) == 0;      // (bulk copies: 16-byte aligned)
  int nslot = 0, state_in_smem = 0;
  size_t dyn = 0;
  auto plan = [&](size_t limit, int most) {
    for (int n = most; n >= 2 && !nslot; --n) {
      const size_t rings = (size_t)MW * n * UNIT;
      if (part_in_ring && (size_t)n * UNIT < (size_t)G * HD * 4) continue;
      if (copyable && rings + fixed + state <= limit) state_in_smem = 1;
      else if (copyable && !grouped && one_unit && state <= rings && rings + fixed <= limit) state_in_smem = 2;
      else if (n == 2 && rings + fixed <= limit) state_in_smem = 0;
      else continue;
      nslot = n;
      dyn = rings + fixed + (state_in_smem == 1 ? state : 0);
    }
  };
  int most = 2 * groups_per_warp;
  most = most < 2 ? 2 : (most > MAX_SLOTS ? MAX_SLOTS : most);
  if (part_in_ring && (size_t)most * UNIT < (size_t)G * HD * 4) most = (G * HD * 4 + UNIT - 1) / UNIT;
  plan(half_sm, most);
  if (!nslot) plan(whole_sm, most);
  if (!nslot) return cudaErrorNotSupported;
  CUtensorMap tm_k, tm_v;
  if (!make_halves_map_bf16(&tm_k, c.k_cache, HD, (uint64_t)s.units * cap, GROUP) ||
      !make_halves_map_bf16(&tm_v, c.v_cache, HD, (uint64_t)s.units * cap, GROUP))
    return cudaErrorInvalidValue;
  const size_t units = (size_t)s.units, slots = units * cap;
  const Range touched[NTOUCHED] = {{(const char*)c.k_cache, slots * ROW_BYTES}, {(const char*)c.v_cache, slots * ROW_BYTES},
                       {(const char*)c.acc, slots * 4}, {(const char*)c.vnorm, slots * 4}, {(const char*)c.pos, slots * 4},
                       {(const char*)c.len, units * 4}, {(const char*)c.free_slot, units * 4},
                       {(const char*)c.next_pos, units * 4}, {(const char*)c.last_slot, units * 4},
                       {(const char*)out, units * G * ROW_BYTES}, {(const char*)evicted, evicted ? units * 4 : 0},
                       {win ? (const char*)c.ring : nullptr, win ? slots * s.window * 4 : 0},
                       {win ? (const char*)c.acc_fixed : nullptr, win ? slots * 8 : 0},
                       {(const char*)q, units * G * ROW_BYTES}, {(const char*)k, units * ROW_BYTES}, {(const char*)v, units * ROW_BYTES}};
  // CTAs with several units have a producer warp.  (One unit a CTA, without it against with it: 32 units x 2049 slots 9.2 and
  // 12.3 us per waiting step, 256 x 1025 24.1 and 26.3; 512 units x 1025 with a history window, two a CTA: 79 and 55.)
  const bool feed = !one_unit;
  auto kern = feed ? (grouped ? (win ? decode_mma_kernel<HD, true, GQ_HEADS, true> : decode_mma_kernel<HD, false, GQ_HEADS, true>)
                              : (win ? decode_mma_kernel<HD, true, 1, true> : decode_mma_kernel<HD, false, 1, true>))
                   : (grouped ? (win ? decode_mma_kernel<HD, true, GQ_HEADS, false> : decode_mma_kernel<HD, false, GQ_HEADS, false>)
                              : (win ? decode_mma_kernel<HD, true, 1, false> : decode_mma_kernel<HD, false, 1, false>));
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)whole_sm);
  if (e != cudaSuccess) return e;
  // share of the machine this launch holds while resident (every CTA waits for the previous launch before it retires): exactly
  // two CTAs of this kernel fit on an SM, or exactly one
  const bool half = dyn <= half_sm;
  const double share_alone = (double)grid / sms, share = half ? share_alone / 2 : share_alone;
  bool alone = false;
  const int independent = independent_of_in_flight(st, capture_of(st), may_overlap, touched, share, share_alone, &alone) ? 1 : 0;
  dyn = half && !alone ? (dyn > third_sm ? dyn : third_sm) : whole_sm;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(feed ? DM_THREADS : WT);
  cfg.dynamicSmemBytes = dyn;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = split;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // may start before the previous launch has drained
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, tm_k, tm_v, independent, G, s.units, state_in_smem, (int)part_in_ring, split, chunk, ld, nslot, B, cap, F, R, s.window,
                            s.norm, s.scale * LOG2E, c, (const __nv_bfloat16*)q, (const __nv_bfloat16*)k, (const __nv_bfloat16*)v,
                            (__nv_bfloat16*)out, evicted, dev_status);
}

}  // namespace

// Returns cudaErrorNotSupported when the shape does not fit this kernel's shared memory (the caller
// then takes the general kernel).
cudaError_t launch_decode_mma(const Shape& s, int B, int F, int R, const vatp_cache& c, const void* q, const void* k,
                              const void* v, void* out, int32_t* evicted, int32_t* dev_status, cudaStream_t st,
                              bool may_overlap, int G) {
  if (!vatp_tc_available() || G < 1 || G > GQ_HEADS) return cudaErrorNotSupported;
  return s.d == 64 ? launch_hd<64>(s, B, F, R, c, q, k, v, out, evicted, dev_status, st, may_overlap, G)
                   : launch_hd<128>(s, B, F, R, c, q, k, v, out, evicted, dev_status, st, may_overlap, G);
}

}  // namespace vatp
