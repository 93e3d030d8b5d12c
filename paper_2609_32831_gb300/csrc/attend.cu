// Fused dequant-and-gather decode attention over heterogeneous segments
// (App. E "Attention over heterogeneous cache segments": one shared softmax
// across segments, chunks merged by log-sum-exp; Eq. 1's per-segment mass as
// a by-product).
//
// Design (GB300, HBM-bound): persistent CTAs walk a static list of work
// items; an item is one chunk of 64-token tiles of one segment of one
// (sequence, KV head). Per CTA one producer warp streams tiles into a
// 2-stage shared-memory ring (TMA 2D loads with 128-byte swizzle for bf16
// rows, 1D bulk copies for packed codes and parameters) and four consumer
// warps compute with mma.sync m16n8k16:
//   bf16 rows:  S = Q K^T in bf16 (exact products), P split into bf16 hi + lo
//               parts so P V keeps ~16 mantissa bits;
//   packed:     each pair of codes -> an exact pair of (subnormal) fp16 values
//               with one LOP3, scales folded into the queries (keys) and the
//               probabilities (values), S and P V in fp16 with fp32
//               accumulation.
// Each item leaves an unnormalised partial (O, m, l); a merge kernel launched
// programmatically behind the call merges a (sequence, KV head)'s items by
// log-sum-exp and writes O, lse and the per-segment probability mass. In
// short calls the items of a (sequence, KV head) run on one thread-block
// cluster instead, which merges them through distributed shared memory; in a
// batch of calls of several n-tiles the last CTA to finish a pair merges it
// and re-arms its counter.
#include <atomic>
#include <mutex>

#include "common.cuh"
#include "internal.h"

namespace uc {

constexpr int kTileTok = 64;
// Ring slots (ST) of a CTA and CTAs per SM the register budget is set for:
// two slots, three CTAs with one query n-tile (128 registers), two with more
// (168; the query buffers of up to seven n-tiles leave room for two CTAs'
// shared memory, eight run one). A launch with several n-tiles and no more
// CTAs than SMs takes three slots and all registers (7 query tokens over 43K
// bf16 tokens, batch 1: 47.5 us otherwise).
constexpr int kStages = 2, kMaxStages = 3;
template <int NTW, int ST>
__host__ __device__ constexpr int ctas_for() { return NTW == 1 ? 3 : (ST == kMaxStages ? 1 : 2); }
constexpr int kConsumers = 4;
constexpr int kAttnThreads = 32 * (kConsumers + 1);
constexpr int kSlotBytes = 32768;
constexpr float kNegInf = -INFINITY;
constexpr float kLn2 = 0.69314718055994530942f;

// slot layout of a packed tile: up to 8 int2 or 4 int4 quantization groups
// (codes 1 KB / 2 KB per group for K and for V, parameters 512 B per group)
constexpr int kSlotKParams = 8192;
constexpr int kSlotVCodes = 12288;
constexpr int kSlotVParams = 20480;

__host__ __device__ constexpr int quant_groups_per_tile(int bits) { return bits == 2 ? 8 : 4; }

constexpr int kMaxItemsPerBh = 64;
constexpr int kMaxPendingMerges = 64;
constexpr int kMaxRows = 64;  // query rows of a KV head (eight n-tiles)
constexpr int kItemQ = 2;  // items handed from the producer to the consumers ahead

struct AttnSmem {
  // one n-tile: the query fragments; a cluster's row sums. Several: m, then
  // weight; l, per (item, row of an 8-row block) of a merge
  alignas(16) float merge_w[kMaxItemsPerBh * 8];
  float merge_l[kMaxItemsPerBh * 8];
  uint64_t full[kMaxStages];
  uint64_t empty[kMaxStages];
  uint64_t item_full[kItemQ];   // producer -> consumers: item position and its query rows
  uint64_t item_empty[kItemQ];  // consumers -> producer: the entry is free again
  int item_pos[kItemQ];         // processing position, -1: no more work
  int n_pending;                    // (sequence, KV head) merges this CTA owes
  int pending[kMaxPendingMerges];
  alignas(16) float row_scale[kMaxRows];  // packed items: logit scale of each query row (see store_q)
  alignas(1024) uint8_t slot[kMaxStages][kSlotBytes];  // as many as the launch has
};

static_assert(offsetof(AttnSmem, row_scale) % 8 == 0, "row scales are read in pairs");

// Query fragments of the current item live in shared memory (2 KB per
// n-tile of 8 query rows): for one n-tile in `merge_w`, keeping three CTAs
// per SM; for more n-tiles after the ring. The bf16 query rows of an
// item as the producer copies them (g * T rows) take as much again per entry
// of the item queue.
constexpr int kQTileBytes = 2048;
static_assert(kQTileBytes == 8 * kHeadDim * 2, "bf16 rows of an n-tile");
__host__ __device__ constexpr int qfrag_tiles(int ntiles) { return ntiles <= 1 ? 0 : ntiles; }

constexpr size_t attend_smem_bytes(int ntiles, int stages = kStages) {
  return offsetof(AttnSmem, slot) + (size_t)stages * kSlotBytes +
         (size_t)(qfrag_tiles(ntiles) + kItemQ * ntiles) * kQTileBytes + 1024;
}

// Shared-memory regions after the ring: query fragments (more than one
// n-tile), then the producer's query-row buffers.
template <int ST>
__device__ __forceinline__ uint8_t* after_ring(AttnSmem& sm) {
  return reinterpret_cast<uint8_t*>(sm.slot) + ST * kSlotBytes;
}
template <int ST>
__device__ __forceinline__ uint8_t* qrows_buf(AttnSmem& sm, int k, int ntiles) {
  return after_ring<ST>(sm) + (qfrag_tiles(ntiles) + k * ntiles) * kQTileBytes;
}

__host__ __device__ size_t attend_part_floats(int ntiles) { return (size_t)ntiles * 8 * (kHeadDim + 2); }

__device__ __forceinline__ bool seg_is_bf16(int kind) {
  return kind == UC_KIND_FULL || kind == UC_KIND_EVICT;
}

// Tiles of a segment holding n tokens; *qtiles = packed tiles before the tail.
__device__ __forceinline__ int seg_tiles(const SegDev& sd, int n, int* qtiles) {
  if (seg_is_bf16(sd.kind)) {
    *qtiles = 0;
    return (n + kTileTok - 1) / kTileTok;
  }
  const int ng = n / kGroup;
  const int tg = quant_groups_per_tile(sd.bits);
  *qtiles = (ng + tg - 1) / tg;
  return *qtiles + ((n % kGroup) ? 1 : 0);
}

struct ItemInfo {
  int bh, b, s, tb, te, qtiles, n;
  bool tail;  // the bf16 residual tail of a packed segment
};

// Item at processing position pos: pair, segment and kept count; *it receives
// its partial-output index, *chunk its place in the segment's split.
__device__ __forceinline__ ItemInfo item_place(const AttnParams& p, int pos, int* it, int* chunk) {
  ItemInfo r;
  const int nbh = p.batch * p.n_kv_heads;
  int local;
  if (pos < p.n_heavy * nbh) {
    r.bh = pos / p.n_heavy;
    local = p.heavy_local[pos % p.n_heavy];
  } else {
    const int q = pos - p.n_heavy * nbh;
    r.bh = q / p.n_light;
    local = p.light_local[q % p.n_light];
  }
  *it = r.bh * p.items_per_bh + local;
  r.b = r.bh / p.n_kv_heads;
  r.s = 0;
  for (int s = 0; s < p.nseg; ++s)
    if (local >= p.seg[s].chunk_begin) r.s = s;
  *chunk = local - p.seg[r.s].chunk_begin;
  r.n = p.seg[r.s].n_kept[r.b];
  return r;
}

// The tiles of an item from its place.
__device__ __forceinline__ void item_range(const AttnParams& p, ItemInfo& r, int c) {
  const SegDev& sd = p.seg[r.s];
  const int nt = seg_tiles(sd, r.n, &r.qtiles);
  r.tail = false;
  if (seg_is_bf16(sd.kind)) {
    r.tb = (int)(((int64_t)c * nt) / sd.n_chunks);
    r.te = (int)(((int64_t)(c + 1) * nt) / sd.n_chunks);
  } else if (c == sd.n_chunks - 1) {  // last chunk: the tail tile (empty if no tail)
    r.tail = true;
    r.tb = r.qtiles;
    r.te = nt;
  } else {
    const int cq = sd.n_chunks - 1;
    r.tb = (int)(((int64_t)c * r.qtiles) / cq);
    r.te = (int)(((int64_t)(c + 1) * r.qtiles) / cq);
  }
}

__device__ __forceinline__ ItemInfo decode_item(const AttnParams& p, int pos, int* it) {
  int c;
  ItemInfo r = item_place(p, pos, it, &c);
  item_range(p, r, c);
  return r;
}

// Work lists. OneCall walks the items of one call; ManyCalls walks several
// calls' items in one launch, the heavy items of every call first, then the
// light tail items. locate() maps a processing position to its call's
// parameters and to the position inside that call's own order.
struct OneCall {
  static constexpr bool kMany = false;
  const AttnParams& p;
  __device__ int n_items() const { return p.n_items; }
  __device__ int n_calls() const { return 1; }
  __device__ const AttnParams& call(int) const { return p; }
  __device__ int items_per_bh(int) const { return p.items_per_bh; }
  __device__ const AttnParams& locate(int pos, int* local, int* c) const {
    *local = pos;
    *c = 0;
    return p;
  }
};

struct ManyCalls {
  static constexpr bool kMany = true;
  const MultiAttnParams& m;
  __device__ int n_items() const { return m.n_items; }
  __device__ int n_calls() const { return m.n_calls; }
  __device__ const AttnParams& call(int c) const { return m.call[c]; }
  __device__ int items_per_bh(int c) const { return m.call[c].items_per_bh; }
  __device__ const AttnParams& locate(int pos, int* local, int* c) const {
    const int nh = m.heavy_begin[m.n_calls];
    int k = 0;
    if (pos < nh) {
      while (k + 1 < m.n_calls && pos >= m.heavy_begin[k + 1]) ++k;
      *local = pos - m.heavy_begin[k];
    } else {
      const int q = pos - nh;
      while (k + 1 < m.n_calls && q >= m.light_begin[k + 1]) ++k;
      const AttnParams& p = m.call[k];
      *local = p.n_heavy * p.batch * p.n_kv_heads + (q - m.light_begin[k]);
    }
    *c = k;
    return m.call[k];
  }
};

template <class P>
struct WorkOf;
template <>
struct WorkOf<AttnParams> {
  using type = OneCall;
};
template <>
struct WorkOf<MultiAttnParams> {
  using type = ManyCalls;
};

__device__ __forceinline__ void consumer_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

// consumer_sync with a vote: true if `ok` holds in every consumer warp.
__device__ __forceinline__ bool consumer_all(bool ok) {
  uint32_t all;
  asm volatile(
      "{\n"
      ".reg .pred p, q;\n"
      "setp.ne.u32 p, %1, 0;\n"
      "barrier.cta.red.and.pred q, 1, 128, p;\n"
      "selp.u32 %0, 1, 0, q;\n"
      "}\n"
      : "=r"(all)
      : "r"((uint32_t)ok)
      : "memory");
  return all != 0;
}

// Arrival on a (sequence, KV head) counter, acquire-release at GPU scope:
// after a CTA barrier, the partial outputs every consumer thread wrote are
// ordered before the increment (release is cumulative over the barrier), and
// the arrival that completes the count has acquired every earlier one, so
// the CTA that merges needs no further fence (a later CTA barrier carries the
// acquire to its other threads).
__device__ __forceinline__ int counter_arrive_acq_rel(int* c) {
  int prev;
  asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(prev) : "l"(c) : "memory");
  return prev;
}

__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(a));
  return v;
}

__device__ __forceinline__ uint2 lds64(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}

// ------------------------------------------------------------- producer
// Items come from a launch-wide counter (the next position to process, in
// the plan's order: heavy items first), so a CTA that finishes early takes
// more. The producer claims its next position once it has issued every tile
// of the current item (the ring still holds work for the consumers, which
// hides the atomic's latency, and no CTA claims work long before it can
// start it), hands each position to the consumers through a two-entry queue
// and copies the item's query rows (the g * T rows of one KV head are
// contiguous) along with it.
//
// In a cluster launch rank r < n_heavy takes its pair's heavy item r, the
// ranks after them (one, or one each) share the pair's light items.
template <int NTW, int ST, bool CLUSTER, class W>
__device__ void produce(const W& w, AttnSmem& sm) {
  const AttnParams& p0 = w.call(0);
  int* sched = p0.sched;
  uint32_t seq = 0;
  bool stop = false;
  // the first item of every CTA is its own index (the grid never exceeds
  // the item count); later items come from the launch-wide counter, so the
  // first copies are issued without waiting for an atomic's round trip
  int pos = blockIdx.x;
  int end = 0;
  if constexpr (CLUSTER) {
    const int pair = blockIdx.x / p0.cluster, rank = blockIdx.x % p0.cluster;
    const int light0 = p0.n_heavy * p0.batch * p0.n_kv_heads + pair * p0.n_light;
    pos = rank < p0.n_heavy ? pair * p0.n_heavy + rank : light0 + rank - p0.n_heavy;
    end = rank < p0.n_heavy ? 0 : light0 + p0.n_light;
  }
  for (uint32_t iseq = 0;; ++iseq) {
    const int k = iseq % kItemQ;
    if (iseq >= kItemQ && !mbar_wait(&sm.item_empty[k], ((iseq / kItemQ) - 1) & 1, p0.status, 12, p0.wait_ns))
      break;
    if (pos >= w.n_items()) {
      sm.item_pos[k] = -1;
      mbar_arrive(&sm.item_full[k]);
      break;
    }
    int it, local, c;
    const AttnParams& p = w.locate(pos, &local, &c);
    int chunk;
    ItemInfo ii = item_place(p, local, &it, &chunk);
    const SegDev& sd = p.seg[ii.s];
    sm.item_pos[k] = pos;
    const uint32_t qbytes = (uint32_t)p.rows * kHeadDim * 2;
    const __nv_bfloat16* qsrc =
        p.q + (size_t)(ii.b * p.n_q_heads + (ii.bh % p.n_kv_heads) * p.group) * p.n_qtok * kHeadDim;
    mbar_arrive_expect_tx(&sm.item_full[k], qbytes);
    bulk_load(qrows_buf<ST>(sm, k, p.mtiles), qsrc, qbytes, &sm.item_full[k]);
    // The kept count is on its way from memory meanwhile: nothing that depends
    // on it moves above the query rows' copy (behind that read, 1K tokens,
    // batch 1, took 7.8 us, 8K int2, batch 8, 14.0; so 7.2 and 13.5).
    asm volatile("" : "+r"(ii.n) : : "memory");
    item_range(p, ii, chunk);
    for (int t = ii.tb; t < ii.te; ++t, ++seq) {
      const int slot = seq % ST;
      if (seq >= ST && !mbar_wait(&sm.empty[slot], ((seq / ST) - 1) & 1, p.status, 10, p.wait_ns)) {
        stop = true;
        break;
      }
      if (pos == p.withhold_pos && t == ii.tb) continue;  // test hook: this tile is never copied
      uint8_t* dst = sm.slot[slot];
      const bool tail = ii.tail;
      if (seg_is_bf16(sd.kind) || tail) {
        int64_t row;
        if (tail)
          row = (int64_t)ii.bh * kGroup;
        else
          row = (int64_t)ii.bh * sd.row_stride + sd.row_offset + (int64_t)t * kTileTok;
        mbar_arrive_expect_tx(&sm.full[slot], kSlotBytes);
        const CUtensorMap* mk = &p.tmap[2 * ii.s];
        const CUtensorMap* mv = &p.tmap[2 * ii.s + 1];
        tma_load_2d(dst, mk, 0, (int)row, &sm.full[slot]);
        tma_load_2d(dst + 8192, mk, 64, (int)row, &sm.full[slot]);
        tma_load_2d(dst + 16384, mv, 0, (int)row, &sm.full[slot]);
        tma_load_2d(dst + 24576, mv, 64, (int)row, &sm.full[slot]);
      } else {
        const int ng = ii.n / kGroup;
        const int tg = quant_groups_per_tile(sd.bits);
        const int g0 = tg * t;
        const int ngt = min(tg, ng - g0);
        const uint32_t kc = 32 * kHeadDim * sd.bits / 8;  // code bytes per group (K or V)
        const uint32_t bytes = (uint32_t)ngt * (2 * kc + 1024);
        mbar_arrive_expect_tx(&sm.full[slot], bytes);
        const size_t blk_codes = (size_t)ii.bh * sd.cap * kHeadDim * sd.bits / 8;
        const size_t blk_kpar = (size_t)ii.bh * (sd.cap / kGroup) * 512;
        const size_t blk_vpar = (size_t)ii.bh * sd.cap * 16;
        bulk_load(dst, sd.k_codes + blk_codes + (size_t)g0 * kc, ngt * kc, &sm.full[slot]);
        bulk_load(dst + kSlotKParams, sd.k_params + blk_kpar + (size_t)g0 * 512, ngt * 512,
                  &sm.full[slot]);
        bulk_load(dst + kSlotVCodes, sd.v_codes + blk_codes + (size_t)g0 * kc, ngt * kc,
                  &sm.full[slot]);
        bulk_load(dst + kSlotVParams, sd.v_params + blk_vpar + (size_t)g0 * 512, ngt * 512,
                  &sm.full[slot]);
      }
    }
    if (stop) break;
    if constexpr (CLUSTER) {
      pos += p0.cluster - p0.n_heavy;
      if (pos >= end) pos = w.n_items();
    } else {
      pos = (int)gridDim.x + atomicAdd(sched, 1);
    }
  }
  // This producer claims nothing more: the last producer of the launch to
  // get here re-arms the work queue for the next launch. Done here rather
  // than at the CTA's exit, so that the fence and the atomic stay off the
  // path of the consumers' final merges.
  if constexpr (!CLUSTER) {
    __threadfence();
    if (atomicAdd(sched + 1, 1) == (int)gridDim.x - 1) {
      sched[0] = 0;
      sched[1] = 0;
    }
  }
  // A consumer that gave up on a bounded wait (the status word is set) no
  // longer waits for the copies this producer issued: they land before the
  // CTA leaves. (Otherwise the consumers have waited for every one.)
  const bool failed = stop || (p0.status != nullptr && *reinterpret_cast<volatile int32_t*>(&p0.status->code) != 0);
  for (uint32_t s = 0; failed && s < ST; ++s) {
    if (seq < s + 1u) break;
    const uint32_t sq = seq - 1u - s;
    if (!mbar_wait(&sm.full[sq % ST], (sq / ST) & 1, p0.status, 15, p0.wait_ns)) break;
  }
}

// ------------------------------------------------------------- consumer
//
// Transposed formulation: with T query tokens the g = Hq / Hkv heads of one
// KV head give 7T query rows, far fewer than the 16 rows of an m16n8k16 A
// operand. Keys therefore take the M role and query rows the N role:
//   S^T [keys x rows]    = K [keys x d] . Q^T [d x rows]
//   O^T [d x rows]      += V^T [d x keys] . P^T [keys x rows]
// An n8 tile of query rows per MMA wastes at most one row for T = 1. P^T
// moves from the accumulator layout into the B-operand layout with one
// movmatrix.trans per 8 x 8 block.
//
// Per thread (g = lane / 4, j = lane % 4), n-tile nt of query rows:
//   Q^T  B fragment: rows nt*8 + g, channels {16i + 2j, +1} and {+8, +9}
//   S^T  accumulator: keys {g, g + 8} x rows nt*8 + {2j, 2j + 1}
//   O^T  accumulator: channels {16mt + g, 16mt + 8 + g} x rows nt*8 + {2j, 2j + 1}

template <int NTW>
struct WarpState {
  float o[NTW][8][4];
  float z[NTW][4];  // packed values: zero-point term per channel group (rows = groups 0..3)
  float m[NTW][2];  // running max per query row (rows 2j, 2j + 1 of each n-tile), log2 units
  float l[NTW][2];  // this thread's share of the row sums
};

template <int NTW>
__device__ __forceinline__ void state_init(WarpState<NTW>& st) {
#pragma unroll
  for (int nt = 0; nt < NTW; ++nt) {
#pragma unroll
    for (int mt = 0; mt < 8; ++mt) st.o[nt][mt][0] = st.o[nt][mt][1] = st.o[nt][mt][2] = st.o[nt][mt][3] = 0.f;
    st.z[nt][0] = st.z[nt][1] = st.z[nt][2] = st.z[nt][3] = 0.f;
    st.m[nt][0] = st.m[nt][1] = kNegInf;
    st.l[nt][0] = st.l[nt][1] = 0.f;
  }
}

template <int NTW>
__device__ __forceinline__ void scale_o(WarpState<NTW>& st, float f) {
#pragma unroll
  for (int nt = 0; nt < NTW; ++nt)
#pragma unroll
    for (int mt = 0; mt < 8; ++mt)
#pragma unroll
      for (int e = 0; e < 4; ++e) st.o[nt][mt][e] *= f;
}

// Online softmax over NB 16-key blocks: x[blk][nt][e] (e: 0/1 key g, 2/3 key
// g+8; e & 1 selects the row), in log2 units. Writes probabilities into pr.
// The reference max m moves only when a row's max exceeds it by more than
// 8, so P = 2^(x - m) <= 2^8 (exact enough in fp16 / bf16 pairs) and o, z, l
// are rescaled only on those (rare) moves. Each lane first tests its own
// logits against m + 8; the row maxima (shuffle reductions) are formed only
// when some lane's test fires.
template <int NTW, int NB>
__device__ __forceinline__ void softmax_rows(WarpState<NTW>& st, const float (&x)[NB][NTW][4],
                                             float (&pr)[NB][NTW][4]) {
#pragma unroll
  for (int nt = 0; nt < NTW; ++nt) {
    bool over = false;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float lim = st.m[nt][h] + 8.f;
#pragma unroll
      for (int k = 0; k < NB; ++k) over |= (x[k][nt][h] > lim) | (x[k][nt][2 + h] > lim);
    }
    if (__any_sync(0xffffffffu, over)) {
      float mx[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float v = fmaxf(x[0][nt][h], x[0][nt][2 + h]);
#pragma unroll
        for (int k = 1; k < NB; ++k) v = fmaxf(v, fmaxf(x[k][nt][h], x[k][nt][2 + h]));
        v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 4));
        v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 8));
        v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 16));
        mx[h] = v;
      }
      const bool g0 = mx[0] > st.m[nt][0] + 8.f, g1 = mx[1] > st.m[nt][1] + 8.f;
      float alpha[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const bool gh = h ? g1 : g0;
        const float nm = gh ? mx[h] : st.m[nt][h];
        alpha[h] = (st.m[nt][h] == kNegInf) ? 0.f : ex2_approx(st.m[nt][h] - nm);
        st.m[nt][h] = nm;
        st.l[nt][h] *= alpha[h];
      }
#pragma unroll
      for (int mt = 0; mt < 8; ++mt) {
        st.o[nt][mt][0] *= alpha[0];
        st.o[nt][mt][1] *= alpha[1];
        st.o[nt][mt][2] *= alpha[0];
        st.o[nt][mt][3] *= alpha[1];
      }
      st.z[nt][0] *= alpha[0];
      st.z[nt][1] *= alpha[1];
      st.z[nt][2] *= alpha[0];
      st.z[nt][3] *= alpha[1];
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float um = (st.m[nt][h] == kNegInf) ? 0.f : st.m[nt][h];
      float sum = 0.f;
#pragma unroll
      for (int k = 0; k < NB; ++k) {
        pr[k][nt][h] = ex2_approx(x[k][nt][h] - um);
        pr[k][nt][2 + h] = ex2_approx(x[k][nt][2 + h] - um);
        sum += pr[k][nt][h] + pr[k][nt][2 + h];
      }
      st.l[nt][h] += sum;
    }
  }
}

__device__ __forceinline__ uint32_t swz(uint32_t base, int key, int chunk) {
  return base + (chunk >> 3) * 8192 + key * 128 + ((((chunk & 7) ^ (key & 7))) << 4);
}

// One 16-key block (keys 16u .. 16u + 15 of a bf16 tile).
template <int NTW>
__device__ __forceinline__ void block_bf16(WarpState<NTW>& st, uint32_t qs,
                                           uint32_t kbase, int u, int valid, float scale) {
  const int lane = threadIdx.x & 31;
  const int mi = lane >> 3, rr = lane & 7, g = lane >> 2;
  float s[NTW][4];
#pragma unroll
  for (int nt = 0; nt < NTW; ++nt) s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
  {
    const int kk = 16 * u + 8 * (mi & 1) + rr;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      uint32_t a[4];
      ldsm_x4(swz(kbase, kk, 2 * i + (mi >> 1)), a[0], a[1], a[2], a[3]);
#pragma unroll
      for (int nt = 0; nt < NTW; ++nt) {
        const uint2 qv = lds64(qs + ((nt * 8 + i) * 32 + lane) * 8);
        mma_bf16(s[nt], a, qv.x, qv.y);
      }
    }
  }
  float x[1][NTW][4], pr[1][NTW][4];
  const bool ok0 = 16 * u + g < valid, ok1 = 16 * u + 8 + g < valid;
#pragma unroll
  for (int nt = 0; nt < NTW; ++nt) {
    x[0][nt][0] = ok0 ? s[nt][0] * scale : kNegInf;
    x[0][nt][1] = ok0 ? s[nt][1] * scale : kNegInf;
    x[0][nt][2] = ok1 ? s[nt][2] * scale : kNegInf;
    x[0][nt][3] = ok1 ? s[nt][3] * scale : kNegInf;
  }
  softmax_rows<NTW, 1>(st, x, pr);
  // P^T as B fragments (bf16 hi + lo parts)
  uint32_t bh[NTW][2], bl[NTW][2];
#pragma unroll
  for (int nt = 0; nt < NTW; ++nt) {
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const float p0 = pr[0][nt][2 * half], p1 = pr[0][nt][2 * half + 1];
      const uint32_t hi = pack_bf16(p0, p1);
      const uint32_t lo = pack_bf16(p0 - bf16_lo(hi), p1 - bf16_hi(hi));
      bh[nt][half] = movmatrix_t(hi);
      bl[nt][half] = movmatrix_t(lo);
    }
  }
  const uint32_t vbase = kbase + 16384;
  const int vk = 16 * u + 8 * (mi >> 1) + rr;
#pragma unroll
  for (int mt = 0; mt < 8; ++mt) {
    uint32_t a[4];
    ldsm_x4_t(swz(vbase, vk, 2 * mt + (mi & 1)), a[0], a[1], a[2], a[3]);
#pragma unroll
    for (int nt = 0; nt < NTW; ++nt) {
      mma_bf16(st.o[nt][mt], a, bh[nt][0], bh[nt][1]);
      mma_bf16(st.o[nt][mt], a, bl[nt][0], bl[nt][1]);
    }
  }
}

// ---- packed codes
//
// A code word holds 16 int2 or 8 int4 codes as pairs: pair p is the code at
// bit p * BITS of the low half and the one at the same bit of the high half.
// Masking a (shifted) copy of the word leaves the codes in the mantissas of
// two subnormal fp16 values: a code at bit B is exactly code * 2^(B - 24), one
// LOP3 per pair and no offset to remove. The tensor cores take subnormal
// operands as they are; the powers of two are put right elsewhere:
//   keys    the query of the pair's channels carries 2^(B0 - B) and the logit
//           scale 2^(24 - B0). int2: copies w << 6, w << 2, w >> 2, w >> 6 with
//           the two pairs of a 16-channel step at bits B0 = 6 and 8 (queries
//           times 1 and 1/4: none overflows for it); int4: copies w << 4, w,
//           w >> 4, w >> 8 with every code at bit B0 = 4. Each halving costs
//           the fp16 queries a bit at their small end, which store_q brings
//           up first, and low codes lose more in the tensor cores' sums. int2
//           at bits 4, 6 and 8 (queries down to 1/16, two shifts per word
//           less, no row scales): 32K layer, batch 16, 64.9 us, now 65.9; lse
//           of 8192 tokens 4.9e-8 off, now 4.3e-8 (bits 4 and 6: 5.7e-8);
//           with queries of 1e-4 on keys of 1e3, 1024 tokens, 1.4e-5 off, now
//           2.7e-7;
//   values  one HFMA2 per pair centres the codes and brings every pair to
//           2^-9 (code - C): copies w and w >> 10 (int2) or w >> 8 (int4).
// (With the exponent 2^(10-B) OR-ed in instead, each pair carried an offset of
// 64, 16 or 4 through the fp32 accumulators, removed by extra rows of the beta
// MMAs; value copies took two or three shifts per word. One 32K layer, batch
// 16: int2 70.1 us; lse of 8192 tokens 2.7e-7 (int2) and 1.2e-7 (int4) off, now
// 4.3e-8 and 4.4e-8.)
struct KeyWords {
  uint32_t l, m, r, r2;
};
template <int BITS>
__device__ __forceinline__ KeyWords key_words(uint32_t w) {
  if constexpr (BITS == 2)
    return KeyWords{w << 6, w << 2, w >> 2, w >> 6};
  else
    return KeyWords{w << 4, w, w >> 4, w >> 8};
}

// Bit of key pair p in its copy and the class of the pair's channels: queries
// scaled by 1 / class_scale.
template <int BITS>
__host__ __device__ constexpr int key_bit0() { return BITS == 4 ? 4 : 6; }
template <int BITS>
__host__ __device__ constexpr int key_bit(int p) { return BITS == 4 ? 4 : 6 + 2 * (p & 1); }
template <int BITS>
__host__ __device__ constexpr int key_class(int p) { return (key_bit<BITS>(p) - key_bit0<BITS>()) / 2; }
__host__ __device__ constexpr float class_scale(int c) { return (float)(1 << (2 * c)); }  // 2^(B - B0)
template <int BITS>
__host__ __device__ constexpr int key_classes() { return BITS == 4 ? 1 : 2; }

template <int BITS, int P>
__device__ __forceinline__ uint32_t key_pair(const KeyWords& c) {
  constexpr uint32_t code = ((1u << BITS) - 1u) << key_bit<BITS>(P);
  constexpr int copy = BITS == 4 ? P : P / 2;
  const uint32_t src = copy == 0 ? c.l : (copy == 1 ? c.m : (copy == 2 ? c.r : c.r2));
  return src & (code | (code << 16));
}

template <int BITS>
struct ValueWords {
  uint32_t m, r;
};
template <int BITS>
__device__ __forceinline__ ValueWords<BITS> value_words(uint32_t w) {
  return ValueWords<BITS>{w, BITS == 2 ? w >> 10 : w >> 8};
}
constexpr float kValueScale = 1.f / 512.f;  // of the codes value_pair returns

// Value pair p: 2^-9 (code - C), C = qmax / 2, exact. Centred, because the
// accumulator sums thousands of tokens: uncentred values would carry
// C * sum(s p) next to the signal.
template <int BITS, int P>
__device__ __forceinline__ uint32_t value_pair(const ValueWords<BITS>& c) {
  constexpr int B = BITS == 4 ? 4 * (P & 1) : 2 * (P % 5);
  constexpr uint32_t code = ((1u << BITS) - 1u) << B;
  const uint32_t x = ((BITS == 2 ? P < 5 : P < 2) ? c.m : c.r) & (code | (code << 16));
  // 2^(15 - B) and -C 2^-9 = -(qmax 2^-10) in fp16 (qmax = 1.1b or 1.111b binary)
  constexpr uint32_t mul = (uint32_t)(15 - B + 15) << 10;
  constexpr uint32_t add = 0x8000u | ((uint32_t)(BITS - 1 - 10 + 15) << 10) |
                           ((((1u << BITS) - 1u) << (11 - BITS)) & 0x3ffu);
  return hfma2_u32(x, mul | (mul << 16), add | (add << 16));
}

// One quantization group (32 keys = two 16-key blocks) of a packed tile;
// row_scale: shared address of the n-tiles' logit scales by query row.
// With x_hat = c * s + z (the powers of two of the codes left out):
//   S^T  = c_K . (s_K (.) Q)^T + beta,  beta = z_K . Q^T
//          (one MMA per 16 channels: A row r holds z over the channels of
//          class r, whose queries carry 1 / class_scale(r): exact fp16
//          products, fp32 sums)
//   O^T += (c - C)_V^T . (s_V (.) P^T) + z'_V^T . P^T,  C = qmax / 2,
//          z' = fp16(z + C s)
// The per-channel key scales fold into the queries as fp16 hi + lo parts (the
// scaled query keeps ~22 bits) and the per-token value scales into the
// probabilities.
// Class rows of a beta accumulator (lanes 4 (first + r) + j) summed with their
// scales: beta of query rows 2j, 2j + 1.
template <int BITS>
__device__ __forceinline__ void beta_rows(const float (&bq)[4], int first, float (&bt)[2]) {
  const int j = threadIdx.x & 3;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    bt[h] = __shfl_sync(0xffffffffu, bq[h], 4 * first + j);
#pragma unroll
    for (int r = 1; r < key_classes<BITS>(); ++r)
      bt[h] = fmaf(class_scale(r), __shfl_sync(0xffffffffu, bq[h], 4 * (first + r) + j), bt[h]);
  }
}

// beta of two groups of one tile with one set of MMAs: A rows 0..3 hold group
// a's zero points by class, rows 4..7 group b's. bt[h][nt] = beta of group h
// for query rows 2j, 2j + 1 of n-tile nt.
template <int NTW, int BITS>
__device__ __forceinline__ void group_beta_pair(uint32_t qsm, uint32_t base, int ga, int gb,
                                                float (&bt)[2][NTW][2]) {
  const int lane = threadIdx.x & 31;
  const int g = lane >> 2, j = lane & 3, gg = g & 3;
  float bq[NTW][4];
#pragma unroll
  for (int nt = 0; nt < NTW; ++nt) bq[nt][0] = bq[nt][1] = bq[nt][2] = bq[nt][3] = 0.f;
  const uint32_t kp = base + kSlotKParams + (g < 4 ? ga : gb) * 512 + j * 16 + 8;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint2 z = lds64(kp + i * 64);  // z(c0 c1), z(c8 c9)
    const uint32_t az[4] = {gg == key_class<BITS>(0) ? z.x : 0u, 0u, gg == key_class<BITS>(1) ? z.y : 0u, 0u};
#pragma unroll
    for (int nt = 0; nt < NTW; ++nt) {
      const uint2 qv = lds64(qsm + ((nt * 8 + i) * 32 + lane) * 8);
      mma_f16(bq[nt], az, qv.x, qv.y);
    }
  }
#pragma unroll
  for (int nt = 0; nt < NTW; ++nt)
#pragma unroll
    for (int h = 0; h < 2; ++h) beta_rows<BITS>(bq[nt], 4 * h, bt[h][nt]);
}

// kBeta = false: the group's beta comes in bt_in (from group_beta_pair)
// instead of its own MMAs.
template <int NTW, int BITS, bool kBeta = true>
__device__ __forceinline__ void group_quant(WarpState<NTW>& st, uint32_t qsm,
                                            uint32_t base, int gl, uint32_t row_scale,
                                            const float (&bt_in)[NTW][2]) {
  const int lane = threadIdx.x & 31;
  const int g = lane >> 2, j = lane & 3;
  constexpr int KW = BITS == 4 ? 4 : 2;  // code words per lane per 8-token tile
  const __half hc = __float2half_rn(0.5f * (float)((1 << BITS) - 1));
  const uint32_t vc_c = pack_h2(hc, hc);  // C = qmax / 2

  // ---- per 16 channels: scaled queries (fp16 hi + lo), beta, and S of both
  // 16-key blocks (four independent MMA chains; beta is added at the end)
  // The lo products have accumulators of their own with one n-tile (four
  // independent MMA chains; one chain per block: 32K int2 68.9 us against
  // 67.0). Two n-tiles are four chains without them, and 16 registers fewer
  // spill less (4 x 16K tokens, 4 query tokens 48.7 -> 46.2 us).
  constexpr bool kLoChain = NTW == 1;
  float bq[NTW][4];
  float sa[2][NTW][4], sl[2][NTW][4];
#pragma unroll
  for (int nt = 0; nt < NTW; ++nt)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      bq[nt][e] = 0.f;
      sa[0][nt][e] = sa[1][nt][e] = sl[0][nt][e] = sl[1][nt][e] = 0.f;
    }
  // key code words of the 8-token tiles 4 gl + t (t = 0..3: keys g, g + 8 of
  // block 0, then of block 1)
  uint32_t kw[4][KW];
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const uint32_t a = base + ((4 * gl + t) * 32 + lane) * (BITS * 4);
    if constexpr (BITS == 4) {
      const uint4 v = lds128(a);
      kw[t][0] = v.x;
      kw[t][1] = v.y;
      kw[t][KW > 2 ? 2 : 0] = v.z;
      kw[t][KW > 3 ? 3 : 1] = v.w;
    } else {
      const uint2 v = lds64(a);
      kw[t][0] = v.x;
      kw[t][1] = v.y;
    }
  }
  const uint32_t kp = base + kSlotKParams + gl * 512 + j * 16;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint4 P = lds128(kp + i * 64);  // s(c0 c1), s(c8 c9), z(c0 c1), z(c8 c9)
    // pairs of channels (16i + 2j, +1) and (16i + 2j + 8, +9)
    const uint32_t az[4] = {kBeta && g == key_class<BITS>(0) ? P.z : 0u, 0u,
                            kBeta && g == key_class<BITS>(1) ? P.w : 0u, 0u};
    // A fragments of both blocks for channels 16 i .. 16 i + 15
    uint32_t af[2][4];
    const int q = BITS == 4 ? (i >> 1) : (i >> 2);
#pragma unroll
    for (int blk = 0; blk < 2; ++blk) {
      const KeyWords w0 = key_words<BITS>(kw[2 * blk][q]), w1 = key_words<BITS>(kw[2 * blk + 1][q]);
      if constexpr (BITS == 4) {
        if ((i & 1) == 0) {
          af[blk][0] = key_pair<4, 0>(w0); af[blk][1] = key_pair<4, 0>(w1);
          af[blk][2] = key_pair<4, 1>(w0); af[blk][3] = key_pair<4, 1>(w1);
        } else {
          af[blk][0] = key_pair<4, 2>(w0); af[blk][1] = key_pair<4, 2>(w1);
          af[blk][2] = key_pair<4, 3>(w0); af[blk][3] = key_pair<4, 3>(w1);
        }
      } else {
        switch (i & 3) {
          case 0:
            af[blk][0] = key_pair<2, 0>(w0); af[blk][1] = key_pair<2, 0>(w1);
            af[blk][2] = key_pair<2, 1>(w0); af[blk][3] = key_pair<2, 1>(w1);
            break;
          case 1:
            af[blk][0] = key_pair<2, 2>(w0); af[blk][1] = key_pair<2, 2>(w1);
            af[blk][2] = key_pair<2, 3>(w0); af[blk][3] = key_pair<2, 3>(w1);
            break;
          case 2:
            af[blk][0] = key_pair<2, 4>(w0); af[blk][1] = key_pair<2, 4>(w1);
            af[blk][2] = key_pair<2, 5>(w0); af[blk][3] = key_pair<2, 5>(w1);
            break;
          default:
            af[blk][0] = key_pair<2, 6>(w0); af[blk][1] = key_pair<2, 6>(w1);
            af[blk][2] = key_pair<2, 7>(w0); af[blk][3] = key_pair<2, 7>(w1);
            break;
        }
      }
    }
#pragma unroll
    for (int nt = 0; nt < NTW; ++nt) {
      const uint2 qv = lds64(qsm + ((nt * 8 + i) * 32 + lane) * 8);
      const uint32_t qs0 = hmul2_u32(qv.x, P.x);
      const uint32_t qs1 = hmul2_u32(qv.y, P.y);
      const uint32_t ql0 = hfms2_u32(qv.x, P.x, qs0);
      const uint32_t ql1 = hfms2_u32(qv.y, P.y, qs1);
      if constexpr (kBeta) mma_f16(bq[nt], az, qv.x, qv.y);
#pragma unroll
      for (int blk = 0; blk < 2; ++blk) {
        mma_f16(sa[blk][nt], af[blk], qs0, qs1);
        mma_f16(kLoChain ? sl[blk][nt] : sa[blk][nt], af[blk], ql0, ql1);
      }
    }
  }
  float x[2][NTW][4];
#pragma unroll
  for (int nt = 0; nt < NTW; ++nt) {
    float bt[2] = {bt_in[nt][0], bt_in[nt][1]};
    if constexpr (kBeta) beta_rows<BITS>(bq[nt], 0, bt);
    const uint2 rs = lds64(row_scale + nt * 32 + j * 8);  // query rows 2j, 2j + 1
    float ks[2] = {__uint_as_float(rs.x), __uint_as_float(rs.y)};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      bt[h] *= ks[h];
      ks[h] *= (float)(1 << (24 - key_bit0<BITS>()));  // the codes' power of two
    }
#pragma unroll
    for (int blk = 0; blk < 2; ++blk)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        x[blk][nt][e] = fmaf(kLoChain ? sa[blk][nt][e] + sl[blk][nt][e] : sa[blk][nt][e], ks[e & 1], bt[e & 1]);
  }

  // ---- softmax over the group's 32 keys
  float pr[2][NTW][4];
  softmax_rows<NTW, 2>(st, x, pr);

  // ---- P V for both blocks
#pragma unroll
  for (int blk = 0; blk < 2; ++blk) {
    const int u = 2 * gl + blk;
    uint32_t b[NTW][2];
#pragma unroll
    for (int nt = 0; nt < NTW; ++nt) {
      b[nt][0] = movmatrix_t(pack_f16(pr[blk][nt][0], pr[blk][nt][1]));
      b[nt][1] = movmatrix_t(pack_f16(pr[blk][nt][2], pr[blk][nt][3]));
    }
    // value parameters of this block's 16 tokens: scales of the 4 channel
    // groups, zero points of groups g / 4 and g / 4 + 2 (rows g and g + 8 of Z)
    const uint32_t vpa = base + kSlotVParams + u * 256 + j * 16;
    uint2 vs[4];
#pragma unroll
    for (int gi = 0; gi < 4; ++gi) vs[gi] = lds64(vpa + gi * 64);  // s(t0 t1), s(t8 t9)
    {
      // Z row gi (lanes g = gi < 4): z' = z + C s of group gi, one MMA
      const uint4 vg = lds128(vpa + (g & 3) * 64);                   // s(t0 t1), s(t8 t9), z(t0 t1), z(t8 t9)
      const uint32_t z0 = g < 4 ? hfma2_u32(vg.x, vc_c, vg.z) : 0u;
      const uint32_t z1 = g < 4 ? hfma2_u32(vg.y, vc_c, vg.w) : 0u;
      const uint32_t az[4] = {z0, 0u, z1, 0u};
#pragma unroll
      for (int nt = 0; nt < NTW; ++nt) mma_f16(st.z[nt], az, b[nt][0], b[nt][1]);
    }
    ValueWords<BITS> vc[2 * KW];
    {
      const uint32_t va = base + kSlotVCodes + (u * 32 + lane) * (BITS * 8);
      const uint4 v0 = lds128(va);
      vc[0] = value_words<BITS>(v0.x);
      vc[1] = value_words<BITS>(v0.y);
      vc[2] = value_words<BITS>(v0.z);
      vc[3] = value_words<BITS>(v0.w);
      if constexpr (BITS == 4) {
        const uint4 v1 = lds128(va + 16);
        vc[2 * KW > 4 ? 4 : 0] = value_words<BITS>(v1.x);
        vc[2 * KW > 5 ? 5 : 1] = value_words<BITS>(v1.y);
        vc[2 * KW > 6 ? 6 : 2] = value_words<BITS>(v1.z);
        vc[2 * KW > 7 ? 7 : 3] = value_words<BITS>(v1.w);
      }
    }
#pragma unroll
    for (int gi = 0; gi < 4; ++gi) {
      uint32_t bs[NTW][2];
#pragma unroll
      for (int nt = 0; nt < NTW; ++nt) {
        bs[nt][0] = hmul2_u32(b[nt][0], vs[gi].x);
        bs[nt][1] = hmul2_u32(b[nt][1], vs[gi].y);
      }
#pragma unroll
      for (int mh = 0; mh < 2; ++mh) {
        const int mt = 2 * gi + mh;
        uint32_t a[4];
        // rows: channels 8m + g with m = 2 mt (a0, a2) and 2 mt + 1 (a1, a3);
        // a0 / a1 tokens 2j, 2j + 1 (pair p0), a2 / a3 tokens 2j + 8, 2j + 9 (p0 + 1)
        if constexpr (BITS == 4) {
          // m = 2mt + h: word m >> 1 = mt, p0 = 2 (m & 1) = 2h
          a[0] = value_pair<4, 0>(vc[mt]);
          a[2] = value_pair<4, 1>(vc[mt]);
          a[1] = value_pair<4, 2>(vc[mt]);
          a[3] = value_pair<4, 3>(vc[mt]);
        } else {
          // word m >> 2 = mt >> 1, p0 = 2 (m & 3) = 4 (mt & 1) + 2h
          const int q = mt >> 1;
          if ((mt & 1) == 0) {
            a[0] = value_pair<2, 0>(vc[q]);
            a[2] = value_pair<2, 1>(vc[q]);
            a[1] = value_pair<2, 2>(vc[q]);
            a[3] = value_pair<2, 3>(vc[q]);
          } else {
            a[0] = value_pair<2, 4>(vc[q]);
            a[2] = value_pair<2, 5>(vc[q]);
            a[1] = value_pair<2, 6>(vc[q]);
            a[3] = value_pair<2, 7>(vc[q]);
          }
        }
#pragma unroll
        for (int nt = 0; nt < NTW; ++nt) mma_f16(st.o[nt][mt], a, bs[nt][0], bs[nt][1]);
      }
    }
  }
}

// Zero the V rows [valid, 64) of a bf16 tile that lie in block u.
__device__ __forceinline__ void zero_v_rows(uint8_t* slot, int u, int valid) {
  const int lane = threadIdx.x & 31;
  const int lo = max(valid, 16 * u), hi = 16 * u + 16;
  for (int r = lo; r < hi; ++r) {
    uint8_t* row0 = slot + 16384 + r * 128;
    if (lane < 8)
      *reinterpret_cast<uint4*>(row0 + lane * 16) = make_uint4(0, 0, 0, 0);
    else if (lane < 16)
      *reinterpret_cast<uint4*>(row0 + 8192 + (lane - 8) * 16) = make_uint4(0, 0, 0, 0);
  }
  __syncwarp();
}

// Partial layout per item: [rows_pad][128] O (unnormalised), [rows_pad] m,
// [rows_pad] l, rows_pad = 8 * (number of n-tiles).

// Output row of query row r of a KV head (r = head * T + token).
template <class P>
__device__ __forceinline__ size_t out_row(const P& p, int b, int kvh, int r) {
  const int hl = p.n_qtok == 1 ? r : r / p.n_qtok, t = p.n_qtok == 1 ? 0 : r % p.n_qtok;
  return (size_t)(b * p.n_q_heads + kvh * p.group + hl) * p.n_qtok + t;
}

// First item of segment q.
__device__ __forceinline__ int segment_begin(const AttnParams& p, int q) { return p.seg[q].chunk_begin; }
__device__ __forceinline__ int segment_begin(const MergeCall& p, int q) { return p.chunk_begin[q]; }

// Log-sum-exp weights of query rows r0 .. r0 + nr - 1 over every item:
// ml[i * stride + rr] holds item i's m, ll[...] its l; the normalised weights
// replace m. PARTS threads per row (128 / PARTS rows at once, stride of them
// real); lse and the per-segment mass are written for the valid rows.
template <int PARTS, class P>
__device__ __forceinline__ void merge_weights(const P& p, float* ml, const float* ll, int stride, int b,
                                              int kvh, int r0, int nr, bool outputs = true) {
  const int I = p.items_per_bh;
  const int rr = threadIdx.x / PARTS, part = threadIdx.x % PARTS;
  const int i0 = PARTS == 16 || rr < stride ? part : I;  // threads past the padded rows have no items
  const bool mass = outputs && p.mass != nullptr;
  float M = kNegInf;
  for (int i = i0; i < I; i += PARTS) M = fmaxf(M, ml[i * stride + rr]);
#pragma unroll
  for (int o = PARTS / 2; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  const float Mu = (M == kNegInf) ? 0.f : M;
  float L = 0.f;
  float Ls[UC_MAX_SEGMENTS];
#pragma unroll
  for (int q = 0; q < UC_MAX_SEGMENTS; ++q) Ls[q] = 0.f;
  for (int i = i0; i < I; i += PARTS) {
    const float mi = ml[i * stride + rr];
    const float w = (mi == kNegInf) ? 0.f : exp2f(mi - Mu);
    const float lw = ll[i * stride + rr] * w;
    L += lw;
    if (mass) {
      int sg = 0;
#pragma unroll
      for (int q = 1; q < UC_MAX_SEGMENTS; ++q) sg += (q < p.nseg && i >= segment_begin(p, q)) ? 1 : 0;
#pragma unroll
      for (int q = 0; q < UC_MAX_SEGMENTS; ++q)
        if (q == sg) Ls[q] += lw;
    }
    ml[i * stride + rr] = w;  // unnormalised weight (this thread's own entry)
  }
#pragma unroll
  for (int o = PARTS / 2; o > 0; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
  const float inv = (L > 0.f) ? 1.f / L : 0.f;
  for (int i = i0; i < I; i += PARTS) ml[i * stride + rr] *= inv;
  if (mass) {
#pragma unroll
    for (int q = 0; q < UC_MAX_SEGMENTS; ++q)
      if (q < p.nseg)
#pragma unroll
        for (int o = PARTS / 2; o > 0; o >>= 1) Ls[q] += __shfl_xor_sync(0xffffffffu, Ls[q], o);
  }
  if (outputs && part == 0 && rr < nr) {
    const size_t orow = out_row(p, b, kvh, r0 + rr);
    if (p.lse) p.lse[orow] = (L > 0.f) ? (M + log2f(L)) * kLn2 : kNegInf;
    if (mass)
      for (int q = 0; q < p.nseg; ++q) p.mass[orow * p.nseg + q] = Ls[q] * inv;
  }
}

// A batch's merge with several n-tiles runs on the 128 consumer threads of the
// CTA that finished the last item of a (sequence, KV head): the weights of
// every item and row, then per 8-row block the weighted sums of the items' O, four channels of two
// rows per thread (16-byte shared-memory reads; one 4-byte read per value
// with its weight held the merge of 13 items for 5 us). After the CTA's last
// item the ring is idle (`seq` given): the row blocks of O stream through it
// back to back, eight items per slot, by bulk copies continuing the consumers'
// tile sequence, the first ones in flight while the weights are formed.
// Without `seq` (a merge between items) the threads load them. Only batches
// merge here: single calls are faster with the merge kernel, and their kernel
// without this code in it (four query tokens, 4 x 16K int2 36.4 -> 35.2 us, 8 x
// 20K int4 70.4 -> 69.3; two, 1 x 300 10.6 -> 10.1; mixed 4 x 16K 33.7 -> 34.1).
template <int NTW, int ST>
__device__ void final_merge(const AttnParams& p, AttnSmem& sm, int bh, uint32_t* seq) {
  const int tid = threadIdx.x;
  const int b = bh / p.n_kv_heads, kvh = bh % p.n_kv_heads;
  const size_t pf = attend_part_floats(p.mtiles);
  const int rows_pad = 8 * p.mtiles;
  const int I = p.items_per_bh;
  const float* base = p.part + (size_t)bh * I * pf;
  constexpr int kPerSlot = kSlotBytes / (8 * kHeadDim * 4);  // 8-row blocks of O per ring slot
  const int nb = (I + kPerSlot - 1) / kPerSlot;
  const int total = nb * p.mtiles;
  auto issue = [&](int n) {  // batch n: eight items of row block n / nb (thread 0)
    const uint32_t sq = *seq + n;
    uint64_t* bar = &sm.full[sq % ST];
    const int i0 = (n % nb) * kPerSlot, cnt = min(kPerSlot, I - i0);
    mbar_arrive_expect_tx(bar, (uint32_t)cnt * 8 * kHeadDim * 4);
    for (int k = 0; k < cnt; ++k)
      bulk_load(sm.slot[sq % ST] + k * 8 * kHeadDim * 4, base + (i0 + k) * pf + (size_t)(n / nb) * 8 * kHeadDim,
                8 * kHeadDim * 4, bar);
  };
  if (seq != nullptr && tid == 0) {
    // the partials were written by other CTAs (generic proxy) and acquired
    // at GPU scope; order that acquire before the copy engine's reads
    fence_proxy_async_global();
    for (int n = 0; n < min(ST, total); ++n) issue(n);
  }
  // rows whose weights are formed at once: every row when the query buffers
  // behind the ring are idle too, else the 8 rows the merge arrays hold
  const int set = seq == nullptr ? 8 : rows_pad;
  float* wts = seq == nullptr ? sm.merge_w : reinterpret_cast<float*>(after_ring<ST>(sm));  // [I][set]
  float* ls = seq == nullptr ? sm.merge_l : wts + I * set;
  const int cq = tid & 31, rg = tid >> 5;  // channels 4 cq .. + 3, rows 2 rg, 2 rg + 1 of a block
  for (int s0 = 0; s0 < p.rows; s0 += set) {
    for (int x = tid; x < I * set; x += 128) {
      const int i = x / set, r = s0 + x % set;
      const float* mp = base + i * pf + rows_pad * kHeadDim + r;
      wts[x] = r < p.rows ? __ldcg(mp) : kNegInf;
      ls[x] = r < p.rows ? __ldcg(mp + rows_pad) : 0.f;
    }
    consumer_sync();
    const int nr = min(set, p.rows - s0);
    if (set == 8)
      merge_weights<16>(p, wts, ls, 8, b, kvh, s0, nr);
    else if (p.mtiles <= 2)
      merge_weights<8>(p, wts, ls, set, b, kvh, s0, nr);
    else if (p.mtiles <= 4)
      merge_weights<4>(p, wts, ls, set, b, kvh, s0, nr);
    else
      merge_weights<2>(p, wts, ls, set, b, kvh, s0, nr);
    consumer_sync();
    for (int r0 = s0; r0 < min(s0 + set, p.rows); r0 += 8) {
      float acc[2][4] = {};
      auto add = [&](int i, float4 x0, float4 x1) {
        const float2 w = *reinterpret_cast<const float2*>(&wts[i * set + (r0 - s0) + 2 * rg]);
        acc[0][0] += w.x * x0.x; acc[0][1] += w.x * x0.y; acc[0][2] += w.x * x0.z; acc[0][3] += w.x * x0.w;
        acc[1][0] += w.y * x1.x; acc[1][1] += w.y * x1.y; acc[1][2] += w.y * x1.z; acc[1][3] += w.y * x1.w;
      };
      if (seq != nullptr) {
        for (int j = 0; j < nb; ++j) {
          const int n = r0 / 8 * nb + j, i0 = j * kPerSlot, cnt = min(kPerSlot, I - i0);
          const uint32_t sq = *seq + n;
          const bool ok = mbar_wait(&sm.full[sq % ST], (sq / ST) & 1, p.status, 14, p.wait_ns);
          const float4* buf = reinterpret_cast<const float4*>(sm.slot[sq % ST]) + 2 * rg * 32 + cq;
          if (ok) {
#pragma unroll
            for (int k = 0; k < kPerSlot; ++k)
              if (k < cnt) add(i0 + k, buf[k * 256], buf[k * 256 + 32]);
          }
          if (n + ST < total) {
            consumer_sync();  // the slot is read: refill it
            if (tid == 0) issue(n + ST);
          }
        }
      } else {
#pragma unroll 4
        for (int i = 0; i < I; ++i) {
          const float4* pi = reinterpret_cast<const float4*>(base + i * pf + (size_t)(r0 + 2 * rg) * kHeadDim) + cq;
          add(i, __ldcg(pi), __ldcg(pi + 32));
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = r0 + 2 * rg + h;
        if (r < p.rows)
          *reinterpret_cast<uint2*>(p.out + out_row(p, b, kvh, r) * kHeadDim + 4 * cq) =
              make_uint2(pack_bf16(acc[h][0], acc[h][1]), pack_bf16(acc[h][2], acc[h][3]));
      }
    }
    consumer_sync();  // the weights and the slots are read
  }
  if (seq != nullptr) *seq += total;
}

// Split-K merge as a kernel of its own: a CTA per (sequence, KV head, 8-row
// block, CW output channels), so the partials of one (b, kvh) are read by
// several SMs at once instead of streaming through one. A thread has four
// channels of one row, so 128 / CW groups of threads share the items; the
// first eight items of each group are fetched before the weights are known.
// One launch serves every call of a batch of one n-tile. What bounds it is the chain launch -> maxima and sums ->
// weights -> sums; with many pairs every CTA's weights would count too (eight
// query tokens, 16 x 300: CW 32 took 31.6 us, 20.1 so), so CW grows with the
// number of CTAs (`merge_width`). The attention launch writes the partials
// while this one is resident, so they are read with ordinary (L2) loads behind
// griddep_wait: the read-only path is for data that no kernel in flight writes.
// The call of row block *blk of a merge launch (then the block's place in it).
__device__ __forceinline__ const MergeCall& merge_call(const MergeCall& p, int*) { return p; }
__device__ __forceinline__ const MergeCall& merge_call(const MultiMerge& m, int* blk) {
  int k = 0;
  for (int n; k + 1 < m.n_calls && *blk >= (n = m.call[k].batch * m.call[k].n_kv_heads * m.call[k].mtiles); ++k)
    *blk -= n;
  return m.call[k];
}

template <int CW, class P>
__global__ void __launch_bounds__(256, kMergePerSm) merge_partials_kernel(const __grid_constant__ P params) {
  constexpr int kCols = CW / 4, kPos = 8 * kCols, G = 256 / kPos, kPre = 8;
  __shared__ float s_m[kMaxItemsPerBh * 8], s_w[kMaxItemsPerBh * 8];  // m, then the weights; l
  __shared__ float4 s_red[G][kPos];
  griddep_wait();  // the attention launch whose partials this merges has completed
  griddep_launch_dependents();
  const int tid = threadIdx.x;
  const int ch = blockIdx.x % (kHeadDim / CW);
  int blk = blockIdx.x / (kHeadDim / CW);
  const MergeCall& p = merge_call(params, &blk);
  const int r0 = (blk % p.mtiles) * 8, bh = blk / p.mtiles;
  const int b = bh / p.n_kv_heads, kvh = bh % p.n_kv_heads;
  const int nr = min(8, p.rows - r0);
  const size_t pf = attend_part_floats(p.mtiles);
  const int rows_pad = 8 * p.mtiles;
  const int I = p.items_per_bh;
  const float* base = p.part + (size_t)bh * I * pf;
  // every (item, row) pair's m and l: at most two pairs per thread
  for (int x = tid; x < I * 8; x += 256) {
    const int i = x >> 3, rr = x & 7;
    float m = kNegInf, l = 0.f;
    if (rr < nr) {
      m = __ldcg(base + i * pf + rows_pad * kHeadDim + r0 + rr);
      l = __ldcg(base + i * pf + rows_pad * kHeadDim + rows_pad + r0 + rr);
    }
    s_m[x] = m;
    s_w[x] = l;
  }
  const int pos = tid % kPos, grp = tid / kPos, rr = pos / kCols, c = ch * CW + 4 * (pos % kCols);
  const float* col = base + (size_t)(r0 + rr) * kHeadDim + c;
  float4 v[kPre];
  auto fetch = [&](int i0) {
#pragma unroll
    for (int k = 0; k < kPre; ++k) {
      const int i = i0 + G * k;
      v[k] = i < I && rr < nr ? __ldcg(reinterpret_cast<const float4*>(col + i * pf)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  fetch(grp);
  __syncthreads();
  if (tid < 128) merge_weights<16>(p, s_m, s_w, 8, b, kvh, r0, nr, ch == 0);
  __syncthreads();
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int i0 = grp; i0 < I; i0 += G * kPre) {
    if (i0 != grp) fetch(i0);
#pragma unroll
    for (int k = 0; k < kPre; ++k) {
      const int i = i0 + G * k;
      if (i < I) {
        const float wt = s_m[i * 8 + rr];
        acc.x += wt * v[k].x; acc.y += wt * v[k].y; acc.z += wt * v[k].z; acc.w += wt * v[k].w;
      }
    }
  }
  if constexpr (G > 1) {
    s_red[grp][pos] = acc;
    __syncthreads();
    if (grp != 0) return;
#pragma unroll
    for (int k = 1; k < G; ++k) {
      const float4 o = s_red[k][pos];
      acc.x += o.x; acc.y += o.y; acc.z += o.z; acc.w += o.w;
    }
  }
  if (rr < nr)
    *reinterpret_cast<uint2*>(p.out + out_row(p, b, kvh, r0 + rr) * kHeadDim + c) =
        make_uint2(pack_bf16(acc.x, acc.y), pack_bf16(acc.z, acc.w));
}

// Query rows of every n-tile as Q^T B fragments in shared memory: word w of
// lane (g, j) for channels 16i + 2j (+8) of row 8 nt + g at
// [((nt * 8 + i) * 32 + lane) * 2 + w], from the bf16 rows the producer copied
// (row r = head * T + token). All consumer threads.
//
// For bf16 rows the words are the queries as they are. For packed keys they
// are fp16, whose step stops shrinking at 2^-24: queries of 1e-4 on keys of
// 1e3 (logits up to 1) lose up to 1e-4 of a logit to it, four times that with
// a class's 1/4. So a row whose largest element is below 1/2 is brought up to
// [1/2, 1) by an exact power of two, which its logit scale takes out again.
// Never above 1: a scaled query q s then stays finite for every fp16 key scale
// s, and rows from 1/2 up stay as they are.
constexpr int kMaxRowShift = 60;  // row scales stay normal fp32 values

template <int BITS>
__device__ __forceinline__ void store_q(const AttnParams& p, uint32_t* qf, const uint8_t* rows, float* row_scale) {
  const int tid = threadIdx.x;
  if constexpr (BITS == 16) {
    for (int x = tid; x < p.mtiles * 512; x += 128) {
      const int nt = x >> 9, i = (x >> 6) & 7, ln = (x >> 1) & 31, w = x & 1;
      const int r = nt * 8 + (ln >> 2);
      const int c = 16 * i + 2 * (ln & 3) + 8 * w;
      qf[x] = r < p.rows ? *reinterpret_cast<const uint32_t*>(rows + (r * kHeadDim + c) * 2) : 0u;
    }
  } else {
    // words t * 128 + tid of an n-tile: one row per thread, i = 2 t + par; the
    // row's other words are in the threads that differ in bits 0-2 (and 6)
    const int ln = (tid >> 1) & 31, w = tid & 1, par = tid >> 6;
    for (int nt = 0; nt < p.mtiles; ++nt) {
      const int r = nt * 8 + (ln >> 2);
      const uint32_t* src = reinterpret_cast<const uint32_t*>(rows) + r * (kHeadDim / 2) + (ln & 3) + 4 * w;
      uint32_t own[4], mx = 0u;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int i = 2 * t + par;
        own[t] = r < p.rows ? src[8 * i] : 0u;
        const uint32_t other = r < p.rows ? src[8 * (i ^ 1)] : 0u;
        mx = __vmaxu2(mx, __vmaxu2(own[t] & 0x7fff7fffu, other & 0x7fff7fffu));
      }
#pragma unroll
      for (int o = 1; o < 8; o *= 2) mx = __vmaxu2(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const int ex = (int)(max(mx & 0xffffu, mx >> 16) >> 7);  // the largest element's exponent field
      const int k = min(max(126 - ex, 0), kMaxRowShift);
      // 2^k / class_scale of the channels' key pair (pairs alternate with w)
      const float f = __uint_as_float((uint32_t)(127 + k) << 23) / (w ? class_scale(key_class<BITS>(1)) : 1.f);
#pragma unroll
      for (int t = 0; t < 4; ++t) qf[nt * 512 + t * 128 + tid] = pack_f16(bf16_lo(own[t]) * f, bf16_hi(own[t]) * f);
      if ((tid & 0x47) == 0) row_scale[r] = p.scale_log2 * __uint_as_float((uint32_t)(127 - k) << 23);
    }
  }
}

// Adds the zero-point term of packed values to O: channel group gi of query
// rows 2j, 2j + 1 sits in lane (gi, j).
template <int NTW>
__device__ __forceinline__ void fold_zero_points(WarpState<NTW>& st) {
  const int j = threadIdx.x & 3;
#pragma unroll
  for (int nt = 0; nt < NTW; ++nt)
#pragma unroll
    for (int gi = 0; gi < 4; ++gi) {
      const float z0 = __shfl_sync(0xffffffffu, st.z[nt][0], 4 * gi + j);
      const float z1 = __shfl_sync(0xffffffffu, st.z[nt][1], 4 * gi + j);
#pragma unroll
      for (int mh = 0; mh < 2; ++mh) {
        st.o[nt][2 * gi + mh][0] += z0;
        st.o[nt][2 * gi + mh][1] += z1;
        st.o[nt][2 * gi + mh][2] += z0;
        st.o[nt][2 * gi + mh][3] += z1;
      }
    }
}

// Full row sums: adds the shares of the 8 key lanes (g).
template <int NTW>
__device__ __forceinline__ void reduce_row_sums(WarpState<NTW>& st) {
#pragma unroll
  for (int nt = 0; nt < NTW; ++nt)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float v = st.l[nt][h];
      v += __shfl_xor_sync(0xffffffffu, v, 4);
      v += __shfl_xor_sync(0xffffffffu, v, 8);
      v += __shfl_xor_sync(0xffffffffu, v, 16);
      st.l[nt][h] = v;
    }
}

// One n-tile: the four consumer warps' states meet in an idle ring slot in one
// step (rows padded by four floats: the fragments' stores and the row reads
// are conflict-free), then 16 threads per query row sum them, eight channels
// each, and store or pass on whole 16-byte pieces. (By a pairwise tree with
// its barriers and 4-byte stores by the last warp 4K int2, batch 1, took 8.8
// us, so 8.3; 32K int2, batch 16, 65.8 and 65.2.)
struct WarpsO {
  float o[kConsumers][8][kHeadDim + 4];
  float m[kConsumers][8], l[kConsumers][8];
};
static_assert(sizeof(WarpsO) <= kSlotBytes, "in a ring slot");

__device__ __forceinline__ void put_warp(WarpsO& b, int warp, const WarpState<1>& st) {
  const int lane = threadIdx.x & 31, g = lane >> 2, j = lane & 3;
#pragma unroll
  for (int mt = 0; mt < 8; ++mt)
#pragma unroll
    for (int e = 0; e < 4; ++e) b.o[warp][2 * j + (e & 1)][16 * mt + g + 8 * (e >> 1)] = st.o[0][mt][e];
  if (g == 0) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      b.m[warp][2 * j + h] = st.m[0][h];
      b.l[warp][2 * j + h] = st.l[0][h];
    }
  }
}

// Maximum of row threadIdx.x / 16 over the warps, their weights, and O of
// channels 4 (threadIdx.x % 16) + {0 .. 3} and the same + 64.
__device__ __forceinline__ float sum_warps(const WarpsO& b, float (&wt)[kConsumers], float4 (&o)[2]) {
  const int row = threadIdx.x >> 4, c = 4 * (threadIdx.x & 15);
  float M = kNegInf;
#pragma unroll
  for (int w = 0; w < kConsumers; ++w) M = fmaxf(M, b.m[w][row]);
#pragma unroll
  for (int w = 0; w < kConsumers; ++w) {
    const float m = b.m[w][row];
    wt[w] = m == kNegInf ? 0.f : exp2f(m - M);
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    o[h] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < kConsumers; ++w) {
      const float4 x = *reinterpret_cast<const float4*>(&b.o[w][row][c + 64 * h]);
      o[h].x += wt[w] * x.x; o[h].y += wt[w] * x.y; o[h].z += wt[w] * x.z; o[h].w += wt[w] * x.w;
    }
  }
  return M;
}

// Merge the warps that share n-tiles (through the item's last slot), then
// write this item's partial.
template <int NTW>
__device__ __forceinline__ void finish_item(const AttnParams& p, AttnSmem& sm, WarpState<NTW>& st,
                                            int it, int last_slot, int NG, int KS, int grp, int ks) {
  const int lane = threadIdx.x & 31;
  const int g = lane >> 2, j = lane & 3;
  fold_zero_points<NTW>(st);
  reduce_row_sums<NTW>(st);
  if constexpr (NTW == 1) {
    float* pi = p.part + (size_t)it * attend_part_floats(1);
    const int row = threadIdx.x >> 4, c = 4 * (threadIdx.x & 15);
    float4 o[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
    float M = kNegInf, l = 0.f;
    if (last_slot >= 0) {
      WarpsO& b = *reinterpret_cast<WarpsO*>(sm.slot[last_slot]);
      consumer_sync();  // every warp has read the slot's tile
      put_warp(b, ks, st);
      consumer_sync();
      float wt[kConsumers];
      M = sum_warps(b, wt, o);
#pragma unroll
      for (int w = 0; w < kConsumers; ++w) l += wt[w] * b.l[w][row];
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.empty[last_slot]);
    }
    *reinterpret_cast<float4*>(pi + row * kHeadDim + c) = o[0];
    *reinterpret_cast<float4*>(pi + row * kHeadDim + c + 64) = o[1];
    if (c == 0) {
      pi[8 * kHeadDim + row] = M;
      pi[8 * kHeadDim + 8 + row] = l;
    }
    return;
  }
  constexpr int kVals = NTW * 36;
  if (KS > 1 && last_slot >= 0) {
    float* buf = reinterpret_cast<float*>(sm.slot[last_slot]);
    consumer_sync();
    for (int step = 1; step < KS; step *= 2) {
      const bool writer = (ks % (2 * step)) == step;
      const bool reader = (ks % (2 * step)) == 0;
      const int region = (ks / (2 * step)) * NG + grp;
      float* rb = buf + region * (kVals * 32);
      if (writer) {
#pragma unroll
        for (int nt = 0; nt < NTW; ++nt) {
#pragma unroll
          for (int mt = 0; mt < 8; ++mt)
#pragma unroll
            for (int e = 0; e < 4; ++e) rb[((nt * 36) + mt * 4 + e) * 32 + lane] = st.o[nt][mt][e];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            rb[(nt * 36 + 32 + h) * 32 + lane] = st.m[nt][h];
            rb[(nt * 36 + 34 + h) * 32 + lane] = st.l[nt][h];
          }
        }
      }
      consumer_sync();
      if (reader) {
#pragma unroll
        for (int nt = 0; nt < NTW; ++nt) {
          float a[2], bb[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float om = rb[(nt * 36 + 32 + h) * 32 + lane];
            const float ol = rb[(nt * 36 + 34 + h) * 32 + lane];
            const float nm = fmaxf(st.m[nt][h], om);
            const float um = (nm == kNegInf) ? 0.f : nm;
            a[h] = exp2f(st.m[nt][h] - um);
            bb[h] = exp2f(om - um);
            st.l[nt][h] = st.l[nt][h] * a[h] + ol * bb[h];
            st.m[nt][h] = nm;
          }
#pragma unroll
          for (int mt = 0; mt < 8; ++mt)
#pragma unroll
            for (int e = 0; e < 4; ++e)
              st.o[nt][mt][e] = st.o[nt][mt][e] * a[e & 1] + rb[(nt * 36 + mt * 4 + e) * 32 + lane] * bb[e & 1];
        }
      }
      consumer_sync();
    }
    fence_proxy_async();
    __syncwarp();
    if (lane == 0) mbar_arrive(&sm.empty[last_slot]);
  }
  if (ks == 0) {
    const size_t pf = attend_part_floats(p.mtiles);
    const int rows_pad = 8 * p.mtiles;
    float* pi = p.part + (size_t)it * pf;
#pragma unroll
    for (int nt = 0; nt < NTW; ++nt) {
      const int ntg = grp * NTW + nt;
      if (ntg >= p.mtiles) continue;
      const int r0 = ntg * 8 + 2 * j;
#pragma unroll
      for (int mt = 0; mt < 8; ++mt) {
        const int c0 = 16 * mt + g;
        pi[(r0) * kHeadDim + c0] = st.o[nt][mt][0];
        pi[(r0 + 1) * kHeadDim + c0] = st.o[nt][mt][1];
        pi[(r0) * kHeadDim + c0 + 8] = st.o[nt][mt][2];
        pi[(r0 + 1) * kHeadDim + c0 + 8] = st.o[nt][mt][3];
      }
      if (g == 0) {
        pi[rows_pad * kHeadDim + r0] = st.m[nt][0];
        pi[rows_pad * kHeadDim + r0 + 1] = st.m[nt][1];
        pi[rows_pad * kHeadDim + rows_pad + r0] = st.l[nt][0];
        pi[rows_pad * kHeadDim + rows_pad + r0 + 1] = st.l[nt][1];
      }
    }
  }
}

// All tiles of one item added to a warp's state: bf16 rows (BITS = 16: bf16
// segments and the tails of packed segments) or packed groups (BITS = 4 / 2).
// With `keep_last` the item's last slot is not handed back; returns it (-1: none).
template <int NTW, int ST, int BITS>
__device__ __forceinline__ int run_tiles(const AttnParams& p, AttnSmem& sm, const ItemInfo& ii, int k, uint32_t& seq,
                                         bool& aborted, int KS, int grp, int ks, bool keep_last,
                                         WarpState<NTW>& st) {
  const int lane = threadIdx.x & 31;
  uint32_t* qf = NTW == 1 ? reinterpret_cast<uint32_t*>(sm.merge_w)
                          : reinterpret_cast<uint32_t*>(after_ring<ST>(sm));
  store_q<BITS>(p, qf, qrows_buf<ST>(sm, k, p.mtiles), sm.row_scale);
  consumer_sync();
  if (lane == 0) mbar_arrive(&sm.item_empty[k]);  // the query rows are no longer needed
  const uint32_t qs = smem_u32(qf) + grp * NTW * 2048, rs = smem_u32(sm.row_scale) + grp * NTW * 32;
  // packed values enter O as kValueScale times theirs
  if constexpr (BITS != 16) scale_o<NTW>(st, kValueScale);
  int last_slot = -1;
  for (int t = ii.tb; t < ii.te; ++t, ++seq) {
    const int slot = seq % ST;
    if (!aborted && !mbar_wait(&sm.full[slot], (seq / ST) & 1, p.status, 11, p.wait_ns)) aborted = true;
    const uint32_t sbase = smem_u32(sm.slot[slot]);
    bool wrote = false;  // generic-proxy writes into the slot (zeroed V rows)
    if (!aborted) {
      if constexpr (BITS == 16) {
        const int valid = ii.tail ? (ii.n % kGroup) : min(kTileTok, ii.n - t * kTileTok);
        wrote = valid < kTileTok;
        for (int u = ks; u < 4; u += KS) {
          if (16 * u >= valid) continue;
          if (valid < 16 * u + 16) zero_v_rows(sm.slot[slot], u, valid);
          block_bf16<NTW>(st, qs, sbase, u, valid, p.scale_log2);
        }
      } else {
        constexpr int kTG = quant_groups_per_tile(BITS);
        const int ng = ii.n / kGroup;
        const int ngt = min(kTG, ng - kTG * t);  // quantization groups in this tile
        int gl = ks;
        if constexpr (NTW == 1 && BITS == 2) {
          // the warp's two groups of a full tile share one set of beta MMAs
          if (gl + KS < ngt) {
            float bt[2][NTW][2];
            group_beta_pair<NTW, BITS>(qs, sbase, gl, gl + KS, bt);
#pragma unroll 1
            for (int h = 0; h < 2; ++h, gl += KS) {
              float bh[NTW][2];
#pragma unroll
              for (int nt = 0; nt < NTW; ++nt) {
                bh[nt][0] = h ? bt[1][nt][0] : bt[0][nt][0];
                bh[nt][1] = h ? bt[1][nt][1] : bt[0][nt][1];
              }
              group_quant<NTW, BITS, false>(st, qs, sbase, gl, rs, bh);
            }
          }
        }
        const float none[NTW][2] = {};
#pragma unroll 1
        for (; gl < ngt; gl += KS) group_quant<NTW, BITS>(st, qs, sbase, gl, rs, none);
      }
    }
    if (t + 1 < ii.te || !keep_last) {
      // reads alone need no proxy fence before the slot is handed back to
      // the copy engine; the zeroed rows of a partial bf16 tile do
      if (wrote) fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.empty[slot]);
    } else {
      last_slot = slot;
    }
  }
  if constexpr (BITS != 16) scale_o<NTW>(st, 1.f / kValueScale);
  return last_slot;
}

template <int NTW, int ST, int BITS>
__device__ __forceinline__ void run_item(const AttnParams& p, AttnSmem& sm, const ItemInfo& ii, int it, int k,
                                         uint32_t& seq, bool& aborted, int NG, int KS, int grp, int ks) {
  WarpState<NTW> st;
  state_init<NTW>(st);
  const int last_slot = run_tiles<NTW, ST, BITS>(p, sm, ii, k, seq, aborted, KS, grp, ks, KS > 1, st);
  finish_item<NTW>(p, sm, st, it, last_slot, NG, KS, grp, ks);
}

// ---- cluster launches (one n-tile): a (sequence, KV head)'s items on the
// CTAs of one cluster. A warp carries its state from item to item (the row
// sums go to its bank per segment, for the masses); the CTA's four warps meet
// in its idle ring, and after one cluster barrier rank r's warps each finish
// query rows of the pair from every CTA's shared memory. No partial output
// goes through global memory, and no CTA waits for an arrival counter's
// answer, copies partials in and weighs them after everyone else has left:
// those took 2 + 5 us at the end of a 20 us call (8K context, batch 8).
struct ClusterPart {
  float o[8][kHeadDim];                // unnormalised O of this CTA's items
  float m[8];                          // per query row, log2 units
  float l[UC_MAX_SEGMENTS][8];         // row sums per segment
};
struct ClusterSmem {
  WarpsO warps;
  ClusterPart part;
};
static_assert(sizeof(ClusterSmem) <= (size_t)kStages * kSlotBytes, "in the idle ring");
// per warp, segment and row: the row sum so far and the maximum it refers to
using RowBank = float2[kConsumers][UC_MAX_SEGMENTS][8];
static_assert(sizeof(RowBank) <= sizeof(float) * kMaxItemsPerBh * 8, "in the merge array the queries leave free");

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// Shared address of the same variable in another CTA of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(const void* local, int rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(local)), "r"(rank));
  return a;
}
__device__ __forceinline__ float ld_cluster(uint32_t a) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a)
               : "memory");
  return v;
}

__device__ __forceinline__ void consume_cluster(const AttnParams& p, AttnSmem& sm) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, j = lane & 3;
  uint32_t seq = 0;
  bool aborted = false;
  RowBank& bank = *reinterpret_cast<RowBank*>(sm.merge_l);
  for (int x = lane; x < UC_MAX_SEGMENTS * 8; x += 32) bank[warp][x >> 3][x & 7] = make_float2(kNegInf, 0.f);
  __syncwarp();
  WarpState<1> st;
  state_init<1>(st);
  for (uint32_t iseq = 0;; ++iseq) {
    const int k = iseq % kItemQ;
    // one decision for the CTA's warps (a wait that ran out in one of them ends
    // the loop in all, so their barriers stay in step); it also separates the
    // last item's reads of the query fragments from this item's writes
    if (!consumer_all(mbar_wait(&sm.item_full[k], (iseq / kItemQ) & 1, p.status, 13, p.wait_ns))) break;
    const int pos = sm.item_pos[k];
    if (pos < 0) break;
    int it;
    const ItemInfo ii = decode_item(p, pos, &it);
    const SegDev& sd = p.seg[ii.s];
    if (seg_is_bf16(sd.kind) || ii.tail)
      run_tiles<1, kStages, 16>(p, sm, ii, k, seq, aborted, kConsumers, 0, warp, false, st);
    else if (sd.bits == 4)
      run_tiles<1, kStages, 4>(p, sm, ii, k, seq, aborted, kConsumers, 0, warp, false, st);
    else
      run_tiles<1, kStages, 2>(p, sm, ii, k, seq, aborted, kConsumers, 0, warp, false, st);
    reduce_row_sums<1>(st);
    if (g == 0) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float2& e = bank[warp][ii.s][2 * j + h];
        const float old = e.y == 0.f ? 0.f : e.y * exp2f(e.x - st.m[0][h]);
        e = make_float2(st.m[0][h], old + st.l[0][h]);
      }
    }
    st.l[0][0] = st.l[0][1] = 0.f;
    __syncwarp();
  }
  // the CTA's part: O of the four warps, row maxima, row sums per segment
  fold_zero_points<1>(st);
  ClusterSmem& cs = *reinterpret_cast<ClusterSmem*>(sm.slot[0]);
  consumer_sync();  // every warp is past its last tile: the ring is idle
  put_warp(cs.warps, warp, st);
  consumer_sync();
  {
    const int row = threadIdx.x >> 4, c = 4 * (threadIdx.x & 15), s = threadIdx.x & 15;
    float wt[kConsumers];
    float4 o[2];
    const float M = sum_warps(cs.warps, wt, o);
    *reinterpret_cast<float4*>(&cs.part.o[row][c]) = o[0];
    *reinterpret_cast<float4*>(&cs.part.o[row][c + 64]) = o[1];
    if (s < p.nseg) {
      float l = 0.f;
#pragma unroll
      for (int w = 0; w < kConsumers; ++w) {
        const float2 e = bank[w][s][row];
        if (e.y != 0.f) l += e.y * exp2f(e.x - M);
      }
      cs.part.l[s][row] = l;
    }
    if (s == 0) cs.part.m[row] = M;
  }
  __syncwarp();
  cluster_arrive();
  cluster_wait();
  // one warp per query row: the rows of the pair over the warps of the cluster
  const int C = p.cluster, rank = blockIdx.x % C;
  const int pair = blockIdx.x / C, b = pair / p.n_kv_heads, kvh = pair % p.n_kv_heads;
  for (int r = rank + C * warp; r < p.rows; r += C * kConsumers) {
    const uint32_t pb = cluster_addr(&cs.part, lane < C ? lane : 0);  // lane c: CTA c's part
    float m = kNegInf, l = 0.f, ls[UC_MAX_SEGMENTS];
#pragma unroll
    for (int s = 0; s < UC_MAX_SEGMENTS; ++s) ls[s] = 0.f;
    if (lane < C) {
      m = ld_cluster(pb + (uint32_t)offsetof(ClusterPart, m) + 4 * r);
#pragma unroll
      for (int s = 0; s < UC_MAX_SEGMENTS; ++s)
        if (s < p.nseg) ls[s] = ld_cluster(pb + (uint32_t)offsetof(ClusterPart, l) + (s * 8 + r) * 4);
    }
    float4 x[16];
#pragma unroll
    for (int c = 0; c < 16; ++c)
      if (c < C) x[c] = ld_cluster4(cluster_addr(&cs.part.o[r][4 * lane], c));
    float M = m;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
    const float w = m == kNegInf ? 0.f : exp2f(m - M);
#pragma unroll
    for (int s = 0; s < UC_MAX_SEGMENTS; ++s) l += ls[s];
    l *= w;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    const float inv = l > 0.f ? 1.f / l : 0.f;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int c = 0; c < 16; ++c)
      if (c < C) {
        const float wc = __shfl_sync(0xffffffffu, w, c) * inv;
        a.x += wc * x[c].x; a.y += wc * x[c].y; a.z += wc * x[c].z; a.w += wc * x[c].w;
      }
    const size_t orow = out_row(p, b, kvh, r);
    *reinterpret_cast<uint2*>(p.out + orow * kHeadDim + 4 * lane) = make_uint2(pack_bf16(a.x, a.y), pack_bf16(a.z, a.w));
    if (lane == 0 && p.lse) p.lse[orow] = l > 0.f ? (M + log2f(l)) * kLn2 : kNegInf;
    if (p.mass) {
#pragma unroll
      for (int s = 0; s < UC_MAX_SEGMENTS; ++s) {
        if (s < p.nseg) {
          ls[s] *= w;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) ls[s] += __shfl_xor_sync(0xffffffffu, ls[s], o);
          if (lane == 0) p.mass[orow * p.nseg + s] = ls[s] * inv;
        }
      }
    }
  }
  __syncwarp();
  cluster_arrive();
  cluster_wait();  // no CTA leaves while another may still read its shared memory
}

template <int NTW, int ST, class W>
__device__ void consume(const W& w, AttnSmem& sm) {
  constexpr bool kMerges = NTW > 1 && W::kMany;  // else the merge kernel does
  const int warp = threadIdx.x >> 5;
  const int mtiles = w.call(0).mtiles;  // the same for every call of a launch
  const int NG = (mtiles + NTW - 1) / NTW <= 1 ? 1 : ((mtiles + NTW - 1) / NTW <= 2 ? 2 : 4);
  const int KS = kConsumers / NG;
  const int grp = warp % NG, ks = warp / NG;
  uint32_t seq = 0;
  bool aborted = false;
  // thread 0: the last arrival (call << 16 | bh), checked one item later
  int prev_key = -1, prev_arrivals = -1;
  if (kMerges && threadIdx.x == 0) sm.n_pending = 0;
  for (uint32_t iseq = 0;; ++iseq) {
    const int k = iseq % kItemQ;
    if (!mbar_wait(&sm.item_full[k], (iseq / kItemQ) & 1, w.call(0).status, 13, w.call(0).wait_ns)) break;
    const int pos = sm.item_pos[k];
    if (pos < 0) break;
    int it, local, c;
    const AttnParams& p = w.locate(pos, &local, &c);
    const ItemInfo ii = decode_item(p, local, &it);
    const SegDev& sd = p.seg[ii.s];
    if (seg_is_bf16(sd.kind) || ii.tail)
      run_item<NTW, ST, 16>(p, sm, ii, it, k, seq, aborted, NG, KS, grp, ks);
    else if (sd.bits == 4)
      run_item<NTW, ST, 4>(p, sm, ii, it, k, seq, aborted, NG, KS, grp, ks);
    else
      run_item<NTW, ST, 2>(p, sm, ii, it, k, seq, aborted, NG, KS, grp, ks);

    consumer_sync();  // the next item's query fragments take this one's place
    if constexpr (!kMerges) continue;
    // A batch: arrive on the item's counter; the CTA whose arrival completes a
    // (sequence, KV head) owes its merge, done after its last item so that
    // no warp waits for the atomic here.
    if (threadIdx.x == 0) {
      if (prev_key >= 0 && prev_arrivals == w.items_per_bh(prev_key >> 16) - 1)
        sm.pending[sm.n_pending++] = prev_key;
      prev_arrivals = counter_arrive_acq_rel(&p.counters[ii.bh]);
      prev_key = (c << 16) | ii.bh;
    }
    if (sm.n_pending == kMaxPendingMerges) {  // list full (not reached for planned grids): merge now
      consumer_sync();
      for (int k = 0; k < kMaxPendingMerges; ++k) {
        const AttnParams& pc = w.call(sm.pending[k] >> 16);
        const int bh = sm.pending[k] & 0xffff;
        final_merge<NTW, ST>(pc, sm, bh, nullptr);
        consumer_sync();
        if (threadIdx.x == 0) pc.counters[bh] = 0;
      }
      if (threadIdx.x == 0) sm.n_pending = 0;
      consumer_sync();
    }
  }
  if constexpr (!kMerges) return;
  if (threadIdx.x == 0) {
    if (prev_key >= 0 && prev_arrivals == w.items_per_bh(prev_key >> 16) - 1)
      sm.pending[sm.n_pending++] = prev_key;
  }
  consumer_sync();
  for (int k = 0; k < sm.n_pending; ++k) {
    const AttnParams& pc = w.call(sm.pending[k] >> 16);
    const int bh = sm.pending[k] & 0xffff;
    final_merge<NTW, ST>(pc, sm, bh, &seq);  // the producer has stopped: the ring is idle
    consumer_sync();
    if (threadIdx.x == 0) pc.counters[bh] = 0;
  }
}

template <int NTW, class P, bool CLUSTER = false, int ST = kStages>
__global__ void __launch_bounds__(kAttnThreads, ctas_for<NTW, ST>()) attend_kernel(const __grid_constant__ P params) {
  const typename WorkOf<P>::type w{params};
  extern __shared__ uint8_t dyn_smem[];
  AttnSmem& sm = *reinterpret_cast<AttnSmem*>(
      (reinterpret_cast<uintptr_t>(dyn_smem) + 1023) & ~static_cast<uintptr_t>(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Launched programmatically, this launch may begin while the kernel before
  // it is finishing: nothing below reads memory before that kernel (the
  // append of this call's layer) has completed, and the next launch may
  // begin as soon as this one runs.
  griddep_wait();
  griddep_launch_dependents();

  if (threadIdx.x == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], kConsumers);
    }
    for (int q = 0; q < kItemQ; ++q) {
      mbar_init(&sm.item_full[q], 1);
      mbar_init(&sm.item_empty[q], kConsumers);
    }
    fence_barrier_init();
  }
  __syncthreads();

  if (warp == kConsumers) {
    if (lane == 0) {
      for (int c = 0; c < w.n_calls(); ++c) {
        const AttnParams& p = w.call(c);
        for (int s = 0; s < p.nseg; ++s) {
          prefetch_tmap(&p.tmap[2 * s]);
          prefetch_tmap(&p.tmap[2 * s + 1]);
        }
      }
      produce<NTW, ST, CLUSTER>(w, sm);
    }
  } else {
    if constexpr (CLUSTER)
      consume_cluster(params, sm);
    else
      consume<NTW, ST>(w, sm);
  }
}

static void attend_setup_once() {
  static std::once_flag once;
  std::call_once(once, [] {
    const int one = (int)attend_smem_bytes(1), most = (int)attend_smem_bytes(8);
    cudaFuncSetAttribute(attend_kernel<1, AttnParams>, cudaFuncAttributeMaxDynamicSharedMemorySize, one);
    cudaFuncSetAttribute(attend_kernel<2, AttnParams>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    cudaFuncSetAttribute(attend_kernel<2, AttnParams, false, kMaxStages>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)attend_smem_bytes(8, kMaxStages));
    cudaFuncSetAttribute(attend_kernel<1, AttnParams, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, one);
    cudaFuncSetAttribute(attend_kernel<1, AttnParams, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaFuncSetAttribute(attend_kernel<1, MultiAttnParams>, cudaFuncAttributeMaxDynamicSharedMemorySize, one);
    cudaFuncSetAttribute(attend_kernel<2, MultiAttnParams>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  });
}

// Resident CTAs per SM of a call with `ntiles` n-tiles (1 .. 8).
int attend_ctas_per_sm(int ntiles) {
  static std::atomic<int> cached[9];
  int n = cached[ntiles].load(std::memory_order_relaxed);
  if (n == 0) {
    attend_setup_once();
    if (ntiles <= 1)
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, attend_kernel<1, AttnParams>, kAttnThreads,
                                                    attend_smem_bytes(1));
    else
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, attend_kernel<2, AttnParams>, kAttnThreads,
                                                    attend_smem_bytes(ntiles));
    n = n > 0 ? n : 1;
    cached[ntiles].store(n, std::memory_order_relaxed);
  }
  return n;
}

static cudaLaunchConfig_t cluster_config(int c, int grid, cudaStream_t st, cudaLaunchAttribute* attr) {
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)c;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = pdl_enabled() ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kAttnThreads);
  cfg.dynamicSmemBytes = attend_smem_bytes(1);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}

// Clusters of c CTAs this device runs at once (0: none).
int attend_clusters(int c) {
  static std::atomic<int> cached[kMaxClusterItems + 1];  // count + 1
  if (c < 1 || c > kMaxClusterItems) return 0;
  int n = cached[c].load(std::memory_order_relaxed) - 1;
  if (n < 0) {
    attend_setup_once();
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_config(c, c, nullptr, attr);
    if (cudaOccupancyMaxActiveClusters(&n, attend_kernel<1, AttnParams, true>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    cached[c].store(n + 1, std::memory_order_relaxed);
  }
  return n;
}

static MergeCall merge_of(const AttnParams& p) {
  MergeCall m;
  m.part = p.part;
  m.out = p.out;
  m.lse = p.lse;
  m.mass = p.mass;
  m.nseg = p.nseg;
  m.batch = p.batch;
  m.n_kv_heads = p.n_kv_heads;
  m.n_q_heads = p.n_q_heads;
  m.n_qtok = p.n_qtok;
  m.group = p.group;
  m.rows = p.rows;
  m.mtiles = p.mtiles;
  m.items_per_bh = p.items_per_bh;
  for (int s = 0; s < p.nseg; ++s) m.chunk_begin[s] = p.seg[s].chunk_begin;
  return m;
}

// The merge of `blocks` (pair, row block)s. Always launched programmatically:
// its CTAs take the SM slots the attention CTAs free and wait
// (griddepcontrol.wait) for that launch to complete, instead of a launch gap
// after it.
template <class P>
static void launch_merge(const P& p, int blocks, int width, cudaStream_t st) {
  if (width == 32)
    launch_maybe_pdl(true, merge_partials_kernel<32, P>, blocks * 4, 256, 0, st, p);
  else if (width == 64)
    launch_maybe_pdl(true, merge_partials_kernel<64, P>, blocks * 2, 256, 0, st, p);
  else
    launch_maybe_pdl(true, merge_partials_kernel<kHeadDim, P>, blocks, 256, 0, st, p);
  count_launch();
}

void launch_attend(const AttnParams& p, int grid, cudaStream_t st) {
  attend_setup_once();
  const bool pdl = pdl_enabled();
  if (p.cluster) {
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_config(p.cluster, p.cluster * p.batch * p.n_kv_heads, st, attr);
    cudaLaunchKernelEx(&cfg, attend_kernel<1, AttnParams, true>, p);
    count_launch();
    return;
  }
  const size_t smem = attend_smem_bytes(p.mtiles, p.stages);
  if (p.mtiles <= 1)
    launch_maybe_pdl(pdl, attend_kernel<1, AttnParams>, grid, kAttnThreads, smem, st, p);
  else if (p.stages == kMaxStages)
    launch_maybe_pdl(pdl, attend_kernel<2, AttnParams, false, kMaxStages>, grid, kAttnThreads, smem, st, p);
  else
    launch_maybe_pdl(pdl, attend_kernel<2, AttnParams>, grid, kAttnThreads, smem, st, p);
  count_launch();
  launch_merge(merge_of(p), p.batch * p.n_kv_heads * p.mtiles, p.merge_width, st);
}

void launch_attend_multi(const MultiAttnParams& m, int grid, cudaStream_t st) {
  attend_setup_once();
  const size_t smem = attend_smem_bytes(m.call[0].mtiles);
  if (m.call[0].mtiles > 1) {
    attend_kernel<2, MultiAttnParams><<<grid, kAttnThreads, smem, st>>>(m);
    count_launch();
    return;
  }
  attend_kernel<1, MultiAttnParams><<<grid, kAttnThreads, smem, st>>>(m);
  count_launch();
  MultiMerge mm;
  mm.n_calls = m.n_calls;
  int blocks = 0;
  for (int c = 0; c < m.n_calls; ++c) {
    mm.call[c] = merge_of(m.call[c]);
    blocks += m.call[c].batch * m.call[c].n_kv_heads;
  }
  launch_merge(mm, blocks, m.merge_width, st);
}

}  // namespace uc

// ------------------------------------------------------ no-allocation variant
//
// uc_attend_static: decode attention for callers that cannot hand the
// library a workspace. Its scratch (status word, work queue, partial
// outputs) is this file-scope device array, reserved on every GPU that loads
// the library for as long as the process lives.
namespace uc {

constexpr size_t kStaticScratchBytes = size_t(8) << 20;  // 8 MiB
static __device__ __align__(256) uint8_t g_attend_scratch[kStaticScratchBytes];

// Device address of g_attend_scratch on the current device. In host code the
// array's name is only a host-side handle, so the address is fetched once per
// device (with that device current) and cached.
constexpr int kMaxDevices = 64;  // devices whose scratch address is cached

static uint8_t* attend_static_scratch(uc_status* status) {
  static std::mutex mu;
  static uint8_t* addr[kMaxDevices] = {};
  int dev = -1, n_dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaGetDeviceCount(&n_dev) != cudaSuccess || dev < 0 ||
      dev >= n_dev || dev >= kMaxDevices) {
    set_error("uc_attend_static: no usable current CUDA device");
    *status = UC_ERR_CUDA;
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(mu);
  if (addr[dev] == nullptr) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_attend_scratch);
    if (e != cudaSuccess || p == nullptr) {
      set_error("uc_attend_static: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
      *status = UC_ERR_CUDA;
      return nullptr;
    }
    addr[dev] = static_cast<uint8_t*>(p);
  }
  return addr[dev];
}

}  // namespace uc

extern "C" uc_status uc_attend_static(const void* q, int32_t n_q_heads, int32_t n_qtok,
                                      const uc_segment* const* segs, int32_t n_seg, void* out, float* lse,
                                      float* mass, void* stream) {
  UC_TRACE();
  using namespace uc;
  // uc_attend's own argument checks come first: the same inputs give the
  // same statuses, and nothing below runs on a rejected call
  size_t need = 0;
  uc_status st = attend_precheck(q, n_q_heads, n_qtok, segs, n_seg, out, "uc_attend_static", &need);
  if (st != UC_OK) return st;
  uint8_t* scratch = attend_static_scratch(&st);
  if (scratch == nullptr) return st;
  if (need > kStaticScratchBytes) {
    set_error("uc_attend_static: this call needs %zu bytes of scratch, more than the %zu of its static "
              "array; use uc_attend with a caller workspace",
              need, kStaticScratchBytes);
    return UC_ERR_OOM;
  }
  // The array keeps the previous call's contents: clear the status word and
  // the work queue's counters (the first 256 bytes), which must start at zero.
  const size_t clear = 256;
  if (cudaMemsetAsync(scratch, 0, clear, reinterpret_cast<cudaStream_t>(stream)) != cudaSuccess) {
    set_error("uc_attend_static: clearing the scratch failed: %s", cudaGetErrorString(cudaGetLastError()));
    return UC_ERR_CUDA;
  }
  return uc_attend(q, n_q_heads, n_qtok, segs, n_seg, out, lse, mass, scratch, kStaticScratchBytes, stream);
}
