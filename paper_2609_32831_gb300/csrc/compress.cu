// Segment compression kernels (§3.4; App. E "Physical, type-aware KV
// storage" and "Batched GQA token selection") and the decode-time append.
//
//  topk            exact per-(sequence, KV head) top-k by radix select on
//                  order-preserving score keys, ties to the lower index,
//                  kept indices written in ascending order
//  gather_rows     compaction of the kept bf16 rows (eviction)
//  quantize_groups int4 / int2 group quantization of the kept sequence and
//                  its bf16 residual tail (n_kept mod 32 last kept tokens)
//  append_token    one decode token per sequence into a segment
#include <algorithm>

#include <cooperative_groups.h>

#include "internal.h"
#include "quant.cuh"

namespace cg = cooperative_groups;

namespace uc {

// ------------------------------------------------------------------ top-k

// Order-preserving key of an fp32 score (ascending key <=> ascending value),
// with -0.0 folded onto +0.0.
__device__ __forceinline__ uint32_t score_key(float f) {
  uint32_t u = __float_as_uint(f);
  if (f == 0.0f) u = 0u;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

constexpr int kTopkThreads = 1024;
constexpr int kTopkWarps = kTopkThreads / 32;
constexpr int kTopkRows = 16;      // 32-candidate rows of a warp kept in registers between the passes
constexpr int kTopkBins = 2048;    // radix digits of 11, 11 and 10 bits
constexpr int kTopkMaxCluster = 8;
// Candidates a CTA takes before the list is spread over a cluster: below, a
// cluster barrier per pass costs more than the shorter lists save.
constexpr int kTopkPerCta = 8192;

// Score of candidate i: scores[i], or scores[idx[i]] through the source's
// logical indices; an index outside the score array flags UC_ERR_RANGE and
// reads nothing.
__device__ __forceinline__ float candidate_score(const float* s, const int32_t* idx, int64_t limit, int i,
                                                 int* bad) {
  if (idx == nullptr) return s[i];
  const int32_t t = idx[i];
  if (t < 0 || t >= limit) {
    *bad = 1;
    return 0.f;
  }
  return s[t];
}

// Exact top-k of one (sequence, KV head) by a cluster of 1 .. 8 CTAs (chosen
// by launch_topk from the list's length). Every warp owns a contiguous run of
// 32-candidate rows whose keys it loads once (coalesced) and keeps in
// registers, so that the three radix passes, the count and the emission read
// no memory (rows past kTopkRows, beyond 131072 candidates per cluster of 8,
// are read again each time). Per pass: a shared-memory histogram, one cluster
// barrier, then every CTA sums the cluster's histograms through distributed
// shared memory and finds the digit with one block scan (each pass has a
// histogram of its own, so no second barrier is needed). Emission order:
// counts of (greater, equal) keys per warp, prefix over the warps and CTAs,
// then per row two ballots give every kept index its ascending place.
// What bounds it is the chain of barriers and the histogram's atomics. An
// eviction of 29492 to 5898 tokens and a re-eviction of those to 2949 (16
// pairs, gather and quantization included) took 161 us with the selection
// that read the scores again in each of five passes and searched its 256 bins
// with one thread (64.5 and 40 us of it), 99.5 us with this one.
__global__ void __launch_bounds__(kTopkThreads) topk_kernel(TopkArgs a) {
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int bh = blockIdx.x / C;
  const int b = bh / a.n_kv_heads;
  const int keep = a.keep[b];
  const float* s = a.scores + (int64_t)bh * a.scores_stride + a.scores_offset;
  int32_t* out = a.kept_idx + (int64_t)bh * a.cap;
  const int32_t* sidx = a.score_idx ? a.score_idx + (int64_t)bh * a.score_idx_stride : nullptr;
  const int r = min(a.n_recent, keep);
  const int n_old = a.src_n[b] - r;
  const int k_old = keep - r;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  __shared__ __align__(16) uint32_t hist[3][kTopkBins];
  __shared__ int warp_cnt[kTopkWarps][2];  // (greater, equal) keys of each warp; scan scratch before
  __shared__ int cta_cnt[2];
  __shared__ uint32_t sh_digit, sh_rem;
  __shared__ int sh_nan;

  if (k_old > 0) {  // the same for every CTA of the cluster (one sequence)
    for (int i = tid; i < 3 * kTopkBins; i += kTopkThreads) hist[0][i] = 0;
    if (tid == 0) sh_nan = 0;
    const int rows = (n_old + 31) / 32;
    const int per_warp = (rows + C * kTopkWarps - 1) / (C * kTopkWarps);
    const int row0 = (rank * kTopkWarps + warp) * per_warp;
    uint32_t keys[kTopkRows];
    int flag = 0;
#pragma unroll
    for (int e = 0; e < kTopkRows; ++e) {
      const int i = (row0 + e) * 32 + lane;
      keys[e] = 0u;
      if (e < per_warp && i < n_old) {
        int bad = 0;
        const float f = candidate_score(s, sidx, a.score_limit, i, &bad);
        if (bad)
          flag = 2;
        else if (isnan(f))
          flag = max(flag, 1);
        keys[e] = score_key(f);
      }
    }
    // body(key, valid, i) over the warp's rows, in index order; every lane
    // of the warp takes every row
    auto each_row = [&](auto&& body) {
#pragma unroll
      for (int e = 0; e < kTopkRows; ++e) {
        if (e < per_warp) {
          const int i = (row0 + e) * 32 + lane;
          body(keys[e], i < n_old, i);
        }
      }
      for (int e = kTopkRows; e < per_warp; ++e) {
        const int i = (row0 + e) * 32 + lane;
        uint32_t key = 0u;
        if (i < n_old) {
          int bad = 0;
          const float f = candidate_score(s, sidx, a.score_limit, i, &bad);
          if (bad)
            flag = 2;
          else if (isnan(f))
            flag = max(flag, 1);
          key = score_key(f);
        }
        body(key, i < n_old, i);
      }
    };
    __syncthreads();
    uint32_t prefix = 0, mask = 0, rem = (uint32_t)k_old;
    int nan = 0;
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
      const int shift = pass == 0 ? 21 : (pass == 1 ? 10 : 0);
      const uint32_t dmask = pass == 2 ? 1023u : 2047u;
      each_row([&](uint32_t key, bool valid, int) {
        if (valid && (key & mask) == prefix) atomicAdd(&hist[pass][(key >> shift) & dmask], 1u);
      });
      if (pass == 0 && flag) atomicMax(&sh_nan, flag);
      if (C > 1)
        cluster.sync();
      else
        __syncthreads();
      // thread t: bins 2047 - 2t and 2046 - 2t (descending keys), summed over the cluster
      uint32_t h1 = 0, h0 = 0;
      for (int q = 0; q < C; ++q) {
        const uint2 v = *reinterpret_cast<const uint2*>(
            (C > 1 ? cluster.map_shared_rank(&hist[pass][0], q) : &hist[pass][0]) + (kTopkBins - 2 - 2 * tid));
        h0 += v.x;
        h1 += v.y;
        if (pass == 0) nan = max(nan, C > 1 ? *cluster.map_shared_rank(&sh_nan, q) : sh_nan);
      }
      const uint32_t c = h1 + h0;
      uint32_t incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      if (lane == 31) warp_cnt[warp][0] = (int)incl;
      __syncthreads();
      uint32_t before = lane < warp ? (uint32_t)warp_cnt[lane][0] : 0u;
      before = __reduce_add_sync(0xffffffffu, before);
      const uint32_t excl = before + incl - c;
      if (excl < rem && rem <= excl + c) {
        const bool hi = rem <= excl + h1;
        sh_digit = (uint32_t)(kTopkBins - 1 - 2 * tid - (hi ? 0 : 1));
        sh_rem = rem - excl - (hi ? 0u : h1);
      }
      __syncthreads();
      prefix |= sh_digit << shift;
      mask |= dmask << shift;
      rem = sh_rem;
    }
    if (nan) {
      // the result is undefined, but later kernels of the call must still find
      // in-range row indices: keep rows 0 .. keep-1
      if (rank == 0) {
        for (int t = tid; t < keep; t += kTopkThreads) out[t] = t;
        if (bh % a.n_kv_heads == 0 && tid == 0) a.n_kept[b] = keep;
        if (tid == 0) set_status(a.status, UC_ERR_RANGE, nan);
      }
      if (C > 1) cluster.sync();  // no CTA leaves while another may still read its shared memory
      return;
    }
    const uint32_t thr = prefix;
    const int need_eq = (int)rem;
    int gt = 0, eq = 0;
    each_row([&](uint32_t key, bool valid, int) {
      gt += __popc(__ballot_sync(0xffffffffu, valid && key > thr));
      eq += __popc(__ballot_sync(0xffffffffu, valid && key == thr));
    });
    // (the last pass's barrier follows its reads of warp_cnt)
    if (lane == 0) {
      warp_cnt[warp][0] = gt;
      warp_cnt[warp][1] = eq;
    }
    __syncthreads();
    const int wg = warp_cnt[lane][0], we = warp_cnt[lane][1];
    int g_before = __reduce_add_sync(0xffffffffu, lane < warp ? wg : 0);
    int e_before = __reduce_add_sync(0xffffffffu, lane < warp ? we : 0);
    if (C > 1) {
      const int g_all = __reduce_add_sync(0xffffffffu, wg), e_all = __reduce_add_sync(0xffffffffu, we);
      if (tid == 0) {
        cta_cnt[0] = g_all;
        cta_cnt[1] = e_all;
      }
      cluster.sync();
      for (int q = 0; q < rank; ++q) {
        const int* cc = cluster.map_shared_rank(&cta_cnt[0], q);
        g_before += cc[0];
        e_before += cc[1];
      }
    }
    int pos = g_before + min(e_before, need_eq);
    int eq_rank0 = e_before;
    const unsigned below = (1u << lane) - 1u;
    each_row([&](uint32_t key, bool valid, int i) {
      const bool is_eq = valid && key == thr;
      const unsigned me = __ballot_sync(0xffffffffu, is_eq);
      const bool take = (valid && key > thr) || (is_eq && eq_rank0 + __popc(me & below) < need_eq);
      const unsigned mt = __ballot_sync(0xffffffffu, take);
      if (take) out[pos + __popc(mt & below)] = i;
      pos += __popc(mt);
      eq_rank0 += __popc(me);
    });
    if (C > 1) cluster.sync();  // no CTA leaves while another may still read its shared memory
  }
  if (rank == 0) {
    for (int t = tid; t < r; t += kTopkThreads) out[k_old + t] = n_old + t;
    if (bh % a.n_kv_heads == 0 && tid == 0) a.n_kept[b] = keep;
  }
}

// -------------------------------------------------- re-compression helpers

// One warp per (b, kvh, 32 kept tokens) of a packed segment: rebuild the K and
// V rows in bf16 (x = code * s + z, exact in fp32, rounded to nearest even);
// the residual tail rows are copied. Lane L handles channels 4L .. 4L + 3.
template <int BITS>
__global__ void dequant_rows_kernel(DequantArgs a) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int nbh = a.batch * a.n_kv_heads;
  if (warp >= nbh * a.max_groups) return;
  const int bh = warp / a.max_groups, g = warp % a.max_groups;
  const int b = bh / a.n_kv_heads;
  const int n = a.n_kept[b];
  const int ng = n / kGroup;
  if (g * kGroup >= n) return;
  __nv_bfloat16* ko = a.k_out + ((size_t)bh * a.cap + (size_t)g * kGroup) * kHeadDim;
  __nv_bfloat16* vo = a.v_out + ((size_t)bh * a.cap + (size_t)g * kGroup) * kHeadDim;
  if (g >= ng) {  // the tail block (n mod 32 rows)
    const __nv_bfloat16* kt = a.k_tail + (size_t)bh * kGroup * kHeadDim;
    const __nv_bfloat16* vt = a.v_tail + (size_t)bh * kGroup * kHeadDim;
    for (int t = 0; t < n - g * kGroup; ++t) {
      reinterpret_cast<uint2*>(ko + t * kHeadDim)[lane] = reinterpret_cast<const uint2*>(kt + t * kHeadDim)[lane];
      reinterpret_cast<uint2*>(vo + t * kHeadDim)[lane] = reinterpret_cast<const uint2*>(vt + t * kHeadDim)[lane];
    }
    return;
  }
  constexpr uint32_t mask = (1u << BITS) - 1u;
  const size_t blk = (size_t)bh * a.cap * kHeadDim * BITS / 8;
  const uint8_t* kc = a.k_codes + blk;
  const uint8_t* vc = a.v_codes + blk;
  const uint8_t* kp = a.k_params + (size_t)bh * (a.cap / kGroup) * 512 + (size_t)g * 512;
  const uint8_t* vp = a.v_params + (size_t)bh * a.cap * 16;
  for (int tg = 0; tg < kGroup; ++tg) {
    const int t = g * kGroup + tg;
    float kx[4], vx[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int c = 4 * lane + e;
      // key code (token tg of group g, channel c) in the fragment layout
      const int nt = tg >> 3, nn = tg & 7, i = c >> 4, cc = c & 15;
      const int j = (cc & 7) >> 1, sub = cc >> 3, ee = cc & 1;
      const int pr = BITS == 4 ? 2 * (i & 1) + sub : 2 * (i & 3) + sub;
      const int wq = BITS == 4 ? (i >> 1) : (i >> 2);
      const uint32_t w =
          *reinterpret_cast<const uint32_t*>(kc + ((size_t)(g * 4 + nt) * 32 + nn * 4 + j) * (BITS * 4) + 4 * wq);
      const uint32_t code = (w >> (BITS * pr + 16 * ee)) & mask;
      const __half* kpar = reinterpret_cast<const __half*>(kp + (i * 4 + j) * 16);
      kx[e] = __fmaf_rn((float)code, __half2float(kpar[sub * 2 + ee]), __half2float(kpar[4 + sub * 2 + ee]));
      // value code (token t, channel c): 16-token tile, lane (c % 8, token pair)
      const int t16 = t >> 4, tt = t & 15, m = c >> 3, gq = c & 7;
      const int vsub = tt >> 3, vj = (tt & 7) >> 1, ve = tt & 1;
      const int vpr = BITS == 4 ? 2 * (m & 1) + vsub : 2 * (m & 3) + vsub;
      const int vwq = BITS == 4 ? (m >> 1) : (m >> 2);
      const uint32_t vw =
          *reinterpret_cast<const uint32_t*>(vc + ((size_t)t16 * 32 + gq * 4 + vj) * (BITS * 8) + 4 * vwq);
      const uint32_t vcode = (vw >> (BITS * vpr + 16 * ve)) & mask;
      const __half* vpar = reinterpret_cast<const __half*>(vp + (size_t)t16 * 256 + ((c >> 5) * 4 + vj) * 16);
      vx[e] = __fmaf_rn((float)vcode, __half2float(vpar[vsub * 2 + ve]), __half2float(vpar[4 + vsub * 2 + ve]));
    }
    const uint2 kw = make_uint2(pack_bf16(kx[0], kx[1]), pack_bf16(kx[2], kx[3]));
    const uint2 vw2 = make_uint2(pack_bf16(vx[0], vx[1]), pack_bf16(vx[2], vx[3]));
    reinterpret_cast<uint2*>(ko + tg * kHeadDim)[lane] = kw;
    reinterpret_cast<uint2*>(vo + tg * kHeadDim)[lane] = vw2;
  }
}

// ----------------------------------------------------------------- gather

// Source row of kept token t of block bh; a re-compression's kept index moves
// on to the logical token of that row (every entry has one reader, the lane
// that also rewrites it), a segment that keeps every token gets its indices
// here (`identity`: row t is kept token t).
// With `write` false the entry stays as it is (no src_idx then).
__device__ __forceinline__ int32_t take_row(const GatherArgs& a, int bh, int t, bool write = true) {
  int32_t* e = a.kept_idx + (int64_t)bh * a.cap + t;
  const int32_t row = a.identity ? t : *e;
  if (a.src_idx != nullptr)
    *e = a.src_idx[(int64_t)bh * a.src_cap + row];
  else if (a.identity && write)
    *e = row;
  return row;
}

// Copy kept tokens t0 .. t0 + cnt - 1 (cnt <= 32) of block bh to the rows
// dst_row .. of k_dst / v_dst. Lane t holds token t0 + t's source row; two
// rows per step (16 lanes x 16 bytes each), eight rows' K and V in flight.
__device__ __forceinline__ void copy_rows(const GatherArgs& a, int bh, int t0, int cnt, int64_t dst_row) {
  const int lane = threadIdx.x & 31;
  const int32_t row = lane < cnt ? take_row(a, bh, t0 + lane) : 0;
  const int64_t src_base = (int64_t)bh * a.src_row_stride + a.src_row_offset;
  const int c = (lane & 15) * 8;
  for (int q0 = 0; q0 < cnt; q0 += 8) {
    uint4 kx[4], vx[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = q0 + 2 * u + (lane >> 4);
      const int64_t sr = (src_base + __shfl_sync(0xffffffffu, row, t & 31)) * kHeadDim + c;
      if (t < cnt) {
        kx[u] = *reinterpret_cast<const uint4*>(a.k_src + sr);
        vx[u] = *reinterpret_cast<const uint4*>(a.v_src + sr);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int t = q0 + 2 * u + (lane >> 4);
      if (t < cnt) {
        *reinterpret_cast<uint4*>(a.k_dst + (dst_row + t) * kHeadDim + c) = kx[u];
        *reinterpret_cast<uint4*>(a.v_dst + (dst_row + t) * kHeadDim + c) = vx[u];
      }
    }
  }
}

// One warp per (b, kvh, 32 kept tokens): copy the kept K and V rows into the
// compacted bf16 storage (rows_per_block = cap, offset 0).
__global__ void gather_rows_kernel(GatherArgs a) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int per_bh = a.max_chunks;
  const int bh = warp / per_bh;
  if (bh >= a.batch * a.n_kv_heads) return;
  const int t0 = (warp % per_bh) * 32;
  const int n = a.keep[bh / a.n_kv_heads];
  if (t0 >= n) return;
  copy_rows(a, bh, t0, min(32, n - t0), (int64_t)bh * a.dst_row_stride + a.dst_row_offset + t0);
}

// ---------------------------------------------------------- quantization

// Persistent: each warp takes the units gw, gw + W, ... (W warps in the grid),
// a unit being a group (32 kept tokens of a (b, kvh)), or its K or V rows
// (`apart`).
// A warp stages a unit's rows in shared memory with one bulk copy per row
// (rows gathered through the kept-index list, 272 bytes apart so that rows of
// the fragment-order reads fall in different banks). One buffer takes unit
// after unit; each warp waits for every copy, but 10 KB of shared memory per
// warp fits 21 warps per SM, which cover each other's waits (buffers of their
// own for K and V with each copy requested half a group ahead fit 12 and were
// 7 % slower). K and V apart halve the latency of calls with no more groups
// than warps (800 tokens, batch 1: 9.6 -> 6.2 us; 7400, batch 1: 10.4 -> 7.8)
// and the uneven last round of slightly longer ones (7400, batch 4: 24.0 ->
// 22.7); from kApartRounds groups per warp up the extra unit costs more (7400,
// batch 8: 39.3 together, 40.9 apart; 32K layer, batch 16: 271 and 280). A re-compression's warp takes
// both, since its kept indices are rewritten as they are read.
constexpr int kQuantWarps = 7;
constexpr int kQuantCtasPerSm = 3;
constexpr int kQuantRowBytes = 272;
constexpr int kApartRounds = 2;

struct QuantWarpSmem {
  alignas(16) uint8_t rows[32 * kQuantRowBytes];
  union {
    QuantStats st;
    QuantStats2 st2;
  };
  uint64_t bar;
};
constexpr size_t kQuantSmemBytes = kQuantWarps * sizeof(QuantWarpSmem);

template <int BITS, bool APART>
__global__ void __launch_bounds__(kQuantWarps * 32, kQuantCtasPerSm) quantize_groups_kernel(GatherArgs a) {
  extern __shared__ __align__(16) uint8_t quant_smem[];
  QuantWarpSmem& sm = reinterpret_cast<QuantWarpSmem*>(quant_smem)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const int n_warps = gridDim.x * kQuantWarps;
  const int per_bh = a.max_chunks;
  const int nbh = a.batch * a.n_kv_heads;
  const int total = (APART ? 2 : 1) * nbh * per_bh;      // apart: every group's K unit, then every V unit
  const int all = total + nbh;                           // then one residual tail per (b, kvh)
  // A work index w with its block ((b, kvh), the V units' after the K units')
  // and group (w < total), stepped by the grid's warps without dividing again.
  struct Work {
    int w, blk, g;
  };
  auto is_v = [&](const Work& k) { return APART && k.blk >= nbh; };
  auto bh_of = [&](const Work& k) { return is_v(k) ? k.blk - nbh : k.blk; };
  const int step_blk = n_warps / per_bh, step_g = n_warps % per_bh;
  auto stepped = [&](Work k) {
    k.w += n_warps;
    k.blk += step_blk;
    k.g += step_g;
    if (k.g >= per_bh) {
      k.g -= per_bh;
      ++k.blk;
    }
    return k;
  };
  // the first valid unit or tail at or after k (groups past a sequence's full
  // groups and empty tails are skipped)
  auto valid_from = [&](Work k) {
    for (; k.w < all; k = stepped(k))
      if (k.w < total ? k.g < a.keep[bh_of(k) / a.n_kv_heads] / kGroup
                      : a.keep[(k.w - total) / a.n_kv_heads] % kGroup != 0)
        break;
    return k;
  };
  if (a.identity && blockIdx.x == 0 && threadIdx.x < a.batch) a.n_kept[threadIdx.x] = a.keep[threadIdx.x];
  if (lane == 0) {
    mbar_init(&sm.bar, 1);
    fence_barrier_init();
  }
  __syncwarp();
  // kept index of this lane's row of unit k (loaded a unit ahead, so that the
  // request does not wait for it)
  auto row_index = [&](const Work& k) {
    return k.w < total ? take_row(a, bh_of(k), k.g * kGroup + lane, !is_v(k)) : 0;
  };
  // K (kv == 0) or V rows of unit k into the buffer
  auto request = [&](const Work& k, int kv, int32_t idx) {
    const int64_t row = (int64_t)bh_of(k) * a.src_row_stride + a.src_row_offset + idx;
    if (lane == 0) mbar_arrive_expect_tx(&sm.bar, kGroup * kHeadDim * 2);
    __syncwarp();
    if (k.w == a.withhold && kv == 0 && lane == 0) return;  // test hook: one K row is never copied
    bulk_load(sm.rows + lane * kQuantRowBytes, (kv ? a.v_src : a.k_src) + row * kHeadDim, kHeadDim * 2, &sm.bar);
  };
  auto row_of = [&](int t) { return reinterpret_cast<const __nv_bfloat16*>(sm.rows + t * kQuantRowBytes); };
  const int w0 = blockIdx.x * kQuantWarps + (threadIdx.x >> 5);
  Work k = valid_from(Work{w0, w0 / per_bh, w0 % per_bh});
  int32_t idx = row_index(k);
  if (k.w < total) request(k, is_v(k), idx);
  uint32_t ph = 0;  // phase of the next completion of the barrier
  bool failed = false;
  auto wait = [&](int where) {
    failed = !__all_sync(0xffffffffu, mbar_wait(&sm.bar, ph, a.status, where, a.wait_ns));
    if (!failed) ph ^= 1u;
    return !failed;
  };
  while (k.w < total) {
    const Work next = valid_from(stepped(k));
    const int32_t next_idx = row_index(next);
    const int bh = bh_of(k), g = k.g;
    QuantOut out;
    out.k_codes = a.k_codes + (size_t)bh * a.cap * kHeadDim * BITS / 8;
    out.k_params = a.k_params + (size_t)bh * (a.cap / kGroup) * 512;
    out.v_codes = a.v_codes + (size_t)bh * a.cap * kHeadDim * BITS / 8;
    out.v_params = a.v_params + (size_t)bh * a.cap * 16;
    bool ok = true, values = is_v(k);
    if (!wait(values ? 21 : 20)) break;
    if (!values) {
      if constexpr (BITS == 2)
        ok = quantize_keys2(sm.rows, kQuantRowBytes, g, out, sm.st2);
      else
        ok = quantize_keys<BITS>(row_of, g, out, sm.st);
      if constexpr (!APART) {  // every lane has read the K rows: the buffer takes the V rows
        request(k, 1, idx);
        if (!wait(21)) break;
        values = true;
      }
    }
    if (values && ok) {
      if constexpr (BITS == 2)
        ok = quantize_values2(sm.rows, kQuantRowBytes, g, out, sm.st2);
      else
        ok = quantize_values<BITS>(row_of, g, out, sm.st);
    }
    if (!ok && lane == 0) set_status(a.status, UC_ERR_RANGE, 2);
    if (next.w < total) request(next, is_v(next), next_idx);
    idx = next_idx;
    k = next;
  }
  if (failed) {
    // copies still in flight must land before the warp's shared memory is
    // released: wait for the barrier's pending phase (bounded again)
    mbar_wait(&sm.bar, ph, nullptr, 0, a.wait_ns);
    return;
  }
  // the residual tails: the last (n mod 32) kept tokens of a (b, kvh), copied
  // to its bf16 tail block of 32 rows
  for (; k.w < all; k = valid_from(stepped(k))) {
    const int bh = k.w - total;
    const int n = a.keep[bh / a.n_kv_heads];
    copy_rows(a, bh, n / kGroup * kGroup, n % kGroup, (int64_t)bh * kGroup);
  }
}

// ---------------------------------------------------------------- append

// One CTA per sequence, one warp per KV head.
template <int BITS>
__global__ void append_token_kernel(AppendArgs a) {
  // Launched programmatically, an append waits for nothing: it writes only
  // its own segment, which the launches it may overlap do not read (the
  // caller orders them so: uc_set_programmatic_launch).
  griddep_launch_dependents();
  const int b = blockIdx.x;
  const int j = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  __shared__ int sh_n;
  if (threadIdx.x == 0) sh_n = a.n_kept[b];
  __syncthreads();
  const int n = sh_n;
  if (n >= a.cap) {
    if (threadIdx.x == 0) set_status(a.status, UC_ERR_BUDGET, 3);
    return;
  }
  if (j < a.n_kv_heads) {
    const int bh = b * a.n_kv_heads + j;
    const __nv_bfloat16* kn = a.k_new + (int64_t)bh * kHeadDim;
    const __nv_bfloat16* vn = a.v_new + (int64_t)bh * kHeadDim;
    int64_t row;
    if (BITS == 16)
      row = (int64_t)bh * a.row_stride + a.row_offset + n;
    else
      row = (int64_t)bh * kGroup + (n % kGroup);
    reinterpret_cast<uint2*>(a.k + row * kHeadDim)[lane] = reinterpret_cast<const uint2*>(kn)[lane];
    reinterpret_cast<uint2*>(a.v + row * kHeadDim)[lane] = reinterpret_cast<const uint2*>(vn)[lane];
    if (a.kept_idx != nullptr && lane == 0)
      a.kept_idx[(int64_t)bh * a.cap + n] = a.position + (a.position_plus_count ? n : 0);
    if (BITS != 16 && (n % kGroup) == kGroup - 1) {
      __syncwarp();
      __threadfence_block();
      const __nv_bfloat16* kt = a.k + (int64_t)bh * kGroup * kHeadDim;
      const __nv_bfloat16* vt = a.v + (int64_t)bh * kGroup * kHeadDim;
      auto krow = [&](int t) { return kt + t * kHeadDim; };
      auto vrow = [&](int t) { return vt + t * kHeadDim; };
      __shared__ QuantStats smem[8];
      QuantOut out;
      out.k_codes = a.k_codes + (size_t)bh * a.cap * kHeadDim * (BITS > 0 ? BITS : 1) / 8;
      out.k_params = a.k_params + (size_t)bh * (a.cap / kGroup) * 512;
      out.v_codes = a.v_codes + (size_t)bh * a.cap * kHeadDim * (BITS > 0 ? BITS : 1) / 8;
      out.v_params = a.v_params + (size_t)bh * a.cap * 16;
      if (!quantize_group_warp<(BITS == 16 ? 4 : BITS)>(krow, vrow, n / kGroup, out, smem[j]))
        if (lane == 0) set_status(a.status, UC_ERR_RANGE, 4);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) a.n_kept[b] = n + 1;
}

// ---------------------------------------------------------------- launchers

static int compress_sms() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    sms = std::max(sms, 1);
  }
  return sms;
}

// CTAs per (sequence, KV head): one up to kTopkPerCta candidates, then as many
// (a power of two up to 8) as share the list at no fewer than that each and
// fit the GPU at one CTA per SM.
void launch_topk(const TopkArgs& a, int n_blocks, cudaStream_t st) {
  int max_src = 0;
  for (int b = 0; b < UC_MAX_BATCH; ++b) max_src = std::max(max_src, a.src_n[b]);
  int c = 1;
  while (c < kTopkMaxCluster && max_src > c * kTopkPerCta && n_blocks * c * 2 <= compress_sms()) c *= 2;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)c;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(n_blocks * c));
  cfg.blockDim = dim3(kTopkThreads);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, topk_kernel, a);
  count_launch();
}

void launch_dequant_rows(const DequantArgs& a, cudaStream_t st) {
  const int warps = a.batch * a.n_kv_heads * a.max_groups;
  if (a.bits == 4)
    dequant_rows_kernel<4><<<(warps + 3) / 4, 128, 0, st>>>(a);
  else
    dequant_rows_kernel<2><<<(warps + 3) / 4, 128, 0, st>>>(a);
  count_launch();
}

void launch_gather(const GatherArgs& a, cudaStream_t st) {
  const int warps = a.batch * a.n_kv_heads * a.max_chunks;
  gather_rows_kernel<<<(warps + 3) / 4, 128, 0, st>>>(a);
  count_launch();
}

template <int BITS, bool APART>
static void quantize(const GatherArgs& a, int blocks, cudaStream_t st) {
  static bool attr = false;
  if (!attr)
    attr = cudaFuncSetAttribute(quantize_groups_kernel<BITS, APART>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kQuantSmemBytes) == cudaSuccess;
  quantize_groups_kernel<BITS, APART><<<blocks, kQuantWarps * 32, kQuantSmemBytes, st>>>(a);
}

void launch_quantize(const GatherArgs& a, int bits, cudaStream_t st) {
  const int nbh = a.batch * a.n_kv_heads, slots = kQuantCtasPerSm * compress_sms();
  const bool apart =
      a.src_idx == nullptr && (int64_t)nbh * a.max_chunks < (int64_t)kApartRounds * kQuantWarps * slots;
  const int warps = nbh * ((apart ? 2 : 1) * a.max_chunks + 1);  // units and tails
  const int blocks = std::min((warps + kQuantWarps - 1) / kQuantWarps, slots);
  if (bits == 4)
    apart ? quantize<4, true>(a, blocks, st) : quantize<4, false>(a, blocks, st);
  else
    apart ? quantize<2, true>(a, blocks, st) : quantize<2, false>(a, blocks, st);
  count_launch();
}

void launch_append(const AppendArgs& a, int bits, cudaStream_t st) {
  const int threads = 32 * ((a.n_kv_heads + 0) > 8 ? 8 : a.n_kv_heads);
  const bool pdl = pdl_enabled();
  if (bits == 4)
    launch_maybe_pdl(pdl, append_token_kernel<4>, a.batch, threads, 0, st, a);
  else if (bits == 2)
    launch_maybe_pdl(pdl, append_token_kernel<2>, a.batch, threads, 0, st, a);
  else
    launch_maybe_pdl(pdl, append_token_kernel<16>, a.batch, threads, 0, st, a);
  count_launch();
}

}  // namespace uc
