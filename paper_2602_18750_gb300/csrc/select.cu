// select.cu -- per-sequence top-k selection (Sec. 3.1 top-alpha retention;
// Sec. 4.2: the global top-alpha after merging every score source).
//
// A row's scores are held on chip as 32-bit order-preserving keys, by one CTA
// of 1024 threads or by a thread-block cluster of C CTAs, each taking a
// contiguous share.  The k-th largest key is found by an MSD radix search with
// digits of 11, 11 and 10 bits that ends as soon as the crossing bin is taken
// whole.  The counts of the leading digit come from the score normalisation
// (SelectArgs::hist0) or are made while the keys are loaded; in a cluster
// every CTA then adds its non-empty bins to all CTAs' sums through distributed
// shared memory.  The keys of the crossing bin (typically 1 to 4 % of a row)
// are put into a list, which a cluster exchanges in one step together with
// the number of keys above the bin: every CTA writes its part into all the
// others, so that after one cluster barrier each holds the whole list, runs
// the remaining digits on its own copy and knows how many tokens the CTAs
// before it keep.  A crossing bin that does not fit the list (heavy ties) is
// searched by histograms over all keys, exchanged like the first one.
//
// Bound by latency on the few SMs that a row occupies: 4 bytes per token are
// read once, and the rest is a chain of block-wide steps.  The length and
// budget are read and the counts cleared before the dependency wait.  The keys
// are read in order (16-byte loads) into shared memory, from where every
// thread takes a run of consecutive ones and makes a bit mask of those above
// and those inside the crossing bin: after that only the few inside it are
// looked at again, and one scan of the threads' counts places the kept tokens.
// The last digits are usually found by ranking at most kFew listed keys
// directly.  What peers need is pushed to them instead of fetched.  Measured
// in the step after the scoring stage (one GPU, before: re-counting loops over
// all keys, fetched histograms): 1 row of 128K 10.9 -> 6.8 us, 4 rows of
// 16-32K 10.4 -> 5.5, 4 of 16K 11.1 -> 7.5, 3 of 12K with window and hits
// (raw scores) about 17 -> 11; alone 17.4 -> 9.4, 12.2 -> 7.4, 11.5 -> 7.6 and
// 10.3 -> 7.2.
//
// Ties at the boundary go to the lowest token index: with tau the k-th key
// and `need` the number of keys equal to tau that must be taken, a token is
// selected iff key > tau, or key == tau and fewer than `need` keys equal to
// tau precede it.  Threads own consecutive runs, so idx comes out in ascending
// order without a sort.
#include <cooperative_groups.h>

#include <algorithm>

#include "hill_internal.h"

namespace cg = cooperative_groups;

namespace hill {
namespace {

constexpr int T = 1024;            // threads
constexpr int kWarps = T / 32;
constexpr int kBins = 2048;
constexpr int kMaxCluster = 8;
constexpr int kPeerThreads = T / kMaxCluster;   // threads that write to one peer
constexpr int kKeysMax = 48128;    // keys per CTA that fit shared memory beside the rest
constexpr int kSelSmem = 225 * 1024;   // dynamic; 1.4 KB static beside it
constexpr int kChunk = 4608;         // keys per CTA that a row is spread to, SMs permitting
constexpr int kChunkMax = 16384;     // and at most, while the cluster can grow
constexpr int kAlone = 8192;       // ranked tokens up to which one CTA is faster than a cluster
// Listed keys that are ranked directly: 64 of them take as long as a histogram
// and its search, 200 take 1.5 us more (a row of 4000 keys with 5 % kept 4.7 us,
// with up to 256 ranked 5.6).
constexpr int kFew = 64;
constexpr int kListMax = 8192;     // crossing-bin keys of a row held by every CTA

// The bin in which the running count from the top bin down reaches `need`,
// what is still needed inside it, and its size.
struct Crossing {
  uint32_t bin, need, count;
};

__device__ __forceinline__ uint32_t warp_scan(uint32_t v) {   // inclusive
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// Called by all threads; two block-wide barriers.  The bins are taken from
// the top down (position p is bin kBins - 1 - p).  Every warp sums a slice of
// them; warp 0 finds the crossing slice and, two bins per lane, the bin.
__device__ __forceinline__ Crossing find_crossing(const uint32_t* counts, uint32_t need, uint32_t* wtot,
                                                  Crossing* found) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  static_assert(kBins == 2 * T, "two bins per thread");
  auto bins = [&](int w) {   // this lane's bins of slice w: .y the upper one
    return *reinterpret_cast<const uint2*>(counts + kBins - (w * 32 + lane + 1) * 2);
  };
  const uint2 b0 = bins(warp);
  const uint32_t mine = __reduce_add_sync(0xffffffffu, b0.x + b0.y);
  if (lane == 0) wtot[warp] = mine;
  __syncthreads();
  if (warp == 0) {
    const uint32_t t = wtot[lane];
    uint32_t inc = warp_scan(t);
    unsigned hit = __ballot_sync(0xffffffffu, inc >= need);
    const int ws = hit ? __ffs(hit) - 1 : kWarps - 1;
    const uint32_t cum = __shfl_sync(0xffffffffu, inc - t, ws);
    const uint2 c = bins(ws);
    inc = cum + warp_scan(c.x + c.y);
    hit = __ballot_sync(0xffffffffu, inc >= need);
    if (lane == (hit ? __ffs(hit) - 1 : 31)) {
      const uint32_t above = inc - c.x - c.y;   // keys above this lane's bins
      const bool low = above + c.y < need;
      *found = Crossing{(uint32_t)(kBins - 1 - (ws * 32 + lane) * 2 - (low ? 1 : 0)), need - above - (low ? c.y : 0u),
                        low ? c.x : c.y};
    }
  }
  __syncthreads();
  return *found;
}

// CL: a cluster of CTAs per row.  Mask: a bit per key of a thread.
template <bool CL, typename Mask>
__global__ void __launch_bounds__(T) hill_select_kernel(const SelectArgs a) {
  int C = 1, r = 0;
  cg::cluster_group cluster = cg::this_cluster();
  if (CL) {
    C = (int)cluster.num_blocks();
    r = (int)cluster.block_rank();
  }
  auto remote = [&](uint32_t* p, int c) -> uint32_t* { return CL ? cluster.map_shared_rank(p, c) : p; };
  // row = one key row; with per-KV-head selection a sequence has
  // rows_per_seq rows that share its length and budget
  const int row = blockIdx.y;
  const int b = row / a.rows_per_seq;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  extern __shared__ __align__(16) uint32_t sm[];
  uint32_t* sums = sm;                      // [3][kBins] counts of each digit over the row
  uint32_t* own = sums + 3 * kBins;         // CL: [kBins] this CTA's counts
  uint32_t* list = own + (CL ? kBins : 0);  // [C][lcap] keys of the crossing bin, by CTA
  uint4* keys = reinterpret_cast<uint4*>(list + a.list_words);   // this CTA's keys in quads (key_quad)
  __shared__ uint32_t wtot[kWarps];         // slice sums of a search
  __shared__ uint32_t wcnt[kWarps];         // kept tokens per warp
  __shared__ Crossing found;
  __shared__ uint32_t s_cnt[kMaxCluster];   // by CTA: (keys above the crossing bin) << 16 | keys in it
  __shared__ uint32_t s_tot[kMaxCluster];   // by CTA: (above tau) << 16 | (equal to tau)
  __shared__ uint32_t my_cnt, s_before, s_few;
  __shared__ __align__(16) uint32_t few[kFew];

  // Before the dependency wait: the length and budget (inputs of the call,
  // complete before the call: include/hill.h) and this CTA's own memory.
  int len = a.lens[b];
  int kk = a.k[b];
  for (int i = tid; i < (3 + (CL ? 1 : 0)) * kBins / 4; i += T)
    reinterpret_cast<uint4*>(sums)[i] = uint4{0u, 0u, 0u, 0u};
  if (tid == 0) my_cnt = s_before = s_few = 0u;
  if (tid < kFew) few[tid] = 0u;
  len = len < 0 ? 0 : (len > a.cap ? a.cap : len);
  // BKP temporal pinning (Sec. 4.2): the most recent tokens [older, len) are
  // kept outright; the ranking runs over [0, older)
  const int rec = a.recent > 0 ? a.recent : 0;
  const int rfull = rec < len ? rec : len;
  const int older = len - rfull;
  int win = rfull;
  kk = kk < 0 ? 0 : (kk > older ? older : kk);
  const bool over = win > a.max_k || kk > a.max_k - min(win, a.max_k);
  if (over) {
    win = min(win, a.max_k);           // the most recent max_k tokens of the window
    kk = min(kk, a.max_k - win);
  }
  const bool search = kk > 0 && kk < older;   // the same in every CTA of the row
  const float* row_key = a.key + (int64_t)row * a.cap;
  const int s0 = (int)((reinterpret_cast<uintptr_t>(row_key) >> 2) & 3u);
  // A short row of a large cache is searched by the cluster's first CTA alone,
  // without the exchanges.  4 rows in a cache of 16K, four CTAs each / alone
  // (us): 1000 tokens 6.4 / 4.6, 6000 6.7 / 5.7, 8000 6.9 / 6.0.
  const bool alone = CL && older + s0 <= a.alone_max;
  const bool multi = CL && !alone;   // the CTAs search together
  const int S = alone ? 1 : C, rs = alone ? 0 : r;   // the CTAs that search; this one among them
  const bool mine_to_search = search && (!alone || r == 0);
  const int lcap = alone ? C * a.lcap : a.lcap;
  if (multi) {
    if (search) cluster.barrier_arrive();   // A: every CTA has started and cleared its memory
  } else {
    __syncthreads();
  }
  // Shares of the ranked tokens: equal ones for the row's CTAs and for a
  // CTA's threads, cut where 16-byte loads may start.  With s0 the place of
  // the row's first key in its 16 bytes, token j is at place j + s0.  The
  // CTA's quads are read from global memory in order and kept in shared
  // memory, from where thread t takes the q quads t * q .. t * q + q - 1; a
  // spare quad in every eight keeps both sides free of bank conflicts.
  const int share = (((older + s0 + S - 1) / S) + 3) & ~3;
  const int nq = share / 4, q = (nq + T - 1) / T;
  const int jc = rs * share - s0;   // the CTA's first token (maybe negative: none there)
  const int hi = min(older, jc + share);
  auto key_quad = [&](int g) { return g + (g >> a.pad_shift); };
  const int j0 = jc + tid * q * 4;   // this thread's first token
  int32_t* out = a.idx + (int64_t)row * a.max_k;
  uint16_t* hits = a.hits ? a.hits + (int64_t)row * a.cap : nullptr;
  // the keys are being written: only their address translation is fetched
  if (mine_to_search && jc + 4 * tid < hi) prefetch_l2(row_key + max(jc + 4 * tid, 0));
  pdl_wait();
  pdl_launch_dependents();

  // The global reads are issued before the first use of any of them.  A key
  // of 0 means no token (a token's key is at least 1).
  uint4 h0v{0u, 0u, 0u, 0u};
  if (mine_to_search && a.hist0 && tid < kBins / 4) h0v = reinterpret_cast<const uint4*>(a.hist0 + (int64_t)row * kBins)[tid];
  // counts of the first digit: taken over, or made from the keys as they come
  uint32_t* h = multi ? own : sums;
  if (mine_to_search) {
    if (multi && !a.hist0) cluster.barrier_wait();   // A
    constexpr int kU = 4;   // quads in flight
    for (int g0 = tid; g0 < nq; g0 += kU * T) {
      float4 f[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int g = g0 + u * T, j = jc + 4 * g;
        f[u] = float4{0.f, 0.f, 0.f, 0.f};
        if (g >= nq) continue;
        if (j >= 0 && j + 3 < hi) {
          f[u] = *reinterpret_cast<const float4*>(row_key + j);
        } else {
          if (j >= 0 && j < hi) f[u].x = row_key[j];
          if (j + 1 >= 0 && j + 1 < hi) f[u].y = row_key[j + 1];
          if (j + 2 >= 0 && j + 2 < hi) f[u].z = row_key[j + 2];
          if (j + 3 >= 0 && j + 3 < hi) f[u].w = row_key[j + 3];
        }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int g = g0 + u * T, j = jc + 4 * g;
        if (g >= nq) continue;
        const float v[4] = {f[u].x, f[u].y, f[u].z, f[u].w};
        uint32_t k[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          k[e] = j + e >= 0 && j + e < hi ? max(ordered_key(v[e]), 1u) : 0u;
          if (!a.hist0 && k[e]) atomicAdd(&h[k[e] >> 21], 1u);
        }
        keys[key_quad(g)] = uint4{k[0], k[1], k[2], k[3]};
      }
    }
  }

  // padding, count and the pinned window (every path)
  if (over && r == 0 && tid == 0) raise_error(a.err, kErrDevArg);
  for (int p = kk + win + r * T + tid; p < a.max_k; p += C * T) out[p] = -1;
  if (r == 0 && tid == 0) a.count[row] = kk + win;
  auto hit = [&](int j) {   // the hit-rate table: +1 per kept token, saturating
    if (hits && hits[j] != 0xffffu) hits[j] = (uint16_t)(hits[j] + 1u);
  };
  for (int j = len - win + r * T + tid; j < len; j += C * T) {
    out[kk + j - (len - win)] = j;
    hit(j);
  }
  if (!search) {
    if (kk > 0)   // every older token is selected
      for (int j = r * T + tid; j < older; j += C * T) {
        out[j] = j;
        hit(j);
      }
    return;
  }
  if (!mine_to_search) return;

  // Add this CTA's non-empty bins to every CTA's sums, and clear them.
  auto push_counts = [&](uint32_t* sum) {
    for (int i = tid; i < kBins; i += T) {
      const uint32_t v = own[i];
      if (v) {
        own[i] = 0u;
        for (int c = 0; c < C; ++c) atomicAdd(remote(sum, c) + i, v);
      }
    }
  };
  if (a.hist0) {
    if (multi) cluster.barrier_wait();   // A
    if (tid < kBins / 4) reinterpret_cast<uint4*>(sums)[tid] = h0v;
  }
  __syncthreads();
  if (multi && !a.hist0) {
    push_counts(sums);
    cluster.sync();
  }
  Crossing x = find_crossing(sums, (uint32_t)kk, wtot, &found);
  uint32_t tau = x.bin << 21;             // the digits found so far
  uint32_t need = x.need;
  bool whole = x.need == x.count;         // the crossing bin is taken whole: keys >= tau are kept
  const bool whole0 = whole;
  // A bit per key of this thread: `gt` above the crossing bin (or in it, when
  // it is kept whole), `in` inside it.
  Mask gt = 0, in = 0;
  const int my_q = min(q, nq - tid * q);
  {
    const uint32_t lo = max(tau, 1u), top = tau + 0x1fffffu;
#pragma unroll 4
    for (int i = 0; i < my_q; ++i) {
      const uint4 v = keys[key_quad(tid * q + i)];
      const uint32_t k[4] = {v.x, v.y, v.z, v.w};
      uint32_t ge4 = 0, gt4 = 0;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        ge4 |= k[e] >= lo ? 1u << e : 0u;
        gt4 |= k[e] > top ? 1u << e : 0u;
      }
      in |= (Mask)ge4 << (4 * i);
      gt |= (Mask)gt4 << (4 * i);
    }
    if (whole) gt = in;
    in ^= gt;
  }
  auto pop = [](Mask m) { return (uint32_t)(sizeof(Mask) == 8 ? __popcll(m) : __popc((uint32_t)m)); };
  auto first = [](Mask m) { return (sizeof(Mask) == 8 ? __ffsll((long long)m) : __ffs((int)(uint32_t)m)) - 1; };
  auto key_of = [&](int i) {   // key i of this thread
    return reinterpret_cast<const uint32_t*>(keys + key_quad(tid * q + (i >> 2)))[i & 3];
  };
  if (multi || !whole) {
    // the crossing bin's keys into the list; (keys above) << 16 | (keys in it)
    const uint32_t cnt = (pop(gt) << 16) | pop(in);
    const uint32_t inc = warp_scan(cnt);
    uint32_t base = 0;
    if (lane == 31 && inc) base = atomicAdd(&my_cnt, inc);
    base = __shfl_sync(0xffffffffu, base, 31);
    uint32_t at = (base + inc - cnt) & 0xffffu;
    for (Mask m = in; m; m &= m - 1, ++at)
      if (at < (uint32_t)lcap) list[rs * lcap + at] = key_of(first(m));
    __syncthreads();
  }
  bool listed = !whole && (my_cnt & 0xffffu) <= (uint32_t)lcap;
  if (multi) {
    const uint32_t nc = my_cnt & 0xffffu;
    if (listed) {
      const int c = tid / kPeerThreads, i0 = tid % kPeerThreads;
      if (c < C && c != r) {
        const uint32_t* src = list + r * lcap;
        uint32_t* dst = remote(list + r * lcap, c);
        for (uint32_t i = i0; i < nc; i += kPeerThreads) dst[i] = src[i];
      }
    }
    if (tid < C) remote(s_cnt, tid)[r] = my_cnt;
    cluster.sync();   // every CTA's list and counts are in place
    listed = !whole;
    for (int c = 0; c < C; ++c) listed = listed && (s_cnt[c] & 0xffffu) <= (uint32_t)lcap;
  }
  // f(key, CTA) for every entry of the list: kWarps / S warps take a CTA's part
  auto each = [&](auto&& f) {
    const int per = kWarps / S, c = warp / per;
    const uint32_t nc = (multi ? s_cnt[c] : my_cnt) & 0xffffu;
    for (uint32_t i = (warp - c * per) * 32 + lane; i < nc; i += per * 32) f(list[c * lcap + i], c);
  };
  // the digits that follow, until the crossing bin is taken whole: from counts
  // of the keys that share those found, or, when few listed keys share them,
  // by ranking these
#pragma unroll 1
  for (int d = 1; d < 3 && !whole; ++d) {
    const uint32_t done = d == 1 ? 0xffe00000u : 0xfffffc00u;
    uint32_t* sum = sums + d * kBins;
    // (the third digit has 10 bits: every other bin)
    auto add = [&](uint32_t* to, uint32_t kv) {
      if ((kv & done) == tau) atomicAdd(&to[(d == 1 ? kv >> 10 : kv << 1) & (kBins - 1)], 1u);
    };
    if (listed && x.count <= kFew) {
      each([&](uint32_t kv, int) {
        if ((kv & done) == tau) few[atomicAdd(&s_few, 1u) & (kFew - 1)] = kv;
      });
      __syncthreads();
      if (tid < kFew && (uint32_t)tid < x.count) {
        const uint32_t kv = few[tid];
        uint32_t ng = 0, ge = 0;   // keys above this one; and not below it
        for (uint32_t i = 0; i < x.count; i += 4) {   // (0 past the end: below every key)
          const uint4 v = *reinterpret_cast<const uint4*>(few + i);
          ng += (v.x > kv ? 1u : 0u) + (v.y > kv ? 1u : 0u) + (v.z > kv ? 1u : 0u) + (v.w > kv ? 1u : 0u);
          ge += (v.x >= kv ? 1u : 0u) + (v.y >= kv ? 1u : 0u) + (v.z >= kv ? 1u : 0u) + (v.w >= kv ? 1u : 0u);
        }
        if (ng < need && need <= ge) found = Crossing{kv, need - ng, ge - ng};   // (equal keys write the same)
      }
      __syncthreads();
      tau = found.bin;
      need = found.need;
      whole = found.need == found.count;
      break;
    }
    if (listed) {
      each([&](uint32_t kv, int) { add(sum, kv); });
    } else {
      for (Mask m = in; m; m &= m - 1) add(multi ? own : sum, key_of(first(m)));
      if (multi) {
        __syncthreads();
        push_counts(sum);
        cluster.sync();
      }
    }
    __syncthreads();
    x = find_crossing(sum, need, wtot, &found);
    tau |= d == 1 ? x.bin << 10 : x.bin >> 1;
    need = x.need;
    whole = x.need == x.count;
  }

  // ---------------------------------------------------------------- compaction
  // Selection rule: whole -> key >= tau (tau > 0); otherwise tau is the k-th
  // key itself and `need` of the keys equal to tau are taken, lowest index
  // first.  Only the crossing bin's keys are looked at again.  Counts are
  // packed as (kept above) << 16 | (equal to tau): a CTA holds fewer than 2^16
  // keys.
  const uint32_t top = whole ? tau - 1u : tau;
  const uint32_t eq = whole ? 0u : tau;   // (no token's key is 0)
  Mask eqm = 0;
  for (Mask m = in; m; m &= m - 1) {
    const uint32_t kv = key_of(first(m));
    if (kv > top) gt |= m & (~m + 1);
    if (kv == eq) eqm |= m & (~m + 1);
  }
  const uint32_t mine = (pop(gt) << 16) | pop(eqm);
  const uint32_t inc = warp_scan(mine);
  if (lane == 31) wcnt[warp] = inc;
  if (multi && listed) {   // the crossing-bin keys that the CTAs before this one keep
    uint32_t v = 0;
    each([&](uint32_t kv, int c) {
      if (c < r) v += (kv > top ? 0x10000u : 0u) + (kv == eq ? 1u : 0u);
    });
    v = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0 && v) atomicAdd(&s_before, v);
  }
  __syncthreads();
  const uint32_t wt = lane < kWarps ? wcnt[lane] : 0u;
  const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? wt : 0u) + inc - mine;
  uint32_t pos = before >> 16, eq_rank = before & 0xffffu;
  if (multi) {
    if (listed || whole0) {
      pos += s_before >> 16;   // (0 when the first digit decided)
      eq_rank += s_before & 0xffffu;
      for (int c = 0; c < r; ++c) pos += s_cnt[c] >> 16;
    } else {
      const uint32_t total = __reduce_add_sync(0xffffffffu, wt);
      if (tid < C) remote(s_tot, tid)[r] = total;
      cluster.sync();
      for (int c = 0; c < r; ++c) {
        pos += s_tot[c] >> 16;
        eq_rank += s_tot[c] & 0xffffu;
      }
    }
  }
  pos += min(eq_rank, need);
  // drop the ties past the budget: the kept keys are then the bits of gt
  for (; eqm && eq_rank < need; ++eq_rank, eqm &= eqm - 1) gt |= eqm & (~eqm + 1);
  if (pos + pop(gt) > (uint32_t)kk) {
    raise_error(a.err, kErrDevArg);   // cannot happen: more picks than the budget
    return;
  }
  if (!hits) {
    for (; gt; gt &= gt - 1) out[pos++] = j0 + first(gt);
    return;
  }
  // with the hit table: four counts are read before any is written
  while (gt) {
    int j[4];
    uint32_t old[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      j[u] = gt ? j0 + first(gt) : -1;
      gt &= gt - 1;
      old[u] = j[u] >= 0 ? hits[j[u]] : 0u;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j[u] >= 0) {
        out[pos++] = j[u];
        if (old[u] != 0xffffu) hits[j[u]] = (uint16_t)(old[u] + 1u);
      }
  }
}

template <bool CL, typename Mask>
cudaError_t launch_select_t(const SelectArgs& a, int C, size_t smem, cudaStream_t st) {
  static int cache[64] = {0};
  auto kern = hill_select_kernel<CL, Mask>;
  cudaError_t e = ensure_smem_attr(reinterpret_cast<const void*>(kern), (int)smem, cache);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(C, a.B * a.rows_per_seq, 1), dim3(T), smem, st, CL ? C : 0, a);
}

}  // namespace

bool select_cap_ok(int cap) { return (cap + kMaxCluster - 1) / kMaxCluster <= kKeysMax; }

int select_hist_bins() { return kBins; }

cudaError_t launch_select(const SelectArgs& a0, int sms, cudaStream_t st) {
  SelectArgs a = a0;
  // CTAs per row: one up to kAlone keys; then more until a CTA has at most
  // kChunk keys, while twice as many still fit `sms`; else as few as hold
  // kChunkMax each.  Measured (us a selection after the scoring, one against four
  // or eight CTAs): 32K x 4 rows 9.8 / 7.4, 64K x 8 13.4 / 11.1, 16K x 4 8.0 / 7.6,
  // per-KV-head 16K x 16 rows -1.5 with 2 -> 4; alone, 16 rows of 8K 6.7 in one
  // CTA and 7.6 in two or four.
  const int rows = a.B * a.rows_per_seq;
  int C = 1;
  while (a.cap > kAlone && C < kMaxCluster && (a.cap + C - 1) / C > (2 * C * rows <= sms ? kChunk : kChunkMax)) C <<= 1;
  int share = (((a.cap + 3 + C - 1) / C) + 3) & ~3;   // of a CTA, at most (see the kernel)
  if (C > 1) share = std::max(share, kAlone);
  const int nq = share / 4, counts = (C > 1 ? 4 : 3) * kBins;
  // the spare quads, where they fit beside a list of full size
  a.pad_shift = (nq + nq / 8 + 1) * 4 + counts + kListMax <= kSelSmem / 4 ? 3 : 31;
  const int key_words = (nq + (nq >> a.pad_shift) + 1) * 4;
  a.lcap = std::min(kListMax, kSelSmem / 4 - counts - key_words) / C;
  a.list_words = (a.lcap * C + 3) & ~3;
  a.alone_max = kAlone;
  const size_t smem = (size_t)(counts + a.list_words + key_words) * 4;
  const bool m32 = nq <= 8 * T;   // at most 32 keys per thread
  if (C > 1) return m32 ? launch_select_t<true, uint32_t>(a, C, smem, st) : launch_select_t<true, uint64_t>(a, C, smem, st);
  return m32 ? launch_select_t<false, uint32_t>(a, C, smem, st) : launch_select_t<false, uint64_t>(a, C, smem, st);
}

}  // namespace hill
