// score.cu -- the K-cache streaming kernel (Eq. 1 over the whole cache) and
// the ATTN-mode normalisation (Sec. 4.1 column sum of softmax weights).
//
// hill_score_kernel: persistent CTAs of kNW warps.  A work item is a tile of
// kT = 32 consecutive tokens of one sequence; CTA x takes the contiguous
// range of items [x * per, (x + 1) * per), so it meets one or two sequences
// and loads their queries and flushes their partials once (measured faster
// than dealing items round robin, by 4 % at 32K and more for short
// sequences, where round robin changes sequence at every item).  Of a long
// 16-bit ATTN stream only the first 13/16 are dealt out so; the rest is
// claimed tile by tile by warps that are free (struct Units).  The KV
// heads g of an item are dealt to the warps (g mod kNW).  Every warp streams
// its own (item, g)
// sequence through a private ring of kSW shared-memory stages: lane 0 issues
// two tiled TMA loads (dims 0-63 and 64-127 of the tile's 32 key rows, 128-
// byte swizzle) completing on the stage's mbarrier.  The warp moves a landed tile into
// registers with ldmatrix (conflict-free thanks to the swizzle), hands the
// slot back to the copy engine for the stage kSW ahead, and computes the
// [32 tokens x 128] . [128 x G heads] product with 16 mma.sync m16n8k16
// (fp32 accumulation; the G query heads fill the N = 8 columns, so one
// instruction stream serves MHA and GQA alike).
//
//   RAW : the per-token sum over heads is reduced across the warps in shared
//         memory at the end of each item (fixed order) and written to scores
//         (and added to accum).
//   ATTN: every logit, pre-scaled by log2 e, is written to a [B][H][cap]
//         buffer; each lane keeps a running (max, sum 2^(z2 - max)) of its
//         own tokens per head in registers, and the lanes of a head are
//         combined once, when the CTA leaves a sequence or a claimed tile,
//         into one partial per (sequence, head, unit of work).
//         hill_attn_finalize_kernel combines the partials and forms s[b,j] =
//         sum_h exp(z[b,h,j] - m_bh) / L_bh; with many such CTAs or partials
//         hill_attn_stats_kernel first combines the partials once per
//         (sequence, head) (launch_attn_finalize).
//
// The query rows of a warp's heads are held as mma B fragments in registers
// for the whole sequence.  Before its dependency wait the kernel builds its
// tile table from the lengths and, with 16-bit keys, starts its first stages
// (inputs of the call only; every global write comes after the wait).
#include "hill_internal.h"

namespace hill {

namespace {

constexpr int kT = 32;                      // tokens per tile (= rows per stage)
constexpr int kNW = 8;                      // warps per CTA
constexpr int kThreads = kNW * 32;
constexpr int kMaxBatchSmem = 512;          // sequences held in the per-CTA tables
constexpr int kTableInts = kMaxBatchSmem + 4;  // B + 1 entries, padded (16-byte alignment)
constexpr int kMaxNg = 4;                   // KV heads per warp per item (Hkv <= kNW * kMaxNg)
constexpr int kBoxBytes = kT * 128;         // one 64-dim half of a tile: 32 swizzled 128-byte rows
constexpr int kKBytes = 2 * kBoxBytes;

constexpr int kShare16 = 13;   // sixteenths of the tiles dealt out in even shares when the rest is claimed
constexpr int kMinShare = 5;   // and the least tiles of such a share: more than a warp's first stages reach
constexpr int kFifo = 8;   // claimed tiles a warp can have in flight: at most kSW + 1

template <int G, bool F8>
struct ScoreCfg {
  // one K tile (a multiple of 1024): 8 KB of 16-bit keys, or 4 KB of E4M3 codes
  static constexpr int kSlotBytes = F8 ? kT * 128 : kKBytes;
  static constexpr int kSW = F8 ? 6 : 3;                   // stages per warp (same bytes in flight)
  static constexpr int kStages = kNW * kSW;
  // shared-memory layout (offsets from a 1024-byte aligned base)
  static constexpr int kOffScale = kStages * kSlotBytes;   // F8: the kT token scales of each stage
  static constexpr int kOffBar = kOffScale + (F8 ? kStages * kT * 4 : 0);
  static constexpr int kOffTab = kOffBar + kStages * 8;
  static constexpr int kOffRed = kOffTab + 2 * kTableInts * 4;
  static constexpr int kOffFlag = kOffRed + 2 * kNW * kT * 4;
  static constexpr int kOffIssued = kOffFlag + kNW * 4;       // warps that issued their last stage
  static constexpr int kOffFifo = kOffIssued + 16;            // [kNW][kFifo] claimed tiles in flight
  static constexpr int kBytes = kOffFifo + kNW * kFifo * 4 + 1024;   // + alignment slack
};

constexpr int kL2Ahead = 4;   // stages per warp brought into L2 before the dependency wait
// Registers per thread of the scoring kernel: at most 192, so that one CTA
// of 256 threads at 64 registers (the two-kernel normalisation's finalize)
// still fits beside it in the SM's 65536 registers and the layer-pipelined
// evaluation can run it during the next layer's K stream.
constexpr int kScoreMaxRegs = 192;

__device__ __forceinline__ int find_seq(const int* tstart, int B, int item) {
  int lo = 0, hi = B;  // tstart[lo] <= item < tstart[hi]
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (tstart[mid] <= item) lo = mid; else hi = mid;
  }
  return lo;
}

// The tiles (items) of all sequences as work units.  Even split: CTA x takes
// unit x, the items [x * per, (x + 1) * per).  With claims: unit x < grid is
// the first share of CTA x, and every item from dyn0 on is a unit of its own,
// claimed (per warp index, for that warp's heads) as warps become free.  A
// sequence's partial slots are its units in order, so what a slot holds does
// not depend on who claimed it.
//
// Why: SMs differ.  Those of a GPC with more SMs get less bandwidth each: per
// CTA an even share of 4 x 16-32K tokens (32 heads) took 112 us in the median,
// 120-127 on 40 of 152 SMs, and those alone do not fill HBM.  With 13/16 dealt
// out and the rest claimed tile by tile: the whole step on 4 x 16-32K tokens
// 178.8 -> 167.9 us, on 8 x 64K 887.9 -> 860.0 (11/16 and 12/16 the same within
// 1 %, 14/16 2 % slower).  Opening the counters and a flush of the statistics
// per claim cost 3-5 us, so short streams keep the even split: claim_min is the
// number of tiles from which the rest is claimed (0: never; claim_min_for in
// api.cu).  The tiles counted are those of the lengths at hand, not of the
// cache's capacity: hill_score on 8 x 1638 tokens in a cache for 8 x 32K takes
// 21.0 us with the even split and 26.1 with claims, on 4096 in one for 128K 9.3
// and 17.0.
struct Units {
  int per, dyn0, grid;   // items of a share; the first item claimed (INT_MAX: none, folded away in kernels without claims)
  __device__ __forceinline__ Units(int n_items, int grid_, int claim_min) {
    grid = grid_;
    const int share = n_items / 16 * kShare16 / grid;
    const bool claims = claim_min > 0 && n_items >= claim_min && share >= kMinShare;
    per = claims ? share : (n_items + grid - 1) / grid;
    dyn0 = claims ? grid * per : 0x7fffffff;
  }
  __device__ __forceinline__ int of(int item) const { return item < dyn0 ? item / per : grid + (item - dyn0); }
};

// The claim counters lie in the caller's workspace, whose contents are
// arbitrary before a call, and no kernel of the call runs before this one.  So
// the first warp that needs a counter opens it: a counter counts only under
// the tag of its launch (odd; the host draws 63 bits), which is put in place in
// two steps (tag - 1 while the count is being zeroed).  The normalisation, which
// runs when every claim is over, takes the tags away again whatever the
// lengths, so that a graph's next replay finds them closed.  A warp waits here
// only for another one that is between two stores; the wait is bounded.
__device__ __noinline__ void open_claims(ClaimCounter* c, unsigned long long tag, unsigned* err) {
  volatile unsigned long long* t = &c->tag;
  unsigned long long cur = *t;
  if (cur != tag && cur != tag - 1) {
    const unsigned long long seen = atomicCAS(&c->tag, cur, tag - 1);
    if (seen == cur) {
      *const_cast<volatile unsigned*>(&c->count) = 0u;
      __threadfence();
      *t = tag;
      return;
    }
  }
  const unsigned long long t0 = global_ns();
  while (*t != tag) {
    if (global_ns() - t0 > kWaitLimitNs) {
      raise_error(err, kErrTimeout);
      break;
    }
  }
  __threadfence();
}

__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Position of a warp in its own stage sequence: item (global tile index), r
// (its r-th KV head of that item, g = goff + warp + r * kNW) and b (the item's
// sequence, advanced incrementally).
struct Cursor {
  int item, r, b;
};

template <int DT, int G, bool RAW, bool F8, bool DEAL, bool CLAIM>
__global__ void __maxnreg__(kScoreMaxRegs) hill_score_kernel(const __grid_constant__ ScoreArgs a) {
  using Cfg = ScoreCfg<G, F8>;
  constexpr int kSlotBytes = Cfg::kSlotBytes;
  constexpr int kSW = Cfg::kSW;
  constexpr int kStages = Cfg::kStages;
  // accumulator columns that can hold a head of the group: 2*tig (+1 when G > 1)
  constexpr int kCols = G >= 2 ? 2 : 1;
  // heads of the group this launch handles (G itself unless G is 4 or 8 and
  // the group is 3, or 5 to 7 heads: the query rows past Gn are zero)
  const int Gn = G <= 2 ? G : a.Gn;

  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw_addr = smem_addr(smem_raw);
  const uint32_t base_addr = (raw_addr + 1023u) & ~1023u;
  unsigned char* base = smem_raw + (base_addr - raw_addr);
  int* tstart = reinterpret_cast<int*>(base + Cfg::kOffTab);          // [B+1] tile prefix
  int* slen = tstart + kTableInts;                                     // [B] clamped lengths
  float* red = reinterpret_cast<float*>(base + Cfg::kOffRed);          // [2][kNW][kT]
  volatile int* abort_flag = reinterpret_cast<int*>(base + Cfg::kOffFlag);   // [kNW]: one per warp group

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int B = a.B, H = a.H, Hkv = a.Hkv, cap = a.cap;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) mbar_init(base_addr + Cfg::kOffBar + s * 8, 1);
    fence_barrier_init();
    for (int w = 0; w < kNW; ++w) abort_flag[w] = 0;
    *reinterpret_cast<int*>(base + Cfg::kOffIssued) = 0;
    prefetch_tmap(&a.kmap);
  }
  // Before the dependency wait this kernel reads only the inputs of the call
  // (lengths, and with 16-bit keys the K cache itself), which the caller has
  // completed before the call (include/hill.h): it builds the tile table and
  // starts the first stages of every warp, so their DRAM latency overlaps the
  // end of the previous kernel.  Every write to global memory (the histogram
  // zeroing, logits, partials, scores) comes after the wait.  The E4M3 shadow
  // is written by hill_quantize_k, possibly the kernel just before, so with
  // F8 the first loads wait too.
  for (int b = threadIdx.x; b < B; b += kThreads) {
    int len = a.lens[b];
    if (len < 0 || len > cap) {
      raise_error(a.err, kErrDevArg);
      len = len < 0 ? 0 : cap;
    }
    slen[b] = len;
  }
  __syncthreads();
  // an item holds every KV head of one tile
  if (threadIdx.x == 0) {
    int acc = 0;
    tstart[0] = 0;
    for (int b = 0; b < B; ++b) {
      acc += (slen[b] + kT - 1) / kT;
      tstart[b + 1] = acc;
    }
  }
  __syncthreads();
  const int n_items = tstart[B];
  static_assert(!CLAIM || (!RAW && !DEAL && !F8), "tiles are claimed on the 16-bit ATTN stream");
  const Units units(n_items, gridDim.x, CLAIM ? a.claim_min : 0);
  const int per = units.per;
  const bool claims = CLAIM && units.dyn0 < n_items;   // (every CTA then has a share)
  const int it_lo = min(n_items, (int)blockIdx.x * per), it_hi = min(n_items, it_lo + per);   // this CTA's share
  // The warps' shares.  Without DEAL (W = 1) the KV heads are dealt to the
  // warps -- warp w takes g0 + r * kNW, r < ng (0 .. kMaxNg) -- and every warp
  // visits every item of the CTA.  With DEAL (launches of at most kNW / 2 KV
  // heads), W = kNW / nkv warps share each head and deal the items instead:
  // warp sub * nkv + i takes head goff + i of items it_lo + sub, + W, ...,
  // so that every warp streams (W * nkv < kNW leaves the rest idle).
  const int W = DEAL ? kNW / a.nkv : 1;
  const int sub = DEAL ? warp / a.nkv : 0;
  const int g0 = a.goff + (DEAL ? warp % a.nkv : warp);
  const int ng = DEAL ? (warp < W * a.nkv ? 1 : 0) : (a.nkv - warp + kNW - 1) / kNW;
  const int it0 = (DEAL && ng == 0) ? it_hi : it_lo + sub;   // this warp's first item
  // With DEAL a warp holds one KV head, and the query heads of its group in
  // up to kMaxNg sub-groups of 8 (a launch covers up to 32 heads per KV head):
  // each K tile is read once and scored for every sub-group, so groups larger
  // than 8 stream their keys once.  Fragment/statistics slot q of a warp is
  // its q-th KV head (no DEAL) or its q-th sub-group (DEAL).
  const int nsub = DEAL ? (a.Gn + 7) / 8 : 1;
  auto head0_of = [&](int q) {   // first query head of slot q
    return (DEAL ? g0 : g0 + q * kNW) * a.Gs + a.hoff + (DEAL ? 8 * q : 0);
  };
  auto gn_of = [&](int q) { return DEAL ? min(8, a.Gn - 8 * q) : Gn; };   // heads of slot q

  const uint64_t pol = l2_evict_first_policy();
  // the logits stay in L2 until the normalisation reads (and discards) them
  const uint64_t pol_keep = l2_evict_last_policy();
  const uint32_t stage0 = base_addr + warp * kSW * kSlotBytes;
  const uint32_t bar0 = base_addr + Cfg::kOffBar + warp * kSW * 8;
  const uint32_t scale0 = base_addr + Cfg::kOffScale + warp * kSW * kT * 4;   // F8 only
  const int b_first = it0 < it_hi ? find_seq(tstart, B, it0) : 0;

  auto advance = [&](Cursor& c) {
    if (++c.r >= ng) {
      c.r = 0;
      c.item += W;
      while (c.b < B - 1 && tstart[c.b + 1] <= c.item) ++c.b;
    }
  };
  // Past its share a warp claims single tiles for its heads from the counter
  // of its warp index (lane 0; the claim made one tile ahead, so that its
  // round trip is over when it is needed), and notes them for the consumer.
  int* fifo = reinterpret_cast<int*>(base + Cfg::kOffFifo) + warp * kFifo;
  unsigned claimed = 0, taken = 0;   // claims of the cursor, and of these taken by the consumer
  unsigned ahead = 0;                // lane 0: the claim made ahead
  auto claim_ahead = [&]() {
    if (lane == 0) ahead = atomicAdd(&a.claim[warp].count, 1u);
  };
  auto claim = [&](Cursor& c) {      // c.item = the next claimed tile, or n_items
    const unsigned u = __shfl_sync(0xffffffffu, ahead, 0);
    c.r = 0;
    if (u >= (unsigned)(n_items - units.dyn0)) {
      c.item = n_items;
      return;
    }
    c.item = units.dyn0 + (int)u;
    while (c.b < B - 1 && tstart[c.b + 1] <= c.item) ++c.b;
    if (lane == 0) fifo[claimed % kFifo] = c.item;
    ++claimed;
    claim_ahead();
  };
  // the cursor's next stage: of its item, its share or a claimed tile.  The
  // first claim is made ahead at the share's last tile, which the prologue's
  // kSW stages never reach (kMinShare).
  static_assert(kMinShare > kSW + 1 || !CLAIM, "a share is longer than the ring");
  const int it_end = claims ? n_items : it_hi;   // where the cursor ends
  auto next_stage = [&](Cursor& c) {
    if (!claims || c.r + 1 < ng || c.item + 1 < it_hi) {
      advance(c);
      if (claims && c.item + 1 == it_hi && c.r == 0) {
        if (lane == 0) open_claims(a.claim + warp, a.claim_tag, a.err);
        claim_ahead();
      }
    } else {
      claim(c);
    }
  };
  // lane 0: load the K tile of position c into slot s
  auto issue = [&](const Cursor& c, uint32_t s) {
    const int j0 = (c.item - tstart[c.b]) * kT;
    const int g = g0 + c.r * kNW;
    const uint32_t fb = bar0 + s * 8;
    const uint32_t dst = stage0 + s * kSlotBytes;
    // tensor-map coordinates: dimension 0 is d, the others are ordered by stride
    const int c1 = a.kdim_tok == 1 ? j0 : (a.kdim_head == 1 ? g : c.b);
    const int c2 = a.kdim_tok == 2 ? j0 : (a.kdim_head == 2 ? g : c.b);
    const int c3 = a.kdim_tok == 3 ? j0 : (a.kdim_head == 3 ? g : c.b);
    if constexpr (F8) {
      // 32 rows of 128 codes (one swizzled box) and the rows' 32 scales
      mbar_arrive_expect_tx(fb, (uint32_t)(kSlotBytes + kT * 4));
      tma_load_4d(dst, &a.kmap, 0, c1, c2, c3, fb, pol);
      bulk_g2s(scale0 + s * kT * 4, a.kscale + ((int64_t)c.b * Hkv + g) * a.cap32 + j0, kT * 4, fb, pol);
    } else {
      mbar_arrive_expect_tx(fb, (uint32_t)kKBytes);
      tma_load_4d(dst, &a.kmap, 0, c1, c2, c3, fb, pol);
      tma_load_4d(dst + kBoxBytes, &a.kmap, 64, c1, c2, c3, fb, pol);
    }
  };

  // prologue: the first kSW stages of this warp
  Cursor pc{it0, 0, b_first};
  uint32_t issued = 0, is_slot = 0;
  // with 16-bit keys, once every warp of the CTA has issued its last stage the
  // next kernel may launch (its CTAs take the SMs this grid's CTAs leave as
  // they drain); the E4M3 path, whose loads wait for the shadow's row of this
  // step, measured slower so and keeps the release at exit
  bool marked = F8;
  auto mark_if_done = [&]() {
    if (!marked && (ng == 0 || pc.item >= it_end)) {
      marked = true;
      if (lane == 0 && atomicAdd(reinterpret_cast<int*>(base + Cfg::kOffIssued), 1) == kNW - 1)
        pdl_launch_dependents();
    }
  };
  auto prologue = [&]() {
    if (ng > 0) {
      for (; issued < (uint32_t)kSW && pc.item < it_hi; ++issued) {
        if (lane == 0) issue(pc, is_slot);
        is_slot = is_slot + 1 == (uint32_t)kSW ? 0u : is_slot + 1;
        advance(pc);
      }
    }
  };
  if constexpr (!F8) {
    prologue();
    // and the next kL2Ahead stages into L2, so that the HBM stream keeps going
    // while the previous kernel finishes
    if (lane == 0 && ng > 0) {
      Cursor lc = pc;
      for (int u = 0; u < kL2Ahead && lc.item < it_hi; ++u) {
        const int j0 = (lc.item - tstart[lc.b]) * kT;
        const int g = g0 + lc.r * kNW;
        const int c1 = a.kdim_tok == 1 ? j0 : (a.kdim_head == 1 ? g : lc.b);
        const int c2 = a.kdim_tok == 2 ? j0 : (a.kdim_head == 2 ? g : lc.b);
        const int c3 = a.kdim_tok == 3 ? j0 : (a.kdim_head == 3 ? g : lc.b);
        tma_prefetch_l2_4d(&a.kmap, 0, c1, c2, c3);
        tma_prefetch_l2_4d(&a.kmap, 64, c1, c2, c3);
        advance(lc);
      }
    }
  }
  pdl_wait();
  // No trigger here: a dependent launches once every CTA has issued its last
  // stage (mark_if_done) or exited.  A trigger at the start would let the next
  // layer's scoring grid (the next launch in this stream) take the SMs this
  // grid leaves free for the normalisation and selection running beside it
  // on another stream; one at the last issued stage lets it start on the SMs
  // this grid's CTAs release as they drain.
  if (a.hist0) {   // this CTA's share of the leading-digit histogram, zeroed for the normalisation
    const int64_t hper = (a.hist0_words + gridDim.x - 1) / gridDim.x;
    const int64_t w0 = min((int64_t)blockIdx.x * hper, a.hist0_words);
    const int64_t w1 = min(w0 + hper, a.hist0_words);
    for (int64_t w = w0 + threadIdx.x; w < w1; w += kThreads) a.hist0[w] = 0u;
  }
  if (it_lo >= it_hi) return;
  if constexpr (F8) prologue();
  mark_if_done();

  // fragment coordinates (mma.sync m16n8k16): C row = token lane/4 (+8),
  // C columns = heads 2*(lane%4) and 2*(lane%4)+1 of the group
  const int grp = lane >> 2, tig = lane & 3;
  // ldmatrix row address pieces: matrix m = lane/8 covers rows (m&1)*8.., k half m>>1
  const int lm_row = (lane & 7) + ((lane >> 3) & 1) * 8;
  const int lm_khalf = lane >> 4;
  uint32_t used = 0, cs = 0, cph = 0;      // stages consumed; slot and phase of the next one
  int item_no = 0;
  bool ok = true;
  int cur_b = -1, cur_unit = -1, cur_slot = 0;

  // q of this warp's heads for the current sequence, as mma B fragments:
  // column grp is query head g*Gs + hoff + grp (zero for grp >= Gn), k = 16*kb + 2*tig (+8)
  // F8: the same rows cast to E4M3 with one scale per head, as m16n8k32 B
  // fragments (k = 32*kb + 4*tig .. +3, and +16), and the scales of this
  // lane's accumulator columns (heads 2*tig and 2*tig + 1)
  uint32_t bq[kMaxNg][F8 ? 4 : 8][2];
  float sqA[kMaxNg], sqB[kMaxNg];
  auto load_q = [&](int b) {
#pragma unroll
    for (int r = 0; r < kMaxNg; ++r) {
      const bool has = (DEAL ? (ng > 0 && r < nsub) : r < ng) && grp < gn_of(r);
      const int64_t row = has ? (int64_t)b * a.q_sb + (int64_t)(head0_of(r) + grp) * a.q_sh : 0;
      if constexpr (F8) {
        const auto* qh = static_cast<const uint16_t*>(a.q) + row;
        float v[4][8];
        float amax = 0.f;
#pragma unroll
        for (int kb = 0; kb < 4; ++kb) {
          uint2 lo{0u, 0u}, hi{0u, 0u};
          if (has) {
            lo = __ldg(reinterpret_cast<const uint2*>(qh + kb * 32 + 4 * tig));
            hi = __ldg(reinterpret_cast<const uint2*>(qh + kb * 32 + 16 + 4 * tig));
          }
          to_float8<DT>(uint4{lo.x, lo.y, hi.x, hi.y}, v[kb]);
#pragma unroll
          for (int i = 0; i < 8; ++i) amax = fmaxf(amax, fabsf(v[kb][i]));
        }
        amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
        amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 2));   // the head's 4 lanes hold all 128 dims
        const float rq = amax > 0.f ? __fdiv_rn(448.f, amax) : 0.f;
#pragma unroll
        for (int kb = 0; kb < 4; ++kb) {
          bq[r][kb][0] = e4m3x2(__fmul_rn(v[kb][0], rq), __fmul_rn(v[kb][1], rq)) |
                         (e4m3x2(__fmul_rn(v[kb][2], rq), __fmul_rn(v[kb][3], rq)) << 16);
          bq[r][kb][1] = e4m3x2(__fmul_rn(v[kb][4], rq), __fmul_rn(v[kb][5], rq)) |
                         (e4m3x2(__fmul_rn(v[kb][6], rq), __fmul_rn(v[kb][7], rq)) << 16);
        }
        const float sq = amax > 0.f ? __fdiv_rn(amax, 448.f) : 0.f;
        sqA[r] = __shfl_sync(0xffffffffu, sq, 8 * tig);
        sqB[r] = __shfl_sync(0xffffffffu, sq, 8 * tig + 4);
      } else {
        const auto* q32 = static_cast<const uint32_t*>(a.q);
#pragma unroll
        for (int kb = 0; kb < 8; ++kb) {
          bq[r][kb][0] = has ? __ldg(q32 + row / 2 + kb * 8 + tig) : 0u;
          bq[r][kb][1] = has ? __ldg(q32 + row / 2 + kb * 8 + 4 + tig) : 0u;
        }
        sqA[r] = sqB[r] = 1.f;
      }
    }
  };
  // ATTN: this lane's running (max, sum 2^(z2 - max)) over its own tokens of
  // the current sequence, per KV head r and column c (z2 = logit * log2 e);
  // lanes are combined only when the CTA leaves the sequence
  float st_m[kMaxNg][kCols], st_l[kMaxNg][kCols];
  auto reset_stat = [&]() {
#pragma unroll
    for (int r = 0; r < kMaxNg; ++r)
#pragma unroll
      for (int c = 0; c < kCols; ++c) {
        st_m[r][c] = kNegHuge;
        st_l[r][c] = 0.f;
      }
  };
  auto flush = [&]() {
#pragma unroll
    for (int r = 0; r < kMaxNg; ++r) {
      if (DEAL ? (ng == 0 || r >= nsub) : r >= ng) break;
#pragma unroll
      for (int c = 0; c < kCols; ++c) {
        float m = st_m[r][c], l = st_l[r][c];
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {   // the 8 lanes of one column
          const float mo = __shfl_xor_sync(0xffffffffu, m, o);
          const float lo = __shfl_xor_sync(0xffffffffu, l, o);
          const float mn = fmaxf(m, mo);
          l = l * ex2(m - mn) + lo * ex2(mo - mn);
          m = mn;
        }
        const int hl = 2 * tig + c;
        if (grp == 0 && hl < gn_of(r))
          a.partials[((int64_t)cur_b * H + head0_of(r) + hl) * a.nslot + cur_slot] = make_float2(m, l);
      }
    }
  };
  // ATTN with DEAL: a warp owns one partial slot in every sequence its CTA
  // meets, and writes a neutral one (-inf, 0) where it visited no tile of it
  // (the normalisation skips entries whose sum is 0).  b_next: the first
  // sequence of the CTA this warp has not written yet.
  const int b_cta_last = it_lo < it_hi ? find_seq(tstart, B, it_hi - 1) : -1;
  int b_next = it_lo < it_hi ? find_seq(tstart, B, it_lo) : 0;
  auto neutral_until = [&](int b_end) {   // sequences [b_next, b_end)
    if constexpr (!RAW && DEAL) {
      if (ng == 0) return;
      for (; b_next < b_end; ++b_next) {
        if (tstart[b_next + 1] == tstart[b_next]) continue;   // empty: no slots
        const int slot = ((int)blockIdx.x - tstart[b_next] / per) * W + sub;
#pragma unroll
        for (int q = 0; q < kMaxNg; ++q) {
          if (q >= nsub) break;
#pragma unroll
          for (int c = 0; c < kCols; ++c) {
            const int hl = 2 * tig + c;
            if (grp == 0 && hl < gn_of(q))
              a.partials[((int64_t)b_next * H + head0_of(q) + hl) * a.nslot + slot] = make_float2(-INFINITY, 0.f);
          }
        }
      }
    }
  };

  for (int own = it0, b = b_first;; own += W, ++item_no) {
    int item = own;
    if (own >= it_hi) {   // the share is done: the claimed tiles, in order
      if constexpr (!CLAIM) break;
      if (taken == claimed) break;
      __syncwarp();
      item = fifo[taken++ % kFifo];
    }
    while (b < B - 1 && tstart[b + 1] <= item) ++b;
    const int tile = item - tstart[b];
    const int j0 = tile * kT;
    const int nv = min(kT, slen[b] - j0);
    float rs[4] = {0.f, 0.f, 0.f, 0.f};   // RAW: token sums of rows grp, grp+8, 16+grp, 24+grp

    const int unit = own < it_hi ? (int)blockIdx.x : units.of(item);
    if (b != cur_b || (CLAIM && unit != cur_unit)) {
      if (!RAW && cur_b >= 0) flush();
      neutral_until(b);
      b_next = b + 1;
      if (b != cur_b) load_q(b);
      if (!RAW) reset_stat();
      cur_b = b;
      cur_unit = unit;
      // this warp's partial slot in b: the unit's rank among the units that
      // meet b, times W, plus the warp's item share
      cur_slot = (unit - units.of(tstart[b])) * W + sub;
    }

    constexpr int kStagesPerItem = DEAL ? 1 : kMaxNg;   // (at most; ng of them)
#pragma unroll
    for (int r = 0; r < kStagesPerItem; ++r) {
      if (r >= ng || !ok) break;
      const int g = DEAL ? g0 : g0 + r * kNW;
      // every lane waits; the warp goes on only if all of them saw the phase
      // complete, so it takes the same path and its shuffles stay converged
      if (!__all_sync(0xffffffffu, mbar_wait(bar0 + cs * 8, cph, a.err))) {
        ok = false;
        abort_flag[sub] = 1;
        break;
      }
      const uint32_t sb = stage0 + cs * kSlotBytes;
      // K tile -> A fragments: 16-bit keys, 2 blocks of 16 tokens x 8 blocks
      // of 16 dims; E4M3 codes, 2 blocks of 16 tokens x 4 blocks of 32 dims
      constexpr int kKB = F8 ? 4 : 8;
      uint32_t af[2][kKB][4];
#pragma unroll
      for (int mb = 0; mb < 2; ++mb) {
        const int t = mb * 16 + lm_row;
#pragma unroll
        for (int kb = 0; kb < kKB; ++kb) {
          const int chunk = kb * 2 + lm_khalf;   // 16-byte chunk of the row
          const uint32_t addr = F8 ? sb + t * 128 + ((chunk ^ (t & 7)) << 4)
                                   : sb + (chunk >> 3) * kBoxBytes + t * 128 + (((chunk & 7) ^ (t & 7)) << 4);
          ldmatrix_x4(addr, af[mb][kb]);
        }
      }
      // F8: the scales of this lane's token rows mb*16 + grp (+8)
      float ksc[4] = {1.f, 1.f, 1.f, 1.f};
      if constexpr (F8) {
        const uint32_t sc = scale0 + cs * kT * 4;
#pragma unroll
        for (int u = 0; u < 4; ++u)
          ksc[u] = __uint_as_float(lds32(sc + ((u >> 1) * 16 + grp + (u & 1) * 8) * 4));
      }
      ++used;
      cph ^= (cs + 1 == (uint32_t)kSW) ? 1u : 0u;
      const uint32_t freed = cs;
      cs = cs + 1 == (uint32_t)kSW ? 0u : cs + 1;
      __syncwarp();
      if (pc.item < it_end) {   // the slot just read takes the stage kSW ahead
        if (lane == 0) {
          fence_proxy_async_smem();
          issue(pc, freed);
        }
        ++issued;
        next_stage(pc);
        mark_if_done();
      }

      // the tile is scored for each fragment slot q: this stage's KV head
      // (no DEAL), or every query sub-group of the warp's KV head (DEAL)
      constexpr int kSlotsPerStage = DEAL ? kMaxNg : 1;
#pragma unroll
      for (int qs = 0; qs < kSlotsPerStage; ++qs) {
      if (DEAL && qs >= nsub) break;
      const int q = DEAL ? qs : r;
      const int hq0 = head0_of(q);    // first query head of the slot
      const int gnq = gn_of(q);       // its heads
      float acc[2][4];
#pragma unroll
      for (int mb = 0; mb < 2; ++mb)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[mb][e] = 0.f;
#pragma unroll
      for (int kb = 0; kb < kKB; ++kb)
#pragma unroll
        for (int mb = 0; mb < 2; ++mb) {
          if constexpr (F8) mma_16832_e4m3(acc[mb], af[mb][kb], bq[q][kb][0], bq[q][kb][1]);
          else mma_16816<DT>(acc[mb], af[mb][kb], bq[q][kb][0], bq[q][kb][1]);
        }
      if constexpr (F8) {   // back to the key and query scales
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          acc[u >> 1][(u & 1) * 2] *= sqA[q] * ksc[u];
          acc[u >> 1][(u & 1) * 2 + 1] *= sqB[q] * ksc[u];
        }
      }

      // acc[mb][c] = token mb*16 + grp, column 2*tig + c; acc[mb][2 + c] = token
      // mb*16 + grp + 8.  Columns >= Gn are zero (their q fragments are zero).
      if constexpr (RAW) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int mb = u >> 1, e = (u & 1) * 2;
          float v = acc[mb][e];
          if constexpr (G >= 2) v += acc[mb][e + 1];
          if constexpr (G >= 4) v += __shfl_xor_sync(0xffffffffu, v, 1);
          if constexpr (G >= 8) v += __shfl_xor_sync(0xffffffffu, v, 2);
          // complete in the tig == 0 lanes
          if (a.kvh) {   // per-KV-head importance: this group's sum is the score of (b, g)
            const int t = mb * 16 + grp + (u & 1) * 8;
            if (tig == 0 && t < nv) {
              const int64_t o = ((int64_t)b * Hkv + g) * cap + j0 + t;
              const float val = v * kInvSqrtD;
              // later sub-groups of the same KV head add to the first one's sum
              if (a.scores) a.scores[o] = (a.raw_add || qs > 0) ? a.scores[o] + val : val;
              if (a.accum) a.accum[o] += val;
            }
          } else {
            rs[u] += v;
          }
        }
      } else {
        float* lg = a.logits + ((int64_t)b * H + hq0) * a.lstride + j0;
#pragma unroll
        for (int c = 0; c < kCols; ++c) {
          const int hl = 2 * tig + c;
          float z[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int mb = u >> 1, e = (u & 1) * 2 + c;
            const int t = mb * 16 + grp + (u & 1) * 8;
            z[u] = t < nv ? acc[mb][e] * kLog2eInvSqrtD : -INFINITY;
            if (t < nv && hl < gnq) st_global_hint(lg + (int64_t)hl * a.lstride + t, z[u], pol_keep);
          }
          const float mn = fmaxf(st_m[q][c], fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3])));
          st_l[q][c] = st_l[q][c] * ex2(st_m[q][c] - mn) +
                       ((ex2(z[0] - mn) + ex2(z[1] - mn)) + (ex2(z[2] - mn) + ex2(z[3] - mn)));
          st_m[q][c] = mn;
        }
      }
      }   // fragment slots
    }
    if (RAW && !a.kvh) {
      // sum over the warps holding the item's heads -- all kNW (W = 1), or
      // the nkv warps of group sub -- in a fixed order, double-buffered by
      // item; a warp whose wait timed out still reaches its group's barrier
      // after raising the group's flag, and the group then leaves together
      const int wg0 = DEAL ? sub * a.nkv : 0, gw = DEAL ? a.nkv : kNW;
      float* rb = red + (item_no & 1) * kNW * kT;
      if (tig == 0) {
#pragma unroll
        for (int u = 0; u < 4; ++u) rb[warp * kT + (u >> 1) * 16 + grp + (u & 1) * 8] = rs[u];
      }
      named_sync(1 + sub, gw * 32);
      if (abort_flag[sub]) break;
      if (warp == wg0 + item_no % gw && lane < nv) {
        float sum = 0.f;
        for (int w = 0; w < gw; ++w) sum += rb[(wg0 + w) * kT + lane];
        sum *= kInvSqrtD;
        const int64_t o = (int64_t)b * cap + j0 + lane;
        if (a.scores) a.scores[o] = a.raw_add ? a.scores[o] + sum : sum;
        if (a.accum) a.accum[o] += sum;
      }
    } else if (!ok) {
      break;
    }
  }
  if (!RAW && cur_b >= 0 && ok) flush();
  if (ok) neutral_until(b_cta_last + 1);
  // after a timeout: give every copy this warp issued and did not consume one
  // more bounded wait before the CTA's shared memory is released
  if (!ok && lane == 0) {
    for (uint32_t u = used; u < issued; ++u) mbar_wait(bar0 + (u % kSW) * 8, (u / kSW) & 1u, a.err);
  }
}

// Combine the per-CTA (max, sum) partials of every head of sequence b, then
// s[b,j] = sum_h 2^(z2[b,h,j] - m_h) / L_h, one token per thread (logits and
// partials are in the base-2 scale z2 = z * log2 e, so each term is the
// softmax weight e^(z - m) / sum e^(z - m)).  All loads are issued before any
// is used: the logits of kFinZ heads of the thread's token (just written and
// mostly L2 resident), its running importance, and the partials, one head per
// warp at a time with a partial per lane.
//
// Bound by latency (and on long caches by the L2 reads of the logits): between
// the loads and the store there must be no chain over the heads.  The weights
// (max, 1/sum) are padded to a multiple of 8 heads whose terms are 0, so that
// the heads are taken 8 at a time without a branch between them; with a
// branch per head the 32 terms took 3600-3900 cycles per CTA, which is more
// than everything else in it (now about 500).  With the partials laid out by
// head and the heads taken without branches, scores to selection went from
// 10.4 to 7.1 us on one 4K sequence and from 14.5 to 7.8 on 4 x 16K of one KV
// head.
constexpr int kFinThreads = 256;                   // threads (= tokens) of a CTA
constexpr int kFinHB = 4;                          // heads of a warp whose partials are combined together
constexpr int kFinU = 5;                           // partials per lane and head held in registers at a time
constexpr int kHistBins = 2048;                    // leading 11 bits of the order-preserving key
constexpr int kFinZ = 32;                          // logits per token held in registers
constexpr int kFinMaxTpt = 16;                     // token blocks per CTA at most (split step)

__device__ __forceinline__ int pad8(int h) { return (h + 7) & ~7; }

// The (max, 1/sum) of every head of sequence b from its ns per-CTA partials:
// a warp takes kFinHB of its heads at a time, kFinU partials per lane and head in
// flight (one KV head has up to 8 partials per scoring CTA: hill_score on 4096
// tokens of 32 query heads 11.8 us; with one partial per lane at a time past the
// first kFinU 39.8).
__device__ __forceinline__ void combine_partials(const FinalizeArgs& a, int b, int ns, float2* wt) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int NW = kFinThreads / 32, HB = kFinHB;
  const float2* pb = a.partials + (int64_t)b * a.H * a.nslot;
  for (int h0 = warp; h0 < a.H; h0 += NW * HB) {
    float m[HB], l[HB];
#pragma unroll
    for (int i = 0; i < HB; ++i) m[i] = -INFINITY, l[i] = 0.f;
    // 32 * kFinU slots of each head at a time, all loads in flight
    for (int s0 = 0; s0 < ns; s0 += 32 * kFinU) {
      float2 p[HB][kFinU];
#pragma unroll
      for (int i = 0; i < HB; ++i)
#pragma unroll
        for (int u = 0; u < kFinU; ++u) {
          const int h = h0 + NW * i, s = s0 + lane + 32 * u;
          p[i][u] = h < a.H && s < ns ? pb[(int64_t)h * a.nslot + s] : make_float2(-INFINITY, 0.f);
        }
#pragma unroll
      for (int i = 0; i < HB; ++i) {
        float mn = m[i];
#pragma unroll
        for (int u = 0; u < kFinU; ++u) mn = fmaxf(mn, p[i][u].x);
        l[i] = l[i] > 0.f ? l[i] * ex2(m[i] - mn) : 0.f;
#pragma unroll
        for (int u = 0; u < kFinU; ++u) l[i] += p[i][u].y > 0.f ? p[i][u].y * ex2(p[i][u].x - mn) : 0.f;
        m[i] = mn;
      }
    }
    float mw[HB];
#pragma unroll
    for (int i = 0; i < HB; ++i) mw[i] = warp_max(m[i]);
#pragma unroll
    for (int i = 0; i < HB; ++i) l[i] = warp_sum(l[i] > 0.f ? l[i] * ex2(m[i] - mw[i]) : 0.f);
#pragma unroll
    for (int i = 0; i < HB; ++i)
      if (lane == 0 && h0 + NW * i < a.H) wt[h0 + NW * i] = make_float2(mw[i], 1.f / l[i]);
  }
}

// STATS: the per-head (max, 1/sum) come from hill_attn_stats_kernel instead of
// every CTA combining the partials itself.  KG: 0: per-sequence importance;
// else per-KV-head importance (a.kvh) for groups of 1, 2 or 4 query heads, of
// any multiple of 8 (KG = 8), or of any size (KG = -1).  Known group sizes
// leave no branch between the heads: with one after each head the sums of 32
// heads in groups of 4 took 2.5 us per CTA (step on 2 x 16K tokens, 8 KV
// heads: 35.2 -> 34.4 us without).
template <bool STATS, int KG>
__global__ void __launch_bounds__(kFinThreads, STATS ? 4 : 2) hill_attn_finalize_kernel(const FinalizeArgs a) {
  constexpr bool KVH = KG != 0;
  extern __shared__ __align__(16) float fsm[];
  const int hp = pad8(a.H);
  float2* wt = reinterpret_cast<float2*>(fsm);                     // [hp] (max, 1/sum)
  uint32_t* hcount = reinterpret_cast<uint32_t*>(fsm + 2 * hp);    // [kHistBins] when a.hist0
  // The lengths are inputs of the call: this kernel only ever follows the
  // scoring kernel of the same call, whose own dependency wait covered every
  // earlier write, so they are read before this kernel's wait and overlap
  // the end of the scoring kernel.  Everything the scoring kernel writes
  // (logits, partials) is read after the wait.
  const int b = blockIdx.y;
  int len = a.lens[b];
  len = len < 0 ? 0 : (len > a.cap ? a.cap : len);
  // this CTA's tokens: a.tpt blocks of kFinThreads from jb
  const int jb = blockIdx.x * kFinThreads * a.tpt;
  // CTA (0, 0) closes the claim counters whatever its sequence's length, and
  // always waits: so this grid never completes before the ones ahead of it,
  // and a later call's claims never meet this call's closing
  auto close_claims = [&]() {
    if (a.claim && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < kNW) a.claim[threadIdx.x].tag = 0ull;
  };
  if (jb >= len) {
    if (blockIdx.x == 0 && blockIdx.y == 0) {
      pdl_wait();
      close_claims();
    }
    return;
  }
  // the scoring CTAs that met b wrote slots 0 .. ns-1
  // (every thread counts the tiles of a share of the sequences)
  __shared__ int s_first, s_total;
  if (threadIdx.x == 0) s_first = s_total = 0;
  if (threadIdx.x < hp - a.H) wt[a.H + threadIdx.x] = make_float2(-kNegHuge, 0.f);   // 0 * 2^(z - huge) = 0
  if (a.hist0)
    for (int i = threadIdx.x; i < kHistBins; i += kFinThreads) hcount[i] = 0u;
  __syncthreads();
  {
    int f = 0, t = 0;
    for (int bb = threadIdx.x; bb < a.B; bb += kFinThreads) {
      int lb = a.lens[bb];
      lb = lb < 0 ? 0 : (lb > a.cap ? a.cap : lb);
      const int tiles = (lb + kT - 1) / kT;
      f += bb < b ? tiles : 0;
      t += tiles;
    }
    if (f) atomicAdd(&s_first, f);
    if (t) atomicAdd(&s_total, t);
  }
  __syncthreads();
  const int first_item = s_first;
  const Units units(s_total, a.score_grid, a.claim_min);
  const int items = (len + kT - 1) / kT;
  const int ns = (units.of(first_item + items - 1) - units.of(first_item) + 1) * a.spc;
  pdl_wait();
  pdl_launch_dependents();
  close_claims();
  // This token's logits of heads [h0, h0 + kFinZ), 8 at a time (those past H
  // repeat the last head, with weight 0).  Threads past the length read the
  // last token's and write nothing.
  int j = jb + threadIdx.x;
  const float* zb = a.logits + (int64_t)b * a.H * a.lstride;
  float zr[kFinZ];
  auto load_z = [&](int h0) {
    const float* zp = zb + min(j, len - 1);
#pragma unroll
    for (int u0 = 0; u0 < kFinZ; u0 += 8)
      if (h0 + u0 < a.H) {
#pragma unroll
        for (int u = u0; u < u0 + 8; ++u) zr[u] = zp[(int64_t)min(h0 + u, a.H - 1) * a.lstride];
      }
  };
  float acc = 0.f;   // the running importance of this token
  auto load_acc = [&]() {
    if (!KVH && a.accum) acc = a.accum[(int64_t)b * a.cap + min(j, len - 1)];
  };
  load_z(0);
  load_acc();
  if constexpr (STATS) {
    for (int h = threadIdx.x; h < a.H; h += kFinThreads) wt[h] = a.stats[(int64_t)b * a.H + h];
  } else {
    combine_partials(a, b, ns, wt);
  }
  __syncthreads();
  for (int blk = 0;;) {   // the CTA's token blocks (one unless a.tpt > 1)
    const bool valid = j < len;
    float s = 0.f;
    int g = 0, in_g = 0;   // KVH: the group being summed and its heads so far
    const int G = KVH ? a.H / a.Hkv : 1;
    for (int h0 = 0;;) {
#pragma unroll
      for (int u0 = 0; u0 < kFinZ; u0 += 8)
        if (h0 + u0 < a.H) {
          float t[8], w[8];
#pragma unroll
          for (int u = 0; u < 8; u += 2) {
            const float4 x = *reinterpret_cast<const float4*>(wt + h0 + u0 + u);   // two heads
            t[u] = ex2(zr[u0 + u] - x.x), w[u] = x.y;
            t[u + 1] = ex2(zr[u0 + u + 1] - x.z), w[u + 1] = x.w;
          }
          if constexpr (KVH) {
            // the sum over each group of G query heads, stored as soon as the
            // group is complete (heads of a group are adjacent)
            auto put = [&]() {
              if (valid) {
                const int64_t o = ((int64_t)b * a.Hkv + g) * a.cap + j;
                if (a.scores) a.scores[o] = s;
                if (a.accum) a.accum[o] += s;
              }
              ++g;
              s = 0.f;
            };
            if constexpr (KG == 1 || KG == 2 || KG == 4) {
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                s = __fmaf_rn(t[u], w[u], s);
                // (Hkv ends the groups where H is no multiple of 8)
                if ((u + 1) % KG == 0 && g < a.Hkv) put();
              }
            } else if constexpr (KG == 8) {
#pragma unroll
              for (int u = 0; u < 8; ++u) s = __fmaf_rn(t[u], w[u], s);
              if ((in_g += 8) == G) {
                put();
                in_g = 0;
              }
            } else {
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                s = __fmaf_rn(t[u], w[u], s);
                if (++in_g == G && h0 + u0 + u < a.H) {
                  put();
                  in_g = 0;
                }
              }
            }
          } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) s = __fmaf_rn(t[u], w[u], s);
          }
        }
      h0 += kFinZ;
      if (h0 >= a.H) break;
      load_z(h0);
    }
    if (!KVH && valid) {
      const int64_t o = (int64_t)b * a.cap + j;
      if (a.scores) a.scores[o] = s;
      float key = s;
      if (a.accum) {
        key = acc + s;
        a.accum[o] = key;
      }
      if (a.hist0 && j < len - min(a.recent, len)) atomicAdd(&hcount[ordered_key(key) >> 21], 1u);
    }
    // The logits are dead once read: drop this warp's lines from L2 without
    // writing them back (each 128-byte line holds the warp's 32 tokens of one
    // head; every lane has consumed its loads before the warp passes the sync).
    // A warp wholly past the length has read the last token's lines, which
    // belong to another warp.
    const int jw = j - (int)(threadIdx.x & 31);
    __syncwarp();
    if (jw < len)
      for (int h = threadIdx.x & 31; h < a.H; h += 32) l2_discard_line(zb + (int64_t)h * a.lstride + jw);
    // the next block of tokens
    if (++blk >= a.tpt || jb + blk * kFinThreads >= len) break;
    j = jb + blk * kFinThreads + threadIdx.x;
    load_z(0);
    load_acc();
  }
  if (a.hist0) {
    __syncthreads();
    uint32_t* hg = a.hist0 + (int64_t)b * kHistBins;
    for (int i = threadIdx.x; i < kHistBins; i += kFinThreads) {
      const uint32_t v = hcount[i];
      if (v) atomicAdd(hg + i, v);
    }
  }
}

// Combine the per-unit (max, sum) partials of one (b, h) into its softmax
// statistics (max, 1 / sum) in the base-2 scale: W warps per pair, each lane
// taking every 32 W-th partial, kStatsPer at a time under their common maximum
// (a running one per partial scales the sum more often: scores of 4 x 16K tokens
// on one KV head were 2.68e-7 from 64 bits by it, 2.60e-7 now), the lanes then
// merged by shuffles and the warps in shared memory.  Used ahead of
// hill_attn_finalize_kernel<true, *> where launch_attn_finalize says; W > 1 when
// tiles were claimed, which leaves a partial per tile.
constexpr int kStatsWarps = 8;
constexpr int kStatsPer = 8;   // partials per lane whose loads are in flight together

template <int W>
__global__ void __launch_bounds__(kStatsWarps * 32) hill_attn_stats_kernel(FinalizeArgs a) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ float2 s_part[kStatsWarps];
  const int pair = (blockIdx.x * kStatsWarps + warp) / W, sub = warp % W;
  const bool live = pair < a.B * a.H;
  const int b = live ? pair / a.H : 0;
  // the slots 0 .. ns-1 of b (lengths are inputs of the call: read before the wait)
  int f = 0, t = 0;
  for (int bb = lane; bb < a.B; bb += 32) {
    int lb = a.lens[bb];
    lb = lb < 0 ? 0 : (lb > a.cap ? a.cap : lb);
    const int tiles = (lb + kT - 1) / kT;
    f += bb < b ? tiles : 0;
    t += tiles;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    f += __shfl_xor_sync(0xffffffffu, f, o);
    t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  int len = a.lens[b];
  len = len < 0 ? 0 : (len > a.cap ? a.cap : len);
  const int items = (len + kT - 1) / kT;
  const Units units(t, a.score_grid, a.claim_min);
  const int ns = items == 0 || !live ? 0 : (units.of(f + items - 1) - units.of(f) + 1) * a.spc;
  pdl_wait();
  pdl_launch_dependents();
  const float2* pb = a.partials + (int64_t)pair * a.nslot;
  float m = -INFINITY, l = 0.f;
  for (int s0 = sub * 32 + lane; s0 < ns; s0 += 32 * W * kStatsPer) {
    float2 p[kStatsPer];
#pragma unroll
    for (int u = 0; u < kStatsPer; ++u) {
      const int s = s0 + 32 * W * u;
      p[u] = s < ns ? pb[s] : make_float2(-INFINITY, 0.f);
    }
    float mn = m;   // (their maximum first, so that every term is scaled once)
#pragma unroll
    for (int u = 0; u < kStatsPer; ++u) mn = fmaxf(mn, p[u].x);
    l = l > 0.f ? l * ex2(m - mn) : 0.f;
#pragma unroll
    for (int u = 0; u < kStatsPer; ++u) l += p[u].y > 0.f ? p[u].y * ex2(p[u].x - mn) : 0.f;
    m = mn;
  }
  auto merge = [&](float mo, float lo) {
    const float mn = fmaxf(m, mo);
    l = (l > 0.f ? l * ex2(m - mn) : 0.f) + (lo > 0.f ? lo * ex2(mo - mn) : 0.f);
    m = mn;
  };
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float mo = __shfl_xor_sync(0xffffffffu, m, o), lo = __shfl_xor_sync(0xffffffffu, l, o);
    merge(mo, lo);
  }
  if constexpr (W > 1) {
    if (lane == 0) s_part[warp] = make_float2(m, l);
    __syncthreads();
    if (sub == 0)
      for (int w = 1; w < W; ++w) merge(s_part[warp + w].x, s_part[warp + w].y);
  }
  if (live && sub == 0 && lane == 0) a.stats[pair] = make_float2(m, 1.f / l);
}

template <int DT, int G, bool RAW, bool F8, bool DEAL, bool CLAIM = false>
cudaError_t launch_score_t(const ScoreArgs& a, int grid, cudaStream_t st) {
  const size_t smem = (size_t)ScoreCfg<G, F8>::kBytes;
  auto kern = hill_score_kernel<DT, G, RAW, F8, DEAL, CLAIM>;
  static int cache[64] = {0};
  cudaError_t e = ensure_smem_attr(reinterpret_cast<const void*>(kern), (int)smem, cache);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(grid), dim3(kThreads), smem, st, 0, a);
}

template <int DT, bool RAW, bool F8>
cudaError_t launch_score_g(const ScoreArgs& a, int G, bool deal, int grid, cudaStream_t st) {
  if (deal) return G == 8 ? launch_score_t<DT, 8, RAW, F8, true>(a, grid, st) : cudaErrorInvalidValue;
  if constexpr (!RAW && !F8) {
    if (a.claim) {
      switch (G) {
        case 1: return launch_score_t<DT, 1, RAW, F8, false, true>(a, grid, st);
        case 2: return launch_score_t<DT, 2, RAW, F8, false, true>(a, grid, st);
        case 4: return launch_score_t<DT, 4, RAW, F8, false, true>(a, grid, st);
        case 8: return launch_score_t<DT, 8, RAW, F8, false, true>(a, grid, st);
      }
      return cudaErrorInvalidValue;
    }
  }
  switch (G) {
    case 1: return launch_score_t<DT, 1, RAW, F8, false>(a, grid, st);
    case 2: return launch_score_t<DT, 2, RAW, F8, false>(a, grid, st);
    case 4: return launch_score_t<DT, 4, RAW, F8, false>(a, grid, st);
    case 8: return launch_score_t<DT, 8, RAW, F8, false>(a, grid, st);
  }
  return cudaErrorInvalidValue;
}

template <int DT, bool F8>
cudaError_t launch_score_m(const ScoreArgs& a, int G, bool raw, bool deal, int grid, cudaStream_t st) {
  return raw ? launch_score_g<DT, true, F8>(a, G, deal, grid, st)
             : launch_score_g<DT, false, F8>(a, G, deal, grid, st);
}

}  // namespace

size_t score_smem_bytes(int G, bool f8) {
  switch (G) {
    case 1: return f8 ? ScoreCfg<1, true>::kBytes : ScoreCfg<1, false>::kBytes;
    case 2: return f8 ? ScoreCfg<2, true>::kBytes : ScoreCfg<2, false>::kBytes;
    case 4: return f8 ? ScoreCfg<4, true>::kBytes : ScoreCfg<4, false>::kBytes;
    default: return f8 ? ScoreCfg<8, true>::kBytes : ScoreCfg<8, false>::kBytes;
  }
}

int64_t score_claim_slots(int64_t n_items, int grid) { return 2 * (int64_t)grid + n_items * 3 / 16 + 32; }
int score_tile_tokens() { return kT; }
int score_warps() { return kNW; }
int score_max_batch() { return kMaxBatchSmem; }
int score_max_kv_heads() { return kMaxNg * kNW; }
int score_deal_warps(int nkv, int G) { return nkv <= kNW / 2 && G >= 5 ? kNW / nkv : 1; }

cudaError_t launch_score(const ScoreArgs& a, int dtype, int G, bool raw, bool f8, bool deal, int grid,
                         cudaStream_t st) {
  if (dtype == 0)
    return f8 ? launch_score_m<0, true>(a, G, raw, deal, grid, st) : launch_score_m<0, false>(a, G, raw, deal, grid, st);
  return f8 ? launch_score_m<1, true>(a, G, raw, deal, grid, st) : launch_score_m<1, false>(a, G, raw, deal, grid, st);
}

template <bool STATS>
static cudaError_t launch_finalize_t(const FinalizeArgs& a, cudaStream_t st) {
  const dim3 grid((a.cap + kFinThreads * a.tpt - 1) / (kFinThreads * a.tpt), a.B);
  const size_t smem = (size_t)((a.H + 7) & ~7) * sizeof(float2) + (a.hist0 ? kHistBins * sizeof(uint32_t) : 0);
  auto launch = [&](auto kern) { return launch_pdl(kern, grid, dim3(kFinThreads), smem, st, 0, a); };
  if (!a.kvh) return launch(hill_attn_finalize_kernel<STATS, 0>);
  switch (a.H / a.Hkv) {
    case 1: return launch(hill_attn_finalize_kernel<STATS, 1>);
    case 2: return launch(hill_attn_finalize_kernel<STATS, 2>);
    case 4: return launch(hill_attn_finalize_kernel<STATS, 4>);
  }
  return (a.H / a.Hkv) % 8 == 0 ? launch(hill_attn_finalize_kernel<STATS, 8>)
                                : launch(hill_attn_finalize_kernel<STATS, -1>);
}

int attn_finalize_waves(int B, int cap, int sms) {
  return (int)(((int64_t)B * ((cap + kFinThreads - 1) / kFinThreads) + sms - 1) / sms);
}

cudaError_t launch_attn_finalize(const FinalizeArgs& a0, int sms, cudaStream_t st, int* kernels,
                                 bool two_kernel) {
  FinalizeArgs a = a0;
  a.tpt = 1;
  // The split step's normalisation runs beside the next layer's scoring
  // kernel, which leaves room for about one such CTA per SM: each thread
  // takes several tokens so that the grid needs at most about two rounds of
  // CTAs instead of trickling through in many.
  if (two_kernel)
    while (a.tpt < kFinMaxTpt &&
           (long long)a.B * ((a.cap + kFinThreads * a.tpt - 1) / (kFinThreads * a.tpt)) > 2LL * sms)
      a.tpt <<= 1;
  // The partials are combined once per (b, h) in a kernel of their own instead
  // of once per CTA with more than two CTAs per SM (attn_finalize_waves), and
  // with more than one where a head has more partials than a warp loads in one
  // round.  Measured, hill_score, one / two kernels (us): 4 x 10K tokens, 8 KV
  // heads (38 partials a head) 18.5 / 19.8, with 1000 tokens in each 6.9 / 6.9 and
  // issued eagerly 11.0 / 12.7; 8 x 6000, 32 KV heads 60.1 / 60.0, with 600 in each
  // 9.8 / 10.3; 1 x 64K, 8 KV heads (152 partials) 25.6 / 26.0; one KV head, 16 x
  // 4K (76) 16.6 / 18.0, 4 x 16K (304) 16.9 / 17.5, the step on 4 of 8-16K 33.0 /
  // 32.6, 2 x 32K (608) 17.8 / 16.8, 1 x 64K (1216) 18.9 / 15.7.
  if (two_kernel || attn_finalize_waves(a.B, a.cap, sms) > 2 ||
      (attn_finalize_waves(a.B, a.cap, sms) > 1 && a.score_grid * a.spc / a.B > 32 * kFinU)) {
    *kernels = 2;
    const int W = a.claim_min > 0 ? 4 : 1;   // warps per (b, h)
    const dim3 sgrid((a.B * a.H * W + kStatsWarps - 1) / kStatsWarps);
    cudaError_t e = W > 1 ? launch_pdl(hill_attn_stats_kernel<4>, sgrid, dim3(kStatsWarps * 32), 0, st, 0, a)
                          : launch_pdl(hill_attn_stats_kernel<1>, sgrid, dim3(kStatsWarps * 32), 0, st, 0, a);
    return e != cudaSuccess ? e : launch_finalize_t<true>(a, st);
  }
  *kernels = 1;
  return launch_finalize_t<false>(a, st);
}

}  // namespace hill
