// attn.cu -- decode attention over the selected tokens only (Sec. 4.1, workflow step 6:
// only the critical KV reaches the attention; Eq. 1 restricted to the set).
//
// Gather + split-K flash decode on persistent CTAs.  The work is a list of
// batches: (sequence b, KV head g, batch bi of 32 consecutive entries of
// b's index list), ordered b, g, bi.  Every warp of the grid owns one
// contiguous segment of that list and streams it through a K region and a V
// region of shared memory.  A batch's 32 K rows and 32 V rows (tokens
// idx[b][32*bi + i]) are gathered with 16-byte asynchronous copies (a
// half-warp per 256-byte row; the K rows and the V rows are separate copy
// groups, so K of the next batch is in flight while this batch's softmax and
// P.V run, and V of the next batch while the next S runs) into an
// XOR-swizzled layout that ldmatrix reads without bank conflicts; rows of
// absent tokens are zero-filled by the copies themselves.  The index entries
// of the batch after next are loaded with the K copies and are checked only
// when that batch is issued.  (TMA
// alternatives were measured slower on the same layout: 256-byte bulk copies
// per row are bound by the copy engine's request rate, and tile::gather4 loads
// reached about 85 % of the cp.async throughput; neither depends on how
// scattered the rows are.)
// Both products run on mma.sync m16n8k16 with fp32 accumulation.  S = q . K^T
// takes the G query heads of the group as the rows of A (held in registers
// for all batches of a (b, g)) and K rows read with ldmatrix as B.  An online
// softmax per head, in base 2 (logits scaled by log2(e)/sqrt(d)), runs across
// the batches of one (b, g).  The output is accumulated transposed, O^T +=
// V^T . P^T: V rows read with transposed ldmatrix form A (16 dims x 16
// tokens), and the weights P -- already laid out as a B fragment by the S
// accumulators -- enter as a 16-bit high part plus its 16-bit residual, so
// every instruction covers 8 heads x 16 dims.  A group of 9 to 16 heads fills
// all 16 rows of A (two row blocks of 8 heads, each with its own softmax state
// and O^T accumulators), so the rows gathered once serve 16 heads; larger
// groups run in passes of 16.  When a warp's segment holds
// all batches of a (b, g) it writes the output; otherwise it writes a partial
// (max, sum, o) that hill_attn_combine_kernel merges.
//
// Small calls are bound by latency, and there the merge is the longest part: a
// second launch, its reads of the counts and of the partials.  With few
// (b, g, pass) triples a cluster of CTAs takes each (CL): its warps share the
// triple's batches, the CTAs merge their warps' partials in shared memory and
// push them to one of them, which writes the output.  Such a CTA knows its
// triple from the start, so the queries are loaded before the dependency wait
// and the first index entries together with the count.  Measured: one 4K sequence of
// 32 heads (k = 819) 7.5 -> 5.0 us, 1 x 128K with 8 KV heads (k = 2048) 8.8 ->
// 6.7, 4 x 16K of one KV head (two passes over 32 heads) 18.3 -> 7.9.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "hill_internal.h"

namespace cg = cooperative_groups;

namespace hill {
namespace {

constexpr int kAW = 8;                               // warps per CTA
constexpr int kAThreads = kAW * 32;
constexpr int kBatch = 32;                           // selected entries per batch
constexpr int kMaxBatchAttn = 512;                   // sequences in the per-CTA table

constexpr int kHalfBytes = kBatch * 128;             // 32 rows x 64 dims, swizzled

struct AttnCfg {
  // K dims 0-63 | K dims 64-127 | V dims 0-63 | V dims 64-127
  static constexpr int kSlotBytes = 4 * kHalfBytes;
  static constexpr int smem(int warps) { return warps * kSlotBytes + 128; }   // + alignment slack
};

constexpr int kPS = 2 + kHeadDim;   // one partial of a head: max, sum, o[kHeadDim]
constexpr int kMaxAttnCluster = 8;

// CL: partials of this CTA's share of the triple's heads, from every CTA of the cluster
template <int G>
constexpr int recv_floats() {
  return (G + kMaxAttnCluster - 1) * kPS;
}

// Position of a batch in the list: table unit u (a sequence b, or with
// per-KV-head selection a pair (b, g)), sequence, KV head, batch within (b, g).
struct Pos {
  int u, b, g, bi;
};

// Selected-token count of table unit u (count[] has one entry per unit).
__device__ __forceinline__ int clamp_count(const AttnArgs& a, int u) {
  const int n = a.count[u];
  return n < 0 ? 0 : (n > a.max_k ? a.max_k : n);
}

// Segment of the batch list owned by global warp w (balanced split).
__device__ __forceinline__ void warp_segment(int total, int nwarps, int w, int& t0, int& t1) {
  const int per = (total + nwarps - 1) / nwarps;
  t0 = min(total, w * per);
  t1 = min(total, t0 + per);
}

template <int DT, int G, bool CL, int NW>
__global__ void __launch_bounds__(NW * 32, kAW / NW) hill_sparse_attn_kernel(const __grid_constant__ AttnArgs a) {
  extern __shared__ unsigned char asmem[];
  __shared__ int s_bstart[CL ? 1 : kMaxBatchAttn + 1];
  __shared__ int s_nbat[CL ? 1 : kMaxBatchAttn];
  __shared__ int s_cnt[CL ? 1 : kMaxBatchAttn];
  __shared__ float s_recv[CL ? recv_floats<G>() : 1];
  __shared__ int s_has[NW];   // CL: the warp has a partial

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = lane >> 2, tig = lane & 3;
  constexpr int kRB = G > 8 ? 2 : 1;          // row blocks of 8 heads
  // CL: the cluster's triple (b, g, pass), its table unit and its heads
  int C = 1, rank = 0, tu = 0, tb = 0, tg = 0;
  int Gn = G <= 2 ? G : a.Gn, hoff = a.hoff;
  if constexpr (CL) {
    C = (int)cg::this_cluster().num_blocks();
    rank = (int)cg::this_cluster().block_rank();
    if (C > 1) cg::this_cluster().barrier_arrive();   // every CTA has started (waited for before the first push)
    const int P = (a.Gs + 15) / 16, triple = blockIdx.x / C, bg = triple / P;
    hoff = 16 * (triple - bg * P);
    Gn = min(16, a.Gs - hoff);
    tb = bg / a.Hkv;
    tg = bg - tb * a.Hkv;
    tu = a.kvh ? bg : tb;
  }
  uint32_t qa[kRB][8][2];                     // q rows of the group as A fragments
  bool head_ok[kRB];
#pragma unroll
  for (int rb = 0; rb < kRB; ++rb) head_ok[rb] = grp + 8 * rb < Gn;
  auto load_q = [&](int b, int g) {
    const auto* q32 = static_cast<const uint32_t*>(a.q);
#pragma unroll
    for (int rb = 0; rb < kRB; ++rb) {
      const bool ok = head_ok[rb];
      const int64_t row = ok ? ((int64_t)b * a.q_sb + (int64_t)(g * a.Gs + hoff + 8 * rb + grp) * a.q_sh) / 2 : 0;
#pragma unroll
      for (int kb = 0; kb < 8; ++kb) {
        qa[rb][kb][0] = ok ? __ldg(q32 + row + kb * 8 + tig) : 0u;
        qa[rb][kb][1] = ok ? __ldg(q32 + row + kb * 8 + 4 + tig) : 0u;
      }
    }
  };
  if constexpr (CL) load_q(tb, tg);   // (an input of the call: include/hill.h)
  pdl_wait();
  // No early trigger (here and in the combine): the attention runs beside
  // the K stream of later layers, and a dependent launched early would hold
  // SMs idle while it waits (measured: the pipelined step is 2 % faster).

  // CL: this cluster's count, and the index entries of warp w's first batch if
  // every warp has one at most
  int n_unit = 0, nb_unit = 0, j_first = -1;
  if constexpr (CL) {
    const int e = (rank * NW + warp) * kBatch + lane;
    if (e < a.max_k) j_first = a.idx[(int64_t)tu * a.max_k + e];
    n_unit = clamp_count(a, tu);
    nb_unit = (n_unit + kBatch - 1) / kBatch;
  }
  auto cnt_of = [&](int u) { return CL ? n_unit : s_cnt[u]; };
  auto nbat_of = [&](int u) { return CL ? nb_unit : s_nbat[u]; };
  // table units: sequences (every KV head reads the same set, Hkv * nbat
  // batches per unit, ordered g, bi), or with per-KV-head selection the pairs
  // (b, g) (nbat batches per unit)
  const int R = a.kvh ? a.B * a.Hkv : a.B;
  const int upb = a.kvh ? 1 : a.Hkv;   // KV heads per unit
  if constexpr (!CL) {
  for (int u = threadIdx.x; u < R; u += (NW * 32)) {
    const int n = clamp_count(a, u);
    s_cnt[u] = n;
    s_nbat[u] = (n + kBatch - 1) / kBatch;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int u = 0; u < R; ++u) {
      s_bstart[u] = acc;
      acc += upb * s_nbat[u];
    }
    s_bstart[R] = acc;
  }
  __syncthreads();
  }
  const int total = CL ? nb_unit : s_bstart[R];
  const int nwarps = (CL ? C : gridDim.x) * NW;
  const int gw = (CL ? rank : blockIdx.x) * NW + warp;
  int t0, t1;
  warp_segment(total, nwarps, gw, t0, t1);
  if (!CL && t0 >= t1) return;

  // 128-byte aligned slots: every swizzled row is one bank-aligned line
  const uint32_t slot0 = ((smem_addr(asmem) + 127u) & ~127u) + warp * AttnCfg::kSlotBytes;
  const uint32_t sk = slot0, sv = slot0 + 2 * kHalfBytes;   // the warp's K rows | V rows
  const auto* kbase = static_cast<const uint16_t*>(a.k);
  const auto* vbase = static_cast<const uint16_t*>(a.v);
  const int ksn = (int)a.k_sn, vsn = (int)a.v_sn;   // the host checks both fit in 32 bits

  // position of batch t0 (binary search once), then advanced one batch at a time
  Pos first;
  if constexpr (CL) {
    first = Pos{tu, tb, tg, t0};
  } else {
    int lo = 0, hi = R;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (s_bstart[mid] <= t0) lo = mid; else hi = mid;
    }
    const int rem = t0 - s_bstart[lo];
    first.u = lo;
    if (a.kvh) {
      first.b = lo / a.Hkv;
      first.g = lo - first.b * a.Hkv;
      first.bi = rem;
    } else {
      first.b = lo;
      first.g = rem / s_nbat[lo];
      first.bi = rem - first.g * s_nbat[lo];
    }
  }
  auto advance = [&](Pos& p) {
    if constexpr (CL) {
      ++p.bi;
      return;
    }
    if (p.u >= R) return;
    if (++p.bi < s_nbat[p.u]) return;
    p.bi = 0;
    if (!a.kvh && ++p.g < a.Hkv) return;
    do {
      ++p.u;
    } while (p.u < R && s_nbat[p.u] == 0);
    p.b = a.kvh ? p.u / a.Hkv : p.u;
    p.g = a.kvh ? p.u - p.b * a.Hkv : 0;
  };

  // raw index entry of this lane for the batch at p (-1 past the count).
  // Nothing here depends on the loaded value, so the load stays in flight
  // until the batch is issued one iteration later, where it is checked.
  auto load_idx = [&](const Pos& p) -> int {
    const int e = p.bi * kBatch + lane;
    return e < cnt_of(p.u) ? a.idx[(int64_t)p.u * a.max_k + e] : -1;
  };
  // An entry of the batch at p that lies outside [0, cap) is reported and
  // skipped (-1: no token).
  auto check = [&](const Pos& p, int jj) -> int {
    if (p.bi * kBatch + lane < cnt_of(p.u) && (jj < 0 || jj >= a.cap)) {
      raise_error(a.err, kErrDevArg);
      jj = -1;
    }
    return jj;
  };
  // Gather the 32 rows of one cache (K or V) for the batch at p into the
  // 8 KB region dst: row r of the batch is token jj of lane r (-1: none,
  // zero-filled).  A half-warp copies one 256-byte row; chunk c (16 bytes)
  // of row r goes to 128-byte line r of half c / 8 at position
  // (c % 8) ^ (r % 8), so the ldmatrix reads below are conflict-free.  One
  // cp.async group per call.
  const int l16 = lane & 15, hrow = lane >> 4;
  const uint32_t dst_lane = (uint32_t)((l16 >> 3) * kHalfBytes + hrow * 128);
  const uint32_t swz_lane = (uint32_t)(((l16 & 7) ^ hrow) << 4);
  auto issue_rows = [&](const Pos& p, uint32_t dst, const uint16_t* base, int64_t sb, int64_t sh, int sn, int jj) {
    const uint16_t* rp = base + (int64_t)p.b * sb + (int64_t)p.g * sh + l16 * 8;
    dst += dst_lane;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int j = __shfl_sync(0xffffffffu, jj, 2 * i + hrow);
      const uint32_t nbytes = j >= 0 ? 16u : 0u;
      const int jc = j >= 0 ? j : 0;
      // row 2i + hrow: (2i + hrow) % 8 = (2i % 8) | hrow
      const uint32_t off = (uint32_t)(i * 256) + (swz_lane ^ (uint32_t)(((2 * i) & 7) << 4));
      cp_async16_zfill(dst + off, rp + (int64_t)jc * sn, nbytes);
    }
    cp_async_commit();
  };

  // Pipeline of one warp over its batches t0 .. t1-1, with one K region and
  // one V region: K rows of batch t + 1 are fetched once S(t) has read the K
  // region (while the softmax and O += P V of batch t run), V rows of batch
  // t + 1 once O += P V(t) has read the V region (while S(t + 1) runs).  The
  // cp.async groups complete in the order K(t), V(t), K(t + 1), V(t + 1), ...
  // The index entries of batch t + 2 are loaded when K(t + 1) is issued.
  Pos pc = first, pi = first, pl = first;
  unsigned vm_cur = 0u, vm_next = 0u;
  int jcur = -1, jnext = -1;                    // entries of the batch being issued, and of the next
  if (!CL || t0 < t1) {
  // (CL, one batch per warp: its entries are here already)
  const bool have = CL && t0 == gw;
  jcur = check(pi, !have ? load_idx(pl) : (pl.bi * kBatch + lane < cnt_of(pl.u) ? j_first : -1));
  advance(pl);
  vm_cur = __ballot_sync(0xffffffffu, jcur >= 0);
  issue_rows(pi, sk, kbase, a.k_sb, a.k_sh, ksn, jcur);
  issue_rows(pi, sv, vbase, a.v_sb, a.v_sh, vsn, jcur);
  advance(pi);
  jnext = t0 + 1 < t1 ? load_idx(pl) : -1;
  advance(pl);
  }

  // mma.sync fragments: grp = lane/4, tig = lane%4.  S accumulators: row grp
  // (+8 with 16 heads: row block rb = 1) = query head grp (+8) of the group
  // (rows >= Gn are zero, and rows 8..15 when G <= 8; Gn = G unless the
  // group has fewer heads than the power-of-two template), columns = tokens
  // nb*8 + 2*tig + {0,1}.  O^T accumulators, one set per row block: rows =
  // dims db*16 + grp (+8), columns = heads 8*rb + 2*tig, 8*rb + 2*tig + 1.
  const int hA = 2 * tig, hB = 2 * tig + 1;   // heads of this lane's O^T columns (in a row block)
  float m_run[kRB], l_run[kRB];               // softmax state of head grp + 8*rb (base 2)
  float oacc[kRB][8][4];
  int cb = -1, cg = -1, cu = -1;              // the (b, g) being accumulated and its unit
  const int per = (total + nwarps - 1) / nwarps;

  auto reset = [&](int b, int g) {
#pragma unroll
    for (int rb = 0; rb < kRB; ++rb) {
      m_run[rb] = -INFINITY;
      l_run[rb] = 0.f;
#pragma unroll
      for (int db = 0; db < 8; ++db)
#pragma unroll
        for (int e = 0; e < 4; ++e) oacc[rb][db][e] = 0.f;
    }
    if constexpr (!CL) load_q(b, g);
  };

  // write the current (b, g): the output itself when this segment holds all
  // of its batches, else a partial for the combine kernel
  float* const staged = reinterpret_cast<float*>(asmem + (slot0 - smem_addr(asmem)));   // CL: in the warp's slot, free by then
  auto flush = [&]() {
    const int nb_ = nbat_of(cu);
    const int firstb = CL ? 0 : s_bstart[cu] + (a.kvh ? 0 : cg * nb_);   // first batch of (cb, cg) in the list
    const bool whole = !CL && firstb / per == (firstb + nb_ - 1) / per;   // one segment holds it all
    const int seg = gw - firstb / per;
#pragma unroll
    for (int rb = 0; rb < kRB; ++rb) {
      // (max, sum) of the heads in this lane's O^T columns of row block rb
      const float mA = __shfl_sync(0xffffffffu, m_run[rb], 8 * tig);
      const float lA = __shfl_sync(0xffffffffu, l_run[rb], 8 * tig);
      const float mB = __shfl_sync(0xffffffffu, m_run[rb], 8 * tig + 4);
      const float lB = __shfl_sync(0xffffffffu, l_run[rb], 8 * tig + 4);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int hl = 8 * rb + (c ? hB : hA);
        if (hl >= Gn) continue;
        const float m = c ? mB : mA, l = c ? lB : lA;
        const int h = cg * a.Gs + hoff + hl;
        if (whole) {
          float* op = a.out + ((int64_t)cb * a.H + h) * kHeadDim + grp;
          const float inv = l > 0.f ? 1.f / l : 0.f;
#pragma unroll
          for (int db = 0; db < 8; ++db) {
            op[db * 16] = oacc[rb][db][c] * inv;
            op[db * 16 + 8] = oacc[rb][db][2 + c] * inv;
          }
        } else {
          float* pp = CL ? staged + hl * kPS : a.part + (((int64_t)cb * a.H + h) * a.splits + seg) * kPS;
          if (grp == 0) {
            pp[0] = m;
            pp[1] = l;
          }
#pragma unroll
          for (int db = 0; db < 8; ++db) {
            pp[2 + db * 16 + grp] = oacc[rb][db][c];
            pp[2 + db * 16 + 8 + grp] = oacc[rb][db][2 + c];
          }
        }
      }
    }
  };

  for (int t = t0; t < t1; ++t) {
    if (pc.b != cb || pc.g != cg) {
      if (cb >= 0) flush();
      cb = pc.b;
      cg = pc.g;
      cu = pc.u;
      reset(cb, cg);
    }
    // K(t) is complete once at most V(t) is pending
    cp_async_wait<1>();
    __syncwarp();
    const unsigned vm = vm_cur;
    const bool more = t + 1 < t1;

    // S = q . K^T: A = q (16 rows = heads), B = K rows (n = 8 tokens)
    float sacc[4][4];
#pragma unroll
    for (int nb = 0; nb < 4; ++nb) {
#pragma unroll
      for (int e = 0; e < 4; ++e) sacc[nb][e] = 0.f;
      const int trow = nb * 8 + (lane & 7);
#pragma unroll
      for (int kp = 0; kp < 4; ++kp) {
        const int c = 4 * kp + (lane >> 3);
        uint32_t bk[4];
        ldmatrix_x4(sk + (c >> 3) * kHalfBytes + trow * 128 + (((c & 7) ^ (trow & 7)) << 4), bk);
        // rows 8..15 of A: the second row block of 16 heads, else zero
        const uint32_t a0[4] = {qa[0][2 * kp][0], kRB > 1 ? qa[kRB - 1][2 * kp][0] : 0u, qa[0][2 * kp][1],
                                kRB > 1 ? qa[kRB - 1][2 * kp][1] : 0u};
        const uint32_t a1[4] = {qa[0][2 * kp + 1][0], kRB > 1 ? qa[kRB - 1][2 * kp + 1][0] : 0u,
                                qa[0][2 * kp + 1][1], kRB > 1 ? qa[kRB - 1][2 * kp + 1][1] : 0u};
        mma_16816<DT>(sacc[nb], a0, bk[0], bk[1]);
        mma_16816<DT>(sacc[nb], a1, bk[2], bk[3]);
      }
    }
    // the K region is free: fetch K(t + 1), and the entries of batch t + 2
    __syncwarp();
    if (more) {
      jcur = check(pi, jnext);
      vm_next = __ballot_sync(0xffffffffu, jcur >= 0);
      issue_rows(pi, sk, kbase, a.k_sb, a.k_sh, ksn, jcur);
      jnext = t + 2 < t1 ? load_idx(pl) : -1;
      advance(pl);
    }
    // online softmax of head grp (+8 for row block 1) over the batch's tokens
    // nb*8 + 2*tig + {0,1}
    uint32_t pb[kRB][2][2][2];   // [row block][k block][hi/lo][tokens 0-7 | 8-15 of the block]
#pragma unroll
    for (int rb = 0; rb < kRB; ++rb) {
      float z[8];
      float tmax = -INFINITY;
#pragma unroll
      for (int nb = 0; nb < 4; ++nb)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int tkn = nb * 8 + 2 * tig + e;
          const float v = ((vm >> tkn) & 1u) ? sacc[nb][2 * rb + e] * kLog2eInvSqrtD : -INFINITY;
          z[nb * 2 + e] = v;
          tmax = fmaxf(tmax, v);
        }
      tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 1));
      tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, 2));
      const float mn = fmaxf(m_run[rb], tmax);   // finite: every batch holds a token
      const float corr = ex2(m_run[rb] - mn);    // 0 on the first batch
      float p[8], psum = 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        p[u] = head_ok[rb] ? ex2(z[u] - mn) : 0.f;
        psum += p[u];
      }
      psum += __shfl_xor_sync(0xffffffffu, psum, 1);
      psum += __shfl_xor_sync(0xffffffffu, psum, 2);
      l_run[rb] = l_run[rb] * corr + psum;
      m_run[rb] = mn;
      // rescale O^T: columns hA, hB take the factor of their head
      const float cA = __shfl_sync(0xffffffffu, corr, 8 * tig);
      const float cB = __shfl_sync(0xffffffffu, corr, 8 * tig + 4);
#pragma unroll
      for (int db = 0; db < 8; ++db) {
        oacc[rb][db][0] *= cA;
        oacc[rb][db][2] *= cA;
        if constexpr (G > 1) {
          oacc[rb][db][1] *= cB;
          oacc[rb][db][3] *= cB;
        }
      }
      // P as B fragments (k = token, n = head grp), split into a 16-bit high
      // part and its 16-bit residual so the weights keep ~22 bits
#pragma unroll
      for (int kt = 0; kt < 2; ++kt)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const float x = p[(2 * kt + hf) * 2], y = p[(2 * kt + hf) * 2 + 1];
          const uint32_t hi = pack2<DT>(x, y);
          const float2 hv = unpack2<DT>(hi);
          pb[rb][kt][0][hf] = hi;
          pb[rb][kt][1][hf] = pack2<DT>(x - hv.x, y - hv.y);
        }
    }
    // V(t) is complete once at most K(t + 1) is pending
    if (more) cp_async_wait<1>();
    else cp_async_wait<0>();
    __syncwarp();
    // O^T += V^T . P^T: A = V^T (16 dims x 16 tokens) by transposed ldmatrix
#pragma unroll
    for (int kt = 0; kt < 2; ++kt) {
      const int trow = kt * 16 + (lane & 7) + ((lane >> 4) & 1) * 8;
#pragma unroll
      for (int db = 0; db < 8; ++db) {
        const int c = 2 * db + ((lane >> 3) & 1);
        uint32_t av[4];
        ldmatrix_x4_trans(sv + (c >> 3) * kHalfBytes + trow * 128 + (((c & 7) ^ (trow & 7)) << 4), av);
#pragma unroll
        for (int rb = 0; rb < kRB; ++rb) {
          mma_16816<DT>(oacc[rb][db], av, pb[rb][kt][0][0], pb[rb][kt][0][1]);
          mma_16816<DT>(oacc[rb][db], av, pb[rb][kt][1][0], pb[rb][kt][1][1]);
        }
      }
    }
    // the V region is free: fetch V(t + 1)
    __syncwarp();
    if (more) {
      issue_rows(pi, sv, vbase, a.v_sb, a.v_sh, vsn, jcur);
      advance(pi);
    }
    vm_cur = vm_next;
    advance(pc);
  }
  if constexpr (!CL) {
    flush();
    return;
  }
  // CL: merge the warps' partials head by head; C > 1: push the CTA's to CTA
  // h % C, which merges the CTAs'
  if (t0 < t1) flush();
  if (lane == 0) s_has[warp] = t0 < t1;
  __syncthreads();
  struct Acc {
    float m = -INFINITY, l = 0.f, o[4] = {0.f, 0.f, 0.f, 0.f};   // dims lane + 32 i
  };
  auto fold = [&](Acc& x, const float* p) {
    const float m = p[0], l = p[1];
    if (m == -INFINITY) return;   // no token
    const float mn = fmaxf(x.m, m), c0 = ex2(x.m - mn), c1 = ex2(m - mn);
    x.l = x.l * c0 + l * c1;
#pragma unroll
    for (int i = 0; i < 4; ++i) x.o[i] = x.o[i] * c0 + p[2 + lane + 32 * i] * c1;
    x.m = mn;
  };
  auto write_out = [&](const Acc& x, int hl) {
    float* op = a.out + ((int64_t)tb * a.H + tg * a.Gs + hoff + hl) * kHeadDim + lane;
    const float inv = x.l > 0.f ? 1.f / x.l : 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) op[32 * i] = x.o[i] * inv;
  };
  const float* const slots_f = staged - warp * (AttnCfg::kSlotBytes / 4);
  if (C > 1) cg::this_cluster().barrier_wait();
  for (int hl = warp; hl < Gn; hl += NW) {
    Acc x;
    for (int w = 0; w < NW; ++w)
      if (s_has[w]) fold(x, slots_f + w * (AttnCfg::kSlotBytes / 4) + hl * kPS);
    if (C == 1) {
      write_out(x, hl);
      continue;
    }
    float* d = cg::this_cluster().map_shared_rank(s_recv, hl % C) + ((hl / C) * C + rank) * kPS;
    if (lane == 0) {
      d[0] = x.m;
      d[1] = x.l;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) d[2 + lane + 32 * i] = x.o[i];
  }
  if (C == 1) return;
  cg::this_cluster().sync();
  for (int i = warp; i * C + rank < Gn; i += NW) {
    Acc x;
    for (int c = 0; c < C; ++c) fold(x, s_recv + (i * C + c) * kPS);
    write_out(x, i * C + rank);
  }
}

// Merge the partials of one (b, h) whose batches were split over several
// warps: out = sum_s 2^{M_s - M} O_s / sum_s 2^{M_s - M} L_s (maxima in the
// base-2 scale of the attention kernel).  Pairs held whole by one warp were
// written directly; sequences with no selected token get zeros.  One CTA per
// (b, h): kCombGroups groups of kHeadDim threads (one per output dimension)
// each merge every kCombGroups-th partial with a running maximum, the loads
// of several partials in flight at once, and the group results are merged in
// shared memory.  A short budget split over many warps (one batch per warp)
// leaves dozens of partials per pair, so their loads must not be serialised.
constexpr int kCombGroups = 4;
constexpr int kCombThreads = kCombGroups * kHeadDim;

__global__ void __launch_bounds__(kCombThreads) hill_attn_combine_kernel(AttnArgs a, int total_warps) {
  __shared__ int s_first, s_nb, s_total;
  __shared__ float s_m[kCombGroups], s_l[kCombGroups];
  __shared__ float s_o[kCombGroups][kHeadDim];
  const int bh = blockIdx.x;
  const int b = bh / a.H, h = bh % a.H;
  const int G = a.H / a.Hkv, g = h / G;
  const int tid = threadIdx.x, dd = tid % kHeadDim, gi = tid / kHeadDim;
  __shared__ int s_nbu[kMaxBatchAttn];
  pdl_wait();
  // the batch layout of the attention kernel (see its table units)
  const int R = a.kvh ? a.B * a.Hkv : a.B;
  for (int u = tid; u < R; u += kCombThreads) s_nbu[u] = (clamp_count(a, u) + kBatch - 1) / kBatch;
  __syncthreads();
  if (tid == 0) {
    const int upb = a.kvh ? 1 : a.Hkv;
    const int mine = a.kvh ? b * a.Hkv + g : b;
    int acc = 0, first = 0, nb = 0;
    for (int u = 0; u < R; ++u) {
      const int nbu = s_nbu[u];
      if (u == mine) {
        first = acc + (a.kvh ? 0 : g * nbu);
        nb = nbu;
      }
      acc += upb * nbu;
    }
    s_first = first;
    s_nb = nb;
    s_total = acc;
  }
  __syncthreads();
  const int nb = s_nb, first = s_first, total = s_total;
  float* op = a.out + (int64_t)bh * kHeadDim + dd;
  if (nb == 0) {
    if (gi == 0) *op = 0.f;
    return;
  }
  const int per = (total + total_warps - 1) / total_warps;
  const int w0 = first / per, w1 = (first + nb - 1) / per;
  if (w0 == w1) return;   // one warp held every batch and wrote the output
  const float* pp = a.part + (int64_t)bh * a.splits * kPS;
  const int nseg = w1 - w0 + 1;
  float M = -INFINITY, L = 0.f, O = 0.f;
  // KU partials per group have their loads issued together; a pair with few
  // partials (nseg is the same for the whole CTA) takes the short variant
  auto merge = [&](auto ku) {
    constexpr int KU = decltype(ku)::value;
    for (int s0 = gi; s0 < nseg; s0 += kCombGroups * KU) {
      float ms[KU], ls[KU], os[KU];
#pragma unroll
      for (int u = 0; u < KU; ++u) {
        const int s = s0 + u * kCombGroups;
        const float* q = pp + (int64_t)s * kPS;
        ms[u] = s < nseg ? q[0] : -INFINITY;
        ls[u] = s < nseg ? q[1] : 0.f;
        os[u] = s < nseg ? q[2 + dd] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < KU; ++u) {
        if (ms[u] == -INFINITY) continue;   // past the end (every written partial holds a token)
        const float mn = fmaxf(M, ms[u]);
        const float c0 = ex2(M - mn), c1 = ex2(ms[u] - mn);   // partial maxima are in the base-2 scale
        L = L * c0 + ls[u] * c1;
        O = O * c0 + os[u] * c1;
        M = mn;
      }
    }
  };
  if (nseg <= kCombGroups * 2) merge(std::integral_constant<int, 2>{});
  else merge(std::integral_constant<int, 16>{});
  s_o[gi][dd] = O;
  if (dd == 0) {
    s_m[gi] = M;
    s_l[gi] = L;
  }
  __syncthreads();
  if (gi == 0) {
    float Mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < kCombGroups; ++i) Mx = fmaxf(Mx, s_m[i]);
    float Ls = 0.f, Os = 0.f;
    if (Mx != -INFINITY) {
#pragma unroll
      for (int i = 0; i < kCombGroups; ++i) {
        const float c = s_m[i] == -INFINITY ? 0.f : ex2(s_m[i] - Mx);
        Ls += s_l[i] * c;
        Os += s_o[i][dd] * c;
      }
    }
    *op = Ls > 0.f ? Os / Ls : 0.f;
  }
}

template <int DT, int G>
cudaError_t launch_attn_t(const AttnArgs& a, int grid, bool combine, cudaStream_t st) {
  static int cache[64] = {0};
  auto kern = hill_sparse_attn_kernel<DT, G, false, kAW>;
  cudaError_t e = ensure_smem_attr(reinterpret_cast<const void*>(kern), AttnCfg::smem(kAW), cache);
  if (e != cudaSuccess) return e;
  e = launch_pdl(kern, dim3(grid), dim3(kAThreads), AttnCfg::smem(kAW), st, 0, a);
  if (e != cudaSuccess || !combine) return e;
  return launch_pdl(hill_attn_combine_kernel, dim3(a.B * a.H), dim3(kCombThreads), 0, st, 0, a, grid * kAW);
}

// Clusters of C CTAs of the cluster form that the current device holds at once.
template <int DT, int G, int NW>
cudaError_t attn_clusters_fit(int C, int* n) {
  static int cache[64] = {0};
  static int fit[64][kMaxAttnCluster + 1];   // (+ 1; 0: not asked yet)
  static std::mutex mu;
  auto kern = hill_sparse_attn_kernel<DT, G, true, NW>;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  e = ensure_smem_attr(reinterpret_cast<const void*>(kern), AttnCfg::smem(NW), cache);   // (checks dev)
  if (e != cudaSuccess) return e;
  int& f = fit[dev][C];
  if (f == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(NW * 32);
    cfg.dynamicSmemBytes = AttnCfg::smem(NW);
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = C;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    e = cudaOccupancyMaxActiveClusters(&f, kern, &cfg);
    if (e != cudaSuccess) return e;
    ++f;
  }
  *n = f - 1;
  return cudaSuccess;
}

// The largest cluster of CTAs of NW warps that all triples can have at once
// (0: none), and the batches that a warp then takes at most.
template <int DT, int G, int NW>
cudaError_t attn_cluster_size(int64_t triples, int nb, int sms, int* C, int* rounds) {
  *C = 0;
  int c = (int)std::min<int64_t>({kMaxAttnCluster, (int64_t)sms * (kAW / NW) / triples, (nb + NW - 1) / NW});
  for (; c >= 1; --c) {
    int n = 0;
    const cudaError_t e = attn_clusters_fit<DT, G, NW>(c, &n);
    if (e != cudaSuccess) return e;
    if (triples > n) continue;
    *C = c;
    *rounds = (nb + c * NW - 1) / (c * NW);
    break;
  }
  return cudaSuccess;
}

// The cluster form, if it is the better one for this call (*done).
template <int DT, int G>
cudaError_t launch_attn_cl(const AttnArgs& a, int sms, cudaStream_t st, bool* done) {
  *done = false;
  const int64_t triples = (int64_t)a.B * a.Hkv * ((a.Gs + 15) / 16);
  const int nb = (a.max_k + kBatch - 1) / kBatch;   // batches of a triple, at most
  if (triples == 0 || nb == 0 || triples > 2 * sms) return cudaSuccess;
  int c8 = 0, r8 = 0, c4 = 0, r4 = 0;
  cudaError_t e = triples <= sms ? attn_cluster_size<DT, G, kAW>(triples, nb, sms, &c8, &r8) : cudaSuccess;
  if (e == cudaSuccess) e = attn_cluster_size<DT, G, kAW / 2>(triples, nb, sms, &c4, &r4);
  if (e != cudaSuccess) return e;
  // with several sequences CTAs of 4 warps, which spread a (b, g) over twice as
  // many SMs, unless they take more rounds (one sequence: its pairs are alike, and
  // beside a K stream fewer, larger CTAs wait less: 1 x 64K, k 50 %, pipelined step
  // 146 us per layer against 151)
  const bool half = c8 == 0 || (c4 > 0 && (a.B > 1 ? r4 <= r8 : r4 < r8));
  const int C = half ? c4 : c8, rounds = half ? r4 : r8;
  const int64_t even = (triples * nb + (int64_t)sms * kAW - 1) / ((int64_t)sms * kAW);
  // A round (one more batch per warp) costs about 1.6 us where latency bounds
  // it, the launches saved about 3.5 us and 8 more for every further pass over
  // the heads; beyond some 10 rounds HBM bounds both forms until the uneven
  // split shows.  Measured, even split / clusters (us, rounds in brackets):
  // 32 heads, 8 x 4K k 20 % 25.0 / 20.0 (6 / 7), 4 x 16-32K k 10 % 34.7 / 32.2
  // (11 / 13), 1 x 64K k 50 % 86.0 / 82.5 (27 / 33); 8 x 16-32K k 50 % 249 /
  // 260 (108 / 129); 7 heads per KV head, 4 KV heads, 64K, k 10 % 12.4 / 10.3
  // (1 / 4), k 20 % 14.2 / 14.9 (2 / 7); 32 heads on one KV head, k 20 % of
  // 64K 24.7 / 18.7 (1 / 7), k 30 % of 128K 32.4 / 41.5 (3 / 20).
  const int64_t passes = (a.Gs + 15) / 16;
  if (C == 0 || even > 32 || rounds > even + even / 4 + 3 * passes) return cudaSuccess;
  // The counts are not known here.  With one sequence at max_k and the others
  // nearly empty the even split has only that one's batches to deal out (`one`
  // rounds), while its clusters still take all their rounds, at 0.5 to 1 us each.
  // Measured, even split / clusters (us) with equal counts, counts of 50-100 %,
  // half of them at 1/8, and one beside 50s; rounds - one in brackets:
  //   32 heads, 8 x 819 (6)  18.9 / 14.7  15.7 / 12.7  13.7 / 10.6  10.3 / 10.2
  //             8 x 947 (7)  24.8 / 20.6  16.0 / 14.4  13.7 / 11.9  10.3 / 11.3
  //             4 x 2300 (7) 30.8 / 26.9  22.0 / 20.1  15.6 / 14.4  12.4 / 13.1
  //             8 x 1100 (8) 29.6 / 25.2  18.8 / 16.9  15.4 / 13.5  10.3 / 12.4
  //             4 x 2600 (8) 34.0 / 30.9  26.9 / 25.5  16.0 / 17.0  12.5 / 15.2
  //             4 x 3277 (10) 40.1 / 37.1  33.2 / 31.4  23.9 / 21.8  12.6 / 17.4
  //   4 heads per KV head, 8 KV heads,
  //             16 x 2200 (8) 34.5 / 26.8  25.0 / 18.9  19.7 / 15.0  11.2 / 13.6
  //             8 x 4600 (8) 32.3 / 27.6  22.1 / 19.5  17.0 / 15.2  11.7 / 13.8
  //             8 x 5600 (10) 37.4 / 32.7  29.1 / 26.3  19.6 / 18.3  12.0 / 15.9
  // (beside empty ones up to 2.7 us lost within the lines).  The lines, 7 and
  // for groups 8, lie where the last column loses less than the others gain.
  const int64_t one = (triples / a.B * nb + (int64_t)sms * kAW - 1) / ((int64_t)sms * kAW);
  if (a.B > 1 && rounds > one + (a.Gs > 1 ? 2 : 1) + 6 * passes) return cudaSuccess;
  *done = true;
  const dim3 grid((unsigned)(triples * C));
  return half ? launch_pdl(hill_sparse_attn_kernel<DT, G, true, kAW / 2>, grid, dim3(kAThreads / 2), AttnCfg::smem(kAW / 2),
                           st, C, a)
              : launch_pdl(hill_sparse_attn_kernel<DT, G, true, kAW>, grid, dim3(kAThreads), AttnCfg::smem(kAW), st, C, a);
}

template <int DT>
cudaError_t launch_attn_cl_d(const AttnArgs& a, int sms, cudaStream_t st, bool* done) {
  if (a.Gs <= 1) return launch_attn_cl<DT, 1>(a, sms, st, done);
  if (a.Gs <= 2) return launch_attn_cl<DT, 2>(a, sms, st, done);
  if (a.Gs <= 4) return launch_attn_cl<DT, 4>(a, sms, st, done);
  if (a.Gs <= 8) return launch_attn_cl<DT, 8>(a, sms, st, done);
  return launch_attn_cl<DT, 16>(a, sms, st, done);
}

template <int DT>
cudaError_t launch_attn_d(const AttnArgs& a, int G, int grid, bool combine, cudaStream_t st) {
  switch (G) {
    case 1: return launch_attn_t<DT, 1>(a, grid, combine, st);
    case 2: return launch_attn_t<DT, 2>(a, grid, combine, st);
    case 4: return launch_attn_t<DT, 4>(a, grid, combine, st);
    case 8: return launch_attn_t<DT, 8>(a, grid, combine, st);
    case 16: return launch_attn_t<DT, 16>(a, grid, combine, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

int attn_batch_tokens() { return kBatch; }
int attn_max_batch() { return kMaxBatchAttn; }

// Partial slots per (b, h): a (b, g) of nb batches meets at most
// ceil(nb / per) + 1 warp segments, and per >= 1.
int attn_max_segments(int max_k) { return (max_k + kBatch - 1) / kBatch + 1; }

cudaError_t launch_sparse_attn_clusters(const AttnArgs& a, int dtype, int sms, cudaStream_t st, bool* done) {
  return dtype == 0 ? launch_attn_cl_d<0>(a, sms, st, done) : launch_attn_cl_d<1>(a, sms, st, done);
}

cudaError_t launch_sparse_attn(const AttnArgs& a, int dtype, int G, int grid, bool combine, cudaStream_t st) {
  return dtype == 0 ? launch_attn_d<0>(a, G, grid, combine, st) : launch_attn_d<1>(a, G, grid, combine, st);
}

}  // namespace hill
