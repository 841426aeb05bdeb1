// quant.cu -- the 8-bit key shadow used by the asymmetric-precision scoring
// (Sec. 4.4: the evaluation ranks tokens with low-precision inner products;
// the attention keeps the original 16-bit keys and values).
//
// Each (b, g, j) row of K (128 dims) becomes 128 E4M3 codes and one float32
// scale: amax = max |K|, r = 448 / amax, code_i = e4m3(K_i * r) (float32
// product, round to nearest even, saturating), scale = amax / 448.
//
// Bound by HBM (256 bytes read and 132 written per row), if enough loads are
// in flight and the per-row work is small.  A warp takes kQRows = 16
// consecutive rows of one (b, g): 8 lanes cover a row with 32 bytes each, and
// a lane's kQU rows are all loaded before the first is used (128 bytes in
// flight per lane, 1024 lanes per SM).  The maximum is taken on the 16-bit
// pairs (exact) and shuffled over 8 lanes; one lane per row does its two
// divisions, and the scales of a quarter-warp leave as 16 contiguous bytes.
// Measured on the shadow of 4 prompts of 8-16K tokens, 32 heads (51.6K x 32
// rows, 640 MB moved): 91 us, 7.07 TB/s, where one row per warp and 8 bytes
// per lane (one CTA per 8 rows) took 280 us.  Other splits: 2 rows per lane
// 96-101 us, 1 row 119; 16 lanes per row 113-126; a persistent grid that
// prefetches the next rows 111-139.  A few rows keep one row per warp
// (launch_quantize_k).
#include <type_traits>

#include "hill_internal.h"

namespace hill {
namespace {

constexpr int kQWarps = 8;
constexpr int kQU = 4;                // rows per quarter-warp
constexpr int kQRows = 4 * kQU;       // rows per warp
constexpr int kQFew = 6144;           // up to this many rows in all: one row per warp

struct Dims16 {
  uint32_t v[8];   // 16 dims of a row
};

// A32: one 32-byte load; else (16-byte aligned rows) two of 16 bytes.
template <bool A32>
__device__ __forceinline__ Dims16 load_dims(const uint16_t* p) {
  Dims16 r;
  if constexpr (A32) {
    asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r.v[0]), "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]), "=r"(r.v[4]), "=r"(r.v[5]), "=r"(r.v[6]),
                   "=r"(r.v[7])
                 : "l"(p));
  } else {
    const uint4 a = ldg_nc128(p), b = ldg_nc128(p + 8);
    r.v[0] = a.x, r.v[1] = a.y, r.v[2] = a.z, r.v[3] = a.w;
    r.v[4] = b.x, r.v[5] = b.y, r.v[6] = b.z, r.v[7] = b.w;
  }
  return r;
}

// max(|a|, |b|) of two pairs; like fmaxf it passes over a NaN.
template <int DT>
__device__ __forceinline__ uint32_t absmax2(uint32_t a, uint32_t b) {
  using T2 = typename std::conditional<DT == 0, __half2, __nv_bfloat162>::type;
  const T2 m = __hmax2(__habs2(*reinterpret_cast<T2*>(&a)), __habs2(*reinterpret_cast<T2*>(&b)));
  return *reinterpret_cast<const uint32_t*>(&m);
}

template <int DT, bool A32>
__global__ void __launch_bounds__(kQWarps * 32, 4) hill_quantize_k_kernel(const QuantArgs a) {
  pdl_wait();
  pdl_launch_dependents();
  const int lane = threadIdx.x & 31, l8 = lane & 7, qt = lane >> 3;
  // warp -> (b, g) and its chunk of kQRows rows
  const int64_t w = (int64_t)blockIdx.x * kQWarps + (threadIdx.x >> 5);
  const int64_t bg = w / a.chunks;
  const int c = (int)(w - bg * a.chunks);
  if (bg >= (int64_t)a.B * a.Hkv) return;
  const int b = (int)(bg / a.Hkv), g = (int)(bg - (int64_t)b * a.Hkv);
  int j0 = a.row_begin[b], j1 = a.row_end[b];
  j0 = j0 < 0 ? 0 : (j0 > a.cap ? a.cap : j0);
  j1 = j1 < j0 ? j0 : (j1 > a.cap ? a.cap : j1);
  const int n = j1 - j0 - c * kQRows;   // rows from this warp's first to the end
  if (n <= 0) return;
  const int64_t j = (int64_t)j0 + c * kQRows + qt * kQU;   // this quarter-warp's first row
  const int nq = n - qt * kQU;                             // its rows (kQU at most)
  const auto* kr = static_cast<const uint16_t*>(a.k) + (int64_t)b * a.k_sb + (int64_t)g * a.k_sh + j * a.k_sn + l8 * 16;
  Dims16 raw[kQU];
#pragma unroll
  for (int u = 0; u < kQU; ++u) raw[u] = u < nq ? load_dims<A32>(kr + u * a.k_sn) : Dims16{};
  float own = 0.f;   // lane l8 < kQU: the maximum of its quarter-warp's row l8
#pragma unroll
  for (int u = 0; u < kQU; ++u) {
    const uint32_t* v = raw[u].v;
    uint32_t m = absmax2<DT>(absmax2<DT>(absmax2<DT>(v[0], v[1]), absmax2<DT>(v[2], v[3])),
                             absmax2<DT>(absmax2<DT>(v[4], v[5]), absmax2<DT>(v[6], v[7])));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) m = absmax2<DT>(m, __shfl_xor_sync(0xffffffffu, m, o));
    const float2 p = unpack2<DT>(m);
    if (l8 == u) own = fmaxf(p.x, p.y);
  }
  // a row without a positive maximum (all zero) has codes and scale 0
  const bool pos = own > 0.f;
  const float r_own = pos ? __fdiv_rn(448.f, own) : 0.f;
  if (l8 < kQU && l8 < nq) a.kscale[bg * a.cap32 + j + l8] = pos ? __fdiv_rn(own, 448.f) : 0.f;
  const unsigned nz = __ballot_sync(0xffffffffu, pos);
  uint8_t* dst = a.k8 + (bg * a.cap + j) * kHeadDim + l8 * 16;
#pragma unroll
  for (int u = 0; u < kQU; ++u) {
    const float r = __shfl_sync(0xffffffffu, r_own, qt * 8 + u);
    if (u >= nq) continue;
    const bool row_pos = (nz >> (qt * 8 + u)) & 1u;
    uint32_t code[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 x = unpack2<DT>(raw[u].v[2 * i]), y = unpack2<DT>(raw[u].v[2 * i + 1]);
      const uint32_t c4 =
          e4m3x2(__fmul_rn(x.x, r), __fmul_rn(x.y, r)) | (e4m3x2(__fmul_rn(y.x, r), __fmul_rn(y.y, r)) << 16);
      code[i] = row_pos ? c4 : 0u;
    }
    *reinterpret_cast<uint4*>(dst + u * kHeadDim) = uint4{code[0], code[1], code[2], code[3]};
  }
}

// One row per warp, 8 bytes per lane, for calls of a few rows (the new tokens
// of a step): bound by latency, they want a short chain in each warp.
template <int DT>
__global__ void __launch_bounds__(kQWarps * 32) hill_quantize_k_rows_kernel(const QuantArgs a) {
  pdl_wait();
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.z, g = blockIdx.y;
  int j0 = a.row_begin[b], j1 = a.row_end[b];
  j0 = j0 < 0 ? 0 : (j0 > a.cap ? a.cap : j0);
  j1 = j1 < j0 ? j0 : (j1 > a.cap ? a.cap : j1);
  const int j = j0 + blockIdx.x * kQWarps + warp;
  if (j >= j1) return;
  const auto* kr = static_cast<const uint16_t*>(a.k) + (int64_t)b * a.k_sb + (int64_t)g * a.k_sh + (int64_t)j * a.k_sn;
  const uint2 raw = *reinterpret_cast<const uint2*>(kr + lane * 4);
  const float2 x = unpack2<DT>(raw.x), y = unpack2<DT>(raw.y);
  float amax = fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(y.x), fabsf(y.y)));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  const int64_t bg = (int64_t)b * a.Hkv + g;
  const bool pos = amax > 0.f;
  const float r = pos ? __fdiv_rn(448.f, amax) : 0.f;
  const uint32_t code =
      e4m3x2(__fmul_rn(x.x, r), __fmul_rn(x.y, r)) | (e4m3x2(__fmul_rn(y.x, r), __fmul_rn(y.y, r)) << 16);
  reinterpret_cast<uint32_t*>(a.k8 + (bg * a.cap + j) * kHeadDim)[lane] = pos ? code : 0u;
  if (lane == 0) a.kscale[bg * a.cap32 + j] = pos ? __fdiv_rn(amax, 448.f) : 0.f;
}

template <int DT>
cudaError_t launch_quantize_rows(const QuantArgs& a, int max_rows, cudaStream_t st) {
  return launch_pdl(hill_quantize_k_rows_kernel<DT>, dim3((max_rows + kQWarps - 1) / kQWarps, a.Hkv, a.B),
                    dim3(kQWarps * 32), 0, st, 0, a);
}

template <int DT, bool A32>
cudaError_t launch_quantize_t(const QuantArgs& a, cudaStream_t st) {
  const int64_t warps = (int64_t)a.B * a.Hkv * a.chunks;
  return launch_pdl(hill_quantize_k_kernel<DT, A32>, dim3((unsigned)((warps + kQWarps - 1) / kQWarps)),
                    dim3(kQWarps * 32), 0, st, 0, a);
}

}  // namespace

cudaError_t launch_quantize_k(const QuantArgs& a0, int dtype, int max_rows, cudaStream_t st) {
  QuantArgs a = a0;
  // one row per warp / 16 rows per warp (us, in a graph): 8 (b, g) of 1 row 1.37 / 1.73, of 128 rows 1.52 / 2.13; 128 of
  // 16 rows 1.59 / 2.16, of 32 1.95 / 2.16, of 64 2.36 / 2.22; 256 of 24 rows 2.25 / 2.21, of 64 3.28 / 2.31: the line
  // is at about 40 rows per SM
  if ((int64_t)a.B * a.Hkv * max_rows <= kQFew)
    return dtype == 0 ? launch_quantize_rows<0>(a, max_rows, st) : launch_quantize_rows<1>(a, max_rows, st);
  a.chunks = (max_rows + kQRows - 1) / kQRows;
  // rows that all start on 32 bytes are read with 32-byte loads (91 us on the
  // case above); the interface asks for 16 only, and those take two 16-byte
  // loads per lane (93 us)
  const bool a32 = (reinterpret_cast<uintptr_t>(a.k) & 31u) == 0 && (a.k_sb % 16) == 0 && (a.k_sh % 16) == 0 &&
                   (a.k_sn % 16) == 0;
  if (dtype == 0) return a32 ? launch_quantize_t<0, true>(a, st) : launch_quantize_t<0, false>(a, st);
  return a32 ? launch_quantize_t<1, true>(a, st) : launch_quantize_t<1, false>(a, st);
}

}  // namespace hill
