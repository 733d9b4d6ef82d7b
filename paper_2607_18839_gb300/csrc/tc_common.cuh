// tc_common.cuh -- pieces of the tcgen05 branch-attention kernel: half of a
// 128-key block of a row's softmax, and TMA tensor-map encoding on
// the host.
#pragma once

#include <cudaTypedefs.h>

#include <mutex>

#include "common.cuh"
#include "sm100.cuh"

namespace hpd {
namespace tc {

// max(a, b, c) in one instruction (three-input max.f32, sm_100 and later).
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

constexpr int kRows = 128;  // stacked query rows of one tile (MMA M)
constexpr int kBlk = 128;   // keys per block (MMA N of S = Q K^T)
constexpr float kRescaleLog2 = 8.0f;  // tolerate a stale row max up to 2^8
// Scores up to this far above a fixed base: their weights, and sums of them,
// stay far from overflow; O = P V overflows where values beyond 2^63 meet them,
// which its reader finds (with running maxima, weights up to 2^8 leave room for
// values up to 2^119).
constexpr float kWindowLog2 = 64.0f;

// A key the row does not see gets the score -inf: 32 columns, visible from
// lo to hi; scale: multiply by mul first.
__device__ __forceinline__ void mask32(uint32_t *v, int lo, int hi, bool scale, float mul) {
  auto below = [](int n) -> uint32_t { return n <= 0 ? 0u : n >= 32 ? ~0u : (1u << n) - 1u; };
  const uint32_t vis = below(hi) & ~below(lo);
  if (scale) {
#pragma unroll
    for (int c = 0; c < 32; ++c) v[c] = __float_as_uint(__uint_as_float(v[c]) * mul);
  }
#pragma unroll
  for (int c = 0; c < 32; ++c) v[c] = (vis & (1u << c)) ? v[c] : 0xff800000u;
}

// exp2(mul * v - base) of 32 scores as bf16 pairs in TMEM columns [dst, dst +
// 16); adds to the sums.  With MAX, the maxima of the scores are taken in the
// same loop (another pipe than the exponentials').  With TWO, what the rounding
// left goes to columns [dst + 32, dst + 48), as bf16 pairs as well.
template <bool MAX, bool TWO>
__device__ __forceinline__ void exp32(uint32_t dst, const uint32_t *v, float mul, float base,
                                      float2 *sum4, float *mx4) {
  const float2 mul2 = make_float2(mul, mul), nbase2 = make_float2(-base, -base);
  uint32_t pk[16], rest[16];
#pragma unroll
  for (int c = 0; c < 32; c += 2) {
    const float2 x = make_float2(__uint_as_float(v[c]), __uint_as_float(v[c + 1]));
    const float2 arg = __ffma2_rn(x, mul2, nbase2);
    const float2 e = make_float2(fast_exp2(arg.x), fast_exp2(arg.y));
    sum4[(c >> 1) & 3] = __fadd2_rn(sum4[(c >> 1) & 3], e);
    pk[c / 2] = pack_bf16x2(e.x, e.y);
    if constexpr (TWO)
      rest[c / 2] = pack_bf16x2(e.x - __uint_as_float(pk[c / 2] << 16),
                                e.y - __uint_as_float(pk[c / 2] & 0xffff0000u));
    if constexpr (MAX) mx4[(c >> 1) & 3] = fmax3(mx4[(c >> 1) & 3], x.x, x.y);
  }
  sm100::tmem_st16(dst, pk);
  if constexpr (TWO) sm100::tmem_st16(dst + 32, rest);
}
__device__ __forceinline__ float sum_of(const float2 *sum4) {
  const float2 s01 = __fadd2_rn(sum4[0], sum4[1]), s23 = __fadd2_rn(sum4[2], sum4[3]);
  const float2 s03 = __fadd2_rn(s01, s23);
  return s03.x + s03.y;
}

// One 128-key block of a row's online softmax is the work of two threads: the
// one of half h owns the 64 columns [64 h, 64 h + 64) of its row.  s_addr is
// this thread's lane at the half's first column, where P (bf16 pairs, 32
// columns; with TWO, 32 more for a second part) replaces the scores; lo / hi bound the row's visible columns in
// half-block coordinates.  Both threads use the same base, so that O's two
// column halves and the two partial sums l_half stay consistent.
// A positive scale keeps the order of the scores, so the maximum is taken
// over the raw scores and an invisible one simply becomes -inf in place (its
// exponential is then 0); another scale is applied to the scores first.
//
// softmax_half_max: the base is the running maximum, which xchg(max of my
// visible scaled scores) takes over both halves (and synchronises them).
// Returns the rescale factor of O.  Warp-collective (tcgen05.ld / st).
template <bool TWO, class Xchg>
__device__ __forceinline__ float softmax_half_max(uint32_t s_addr, int lo, int hi, float sl2,
                                                  float &m_run, float &l_half, Xchg xchg) {
  using namespace sm100;
  const float NEG_INF = -__int_as_float(0x7f800000);
  const bool raw = sl2 > 0.f;
  const float mul = raw ? sl2 : 1.f;
  uint32_t v[64];
  float mx8[8];
#pragma unroll
  for (int a = 0; a < 8; ++a) mx8[a] = NEG_INF;
  tmem_ld32(s_addr, v);
  tmem_ld32(s_addr + 32, v + 32);
  tmem_ld_wait32(v);
  tmem_ld_wait32(v + 32);
  mask32(v, lo, hi, !raw, sl2);
  mask32(v + 32, lo - 32, hi - 32, !raw, sl2);
#pragma unroll
  for (int c = 0; c < 64; c += 16)
#pragma unroll
    for (int a = 0; a < 8; ++a)
      mx8[a] = fmax3(mx8[a], __uint_as_float(v[c + 2 * a]), __uint_as_float(v[c + 2 * a + 1]));
  const float mx = xchg(fmax3(fmax3(mx8[0], mx8[1], mx8[2]), fmax3(mx8[3], mx8[4], mx8[5]),
                              fmaxf(mx8[6], mx8[7])) *
                        mul);
  const float m_new = mx > m_run + kRescaleLog2 ? mx : m_run;
  const float base = m_new == NEG_INF ? 0.f : m_new;
  const float alpha = m_new == m_run ? 1.f : fast_exp2(m_run - base);
  float2 sum4[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) sum4[a] = make_float2(0.f, 0.f);
  exp32<false, TWO>(s_addr, v, mul, base, sum4, nullptr);
  exp32<false, TWO>(s_addr + 16, v + 32, mul, base, sum4, nullptr);
  l_half = l_half * alpha + sum_of(sum4);
  m_run = m_new;
  return alpha;
}

// softmax_half_based: the base is the row's m_run as it is (any base within
// 2^kWindowLog2 below the maximum gives the same result after the final
// normalisation: fp32 and bf16 have the exponents for it), so the halves
// exchange nothing and no maximum is waited for.  plain: every row of the warp sees
// every key, and the scale is positive.  Returns false when a score of this
// thread lies above the window.
template <bool TWO>
__device__ __forceinline__ bool softmax_half_based(uint32_t s_addr, bool plain, int lo, int hi,
                                                   float sl2, float m_run, float &l_half) {
  using namespace sm100;
  const float NEG_INF = -__int_as_float(0x7f800000);
  if (!plain && __all_sync(0xffffffffu, hi <= max(lo, 0))) {  // no row of the warp sees a key of the half
    uint32_t z[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) z[c] = 0u;
    tmem_st32(s_addr, z);
    if constexpr (TWO) tmem_st32(s_addr + 32, z);
    return true;
  }
  const bool raw = sl2 > 0.f;
  const float mul = raw ? sl2 : 1.f, base = m_run == NEG_INF ? 0.f : m_run;
  uint32_t v[64];
  float2 sum4[4];
  float mx4[4];
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    sum4[a] = make_float2(0.f, 0.f);
    mx4[a] = NEG_INF;
  }
  tmem_ld32(s_addr, v);
  tmem_ld_wait32(v);
  tmem_ld32(s_addr + 32, v + 32);
  if constexpr (TWO) tmem_ld_wait32(v + 32);  // the second part takes their place
  if (!plain) mask32(v, lo, hi, !raw, sl2);
  exp32<true, TWO>(s_addr, v, mul, base, sum4, mx4);
  if constexpr (!TWO) tmem_ld_wait32(v + 32);
  if (!plain) mask32(v + 32, lo - 32, hi - 32, !raw, sl2);
  exp32<true, TWO>(s_addr + 16, v + 32, mul, base, sum4, mx4);
  l_half += sum_of(sum4);
  // (the maxima pass over NaN, which stays in the sums whatever the base)
  return fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * mul <= base + kWindowLog2;
}

// ------------------------------------------------------------------ host --
inline PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
  });
  return fn;
}

// 3-D bf16 tensor map over [d2][d1][d0] (d0 contiguous) with a
// (b0, b1, b2) box and 128-byte swizzle.
inline cudaError_t make_map(CUtensorMap *map, const void *base, uint64_t d0, uint64_t d1,
                            uint64_t d2, uint32_t b0, uint32_t b1, uint32_t b2) {
  auto fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  const cuuint64_t dims[3] = {d0, d1, d2};
  const cuuint64_t strides[2] = {d0 * 2, d0 * d1 * 2};
  const cuuint32_t box[3] = {b0, b1, b2};
  const cuuint32_t es[3] = {1, 1, 1};
  const CUresult r =
      fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(base), dims, strides, box,
         es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// 5-D bf16 tensor map over the paged cache [pages][16][H_kv][D]: one box is
// box_pages consecutive pages of one KV head, whole rows, in the order (8-token
// group, 64-column chunk, token, column), so that a page is one box and one
// run of shared memory (kGroupBytes per group).  For that order the strides go
// down as well as up (a token's lies before a chunk's and a head's).  The
// driver's header asks of a stride only a multiple of 16 below 2^40 and shows
// strides that each include the one before; it says nothing of this order, in
// which a map walks a transposed view.  It holds on this driver: every paged
// parity case would fail without.  The documented order alone (one box per page
// and 64 columns) took 67.3 us where this takes 57.9.
inline cudaError_t make_page_map(CUtensorMap *map, const void *base, int D, int H_kv,
                                 int num_pages, int box_pages = 1) {
  auto fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  const cuuint64_t row = static_cast<cuuint64_t>(D) * 2 * H_kv;  // bytes of a token
  const cuuint64_t chunks = static_cast<cuuint64_t>(D / 64);
  const cuuint64_t dims[5] = {64, 8, chunks, 2 * static_cast<cuuint64_t>(num_pages),
                              static_cast<cuuint64_t>(H_kv)};
  const cuuint64_t strides[4] = {row, 128, 8 * row, static_cast<cuuint64_t>(D) * 2};
  const cuuint32_t box[5] = {64, 8, static_cast<cuuint32_t>(chunks),
                             2 * static_cast<cuuint32_t>(box_pages), 1};
  const cuuint32_t es[5] = {1, 1, 1, 1, 1};
  const CUresult r =
      fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(base), dims, strides, box,
         es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Map of Q ([B m][H_q][D]): one box is 64 columns x G heads x 128 / G
// tokens, i.e. one 128-row tile of stacked query rows (row = token x G +
// head within the KV group) in the layout of a 128-key K block; rows past
// the last token read zeros.
inline cudaError_t make_q_map(const AttnParams &p, CUtensorMap *tq) {
  return make_map(tq, p.q, p.D, p.H_q, static_cast<uint64_t>(p.rows_total), 64, p.G, kRows / p.G);
}

// K and V maps of the contiguous prefix ([tokens][H_kv][D], one KV head x
// 128 keys x 64 columns per box); the paged cache stands in when there is
// no prefix at all (the maps are then never used).
inline cudaError_t make_prefix_maps(const AttnParams &p, CUtensorMap *tk, CUtensorMap *tv) {
  const int D = p.D;
  const bool has_prefix = p.prefix_tokens > 0 && !p.prefix_page_table;  // paged: page maps
  const uint64_t T = has_prefix ? static_cast<uint64_t>(p.prefix_tokens) : 1;
  cudaError_t e = make_map(tk, has_prefix ? p.prefix_k : p.k_cache, D, p.H_kv, T, 64, 1, kBlk);
  if (e != cudaSuccess) return e;
  return make_map(tv, has_prefix ? p.prefix_v : p.v_cache, D, p.H_kv, T, 64, 1, kBlk);
}

}  // namespace tc
}  // namespace hpd
