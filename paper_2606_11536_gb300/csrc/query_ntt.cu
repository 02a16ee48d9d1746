// query_ntt.cu -- the forward NTT of a batch's queries straight into the GEMMs' digit operand.
//
// The tensor GEMMs read the queries as 16-bit digits in core-matrix blocks, 16 bytes of
// eight ciphertexts' digits each (gemm_digit.cu, gemm_tc.cu).  A CTA transforms those eight rows
// of one query component and prime and writes 64 bytes (the four digits) per slot, so that
// the NTT-form residues never reach memory: per residue 4 bytes are read and 8 written where the
// separate transpose wrote and read 4 more.
//
// Eight rows of n words do not leave room for several CTAs per SM, which writing while others
// compute needs.  The passes below the top four bits stay within blocks of n/16 elements, so a
// CTA takes 2048 slots: it reads whole rows, and of the stages on the top bits computes the one
// output of each butterfly that leads to its slots (n = 2^12: 40 butterfly outputs' products
// where one CTA would take 32).  The CTAs of a row are neighbours and share its read in L2.
//
// No unit is full (n = 2^11: shared-memory wavefronts 65%, issue 47%, multiply-add pipe 46%, DRAM
// 44%): phases of loads, transform, digits and stores between block barriers.
// Transform and transpose -> this: n = 2^12, 32 queries x 2048 x L = 2 4.80 -> 4.04 ms (12.9 GB), bf16
// 32 x 512 1201 -> 993 us; n = 2^11, 32 x 512 605 -> 489 us; L = 3, 3 x 301 134 -> 101 us.  Three CTAs per SM
// at 40 registers for n >= 2^12; n = 2^11 spills there and takes two (620 -> 489 us).
#include <atomic>

#include <cuda_fp16.h>

#include "ntt_row.cuh"

namespace gbpir {
namespace {

constexpr int kSlots = 2048, kPadSlots = kSlots + kSlots / 16, kCtaThreads = 512, kRowThreads = 128;

struct QueryArgs {
  const uint32_t *queries;  // [B][D1][2][L][n], coefficient form
  uint16_t *qt;             // [L n][Uc][4 Mp][16]
  uint32_t M, Mp, D1, i0, Kc, L;
  NttConst ntt;
};

// One output of a butterfly with the pair p: x + t, or x - t + 2q.
__device__ __forceinline__ uint32_t bfly_half(uint32_t x, uint32_t y, uint2 p, bool upper, uint32_t q) {
  const uint32_t t = shoup_mul(y, p.x, p.y, q);
  return csub(x, 2 * q) + (upper ? 2 * q - t : t);
}

// Bits LOGN - 1 .. LOGN - 4 of unit lo, the 16 >> (LOGN - 11) outputs among slots 2048 part ...
template <int LOGN>
__device__ __forceinline__ void first_pass(uint32_t *row, const uint32_t *src, bool valid, uint32_t part,
                                           uint32_t lo, const uint2 *__restrict__ tw, uint32_t q) {
  constexpr int BLO = LOGN - 4, TOP = LOGN - 11, OUT = 16 >> TOP;
  uint32_t v[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) v[e] = valid ? src[lo + ((uint32_t)e << BLO)] : 0u;
#pragma unroll
  for (int t = 0; t < TOP; ++t) {
    const uint2 p = __ldg(tw + (1u << t) + (part >> (TOP - t)));
    const bool upper = (part >> (TOP - 1 - t)) & 1;
#pragma unroll
    for (int e = 0; e < (8 >> t); ++e) v[e] = bfly_half(v[e], v[e + (8 >> t)], p, upper, q);
  }
  uint32_t w[OUT];
#pragma unroll
  for (int e = 0; e < OUT; ++e) w[e] = v[e];
  fwd_stages<4 - TOP, BLO, LOGN>(w, part, tw, q);
  const uint32_t base = part * kSlots + lo, pbase = padx<LOGN>(base);
#pragma unroll
  for (int e = 0; e < OUT; ++e) row[pidx<LOGN, BLO>(pbase, base, e)] = w[e];
}

// BF16: the tensor layout's digits (k in order); else f16, in order or as k_query_digits pairs them.
template <int LOGN, bool BF16, bool IN_ORDER>
__global__ void __launch_bounds__(kCtaThreads, LOGN == 11 ? 2 : 3) k_ntt_query_digits(const QueryArgs a) {
  constexpr int N = 1 << LOGN, PARTS = N / kSlots;
  extern __shared__ uint32_t sm[];
  const uint32_t part = blockIdx.x % PARTS, mh = blockIdx.x / PARTS, h = mh & 1, m = mh >> 1;
  const uint32_t u = blockIdx.y, j = blockIdx.z, tid = threadIdx.x;
  const auto ciphertext = [&](uint32_t e) {  // of position 8h + e of the 16
    return 16 * u + (IN_ORDER ? 8 * h + e : 4 * h + 2 * (e >> 2) + (e & 1) + 8 * ((e >> 1) & 1));
  };
  chain_wait();
  const bool any = m < a.M && ciphertext(0) < a.Kc;  // the least of the eight
  const uint32_t slot0 = tid >> 1, dig = 2 * (tid & 1);  // two digits of a slot per thread
  const uint64_t slot_step = (uint64_t)gridDim.y * a.Mp * 64;
  uint16_t *dst = a.qt + ((uint64_t)j * N + part * kSlots + slot0) * slot_step + (uint64_t)u * a.Mp * 64 +
                  (m >> 1) * 128 + h * 64 + (m & 1) * 32 + 8 * dig;
  if (!any) {
    const uint32_t zero[8] = {};
#pragma unroll 4
    for (uint32_t k = 0; k < kSlots / (kCtaThreads / 2); ++k, dst += (kCtaThreads / 2) * slot_step)
      st_global32(reinterpret_cast<uint32_t *>(dst), zero);
    return;
  }
  const uint32_t q = pick(a.ntt.q, j), grp = tid / kRowThreads, t = tid % kRowThreads;
  const uint2 *tw = pick(a.ntt.fwd, j);
  const uint32_t back = padx<LOGN>(part * kSlots);  // slot 2048 part is the buffer's first
#pragma unroll 1
  for (uint32_t e = grp; e < 8; e += kCtaThreads / kRowThreads) {
    const uint32_t i = ciphertext(e);
    const uint32_t *src = a.queries + ((((uint64_t)(m >> 1) * a.D1 + a.i0 + i) * 2 + (m & 1)) * a.L + j) * N;
#pragma unroll 1
    for (uint32_t it = 0; it < PARTS; ++it)
      first_pass<LOGN>(sm + e * kPadSlots - back, src, i < a.Kc, part, t + it * kRowThreads, tw, q);
  }
  __syncthreads();
#pragma unroll 1
  for (uint32_t e = grp; e < 8; e += kCtaThreads / kRowThreads) {
    uint32_t *row = sm + e * kPadSlots - back, v[16];
    const uint32_t unit = part * kRowThreads + t;
    mid_pass<LOGN, LOGN - 8, true>(row, tw, q, unit);
    __syncwarp();
    fwd_last<LOGN>(row, tw, q, unit, v);
    __syncwarp();  // n = 2^13 reads its neighbours' words in the last pass
#pragma unroll
    for (int k = 0; k < 16; ++k) row[padx<LOGN>(16 * unit) + k] = v[k] + 0x00808080u;
  }
  __syncthreads();
  // two lanes a slot, two digit rows each: whole sectors
#pragma unroll 2
  for (uint32_t k = 0; k < kSlots / (kCtaThreads / 2); ++k, dst += (kCtaThreads / 2) * slot_step) {
    const uint32_t *x = sm + padx<LOGN>(slot0 + k * (kCtaThreads / 2));
    uint32_t b[8], o[8];  // 128 + signed digit in bytes 0..2, the top digit in byte 3
#pragma unroll
    for (int e = 0; e < 8; ++e) b[e] = x[e * kPadSlots];
#pragma unroll
    for (uint32_t r = 0; r < 2; ++r) {
      const uint32_t d = dig + r;
      if (BF16) {
        // the byte as the low bits of 2^23, less 2^23 and the bias: at most 8 significant bits,
        // so the top half of the f32 is the bf16 value
        const float bias = d == 3 ? 8388608.0f : 8388736.0f;
        const uint32_t sel = d | 0x7550;  // byte 0 = the digit, then zeros and the exponent
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float f0 = __uint_as_float(__byte_perm(b[2 * e], 0x4B000000u, sel)) - bias;
          const float f1 = __uint_as_float(__byte_perm(b[2 * e + 1], 0x4B000000u, sel)) - bias;
          o[4 * r + e] = __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
        }
      } else {
        const uint32_t sel = d | (4 + d) << 8;
        const __half2 bias = d == 3 ? __float2half2_rn(1024.0f) : __float2half2_rn(1152.0f);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          // two bytes under the exponent of 1024, less 1024 and the bias: exact in f16
          const uint32_t bits = (__byte_perm(b[2 * e], b[2 * e + 1], sel) & 0x00FF00FFu) | 0x64006400u;
          const __half2 f = __hsub2(*reinterpret_cast<const __half2 *>(&bits), bias);
          o[4 * r + e] = *reinterpret_cast<const uint32_t *>(&f);
        }
      }
    }
    st_global32(reinterpret_cast<uint32_t *>(dst), o);
  }
}

template <int LOGN, bool BF16, bool IN_ORDER>
cudaError_t query_launch(const QueryArgs &a, uint32_t Uc, cudaStream_t s) {
  constexpr int smem = 8 * kPadSlots * 4;
  const auto kernel = k_ntt_query_digits<LOGN, BF16, IN_ORDER>;
  static std::atomic<uint64_t> known{0};  // devices whose limit is raised
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 64 || !(known.load(std::memory_order_acquire) >> dev & 1)) {
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) return e;
    if (dev < 64) known.fetch_or(1ull << dev, std::memory_order_acq_rel);
  }
  return launch_chained(kernel, dim3((1u << LOGN) / kSlots * 2 * a.Mp, Uc, a.L), kCtaThreads, smem, s, a);
}

template <int LOGN>
cudaError_t query_layout(int layout, const QueryArgs &a, uint32_t Uc, cudaStream_t s) {
  if (layout == PIR_LAYOUT_TENSOR) return query_launch<LOGN, true, true>(a, Uc, s);
  if (layout == PIR_LAYOUT_LIMB) return query_launch<LOGN, false, true>(a, Uc, s);
  return query_launch<LOGN, false, false>(a, Uc, s);
}

}  // namespace

// Eight rows a CTA fill the SMs twice from 4096 rows on (5418: 134 -> 101 us); below, a transform
// of one row a CTA and the transpose are the shorter chain.
bool query_ntt_fuses(uint32_t L, uint32_t B, uint32_t Kc) { return (uint64_t)B * Kc * 2 * L >= 4096; }

cudaError_t launch_ntt_query_digits(const ParamCtx &c, int layout, const uint32_t *queries, uint32_t B, uint32_t D1,
                                    uint32_t i0, uint32_t Kc, uint32_t Mp, uint16_t *qt, cudaStream_t s) {
  const uint32_t Uc = layout == PIR_LAYOUT_TENSOR ? Kc / 16 : (Kc + 63) / 64 * 4;
  if (Mp % 4 != 0 || Kc == 0 || (layout == PIR_LAYOUT_TENSOR && Kc % 16 != 0) || Uc > 65535) return cudaErrorInvalidValue;
  QueryArgs a = {};
  a.queries = queries;
  a.qt = qt;
  a.M = 2 * B;
  a.Mp = Mp;
  a.D1 = D1;
  a.i0 = i0;
  a.Kc = Kc;
  a.L = c.p.L;
  a.ntt = c.ntt;
  switch (c.logn) {
    case 11: return query_layout<11>(layout, a, Uc, s);
    case 12: return query_layout<12>(layout, a, Uc, s);
    case 13: return query_layout<13>(layout, a, Uc, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace gbpir
