// ntt_row.cuh -- the radix-16 passes of a negacyclic NTT row, for the kernels that transform
// rows: a row's n/16 threads hold 16 residues each.  Included by one kernel file at a time.
#pragma once
#include "common.cuh"

namespace gbpir {
namespace {

// Shared positions are padded: one word in sixteen, or for n = 2^13 two in thirty-two, which
// is free of bank conflicts in every pass there (32 neighbours; 16 blocks of 32 by parity;
// the first leaves one lane pair in two wavefronts where a warp takes 32 neighbours).
template <int LOGN>
__device__ __forceinline__ uint32_t padx(uint32_t i) {
  return LOGN == 13 ? i + 2 * (i >> 5) : i + (i >> 4);
}

// Padded position of element e of a unit whose base index has bits [BLO, BLO + 4) clear:
// that of its base plus a constant where the padding adds up, so that the address is the
// unit's plus a compile-time offset.
template <int LOGN, int BLO>
__device__ __forceinline__ uint32_t pidx(uint32_t pbase, uint32_t base, int e) {
  if constexpr (LOGN == 13 ? BLO <= 1 || BLO >= 5 : BLO == 0 || BLO >= 4)
    return pbase + padx<LOGN>((uint32_t)e << BLO);
  else
    return padx<LOGN>(base + ((uint32_t)e << BLO));
}

// x - m if x >= m, else x (x < 2m <= 2^32): as unsigned values x - m wraps above x
// exactly when x < m, so the minimum picks the right one: one add-and-minimum instruction.
__device__ __forceinline__ uint32_t csub(uint32_t x, uint32_t m) { return __viaddmin_u32(x, 0u - m, x); }

// Element j < L of a per-prime parameter array, by compare and select: indexing a
// kernel parameter array with a run-time j makes the compiler copy the whole
// parameter block to local memory first.
template <typename T>
__device__ __forceinline__ T pick(const T (&a)[PIR_MAX_L], uint32_t j) {
  T r = a[0];
#pragma unroll
  for (uint32_t i = 1; i < PIR_MAX_L; ++i) r = j == i ? a[i] : r;
  return r;
}

// 32 bytes at once (a whole sector per thread; the address 32-byte aligned)
__device__ __forceinline__ void ld_global32(const uint32_t *p, uint32_t *v) {
  asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void st_global32(uint32_t *p, const uint32_t *v) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
               "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
// 16 consecutive words of a row: rows start on 16-byte boundaries only
__device__ __forceinline__ void load16(const uint32_t *p, uint32_t (&v)[16], bool wide) {
  if (wide) {
    ld_global32(p, v);
    ld_global32(p + 8, v + 8);
  } else {
#pragma unroll
    for (int e = 0; e < 16; e += 4) {
      const uint4 x = *reinterpret_cast<const uint4 *>(p + e);
      v[e] = x.x, v[e + 1] = x.y, v[e + 2] = x.z, v[e + 3] = x.w;
    }
  }
}
__device__ __forceinline__ void store16(uint32_t *p, const uint32_t (&v)[16], bool wide) {
  if (wide) {
    st_global32(p, v);
    st_global32(p + 8, v + 8);
  } else {
#pragma unroll
    for (int e = 0; e < 16; e += 4) *reinterpret_cast<uint4 *>(p + e) = make_uint4(v[e], v[e + 1], v[e + 2], v[e + 3]);
  }
}
__device__ __forceinline__ bool wide_ok(const void *p) { return ((uintptr_t)p & 31u) == 0; }

// Twiddle pairs {w, Shoup companion} used by one stage of one radix-2^RB unit.
// Stage bit b pairs (x, x + 2^b); the pair belongs to block g = index >> (b+1) and
// uses twiddle m + g, m = n >> (b+1).  Within a unit the blocks of stage LB are the
// 2^(RB-1-LB) consecutive entries from m + (hi << (RB-1-LB)), a run aligned to its
// own length, so they arrive in 16-byte loads (8 bytes for a single pair).
template <int CNT>
struct Pairs {  // CNT twiddle pairs held as whole 16-byte vectors (8 bytes when CNT = 1)
  uint4 v[(CNT + 1) / 2];
  __device__ __forceinline__ void load(const uint2 *__restrict__ src) {
    if constexpr (CNT == 1) {
      const uint2 x = __ldg(src);
      v[0] = make_uint4(x.x, x.y, 0u, 0u);
    } else {
#pragma unroll
      for (int i = 0; i < CNT / 2; ++i) v[i] = __ldg(reinterpret_cast<const uint4 *>(src) + i);
    }
  }
  // CNT pairs as CNT/2 16-byte loads spaced `stride` 16-byte words apart (the
  // lane-major copy: load i of every thread is one contiguous run)
  __device__ __forceinline__ void load_lane_major(const uint4 *__restrict__ src, uint32_t stride) {
#pragma unroll
    for (int i = 0; i < CNT / 2; ++i) v[i] = __ldg(src + (size_t)i * stride);
  }
  template <int I>
  __device__ __forceinline__ uint32_t w() const { return (I & 1) ? v[I / 2].z : v[I / 2].x; }
  template <int I>
  __device__ __forceinline__ uint32_t ws() const { return (I & 1) ? v[I / 2].w : v[I / 2].y; }
};

// One forward (Cooley-Tukey) butterfly of stage LB on elements E and E + 2^LB.
template <int RB, int LB, int E, int CNT>
__device__ __forceinline__ void fwd_bfly(uint32_t (&v)[1 << RB], const Pairs<CNT> &p, uint32_t q) {
  if constexpr (E < (1 << RB)) {
    if constexpr ((E & (1 << LB)) == 0) {
      const uint32_t q2 = 2 * q;
      uint32_t x = v[E];
      const uint32_t y = v[E | (1 << LB)];
      x = csub(x, q2);                                                              // [0, 2q)
      const uint32_t t = shoup_mul(y, p.template w<(E >> (LB + 1))>(), p.template ws<(E >> (LB + 1))>(), q);  // [0, 2q)
      // x - t + 2q as 2x + 2q - (x + t): two instructions either way, but in this form the
      // compiler's butterfly issues in 3.9 cycles per warp against 5.8
      const uint32_t s = x + t;
      v[E] = s;                                                                     // [0, 4q)
      v[E | (1 << LB)] = x + x + q2 - s;                                            // (0, 4q)
    }
    fwd_bfly<RB, LB, E + 1, CNT>(v, p, q);
  }
}

// One forward stage on the unit's bit BLO + LB.
template <int RB, int BLO, int LOGN, int LB>
__device__ __forceinline__ void fwd_stage(uint32_t (&v)[1 << RB], uint32_t hi, const uint2 *__restrict__ tw,
                                          uint32_t q) {
  constexpr int CNT = 1 << (RB - 1 - LB);
  constexpr uint32_t m = 1u << (LOGN - 1 - (BLO + LB));
  Pairs<CNT> p;
  if constexpr (BLO == 0 && RB == 4 && LB <= 1) {  // the lane-major copy after the table
    constexpr uint32_t units = 1u << (LOGN - 4);
    p.load_lane_major(reinterpret_cast<const uint4 *>(tw + (1u << LOGN)) + (LB == 0 ? 0u : 4 * units) + hi, units);
  } else {
    p.load(tw + m + (hi << (RB - 1 - LB)));
  }
  fwd_bfly<RB, LB, 0, CNT>(v, p, q);
}

// Forward stages on one unit: bits BLO+RB-1 down to BLO of the element index.
template <int RB, int BLO, int LOGN, int LB = RB - 1>
__device__ __forceinline__ void fwd_stages(uint32_t (&v)[1 << RB], uint32_t hi, const uint2 *__restrict__ tw,
                                           uint32_t q) {
  fwd_stage<RB, BLO, LOGN, LB>(v, hi, tw, q);
  if constexpr (LB > 0) fwd_stages<RB, BLO, LOGN, LB - 1>(v, hi, tw, q);
}

// One inverse (Gentleman-Sande) butterfly of stage LB; values in [0, 2q).
template <int RB, int LB, int E, int CNT>
__device__ __forceinline__ void inv_bfly(uint32_t (&v)[1 << RB], const Pairs<CNT> &p, uint32_t q) {
  if constexpr (E < (1 << RB)) {
    if constexpr ((E & (1 << LB)) == 0) {
      const uint32_t q2 = 2 * q;
      const uint32_t x = v[E], y = v[E | (1 << LB)];
      const uint32_t s = x + y;
      v[E] = csub(s, q2);
      v[E | (1 << LB)] = shoup_mul(x + x + q2 - s, p.template w<(E >> (LB + 1))>(), p.template ws<(E >> (LB + 1))>(), q);
    }
    inv_bfly<RB, LB, E + 1, CNT>(v, p, q);
  }
}

// One inverse stage on bit BLO + LB.
template <int RB, int BLO, int LOGN, int LB>
__device__ __forceinline__ void inv_stage(uint32_t (&v)[1 << RB], uint32_t hi, const uint2 *__restrict__ tw,
                                          uint32_t q) {
  constexpr int CNT = 1 << (RB - 1 - LB);
  constexpr uint32_t m = 1u << (LOGN - 1 - (BLO + LB));
  Pairs<CNT> p;
  if constexpr (BLO == 0 && RB == 4 && LB <= 1) {  // the lane-major copy after the table
    constexpr uint32_t units = 1u << (LOGN - 4);
    p.load_lane_major(reinterpret_cast<const uint4 *>(tw + (1u << LOGN)) + (LB == 0 ? 0u : 4 * units) + hi, units);
  } else {
    p.load(tw + m + (hi << (RB - 1 - LB)));
  }
  inv_bfly<RB, LB, 0, CNT>(v, p, q);
}

// Inverse stages on one unit: bits BLO up to BLO+RB-1.
template <int RB, int BLO, int LOGN, int LB = 0>
__device__ __forceinline__ void inv_stages(uint32_t (&v)[1 << RB], uint32_t hi, const uint2 *__restrict__ tw,
                                           uint32_t q) {
  inv_stage<RB, BLO, LOGN, LB>(v, hi, tw, q);
  if constexpr (LB < RB - 1) inv_stages<RB, BLO, LOGN, LB + 1>(v, hi, tw, q);
}

// The passes of one row by T = n/16 threads, 16 residues v each.  sm is the row's shared
// buffer (padded).

// Forward, bits LOGN - 1 .. LOGN - 4 of the elements load(idx), into shared memory.
template <int LOGN, typename Load>
__device__ __forceinline__ void fwd_first(uint32_t *sm, Load load, const uint2 *__restrict__ tw, uint32_t q,
                                          uint32_t tid) {
  constexpr int BLO = LOGN - 4;
  uint32_t v[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) v[e] = load(tid + ((uint32_t)e << BLO));
  fwd_stages<4, BLO, LOGN>(v, 0, tw, q);
  const uint32_t pbase = padx<LOGN>(tid);
#pragma unroll
  for (int e = 0; e < 16; ++e) sm[pidx<LOGN, BLO>(pbase, tid, e)] = v[e];
}

// A radix-16 pass on bits BLO .. BLO + 3, shared memory to shared memory.
template <int LOGN, int BLO, bool FWD>
__device__ __forceinline__ void mid_pass(uint32_t *sm, const uint2 *__restrict__ tw, uint32_t q, uint32_t tid) {
  const uint32_t lo = tid & ((1u << BLO) - 1), hi = tid >> BLO, base = (hi << (BLO + 4)) | lo, pbase = padx<LOGN>(base);
  uint32_t v[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) v[e] = sm[pidx<LOGN, BLO>(pbase, base, e)];
  if constexpr (FWD)
    fwd_stages<4, BLO, LOGN>(v, hi, tw, q);
  else
    inv_stages<4, BLO, LOGN>(v, hi, tw, q);
#pragma unroll
  for (int e = 0; e < 16; ++e) sm[pidx<LOGN, BLO>(pbase, base, e)] = v[e];
}

// The 8 twiddle pairs of bit 0 for elements 16 tid .. 16 tid + 15 (the lane-major copy).
template <int LOGN>
__device__ __forceinline__ void bit0_twiddles(Pairs<8> &p, const uint2 *__restrict__ tw, uint32_t tid) {
  p.load_lane_major(reinterpret_cast<const uint4 *>(tw + (1u << LOGN)) + tid, 1u << (LOGN - 4));
}

// Forward, the bits below; v becomes elements 16 tid .. 16 tid + 15 of the result, canonical.
// n = 2^13: bits 4..1 give thread tid the elements of one parity of 32 consecutive ones;
// neighbours trade halves and take the pairs of bit 0.
template <int LOGN>
__device__ __forceinline__ void fwd_last(const uint32_t *sm, const uint2 *__restrict__ tw, uint32_t q, uint32_t tid,
                                         uint32_t (&v)[16]) {
  if constexpr (LOGN == 13) {
    const uint32_t lo = tid & 1, hi = tid >> 1, base = (hi << 5) | lo, pbase = padx<LOGN>(base);
    uint32_t w[16];
#pragma unroll
    for (int e = 0; e < 16; ++e) w[e] = sm[pidx<LOGN, 1>(pbase, base, e)];
    fwd_stages<4, 1, LOGN>(w, hi, tw, q);
    Pairs<8> p;
    bit0_twiddles<LOGN>(p, tw, tid);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t got = __shfl_xor_sync(0xffffffffu, lo ? w[i] : w[i + 8], 1);
      v[2 * i] = lo ? got : w[i];
      v[2 * i + 1] = lo ? w[i + 8] : got;
    }
    fwd_bfly<4, 0, 0, 8>(v, p, q);
  } else {
    const uint32_t pbase = padx<LOGN>(16 * tid);
#pragma unroll
    for (int e = 0; e < 16; ++e) v[e] = sm[pbase + e];
    if constexpr (LOGN == 12) {
      fwd_stages<4, 0, LOGN>(v, tid, tw, q);
    } else {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        uint32_t w[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) w[e] = v[8 * r + e];
        fwd_stages<3, 0, LOGN>(w, 2 * tid + r, tw, q);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[8 * r + e] = w[e];
      }
    }
  }
#pragma unroll
  for (int e = 0; e < 16; ++e) v[e] = csub(csub(v[e], 2 * q), q);
}

// The forward transform of one row; v as fwd_last leaves it.
template <int LOGN, typename Load>
__device__ __forceinline__ void fwd_row(uint32_t *sm, Load load, const uint2 *__restrict__ tw, uint32_t q, uint32_t tid,
                                        uint32_t (&v)[16]) {
  fwd_first<LOGN>(sm, load, tw, q, tid);
  __syncthreads();
  mid_pass<LOGN, LOGN - 8, true>(sm, tw, q, tid);
  __syncwarp();
  fwd_last<LOGN>(sm, tw, q, tid, v);
}

// Inverse, bits 0 .. 3 (n = 2^13: 0 .. 4) of elements 16 tid .. 16 tid + 15 in v, into shared
// memory.
template <int LOGN>
__device__ __forceinline__ void inv_first(uint32_t *sm, const uint2 *__restrict__ tw, uint32_t q, uint32_t tid,
                                          uint32_t (&v)[16]) {
  if constexpr (LOGN == 13) {
    const uint32_t lo = tid & 1, hi = tid >> 1, base = (hi << 5) | lo, pbase = padx<LOGN>(base);
    Pairs<8> p;
    bit0_twiddles<LOGN>(p, tw, tid);
    inv_bfly<4, 0, 0, 8>(v, p, q);
    uint32_t w[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t got = __shfl_xor_sync(0xffffffffu, lo ? v[2 * i] : v[2 * i + 1], 1);
      w[i] = lo ? got : v[2 * i];
      w[i + 8] = lo ? v[2 * i + 1] : got;
    }
    inv_stages<4, 1, LOGN>(w, hi, tw, q);
#pragma unroll
    for (int e = 0; e < 16; ++e) sm[pidx<LOGN, 1>(pbase, base, e)] = w[e];
  } else {
    inv_stages<4, 0, LOGN>(v, tid, tw, q);
    const uint32_t pbase = padx<LOGN>(16 * tid);
#pragma unroll
    for (int e = 0; e < 16; ++e) sm[pbase + e] = v[e];
  }
}

// Inverse, the top bits, times n^-1, canonical; element idx goes to out(idx, value).
template <int LOGN, typename Out>
__device__ __forceinline__ void inv_last(const uint32_t *sm, const uint2 *__restrict__ tw, uint32_t q, uint32_t ninv,
                                         uint32_t ninv_sh, uint32_t tid, Out out) {
  constexpr int RB = LOGN == 11 ? 3 : 4, BLO = LOGN - RB, PER = 16 >> RB, T = 1 << (LOGN - 4);
#pragma unroll
  for (int r = 0; r < PER; ++r) {
    const uint32_t lo = tid + r * T, pbase = padx<LOGN>(lo);
    uint32_t v[1 << RB];
#pragma unroll
    for (int e = 0; e < (1 << RB); ++e) v[e] = sm[pidx<LOGN, BLO>(pbase, lo, e)];
    inv_stages<RB, BLO, LOGN>(v, 0, tw, q);
#pragma unroll
    for (int e = 0; e < (1 << RB); ++e)
      out(lo + ((uint32_t)e << BLO), csub(shoup_mul(v[e], ninv, ninv_sh, q), q));
  }
}

}  // namespace
}  // namespace gbpir
