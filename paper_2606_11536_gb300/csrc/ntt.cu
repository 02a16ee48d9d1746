// ntt.cu -- forward / inverse negacyclic NTT over 30-bit primes (Sec. 2.3; the
// paper's single-kernel, on-chip NTT, Sec. 4.3).
//
// One CTA transforms one polynomial row of n residues (row r uses prime r % L).
// Each thread holds 16 residues in registers and applies four butterfly stages
// to them; the rows pass through shared memory (padded one word in sixteen) between
// such radix-16 passes: n = 2^11 -> 4+4+3 bits, 2^12 -> 4+4+4, 2^13 -> 4+4+4+1 (the last
// bit between neighbouring threads, by shuffles).  Only the pass over the top bits mixes
// elements of different warps: the others stay within blocks of n/16 elements that one
// warp holds, so a row takes one block barrier and a warp barrier per further pass.
//
// Arithmetic: twiddles are psi^brv(i) (forward) and psi^-brv(i) (inverse) with
// Shoup companions floor(w * 2^32 / q), so each twiddle product is one high and
// two low 32-bit multiplies.  Butterflies keep values lazily reduced (Harvey):
// forward values live in [0, 4q), inverse values in [0, 2q); 4q < 2^32 because
// q < 2^30.  The last pass reduces to canonical [0, q) (and, for the inverse,
// multiplies by n^-1).
//
// Output order: forward NTT(a)[k] = sum_t a_t psi^((2 brv(k) + 1) t), the natural
// result of decimation in time with psi powers in bit-reversed order.
//
// Bound by the multiply-add pipe (a butterfly's high product and two low ones; 71 to 73% active),
// the shared-memory wavefronts (64 to 70%) and the issue slots (66%) together: 2 GiB of rows,
// n = 2^12, forward 1393 -> 1140 us (3.8 TB/s), n = 2^13, inverse 1610 -> 1315 us, with row numbers
// divided by multiplication instead of 64-bit divisions (a sixth of all instructions), one block
// barrier a row, whole-sector stores.
#include "ntt_row.cuh"

namespace gbpir {
namespace {

// Source kinds of the first pass.
enum { SRC_U32 = 1, SRC_RAW = 2 };

struct RawSrc {
  const uint8_t *raw;  // little-endian bit stream of log2p-bit coefficients
  uint64_t poly0;      // row-major order: local polynomial p is poly0 + p
  uint32_t log2p;
  uint32_t col_major;  // 1: local polynomial p is (i, c) = (p % D1, c0 + p / D1)
  uint32_t D1, D2;
  uint64_t c0;
  __device__ __forceinline__ uint64_t poly(uint64_t p) const {
    return col_major ? (p % D1) * D2 + (c0 + p / D1) : poly0 + p;
  }
};

// Source rows of a launch: local row r reads source row off + (r / G) * S + (r % G) * T, so
// a chunk of ciphertexts can be taken out of every query of a batch without a copy.  Row
// numbers stay below 2^31 (a row is 8 KiB at least).
struct RowMap {
  uint32_t off, S, T;
  FastDiv G, L;  // L: the row's prime is r % L
  RowMap() = default;
  RowMap(uint64_t o, uint64_t g, uint64_t s, uint64_t t, uint32_t l)
      : off((uint32_t)o), S((uint32_t)s), T((uint32_t)t), G(g), L(l) {}
  __device__ __forceinline__ uint64_t operator()(uint32_t r) const {
    const uint32_t g = G.div(r);
    return off + (uint64_t)g * S + (r - g * G.d) * T;
  }
};

// Coefficient `t` of plaintext polynomial `poly` from the raw bit stream.
__device__ __forceinline__ uint32_t raw_coeff(const RawSrc &rs, uint64_t poly, uint32_t t, uint32_t logn) {
  const uint64_t bit0 = ((poly << logn) + t) * rs.log2p;
  const uint64_t byte0 = bit0 >> 3;
  const uint32_t nbytes = (uint32_t)(((bit0 & 7) + rs.log2p + 7) >> 3);
  uint64_t w = 0;
  for (uint32_t b = 0; b < nbytes; ++b) w |= (uint64_t)rs.raw[byte0 + b] << (8 * b);
  return (uint32_t)((w >> (bit0 & 7)) & ((1ull << rs.log2p) - 1));
}

// CTAs per SM: 1280 threads for n = 2^11 and 2^12 (48 registers), 1536 for 2^13 (40; with two
// CTAs of 512 the inverse took 1562 instead of 1315 us on 2 GiB).
template <int LOGN>
constexpr int kNttCtas = LOGN == 13 ? 3 : 20480 >> LOGN;

template <int LOGN, int SRC>
__global__ void __launch_bounds__((1 << LOGN) / 16, kNttCtas<LOGN>)
    k_ntt_fwd(const uint32_t *src, RowMap rm, RawSrc rs, uint32_t *dst, NttConst C, uint32_t rows) {
  constexpr int N = 1 << LOGN;
  extern __shared__ uint32_t sm[];
  const bool wide = wide_ok(dst);
  chain_wait();
  for (uint32_t row = blockIdx.x; row < rows; row += gridDim.x) {
    const uint32_t p = rm.L.div(row), j = row - p * rm.L.d;
    const uint64_t poly = SRC == SRC_RAW ? rs.poly(p) : 0;
    uint32_t v[16];
    const uint32_t *gin = SRC == SRC_U32 ? src + rm(row) * N : nullptr;
    const auto load = [&](uint32_t i) { return SRC == SRC_U32 ? gin[i] : raw_coeff(rs, poly, i, LOGN); };
    fwd_row<LOGN>(sm, load, pick(C.fwd, j), pick(C.q, j), threadIdx.x, v);
    store16(dst + (uint64_t)row * N + 16 * threadIdx.x, v, wide);
    if (row + gridDim.x < rows) __syncthreads();  // the next row reuses shared memory
  }
}

template <int LOGN>
__global__ void __launch_bounds__((1 << LOGN) / 16, kNttCtas<LOGN>)
    k_ntt_inv(const uint32_t *src, RowMap rm, uint32_t *dst, NttConst C, uint32_t rows) {
  constexpr int N = 1 << LOGN;
  extern __shared__ uint32_t sm[];
  const uint32_t tid = threadIdx.x;
  const bool wide = wide_ok(src);
  chain_wait();
  for (uint32_t row = blockIdx.x; row < rows; row += gridDim.x) {
    const uint32_t j = rm.L.mod(row);
    const uint32_t q = pick(C.q, j);
    const uint2 *tw = pick(C.inv, j);
    uint32_t *gout = dst + (uint64_t)row * N;
    uint32_t v[16];
    load16(src + rm(row) * N + 16 * tid, v, wide);
    inv_first<LOGN>(sm, tw, q, tid, v);
    __syncwarp();
    mid_pass<LOGN, LOGN == 13 ? 5 : 4, false>(sm, tw, q, tid);
    __syncthreads();
    inv_last<LOGN>(sm, tw, q, pick(C.ninv, j), pick(C.ninv_sh, j), tid, [&](uint32_t i, uint32_t x) { gout[i] = x; });
    if (row + gridDim.x < rows) __syncthreads();
  }
}

// One coefficient switched to q_0 from its L canonical residues in shared memory
// (row j at sm + j * padn, position pt): Garner digits a_k of x mod Q', that value
// mod q_0 and its comparison with (Q' - 1) / 2 (digit by digit from the top), then
// y = (x_0 - (x mod Q')) Q'^-1 + [x mod Q' > (Q' - 1) / 2]  (mod q_0),
// which is round(x / Q') mod q_0: x = Q' floor(x / Q') + (x mod Q').  Every residue
// is below 2^30 < 2 q_k, so one conditional subtraction brings it under any q_k.
__device__ __forceinline__ uint32_t switch_coeff(const uint32_t *sm, uint32_t padn, uint32_t pt, const NttConst &C,
                                                 const SwitchConst &W, uint32_t L) {
  const uint32_t q0 = C.q[0];
  uint32_t a[PIR_MAX_L];
  uint32_t xm = 0;
#pragma unroll
  for (int k = 1; k < PIR_MAX_L; ++k) {
    a[k] = 0;
    if ((uint32_t)k < L) {
      const uint32_t qk = C.q[k];
      uint32_t t = sm[k * padn + pt];
#pragma unroll
      for (int i = 1; i < k; ++i) {
        const uint32_t ai = a[i] >= qk ? a[i] - qk : a[i];
        t = shoup_mul(t + qk - ai, W.c[k][i], W.c_sh[k][i], qk);
        t = t >= qk ? t - qk : t;
      }
      a[k] = t;
      const uint32_t ak = t >= q0 ? t - q0 : t;
      uint32_t pr = shoup_mul(ak, W.w[k], W.w_sh[k], q0);
      pr = pr >= q0 ? pr - q0 : pr;
      xm += pr;
      xm = xm >= q0 ? xm - q0 : xm;
    }
  }
  bool up = false, eq = true;
#pragma unroll
  for (int k = PIR_MAX_L - 1; k >= 1; --k)
    if ((uint32_t)k < L && eq && a[k] != W.h[k]) {
      up = a[k] > W.h[k];
      eq = false;
    }
  uint32_t y = shoup_mul(sm[pt] + q0 - xm, W.qinv, W.qinv_sh, q0);
  y = y >= q0 ? y - q0 : y;
  y += up ? 1u : 0u;
  return y >= q0 ? y - q0 : y;
}

// Inverse NTT with modulus switching fused into its epilogue (Sec. 4.3 fuses the
// modulus reduction into the inverse NTT; App. D.5 defines the switch): block c
// takes the L residue rows src + (c L + j) n of one polynomial (NTT form) and
// writes dst + c n, its coefficients over the single prime q_0.  2 x n/16 threads:
// half h inverts rows h, h + 2, ... into their own shared buffers (canonical), then
// all threads switch the coefficients, four per 16-byte store.
template <int LOGN>
__global__ void __launch_bounds__((1 << LOGN) / 8, LOGN == 13 ? 1 : 12288 >> LOGN)  // 1024 or 1536 threads per SM
    k_ntt_inv_switch(const uint32_t *src, uint32_t *dst, NttConst C, SwitchConst W, uint32_t L) {
  constexpr int N = 1 << LOGN, PADN = N + N / 16, T = N / 16;
  extern __shared__ uint32_t sm[];
  const uint32_t half = threadIdx.x / T, tid = threadIdx.x % T;
  const bool wide = wide_ok(src);
  chain_wait();
  for (uint32_t r = 0; r < (L + 1) / 2; ++r) {
    const uint32_t j = 2 * r + half;
    const bool act = j < L;  // the barriers below are reached by both halves
    const uint32_t jj = act ? j : 0;
    uint32_t *smh = sm + jj * PADN;
    const uint32_t q = pick(C.q, jj);
    const uint2 *tw = pick(C.inv, jj);
    if (act) {
      uint32_t v[16];
      load16(src + ((uint64_t)blockIdx.x * L + jj) * N + 16 * tid, v, wide);
      inv_first<LOGN>(smh, tw, q, tid, v);
      __syncwarp();
      mid_pass<LOGN, LOGN == 13 ? 5 : 4, false>(smh, tw, q, tid);
    }
    __syncthreads();
    // (the last pass reads and writes the same elements of a thread)
    if (act)
      inv_last<LOGN>(smh, tw, q, pick(C.ninv, jj), pick(C.ninv_sh, jj), tid,
                     [&](uint32_t i, uint32_t x) { smh[padx<LOGN>(i)] = x; });
    __syncthreads();
  }
  uint32_t *out = dst + (uint64_t)blockIdx.x * N;
  for (uint32_t g = threadIdx.x; g < (uint32_t)N / 4; g += blockDim.x) {
    const uint32_t pt = padx<LOGN>(4 * g);  // four consecutive positions stay consecutive
    uint4 y;
    y.x = switch_coeff(sm, PADN, pt + 0, C, W, L);
    y.y = switch_coeff(sm, PADN, pt + 1, C, W, L);
    y.z = switch_coeff(sm, PADN, pt + 2, C, W, L);
    y.w = switch_coeff(sm, PADN, pt + 3, C, W, L);
    *reinterpret_cast<uint4 *>(out + 4 * g) = y;
  }
}

// Forward NTT of the a- and b-polynomial of one ciphertext (rows (i, comp 0) and
// (i, comp 1) of prime j of a batch-1 query chunk), written straight into the
// slot-major layout [L*n][stride][2] that the batch-1 scan reads (column col0 + i): the transpose of
// Sec. 4.2 fused into the NTT.  Block = i * L + j, 2 x n/16 threads: each half
// transforms one row in its own shared buffer, then all threads write the pairs.
template <int LOGN>
__global__ void __launch_bounds__((1 << LOGN) / 8)
    k_ntt_fwd_pair_slots(const uint32_t *src, uint64_t row0, NttConst C, uint32_t L, uint32_t stride, uint32_t col0,
                         uint32_t *slots) {
  constexpr int N = 1 << LOGN, PADN = N + N / 16, T = N / 16;
  extern __shared__ uint32_t sm[];
  const uint32_t i = blockIdx.x / L, j = blockIdx.x % L;
  const uint32_t half = threadIdx.x / T, tid = threadIdx.x % T;
  uint32_t *smh = sm + half * PADN;
  const uint32_t q = pick(C.q, j);
  const uint2 *tw = pick(C.fwd, j);
  const uint32_t *gin = src + (row0 + (uint64_t)i * 2 * L + (uint64_t)half * L + j) * N;
  chain_wait();
  uint32_t v[16];
  fwd_row<LOGN>(smh, [&](uint32_t i) { return gin[i]; }, tw, q, tid, v);
  // n = 2^13 reads its neighbours' words in the last pass
  __syncwarp();
#pragma unroll
  for (int e = 0; e < 16; ++e) smh[padx<LOGN>(16 * tid) + e] = v[e];
  __syncthreads();
  uint32_t *dst = slots + ((uint64_t)j * N * stride + col0 + i) * 2;
  for (uint32_t k = threadIdx.x; k < (uint32_t)N; k += 2 * T)
    *reinterpret_cast<uint2 *>(dst + (uint64_t)k * stride * 2) = make_uint2(sm[padx<LOGN>(k)], sm[PADN + padx<LOGN>(k)]);
}

constexpr uint64_t kMaxGrid = 1u << 30, kMaxRows = 0x7fffffffull;

template <int LOGN>
cudaError_t fwd_launch(const ParamCtx &c, const uint32_t *src, const RowMap &rm, const RawSrc &rs, uint32_t *dst,
                       uint64_t rows, cudaStream_t s, bool raw) {
  const int T = (1 << LOGN) / 16;
  const size_t smem = ((1u << LOGN) + (1u << LOGN) / 16) * sizeof(uint32_t);
  const unsigned grid = (unsigned)(rows < kMaxGrid ? rows : kMaxGrid);
  if (raw)
    return launch_chained(k_ntt_fwd<LOGN, SRC_RAW>, grid, T, smem, s, nullptr, rm, rs, dst, c.ntt, (uint32_t)rows);
  return launch_chained(k_ntt_fwd<LOGN, SRC_U32>, grid, T, smem, s, src, rm, rs, dst, c.ntt, (uint32_t)rows);
}

template <int LOGN>
cudaError_t inv_launch(const ParamCtx &c, const uint32_t *src, const RowMap &rm, uint32_t *dst, uint64_t rows,
                       cudaStream_t s) {
  const int T = (1 << LOGN) / 16;
  const size_t smem = ((1u << LOGN) + (1u << LOGN) / 16) * sizeof(uint32_t);
  const unsigned grid = (unsigned)(rows < kMaxGrid ? rows : kMaxGrid);
  return launch_chained(k_ntt_inv<LOGN>, grid, T, smem, s, src, rm, dst, c.ntt, (uint32_t)rows);
}

cudaError_t fwd_any(const ParamCtx &c, const uint32_t *src, const RowMap &rm, const RawSrc &rs, uint32_t *dst,
                    uint64_t rows, cudaStream_t s, bool raw) {
  if (rows == 0) return cudaSuccess;
  if (rows > kMaxRows) return cudaErrorInvalidValue;
  switch (c.logn) {
    case 11: return fwd_launch<11>(c, src, rm, rs, dst, rows, s, raw);
    case 12: return fwd_launch<12>(c, src, rm, rs, dst, rows, s, raw);
    case 13: return fwd_launch<13>(c, src, rm, rs, dst, rows, s, raw);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_ntt_fwd(const ParamCtx &c, const uint32_t *src, uint32_t *dst, uint64_t rows, cudaStream_t s) {
  if (rows > kMaxRows) return cudaErrorInvalidValue;  // (a divisor past 2^31 has no FastDiv)
  const RawSrc rs = {};
  const RowMap rm(0, rows ? rows : 1, 0, 1, c.p.L);
  return fwd_any(c, src, rm, rs, dst, rows, s, false);
}

cudaError_t launch_ntt_fwd_rows(const ParamCtx &c, const uint32_t *src, uint64_t off, uint64_t G, uint64_t S,
                                uint32_t *dst, uint64_t rows, cudaStream_t s) {
  const RawSrc rs = {};
  const RowMap rm(off, G, S, 1, c.p.L);
  return fwd_any(c, src, rm, rs, dst, rows, s, false);
}

cudaError_t launch_ntt_fwd_raw(const ParamCtx &c, const uint8_t *raw, int col_major, uint32_t D1, uint32_t D2,
                               uint64_t first, uint64_t npolys, uint32_t *dst, cudaStream_t s) {
  RawSrc rs = {};
  rs.raw = raw;
  rs.log2p = c.p.log2p;
  rs.col_major = col_major ? 1u : 0u;
  rs.D1 = D1;
  rs.D2 = D2;
  if (col_major)
    rs.c0 = first;
  else
    rs.poly0 = first;
  const RowMap rm(0, 1, 1, 1, c.p.L);
  return fwd_any(c, nullptr, rm, rs, dst, npolys * c.p.L, s, true);
}

template <int LOGN>
cudaError_t pair_launch(const ParamCtx &c, const uint32_t *src, uint64_t row0, uint32_t kc, uint32_t stride,
                        uint32_t col0, uint32_t *slots, cudaStream_t s) {
  const int T = (1 << LOGN) / 8;  // two rows in parallel
  const int smem = 2 * ((1 << LOGN) + (1 << LOGN) / 16) * (int)sizeof(uint32_t);
  cudaError_t e = cudaSuccess;
  if (smem > 48 * 1024 &&  // above the limit a kernel has without asking
      (e = cudaFuncSetAttribute(k_ntt_fwd_pair_slots<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess)
    return e;
  return launch_chained(k_ntt_fwd_pair_slots<LOGN>, kc * c.p.L, T, smem, s, src, row0, c.ntt, c.p.L, stride, col0, slots);
}

cudaError_t launch_ntt_fwd_pair_slots(const ParamCtx &c, const uint32_t *queries, uint32_t i0, uint32_t kc,
                                      uint32_t stride, uint32_t col0, uint32_t *slots, cudaStream_t s) {
  if (kc == 0) return cudaSuccess;
  if (col0 + (uint64_t)kc > stride) return cudaErrorInvalidValue;
  const uint64_t row0 = (uint64_t)i0 * 2 * c.p.L;  // row (b = 0, i0, comp 0, j = 0)
  switch (c.logn) {
    case 11: return pair_launch<11>(c, queries, row0, kc, stride, col0, slots, s);
    case 12: return pair_launch<12>(c, queries, row0, kc, stride, col0, slots, s);
    case 13: return pair_launch<13>(c, queries, row0, kc, stride, col0, slots, s);
  }
  return cudaErrorInvalidValue;
}

template <int LOGN>
cudaError_t switch_launch(const ParamCtx &c, const uint32_t *src, uint32_t *dst, uint64_t count, cudaStream_t s) {
  constexpr int N = 1 << LOGN, PADN = N + N / 16;
  const uint32_t L = c.p.L;
  const int smem = (int)(L * PADN * sizeof(uint32_t));
  cudaError_t e = cudaSuccess;
  if (smem > 48 * 1024 &&  // above the limit a kernel has without asking
      (e = cudaFuncSetAttribute(k_ntt_inv_switch<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess)
    return e;
  for (uint64_t first = 0; first < count; first += kMaxGrid) {
    const uint64_t nb = count - first < kMaxGrid ? count - first : kMaxGrid;
    if ((e = launch_chained(k_ntt_inv_switch<LOGN>, (unsigned)nb, N / 8, smem, s, src + first * L * N, dst + first * N,
                            c.ntt, c.sw, L)) != cudaSuccess)
      return e;
  }
  return cudaSuccess;
}

cudaError_t launch_ntt_inv_switch(const ParamCtx &c, const uint32_t *src, uint32_t *dst, uint64_t count,
                                  cudaStream_t s) {
  if (count == 0) return cudaSuccess;
  switch (c.logn) {
    case 11: return switch_launch<11>(c, src, dst, count, s);
    case 12: return switch_launch<12>(c, src, dst, count, s);
    case 13: return switch_launch<13>(c, src, dst, count, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_ntt_inv(const ParamCtx &c, const uint32_t *src, uint32_t *dst, uint64_t rows, cudaStream_t s) {
  if (rows == 0) return cudaSuccess;
  if (rows > kMaxRows) return cudaErrorInvalidValue;
  const RowMap rm(0, rows, 0, 1, c.p.L);
  switch (c.logn) {
    case 11: return inv_launch<11>(c, src, rm, dst, rows, s);
    case 12: return inv_launch<12>(c, src, rm, dst, rows, s);
    case 13: return inv_launch<13>(c, src, rm, dst, rows, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_ntt_fwd_rows_t(const ParamCtx &c, const uint32_t *src, uint64_t off, uint64_t G, uint64_t S,
                                  uint64_t T, uint32_t *dst, uint64_t rows, cudaStream_t s) {
  const RawSrc rs = {};
  const RowMap rm(off, G, S, T, c.p.L);
  return fwd_any(c, src, rm, rs, dst, rows, s, false);
}

}  // namespace gbpir
