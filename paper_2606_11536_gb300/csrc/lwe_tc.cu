// lwe_tc.cu -- the scalar-HE (LWE) DB GEMM of SimplePIR's online step (Sec. 2.5) on the
// fifth-generation tensor cores:
//     out[b][i] = sum_j A[i][j] * Q[b][j]   (mod 2^32)
// with A the raw DB (D1 x D0 signed INT8 plaintexts) and Q the B query vectors.
//
// This chip's INT8 tensor rate (mma.sync, 158 TOPS; tcgen05 has no INT8 form here) is a
// twelfth of its f16 one, so Sec. 4.1's byte decomposition is carried by f16.  A query
// word is four signed base-256 digits mod 2^32, d_p in [-128, 127]; digits and plaintexts
// are exact in f16, a product is at most 2^14, and a sum of 1024 of them is an integer of
// at most 2^24 that the f32 accumulator holds exactly.  The epilogue converts the sums,
// shifts them by their digit's place and adds them in wrapping 32-bit registers.
//
// One MMA: M = 128 DB rows per CTA (two CTAs with CG = 2), N = 4 * queries <= 128, K = 16.
// A lives in tensor memory: a row is a lane, and 128 bytes of a row become 64 columns of
// f16 pairs in five operations per four bytes (flip the sign bits, put two bytes under the
// exponent of 1024, subtract 1152).  With CG = 2 each CTA holds half of the query digits:
// their way from L2 to the SMs is what more queries would run into.
//
// The (row tile, K chunk) units lie in one line, cut into equal ranges, one per CTA (or
// pair): a CTA adds its sums to the zeroed output when it leaves a tile.  Wrapping adds
// give the same words in any order.  Tiles of one chunk are stored instead, and nothing is
// zeroed.  Warps:
//   0..7    epilogue (two sets of the four lane quarters);
//   8..23   converters, four warpgroups taking stages of 128 rows x 128 bytes in turn;
//   24, 25  stream the DB and the query digits (tensor maps);
//   26      issues the MMAs.
// Measured (whole calls, against mma.sync INT8, which this replaced): 1 GiB DB (32768 x 32768), 32
// queries 2265 -> 215 us, 5.0 TB/s of DB; 8 GiB DB, 16 queries 1273 us, 6.7 TB/s = the measured
// copy rate.  Bound by HBM up to 16 queries; at 32 an MMA (74 cycles per 2 KiB of DB) is close
// behind the stream (87).
// Every barrier wait is bounded; one that runs out sets the device error word.
#include "async.cuh"
#include "common.cuh"
#include "stage_drain.h"
#include "tcgen.cuh"

#include <cuda_fp16.h>

namespace gbpir {
namespace {

using async::mbar_arrive;
using async::mbar_expect_tx;
using async::mbar_init;
using async::saddr;
using async::wait_bounded;
using namespace tcgen;

constexpr uint32_t kEpi = 8, kCvt = 16, kGroups = kCvt / 4;
constexpr uint32_t kDbWarp = kEpi + kCvt, kQueryWarp = kDbWarp + 1, kMmaWarp = kDbWarp + 2;
constexpr uint32_t kThreads = (kMmaWarp + 1) * 32;
constexpr uint32_t kK = 128;                      // DB bytes of a row per stage
constexpr uint32_t kRawBytes = 128 * kK;
constexpr uint32_t kStageCols = kK / 2;           // tensor-memory columns of a stage
constexpr uint32_t kMaxN = 128;                   // accumulator columns
constexpr uint32_t kA0 = 2 * kMaxN, kSA = (512 - kA0) / kStageCols;  // the A ring above two accumulators
static_assert(kSA == kGroups, "a slot of the A ring stays with one converter group");
constexpr uint32_t kMaxRaw = 12, kMaxB = 4;
constexpr uint32_t kBars = 2 * kMaxRaw + 2 * kMaxB + 2 * kSA + 2 * 2 + 1;

struct LweArgs {
  uint32_t *out, *err;
  uint32_t D1, B, NT, mtiles;   // rows, queries, accumulator columns, query tiles
  uint32_t chunk, nchunks;      // stages per chunk, chunks per tile
  uint32_t nks;                 // stages per tile
  uint64_t units;               // row tiles x mtiles x nchunks, chunks fastest
  uint32_t SR, SB, bstage;
};

template <int CG>
__global__ void __launch_bounds__(kThreads, 1)
    k_lwe_tc(LweArgs a, const __grid_constant__ CUtensorMap tm_db, const __grid_constant__ CUtensorMap tm_q) {
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t *bsm = smem + a.SR * kRawBytes;
  uint64_t *bars = reinterpret_cast<uint64_t *>(bsm + a.SB * a.bstage);
  const uint32_t raw0 = saddr(smem), fullR = saddr(bars), emptyR = fullR + 8 * kMaxRaw;
  const uint32_t fullB = emptyR + 8 * kMaxRaw, emptyB = fullB + 8 * kMaxB;
  const uint32_t fullA = emptyB + 8 * kMaxB, emptyA = fullA + 8 * kSA;
  const uint32_t tfull = emptyA + 8 * kSA, tempty = tfull + 16, done = tempty + 16;
  uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + kBars);
  // (through a shuffle: the compiler then knows the roles' code to be warp-uniform)
  const uint32_t warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t rank = CG == 2 ? cluster_rank() : 0;
  const uint64_t me = blockIdx.x / CG, all = gridDim.x / CG;
  const uint64_t u0 = a.units * me / all, u1 = a.units * (me + 1) / all;

  if (threadIdx.x == 0) {
    for (uint32_t k = 0; k < kMaxRaw; ++k) {
      mbar_init(fullR + 8 * k, 1);
      mbar_init(emptyR + 8 * k, 4);
    }
    for (uint32_t k = 0; k < kMaxB; ++k) {
      mbar_init(fullB + 8 * k, 1);
      mbar_init(emptyB + 8 * k, 1);
    }
    for (uint32_t k = 0; k < kSA; ++k) {
      mbar_init(fullA + 8 * k, CG * 4);
      mbar_init(emptyA + 8 * k, 1);
    }
    for (uint32_t k = 0; k < 2; ++k) {
      mbar_init(tfull + 8 * k, 1);
      mbar_init(tempty + 8 * k, CG * kEpi);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kMmaWarp) tmem_alloc<CG>(saddr(tslot), 512);
  fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();
  fence_after();
  const uint32_t tmem = *tslot;

  // stages of unit u: its chunk's, fewer in a tile's last chunk
  auto stages_of = [&](uint32_t ch) { return a.nks - ch * a.chunk < a.chunk ? a.nks - ch * a.chunk : a.chunk; };

  if (warp >= kEpi && warp < kEpi + kCvt) {
    // ---------------- converters ----------------
    const uint32_t quarter = warp & 3, group = (warp - kEpi) >> 2, row = 32 * quarter + lane;
    const uint32_t ta = tmem + kA0 + ((32 * quarter) << 16);
    const uint32_t fullA_lead = CG == 2 ? map_to_rank(fullA, 0) : fullA;
    const uint32_t bias = 0x64806480u;  // f16 1152 | 1152
    // all stages of this CTA's units, in order
    const uint64_t t0 = u0 / a.nchunks, t1 = u1 / a.nchunks;
    const uint64_t stages = t1 * a.nks + (u1 % a.nchunks) * a.chunk - (t0 * a.nks + (u0 % a.nchunks) * a.chunk);
    Ring rr, ra;
    rr.skip(group, a.SR);
    ra.skip(group, kSA);
    bool ok = true;
    for (uint64_t g = group; g < stages; g += kGroups, rr.skip(kGroups, a.SR), ra.skip(kGroups, kSA)) {
      if (!__all_sync(0xffffffffu, wait_bounded(fullR + 8 * rr.slot, rr.phase))) {
        ok = false;
        break;
      }
      const uint32_t base = raw0 + rr.slot * kRawBytes + row * 128;
#pragma unroll
      for (int half = 0; half < 2; ++half) {  // 64 bytes of the row: 32 columns
        uint32_t f[32];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint4 w;
          asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                       : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w)
                       : "r"(base + (((4 * half + c) ^ (row & 7)) << 4))
                       : "memory");
          const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint32_t y = x[i] ^ 0x80808080u;
            f[8 * c + 2 * i] = half2_sub(__byte_perm(y, 0x64646464u, 0x4140), bias);
            f[8 * c + 2 * i + 1] = half2_sub(__byte_perm(y, 0x64646464u, 0x4342), bias);
          }
        }
        if (half == 1) {
          __syncwarp();
          if (lane == 0) mbar_arrive(emptyR + 8 * rr.slot);
        } else {
          if (!__all_sync(0xffffffffu, wait_bounded(emptyA + 8 * ra.slot, ra.phase ^ 1))) {
            ok = false;
            break;
          }
          fence_after();
        }
        tmem_st_32x32b_x32(ta + ra.slot * kStageCols + 32 * half, f);
      }
      if (!ok) break;
      tmem_st_wait();
      fence_before();
      __syncwarp();
      if (lane == 0) {
        if (CG == 2)
          mbar_arrive_at(fullA_lead + 8 * ra.slot);
        else
          mbar_arrive(fullA + 8 * ra.slot);
      }
    }
    // the MMAs have read the ring's last stages: no commit is still on its way here
    for (uint64_t g = first_undrained(stages, group, kGroups, kSA); ok && g < stages; g += kGroups)
      ok = __all_sync(0xffffffffu, wait_bounded(emptyA + 8 * (uint32_t)(g % kSA), (uint32_t)(g / kSA) & 1));
    if (!ok && lane == 0) atomicExch(a.err, 1u);
  } else if (warp == kDbWarp || warp == kQueryWarp) {
    // ---------------- DB bytes, query digits ----------------
    if (lane == 0) {
      const bool db = warp == kDbWarp;
      const uint64_t pol = db ? async::policy_evict_first() : async::policy_evict_last();
      const uint32_t size = db ? a.SR : a.SB, rows = a.NT / CG;
      const uint32_t full = db ? fullR : fullB, empty = db ? emptyR : emptyB;
      Ring r;
      uint32_t n = 0;
      bool ok = true;
      for (uint64_t u = u0; ok && u < u1; ++u) {
        const uint64_t tile = u / a.nchunks;
        const uint32_t ch = (uint32_t)(u % a.nchunks), mt = (uint32_t)(tile % a.mtiles);
        const uint32_t row0 = ((uint32_t)(tile / a.mtiles) * CG + rank) * 128, ns = stages_of(ch);
        for (uint32_t k = 0; k < ns; ++k, r.next(size), ++n) {
          if (!wait_bounded(empty + 8 * r.slot, r.phase ^ 1)) {
            atomicExch(a.err, 1u);
            ok = false;
            break;
          }
          const uint32_t ks = ch * a.chunk + k;
          if (db) {
            mbar_expect_tx(full + 8 * r.slot, kRawBytes);
            tma_load_2d(raw0 + r.slot * kRawBytes, &tm_db, ks * kK, row0, full + 8 * r.slot, pol);
          } else {
            if (rank == 0) mbar_expect_tx(full + 8 * r.slot, CG * a.bstage);
            tma_load_3d<CG>(saddr(bsm) + r.slot * a.bstage, &tm_q, 0, (mt * a.NT + rank * rows) / 8, ks * (kK / 16),
                            CG == 2 ? map_to_rank(full + 8 * r.slot, 0) : full + 8 * r.slot, pol);
          }
        }
      }
      const uint32_t back = n < size ? n : size;
      for (uint32_t k = 0; k < back; ++k) {
        r.slot = r.slot ? r.slot - 1 : size - 1;
        if (r.slot == size - 1) r.phase ^= 1;
        // never leave with copies in flight, nor with a commit on its way to this CTA
        if ((db || rank == 0) && !wait_bounded(full + 8 * r.slot, r.phase)) atomicExch(a.err, 1u);
        if (!db && !wait_bounded(empty + 8 * r.slot, r.phase)) atomicExch(a.err, 1u);
      }
    }
    __syncwarp();
  } else if (warp == kMmaWarp) {
    // ---------------- MMAs ----------------
    if (rank == 0) {
      const uint32_t idesc = instr_desc_f16(128 * CG, a.NT), rows = a.NT / CG;
      const uint64_t bstep = rows * 32 >> 4;
      Ring rb, ra, rt;
      bool ok = true, rdyA = false, rdyB = false;  // looked up before the MMAs that precede them
      auto wait = [&](uint32_t bar, uint32_t parity) {
        ok = __all_sync(0xffffffffu, wait_bounded(bar, parity)) && ok;
      };
      uint32_t ch = (uint32_t)(u0 % a.nchunks);
      for (uint64_t u = u0; ok && u < u1; ++u) {
        const uint32_t ns = stages_of(ch), d = tmem + rt.slot * kMaxN;
        wait(tempty + 8 * rt.slot, rt.phase ^ 1);
        for (uint32_t k = 0; k < ns; ++k) {
          if (!rdyB) wait(fullB + 8 * rb.slot, rb.phase);
          if (!rdyA) wait(fullA + 8 * ra.slot, ra.phase);
          if (!ok) break;
          fence_after();
          const uint32_t slotA = ra.slot, slotB = rb.slot, ad = tmem + kA0 + slotA * kStageCols;
          const uint64_t bd = smem_desc(saddr(bsm) + slotB * a.bstage, 128, 256);
          ra.next(kSA);
          rb.next(a.SB);
          const bool nextA = mbar_test(fullA + 8 * ra.slot, ra.phase);
          const bool nextB = mbar_test(fullB + 8 * rb.slot, rb.phase);
          if (elect_one()) {
#pragma unroll
            for (int v = 0; v < (int)kK / 16; ++v) mma_f16_ts<CG>(d, ad + 8 * v, bd + v * bstep, idesc, k || v);
            mma_commit<CG>(emptyA + 8 * slotA);
            mma_commit<CG>(emptyB + 8 * slotB);
          }
          rdyA = __all_sync(0xffffffffu, nextA);
          rdyB = __all_sync(0xffffffffu, nextB);
        }
        if (!ok) break;
        if (elect_one()) mma_commit<CG>(tfull + 8 * rt.slot);
        rt.next(2);
        if (++ch == a.nchunks) ch = 0;
      }
      if (!ok && elect_one()) atomicExch(a.err, 1u);
      // on every path: no MMA may still be running when the tensor memory is freed
      if (elect_one()) mma_commit_local<CG>(done);
      if (!wait_bounded(done, 0)) atomicExch(a.err, 1u);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue ----------------
    const uint32_t quarter = warp & 3, set = warp >> 2, G = a.NT / 16;  // groups of 4 queries x 4 digits
    const uint32_t tempty_lead = CG == 2 ? map_to_rank(tempty, 0) : tempty;
    Ring rt;
    bool ok = true;
    uint32_t sum[4][4];  // [group set, set + 2, ..][query]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int b = 0; b < 4; ++b) sum[i][b] = 0;
    uint32_t ch = (uint32_t)(u0 % a.nchunks);
    for (uint64_t u = u0; u < u1; ++u) {
      if (!__all_sync(0xffffffffu, wait_bounded(tfull + 8 * rt.slot, rt.phase))) {
        ok = false;
        break;
      }
      fence_after();
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t g = set + 2 * i;
        if (g < G) {
          uint32_t f[16];
          tmem_ld16(tmem + rt.slot * kMaxN + ((32 * quarter) << 16) + 16 * g, f);
#pragma unroll
          for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int p = 0; p < 4; ++p)
              sum[i][b] += (uint32_t)__float2int_rn(__uint_as_float(f[4 * b + p])) << (8 * p);
        }
      }
      fence_before();
      __syncwarp();
      if (lane == 0) {
        if (CG == 2)
          mbar_arrive_at(tempty_lead + 8 * rt.slot);
        else
          mbar_arrive(tempty + 8 * rt.slot);
      }
      rt.next(2);
      if (++ch == a.nchunks || u + 1 == u1) {  // leaving the tile
        const uint64_t tile = u / a.nchunks;
        const uint64_t i0 = ((tile / a.mtiles) * CG + rank) * 128 + 32 * quarter + lane;
        const uint32_t q0 = (uint32_t)(tile % a.mtiles) * (a.NT / 4);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const uint32_t g = set + 2 * i, q = q0 + 4 * g + b;
            if (g < G && q < a.B && i0 < a.D1) {
              uint32_t *o = a.out + (uint64_t)q * a.D1 + i0;
              if (a.nchunks == 1)
                *o = sum[i][b];
              else
                atomicAdd(o, sum[i][b]);
            }
            sum[i][b] = 0;
          }
        if (ch == a.nchunks) ch = 0;
      }
    }
    if (!ok && lane == 0) atomicExch(a.err, 1u);
  }

  fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();
  if (warp == kMmaWarp) {
    fence_after();
    tmem_dealloc<CG>(tmem, 512);
  }
}

// Query words [B][D0] -> f16 digits qt [u = j / 16][rows][16] in core-matrix blocks (element
// (row r, k) at (r / 8) * 128 + (k / 8) * 64 + (r % 8) * 8 + k % 8), row r = 4b + p; rows
// past the queries and words past D0 are zero.  Thread = (query, 8 words).  The threads
// also clear `words` words of the output that the GEMM adds to (a launch less than a memset).
__global__ void __launch_bounds__(256) k_lwe_digits(const uint32_t *__restrict__ Q, uint32_t B, uint32_t D0,
                                                    uint32_t Bp, uint32_t nh, uint16_t *__restrict__ qt,
                                                    uint32_t *__restrict__ out, uint64_t words) {
  const uint32_t t = blockIdx.x * 256 + threadIdx.x, b = t % Bp, h = t / Bp;  // half block h: words 8h .. 8h + 7
  for (uint64_t w = t; w < words; w += (uint64_t)gridDim.x * 256) out[w] = 0;
  if (h >= nh) return;
  uint4 w0 = make_uint4(0, 0, 0, 0), w1 = w0;
  if (b < B && 8 * h < D0) {
    const uint4 *src = reinterpret_cast<const uint4 *>(Q + (uint64_t)b * D0 + 8 * h);
    w0 = __ldg(src);
    w1 = __ldg(src + 1);
  }
  const uint32_t y[8] = {w0.x + 0x80808080u, w0.y + 0x80808080u, w0.z + 0x80808080u, w0.w + 0x80808080u,
                         w1.x + 0x80808080u, w1.y + 0x80808080u, w1.z + 0x80808080u, w1.w + 0x80808080u};
  uint16_t *dst = qt + (uint64_t)(h >> 1) * Bp * 64 + (b >> 1) * 128 + (h & 1) * 64 + (b & 1) * 32;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    uint32_t o[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      o[e] = half2_sub((__byte_perm(y[2 * e], y[2 * e + 1], p | (4 + p) << 8) & 0x00FF00FFu) | 0x64006400u, 0x64806480u);
    *reinterpret_cast<uint4 *>(dst + 8 * p) = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

uint32_t padded_queries(uint32_t B) { return (B + 3u) & ~3u; }
uint32_t padded_words(uint32_t D0) { return (D0 + kK - 1) / kK * kK; }

}  // namespace

// Tensor-map coordinates are signed 32-bit: the last row of the last tile has to lie below
// 2^31 (tiles of 256 rows where CTAs work in pairs).  Past it a box reads as zeros.
bool lwe_tc_addresses(uint32_t D1) { return (D1 + 255ull) / 256 * 256 <= 1ull << 31; }

size_t lwe_tc_scratch_bytes(uint32_t D0, uint32_t B) { return (size_t)padded_words(D0) * padded_queries(B) * 8; }

cudaError_t launch_lwe_tc(const int8_t *A, uint32_t D1, uint32_t D0, const uint32_t *Q, uint32_t B, uint32_t *out,
                          uint16_t *qt, cudaStream_t s) {
  if (!lwe_tc_addresses(D1)) return cudaErrorInvalidValue;
  LweArgs a = {};
  cudaError_t e = device_error_word(&a.err);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const uint32_t Bp = padded_queries(B), Ntot = 4 * Bp;
  a.out = out;
  a.D1 = D1;
  a.B = B;
  a.mtiles = (Ntot + kMaxN - 1) / kMaxN;
  a.NT = ((Ntot + a.mtiles - 1) / a.mtiles + 15u) & ~15u;
  a.nks = padded_words(D0) / kK;
  const uint32_t CG = a.NT > 32 && D1 > 128 ? 2 : 1;
  const uint64_t tiles = (D1 + 128ull * CG - 1) / (128 * CG) * a.mtiles;
  // chunks of 1024 bytes, shorter where there would be fewer than one a CTA
  a.chunk = 1024 / kK;
  while (a.chunk > 1 && tiles * ((a.nks + a.chunk - 1) / a.chunk) < (uint64_t)sms / CG) a.chunk /= 2;
  a.nchunks = (a.nks + a.chunk - 1) / a.chunk;
  a.units = tiles * a.nchunks;
  a.bstage = (a.NT / CG) * kK * 2;
  const size_t fixed = kBars * 8 + 16;
  a.SB = kMaxB;
  a.SR = (uint32_t)((kSmemMax - fixed - a.SB * a.bstage) / kRawBytes);
  if (a.SR > kMaxRaw) a.SR = kMaxRaw;
  a.SR = a.SR / kGroups * kGroups;  // a DB slot stays with one converter group
  size_t smem = a.SR * kRawBytes + a.SB * a.bstage + fixed;
  if (smem < kSmemMin) smem = kSmemMin;
  alignas(64) CUtensorMap tm_db = {}, tm_q = {};
  if (!byte_tensor_map(&tm_db, A, D0, D1, kK, 128) ||
      !digit_tensor_map(&tm_q, qt, Ntot / 8, padded_words(D0) / 16, a.NT / CG / 8, kK / 16))
    return cudaErrorInvalidValue;
  const uint32_t nh = padded_words(D0) / 8;
  const uint64_t words = a.nchunks == 1 ? 0 : (uint64_t)B * D1;
  uint64_t grid = ((uint64_t)nh * Bp + 255) / 256;
  if (grid < 152 && words > grid * 2048) grid = 152;  // enough threads for the output too
  k_lwe_digits<<<(unsigned)grid, 256, 0, s>>>(Q, B, D0, Bp, nh, qt, out, words);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return CG == 2 ? launch_persistent<k_lwe_tc<2>, 2>(a.units, kThreads, smem, s, a, tm_db, tm_q)
                 : launch_persistent<k_lwe_tc<1>, 1>(a.units, kThreads, smem, s, a, tm_db, tm_q);
}

}  // namespace gbpir
