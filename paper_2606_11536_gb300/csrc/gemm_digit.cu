// gemm_digit.cu -- the batched first-dimension modular GEMM of the plain and limb layouts
// on the tensor cores: the resident residues are split into digits on the way to the MMA.
//
//   out[s][m][c] = sum_{i < Kc} qs[s][i][m] * db[s][i0 + i][c]   (mod q_j),  s = j*n + k
//
// Digits, and why the sums are exact.  A residue x < 2^30 is sum_l 256^l d_l with signed
// digits d_0..d_2 in [-128, 127] and d_3 in [0, 64], exact in f16.  The 16 digit products
//     P_la[c][m] = sum_{i < 1024} d_l(db[i][c]) * d_a(qs[i][m]),  |P_la| <= 1024 * 2^14 = 2^24,
// are integers that an f32 accumulator holds exactly in any order of summation.
// The bytes of x + 0x808080 are d_l + 128 (the top one d_3); a byte under the exponent of
// 1024 is the f16 1024 + byte, less a constant the digit.  That is 7 operations per
// residue, two bytes at a time.
// Every 1024 rows the epilogue reads P back, weights digit pair (l, a) with
// 2^(8 (l + a)) mod q, sums in int64 and keeps the sum in registers across the chunks;
// it reduces mod q once per output.
//
// The limb layout's residues are their four bytes already, digits in [0, 255]: a byte under
// the exponent of 1024, less 1024.  Its sums take 512 rows (512 * 255 * 128 < 2^24), and its
// K positions are the rows in order.
//
// One MMA (M = 128 per CTA, N = 4 * query rows, K = 16) forms all 16 products.  A rows are
// (DB column, digit) pairs, B rows (query row, digit) pairs n = 4 * m + a.  A lives in
// tensor memory: with A in shared memory an MMA takes 43 + N / 2 cycles on this chip
// (measured back to back, any layout), from tensor memory 11 + N / 2, and the shared
// memory keeps its bandwidth for the query digits.  With CG = 2 a CTA pair runs M = 256
// MMAs: each CTA converts its own 32 columns per tile and holds half of the query digits.
//
// Work unit = (slot, T tiles of 32 columns, up to 256 B rows as H = 1 or 2 halves); a
// block is 64 rows of one tile, an A stage SUB = 2 / H blocks: the MMA warp spends about
// 300 cycles a stage on its barriers, as much as 16 small MMAs take.  One persistent CTA
// per SM:
//   warps 0..7 (H = 2: 0..15)   epilogue, sets of the four tensor-memory lane quarters;
//   warps up to 23   converters, warpgroups taking stages in turn; a warp owns a lane
//                 quarter = 8 columns x 4 digits: words from the swizzled block, digits
//                 to registers, tcgen05.st into the A ring;
//   warp  24      streams the DB words into a ring of 8 KiB blocks (tensor map);
//   warp  25      streams the query digits, as many rows at a time as an A stage;
//   warp  26      issues the MMAs.
// Tensor memory: R accumulators (2 for H = 1, 3 for H = 2) and the A ring above them.
// Lane lambda of quarter w holds digit lambda / 8 of column 8 w + lambda % 8, which is
// how tcgen05.st.16x256b lays a thread's four words out.  Its K positions 4j .. 4j + 3 are
// rows 2j, 2j + 1, 2j + 8, 2j + 9 of each 16 (the query digits are stored in that order),
// so that the four row groups a warp reads at once fall into different swizzled chunks:
// no bank conflicts.  (LIMB: a block is 64 bytes of 128 (limb, column) rows, a lane reads its
// own row, tcgen05.st.32x32b.)
//
// Measured (GB300, 2.07 GHz, against the CUDA-core tiles): 8 GiB DB (n = 4096, 2048 x 512),
// batch 32: 69.4 -> 12.2 ms, 0.85 of the sustained bf16 rate as 16 digit products; 1 GiB DB
// (n = 2048, 512 x 512), batch 8: 2.3 -> 0.81 ms, 5.3 TB/s of DB words; 1 GiB DB (n = 4096),
// batch 4: 1.38 -> 0.73 ms; limb layout (n = 2048, 512 x 256), batch 32: 7.8 (INT8 mma.sync) ->
// 0.89 ms.  With few query rows it is bound by HBM, from 2B = 32 by the
// MMAs (and, where D1 is short, by the epilogue's serial parts).  Handing the accumulators back
// before the arithmetic on their copies took the limb case from 1.00 ms there, the 8 GiB one
// from 12.8.  The second half's MMAs one stage behind the first's, so that the next unit's first
// half would not wait at all, were slower (16.3 ms): the A ring loses the slot its converters need.
//
// Every barrier wait is bounded; one that runs out sets the device error word.
#include "async.cuh"
#include "common.cuh"
#include "stage_drain.h"
#include "tcgen.cuh"

#include <type_traits>

namespace gbpir {
namespace {

using async::mbar_arrive;
using async::mbar_expect_tx;
using async::mbar_init;
using async::saddr;
using async::wait_bounded;
using namespace tcgen;

constexpr uint32_t kWorkers = 24;  // epilogue and converter warps
constexpr uint32_t kDbWarp = kWorkers, kQueryWarp = kDbWarp + 1, kMmaWarp = kDbWarp + 2;
constexpr uint32_t kThreads = (kMmaWarp + 1) * 32;
constexpr uint32_t kRows = 64;                    // DB rows per block
constexpr uint32_t kRawBytes = kRows * 32 * 4;    // one block of DB words
constexpr uint32_t kBlockCols = kRows / 2;        // tensor-memory columns of one block's digits
constexpr uint32_t kMaxRaw = 16, kMaxB = 4, kMaxA = 4;
constexpr uint32_t kTmem = 512;
constexpr uint32_t kBars = 2 * kMaxRaw + 2 * kMaxB + 2 * kMaxA + 2 * 3 + 1;

struct DigArgs {
  uint32_t *out;  // [L*n][M][D2]
  uint32_t *err;
  uint32_t M, D2, i0, Kc, Uc;
  uint32_t T, NH;                    // column tiles, B rows per half
  uint32_t W, R, SA, a0;             // accumulator columns and count; A ring stages and first column
  uint32_t cgroups, mtiles, nunits;  // units = slots x mtiles x cgroups, cgroups fastest
  uint32_t SR, SB, bstage;           // DB-word blocks, query stages, bytes of the latter in this CTA
  uint32_t logn;
  int acc_in;
};

template <typename T>
__device__ __forceinline__ T pick(const T (&v)[PIR_MAX_L], uint32_t j) {
  T r = v[0];
#pragma unroll
  for (uint32_t i = 1; i < PIR_MAX_L; ++i) r = j == i ? v[i] : r;
  return r;
}

__device__ __forceinline__ int64_t mad_wide(int32_t x, int32_t y, int64_t acc) {
  int64_t d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(x), "r"(y), "l"(acc));
  return d;
}

__device__ __forceinline__ void ld_shared16(uint32_t addr, uint32_t (&v)[4]) {
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(addr)
               : "memory");
}

__device__ __forceinline__ uint32_t ld_shared(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

// The units first, first + step, ... of a CTA (or pair), divided out once.
struct UnitWalk {
  uint32_t cg, mt, s, dcg, dmt, ds;
  __device__ __forceinline__ UnitWalk(const DigArgs &a, uint32_t first, uint32_t step) {
    cg = first % a.cgroups, mt = first / a.cgroups % a.mtiles, s = first / (a.cgroups * a.mtiles);
    dcg = step % a.cgroups, dmt = step / a.cgroups % a.mtiles, ds = step / (a.cgroups * a.mtiles);
  }
  __device__ __forceinline__ void next(const DigArgs &a) {
    cg += dcg, mt += dmt, s += ds;
    if (cg >= a.cgroups) cg -= a.cgroups, ++mt;
    if (mt >= a.mtiles) mt -= a.mtiles, ++s;
  }
};

template <int CG, int SUB, bool LIMB>
__global__ void __launch_bounds__(kThreads, 1)
    k_gemm_digit(DigArgs a, ModConst mc, const __grid_constant__ CUtensorMap tm_db,
                 const __grid_constant__ CUtensorMap tm_q) {
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t *bsm = smem + a.SR * kRawBytes;  // query stages after the DB-word stages
  uint64_t *bars = reinterpret_cast<uint64_t *>(bsm + a.SB * a.bstage);
  const uint32_t raw0 = saddr(smem), fullR = saddr(bars), emptyR = fullR + 8 * kMaxRaw;
  const uint32_t fullB = emptyR + 8 * kMaxRaw, emptyB = fullB + 8 * kMaxB;
  const uint32_t fullA = emptyB + 8 * kMaxB, emptyA = fullA + 8 * kMaxA;
  const uint32_t tfull = emptyA + 8 * kMaxA, tempty = tfull + 8 * 3, done = tempty + 8 * 3;
  uint32_t *tslot = reinterpret_cast<uint32_t *>(bars + kBars);
  int32_t *wtab = reinterpret_cast<int32_t *>(tslot + 4);  // [L][8]: 2^(8 t) mod q_j
  // (through a shuffle: the compiler then knows the roles' code to be warp-uniform)
  const uint32_t warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t rank = CG == 2 ? cluster_rank() : 0;
  const uint32_t first = blockIdx.x / CG, step = gridDim.x / CG;
  constexpr uint32_t kStageRows = SUB * kRows, H = 2 / SUB;
  constexpr uint32_t kChunkRows = LIMB ? 512 : 1024;  // rows per exact f32 sum
  constexpr uint32_t kSets = 2 * H, kEpi = 4 * kSets, kCvt = kWorkers - kEpi, kGroups = kCvt / 4;
  constexpr int kPer = H == 1 ? 6 : 2, kItems = H * kPer;  // accumulator groups per epilogue set: a half's, a unit's
  const uint32_t nks = (a.Kc + kStageRows - 1) / kStageRows;  // stages of a tile per unit
  const uint32_t units = (a.nunits - first + step - 1) / step;

  if (threadIdx.x == 0) {
    for (uint32_t k = 0; k < kMaxRaw; ++k) {
      mbar_init(fullR + 8 * k, 1);
      mbar_init(emptyR + 8 * k, 4);
    }
    for (uint32_t k = 0; k < kMaxB; ++k) {
      mbar_init(fullB + 8 * k, 1);
      mbar_init(emptyB + 8 * k, 1);
    }
    for (uint32_t k = 0; k < kMaxA; ++k) {
      mbar_init(fullA + 8 * k, CG * 4);
      mbar_init(emptyA + 8 * k, 1);
    }
    for (uint32_t k = 0; k < 3; ++k) {
      mbar_init(tfull + 8 * k, 1);
      mbar_init(tempty + 8 * k, CG * kEpi);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0 && lane < PIR_MAX_L) {
    const uint32_t q = pick(mc.q, lane);
    const uint64_t mu = pick(mc.mu, lane);
    uint32_t pw = 1;
    for (int t = 0; t < 7; ++t) {
      wtab[8 * lane + t] = (int32_t)pw;
      pw = q ? reduce64((uint64_t)pw << 8, q, mu) : 0;
    }
  }
  if (warp == kMmaWarp) tmem_alloc<CG>(saddr(tslot), kTmem);
  fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();
  fence_after();
  const uint32_t tmem = *tslot;

  if (warp >= kEpi && warp < kEpi + kCvt) {
    // ---------------- converters ----------------
    const uint32_t quarter = warp & 3, group = (warp - kEpi) >> 2;
    const uint32_t rho = lane >> 2, j = lane & 3, ch = 2 * quarter + (rho >> 2);
    // LIMB: this lane's row and the swizzle of its 16-byte chunks; else the words of the
    // even and the odd rows
    const uint32_t lrow = 32 * (lane >> 3) + 8 * quarter + (lane & 7);
    const uint32_t off0 = LIMB ? lrow * 64 : 2 * j * 128 + ((ch ^ (2 * j)) << 4) + (rho & 3) * 4;
    const uint32_t off1 = LIMB ? (lrow >> 1 & 3) << 4
                               : (2 * j + 1) * 128 + ((ch ^ (2 * j + 1)) << 4) + (rho & 3) * 4;
    const uint32_t bias = 0x64806480u, bias3 = 0x64006480u;  // f16 1152 | 1152 and 1152 | 1024
    const uint32_t ta = tmem + a.a0 + ((32 * quarter) << 16);
    const uint32_t fullA_lead = CG == 2 ? map_to_rank(fullA, 0) : fullA;
    // no more groups than A slots: a slot then stays with one group, which sees its rounds
    // one by one (a parity tells apart neighbouring rounds only)
    const uint32_t groups = kGroups < a.SA ? kGroups : a.SA;
    const uint64_t stages = group < groups ? (uint64_t)units * nks * a.T : 0;
    Ring rr, ra;
    rr.skip(group * SUB, a.SR);
    ra.skip(group, a.SA);
    bool ok = true;
    for (uint64_t g = group; ok && g < stages; g += groups, rr.skip((groups - 1) * SUB, a.SR), ra.skip(groups, a.SA)) {
#pragma unroll
      for (int sub = 0; sub < SUB; ++sub, rr.next(a.SR)) {
        if (!__all_sync(0xffffffffu, wait_bounded(fullR + 8 * rr.slot, rr.phase))) {
          ok = false;
          break;
        }
        const uint32_t base = raw0 + rr.slot * kRawBytes;
        uint32_t f[32];  // LIMB: this lane's 64 digits; else digits 0, 1 and 2, 3 of its column
        if constexpr (LIMB) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint32_t x[4];
            ld_shared16(base + off0 + ((c << 4) ^ off1), x);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              f[8 * c + 2 * i] = half2_sub(__byte_perm(x[i], 0x64646464u, 0x4140), 0x64006400u);
              f[8 * c + 2 * i + 1] = half2_sub(__byte_perm(x[i], 0x64646464u, 0x4342), 0x64006400u);
            }
          }
        } else {
#pragma unroll
          for (int kb = 0; kb < 4; ++kb) {
            uint32_t e[4], o[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              const uint32_t y = ld_shared(base + (t & 1 ? off1 : off0) + (t >> 1) * 1024 + kb * 2048) + 0x00808080u;
              e[t] = half2_sub((y & 0x00FF00FFu) | 0x64006400u, bias);
              o[t] = half2_sub(__byte_perm(y, 0x64646464u, 0x4341), bias3);
            }
#pragma unroll
            for (int v = 0; v < 2; ++v) {
              f[4 * kb + v] = __byte_perm(e[2 * v], e[2 * v + 1], 0x5410);
              f[4 * kb + 2 + v] = __byte_perm(o[2 * v], o[2 * v + 1], 0x5410);
              f[16 + 4 * kb + v] = __byte_perm(e[2 * v], e[2 * v + 1], 0x7632);
              f[16 + 4 * kb + 2 + v] = __byte_perm(o[2 * v], o[2 * v + 1], 0x7632);
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(emptyR + 8 * rr.slot);
        if (sub == 0) {
          if (!__all_sync(0xffffffffu, wait_bounded(emptyA + 8 * ra.slot, ra.phase ^ 1))) {
            ok = false;
            break;
          }
          fence_after();
        }
        const uint32_t dst = ta + (ra.slot * SUB + sub) * kBlockCols;
        if constexpr (LIMB) {
          tmem_st_32x32b_x32(dst, f);
        } else {
          tmem_st_16x256b_x4(dst, f);
          tmem_st_16x256b_x4(dst + (16 << 16), f + 16);
        }
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
    // the MMAs have read the ring's last stages: no commit is still on its way here (with fewer
    // groups than slots, a group has several of those)
    for (uint64_t g = first_undrained(stages, group, groups, a.SA); ok && g < stages; g += groups)
      ok = __all_sync(0xffffffffu, wait_bounded(emptyA + 8 * (uint32_t)(g % a.SA), (uint32_t)(g / a.SA) & 1));
    if (!ok && lane == 0) atomicExch(a.err, 1u);
  } else if (warp == kDbWarp) {
    // ---------------- DB words ----------------
    if (lane == 0) {
      const uint64_t pol = async::policy_evict_first();
      Ring r;
      uint32_t n = 0;
      bool ok = true;
      UnitWalk w(a, first, step);
      for (uint32_t u = 0; ok && u < units; ++u, w.next(a)) {
        const uint32_t c0 = (w.cg * CG + rank) * a.T * 32;
        for (uint32_t ks = 0; ok && ks < nks; ++ks)
          for (uint32_t t = 0; t < a.T * SUB; ++t, r.next(a.SR), ++n) {
            if (!wait_bounded(emptyR + 8 * r.slot, r.phase ^ 1)) {
              atomicExch(a.err, 1u);
              ok = false;
              break;
            }
            mbar_expect_tx(fullR + 8 * r.slot, kRawBytes);
            const uint32_t c = c0 + t / SUB * 32, i = a.i0 + ks * kStageRows + t % SUB * kRows;
            if (LIMB)
              tma_load_4d(raw0 + r.slot * kRawBytes, &tm_db, i, c, 0, w.s, fullR + 8 * r.slot, pol);
            else
              tma_load_3d<1>(raw0 + r.slot * kRawBytes, &tm_db, c, i, w.s, fullR + 8 * r.slot, pol);
          }
      }
      // never leave with copies in flight
      const uint32_t back = n < a.SR ? n : a.SR;
      for (uint32_t k = 0; k < back; ++k) {
        r.slot = r.slot ? r.slot - 1 : a.SR - 1;
        if (r.slot == a.SR - 1) r.phase ^= 1;
        if (!wait_bounded(fullR + 8 * r.slot, r.phase)) atomicExch(a.err, 1u);
      }
    }
    __syncwarp();
  } else if (warp == kQueryWarp) {
    // ---------------- query digits ----------------
    if (lane == 0) {
      const uint64_t pol = async::policy_evict_last();
      const uint32_t rows = a.NH / CG;
      Ring r;
      uint32_t n = 0;
      bool ok = true;
      UnitWalk w(a, first, step);
      for (uint32_t u = 0; ok && u < units; ++u, w.next(a)) {
        for (uint32_t r0 = 0; r0 < a.Kc; r0 += kStageRows, r.next(a.SB), ++n) {
          if (!wait_bounded(emptyB + 8 * r.slot, r.phase ^ 1)) {
            atomicExch(a.err, 1u);
            ok = false;
            break;
          }
          const uint32_t bar = CG == 2 ? map_to_rank(fullB + 8 * r.slot, 0) : fullB + 8 * r.slot;
          if (rank == 0) mbar_expect_tx(fullB + 8 * r.slot, CG * a.bstage);
          const uint32_t dst = saddr(bsm + r.slot * a.bstage);
          for (uint32_t hf = 0; hf < H; ++hf)
            tma_load_3d<CG>(dst + hf * (kStageRows / 16) * rows * 32, &tm_q, 0, ((w.mt * H + hf) * a.NH + rank * rows) / 8,
                            w.s * a.Uc + r0 / 16, bar, pol);
        }
      }
      const uint32_t back = n < a.SB ? n : a.SB;
      for (uint32_t k = 0; k < back; ++k) {
        r.slot = r.slot ? r.slot - 1 : a.SB - 1;
        if (r.slot == a.SB - 1) r.phase ^= 1;
        // never leave with copies in flight, nor with a commit on its way to this CTA
        if (rank == 0 && !wait_bounded(fullB + 8 * r.slot, r.phase)) atomicExch(a.err, 1u);
        if (!wait_bounded(emptyB + 8 * r.slot, r.phase)) atomicExch(a.err, 1u);
      }
    }
    __syncwarp();
  } else if (warp == kMmaWarp) {
    // ---------------- MMAs ----------------
    // the whole warp runs the loop, so that its state stays warp-uniform; one lane issues
    if (rank == 0) {
      const uint32_t idesc = instr_desc_f16(128 * CG, a.NH), rows = a.NH / CG;
      const uint64_t bstep = rows * 32 >> 4;  // one K = 16 block of query digits
      Ring rb, ra, rt;
      bool ok = true;
      // The next stages' barriers are looked up before the MMAs of this one are issued and
      // the answers read after them: a wait costs about 100 cycles even where it is over.
      bool rdyA = false, rdyB = false;
      auto wait = [&](uint32_t bar, uint32_t parity) {
        ok = __all_sync(0xffffffffu, wait_bounded(bar, parity)) && ok;
      };
      for (uint32_t u = 0; ok && u < units; ++u) {
        uint32_t left = 0;  // stages of a tile left in the chunk
        for (uint32_t ks = 0; ks < nks; ++ks) {
          const bool head = left == 0;
          Ring rt2 = rt;
          rt2.next(a.R);
          if (head) {
            wait(tempty + 8 * rt.slot, rt.phase ^ 1);
            if (H == 2) wait(tempty + 8 * rt2.slot, rt2.phase ^ 1);
            left = kChunkRows / kStageRows;
          }
          if (!rdyB) wait(fullB + 8 * rb.slot, rb.phase);
          if (!ok) break;
          // the last stage may hold one block only: its second half is not this chunk's
          const bool whole = SUB == 1 || ks * kStageRows + kRows < a.Kc;
          const uint64_t bd0 = smem_desc(saddr(bsm) + rb.slot * a.bstage, 128, 256);
          const uint32_t slotB = rb.slot;
          rb.next(a.SB);
          uint32_t d0 = tmem + rt.slot * a.W;
          for (uint32_t t = 0; t < a.T; ++t, d0 += a.NH) {
            if (!rdyA) wait(fullA + 8 * ra.slot, ra.phase);
            if (!ok) break;
            fence_after();
            const uint32_t slot = ra.slot, ad = tmem + a.a0 + slot * (SUB * kBlockCols);
            ra.next(a.SA);
            const bool nextA = mbar_test(fullA + 8 * ra.slot, ra.phase);
            const bool nextB = t + 1 == a.T && mbar_test(fullB + 8 * rb.slot, rb.phase);
            if (elect_one()) {
#pragma unroll
              for (int v = 0; v < 4 * SUB; ++v)
                if (v < 4 || whole) mma_f16_ts<CG>(d0, ad + 8 * v, bd0 + v * bstep, idesc, !head || v);
              if (H == 2) {
                const uint32_t d1 = tmem + rt2.slot * a.W;
                const uint64_t bd1 = bd0 + 4 * bstep;
#pragma unroll
                for (int v = 0; v < 4; ++v) mma_f16_ts<CG>(d1, ad + 8 * v, bd1 + v * bstep, idesc, !head || v);
              }
              mma_commit<CG>(emptyA + 8 * slot);
            }
            rdyA = __all_sync(0xffffffffu, nextA);
            rdyB = __all_sync(0xffffffffu, nextB);
          }
          if (!ok) break;
          if (elect_one()) mma_commit<CG>(emptyB + 8 * slotB);
          if (--left == 0 || ks + 1 == nks) {
            if (elect_one()) mma_commit<CG>(tfull + 8 * rt.slot);
            if (H == 2) {
              if (elect_one()) mma_commit<CG>(tfull + 8 * rt2.slot);
              rt.next(a.R);
            }
            rt.next(a.R);
            left = 0;
          }
        }
      }
      if (!ok && elect_one()) atomicExch(a.err, 1u);
      // on every path: no MMA may still be running when the tensor memory is freed
      if (elect_one()) mma_commit_local<CG>(done);
      if (!wait_bounded(done, 0)) atomicExch(a.err, 1u);
    }
    __syncwarp();
  } else {
    // ---------------- epilogue ----------------
    const uint32_t quarter = warp & 3, set = warp >> 2;
    // A thread reads all four DB digits of its column but only query digits 2p, 2p + 1 (p
    // the lane's parity) of two rows out of each group of four; it trades one row's half
    // with its neighbour and keeps row 2p + (lane / 2) % 2.
    const uint32_t p = lane & 1, b = 2 * p + ((lane >> 1) & 1), col = 8 * quarter + (lane >> 2);
    const uint32_t G = a.NH / 16, items = a.T * G;  // groups of 16 accumulator columns (4 query rows), per half
    const uint32_t nchunk = (a.Kc + kChunkRows - 1) / kChunkRows;
    // This lane's outputs, one per group set, set + kSets, ... of each half: the query row
    // above the column, or all ones.
    uint32_t place[kItems];
#pragma unroll
    for (int it = 0; it < kItems; ++it) {
      const uint32_t item = set + kSets * (it % kPer), t = H == 2 ? 0 : item / G, g = item - t * G;
      const uint32_t m = (uint32_t)(it / kPer) * (a.NH / 4) + 4 * g + b;
      place[it] = item < items ? m << 16 | (32 * t + col) : ~0u;
    }
    const uint32_t tempty_lead = CG == 2 ? map_to_rank(tempty, 0) : tempty;
    Ring rt;
    bool ok = true;
    UnitWalk w(a, first, step);
    for (uint32_t u = 0; ok && u < units; ++u, w.next(a)) {
      const uint32_t j = w.s >> a.logn;
      const uint32_t q = pick(mc.q, j);
      const uint64_t mu = pick(mc.mu, j);
      int32_t wgt[5];  // digit-pair weights 2^(8 (l + a)) mod q, a = 2p or 2p + 1
#pragma unroll
      for (int d = 0; d < 5; ++d) wgt[d] = wtab[8 * j + 2 * p + d];
      const uint32_t m0 = w.mt * (H * a.NH / 4), c0 = (w.cg * CG + rank) * a.T * 32;
      uint32_t *const out = a.out + ((uint64_t)w.s * a.M + m0) * a.D2 + c0;
      auto output = [&](int it) -> uint32_t * {  // null: none
        const uint32_t m = place[it] >> 16, c = place[it] & 0xFFFF;
        return place[it] != ~0u && m0 + m < a.M && c0 + c < a.D2 ? out + (m * a.D2 + c) : nullptr;
      };
      int64_t tot[kItems];
      uint32_t prev[kItems];  // what the outputs hold already, fetched ahead of the chunk
#pragma unroll
      for (int it = 0; it < kItems; ++it) {
        const uint32_t *o = a.acc_in ? output(it) : nullptr;
        tot[it] = 0;
        prev[it] = o ? *o : 0u;
      }
      for (uint32_t ch = 0; ok && ch < nchunk; ++ch) {
#pragma unroll
        for (int it = 0; it < kItems; it += 2) {
          if (it % kPer == 0) {
            if (!__all_sync(0xffffffffu, wait_bounded(tfull + 8 * rt.slot, rt.phase))) {
              ok = false;
              break;
            }
            fence_after();
          }
          const uint32_t item = set + kSets * (it % kPer);
          uint32_t f[4][8];
          if (item < items) {  // two groups in flight; a missing second one is the first again
            const uint32_t src = tmem + rt.slot * a.W + ((32 * quarter) << 16) + 16 * item;
            const uint32_t src2 = item + kSets < items ? src + 16 * kSets : src;
            tmem_ld_16x256b_x2(src, f[0]);
            tmem_ld_16x256b_x2(src + (16 << 16), f[1]);
            tmem_ld_16x256b_x2(src2, f[2]);
            tmem_ld_16x256b_x2(src2 + (16 << 16), f[3]);
            tmem_ld_wait(f[0], f[1], f[2], f[3]);
          }
          // the accumulators are handed back before the arithmetic on their copies: the next
          // unit's MMAs wait for them
          if (it % kPer == kPer - 2) {
            fence_before();
            __syncwarp();
            if (lane == 0) {
              if (CG == 2)
                mbar_arrive_at(tempty_lead + 8 * rt.slot);
              else
                mbar_arrive(tempty + 8 * rt.slot);
            }
            rt.next(a.R);
          }
          if (item < items) {
#pragma unroll
            for (int g2 = 0; g2 < 2; ++g2) {
              int64_t sum[2];
#pragma unroll
              for (int v = 0; v < 2; ++v) {
                int64_t x = 0;
#pragma unroll
                for (int l = 0; l < 4; ++l)
#pragma unroll
                  for (int d = 0; d < 2; ++d)
                    x = mad_wide(__float2int_rn(__uint_as_float(f[2 * g2 + (l >> 1)][4 * v + 2 * (l & 1) + d])),
                                 wgt[l + d], x);
                sum[v] = x;
              }
              // 16 products of 2^24 * 2^30 a chunk: below 2^62 after 16 chunks
              tot[it + g2] += (p ? sum[1] : sum[0]) + __shfl_xor_sync(0xffffffffu, p ? sum[0] : sum[1], 1);
            }
          }
        }
      }
      if (!ok) break;
      // all reductions side by side, outside the stores' branches: one after the other
      // they took longer than the chunk's own arithmetic
      const uint64_t off = (uint64_t)q << 33;  // a multiple of q above 2^62
      uint32_t r[kItems];
#pragma unroll
      for (int it = 0; it < kItems; ++it) {
        r[it] = reduce64((uint64_t)tot[it] + off, q, mu) + prev[it];
        r[it] = min(r[it], r[it] - q);
      }
#pragma unroll
      for (int it = 0; it < kItems; ++it)
        if (uint32_t *o = output(it)) *o = r[it];
    }
    if (!ok && lane == 0) atomicExch(a.err, 1u);
  }

  fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync();
  if (warp == kMmaWarp) {
    fence_after();
    tmem_dealloc<CG>(tmem, kTmem);
  }
}

// qhat rows [B][Ks][2][L][n], ciphertexts k0 .. k0 + Kc - 1 of every query -> f16 digits
// qt [s][u = i / 16][4 * Mp rows][16] in core-matrix blocks (element (row r, position k)
// of a block at (r / 8) * 128 + (k / 8) * 64 + (r % 8) * 8 + k % 8), row r = 4m + a.
// Position k = 4j + t holds ciphertext 2j + t % 2 + 8 (t / 2) of the 16 (in_order: k); rows
// m >= M and the ciphertexts from Kc up to a multiple of 64 are zero.
// CTA = 32 slots x 16 ciphertexts x 8 query rows, as k_query_to_tensor: residues are
// staged in shared memory with coalesced reads along the slots; then a thread takes
// (slot, m, K half) and writes the four 16-byte digit rows of its 8 residues.
__global__ void __launch_bounds__(256) k_query_digits(const uint32_t *__restrict__ qhat, uint32_t M, uint32_t Mp,
                                                      uint32_t Ks, uint32_t k0, uint32_t Kc, uint32_t L, uint32_t logn,
                                                      int in_order, uint16_t *__restrict__ qt) {
  __shared__ uint32_t vals[16][8][33];
  const uint32_t n = 1u << logn;
  const uint32_t s0 = blockIdx.x * 32, u = blockIdx.y, mb = blockIdx.z;
  const uint32_t j = s0 >> logn, slot0 = s0 & (n - 1);
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t v[16];
#pragma unroll
  for (uint32_t r = 0; r < 16; ++r) {
    const uint32_t p = warp + 8 * r, il = p >> 3, ml = p & 7, m = mb * 8 + ml, i = u * 16 + il;
    v[r] = m < M && i < Kc ? __ldg(qhat + ((uint64_t)((uint64_t)(m >> 1) * Ks + k0 + i) * 2 + (m & 1)) * L * n +
                                   (uint64_t)j * n + slot0 + lane)
                           : 0u;
  }
#pragma unroll
  for (uint32_t r = 0; r < 16; ++r) {
    const uint32_t p = warp + 8 * r;
    vals[p >> 3][p & 7][lane] = v[r];
  }
  __syncthreads();
  const uint32_t Ntot = 4 * Mp, Uc = gridDim.y;
  for (uint32_t w = threadIdx.x; w < 32 * 16; w += 256) {
    const uint32_t sl = w >> 4, t = w & 15;
    const uint32_t ml = ((t >> 2) << 1) | (t & 1), h = (t >> 1) & 1;
    if (mb * 8 + ml >= Mp) continue;
    uint32_t b[8];  // 128 + signed digit in bytes 0..2, the top digit in byte 3
#pragma unroll
    for (int e = 0; e < 8; ++e)  // position 8h + e: j = 2h + e / 4, t = e % 4
      b[e] = vals[in_order ? 8 * h + e : 2 * (2 * h + e / 4) + (e & 1) + 8 * ((e >> 1) & 1)][ml][sl] + 0x00808080u;
    const uint64_t s = s0 + sl;
    uint16_t *dst = qt + (s * Uc + u) * (uint64_t)Ntot * 16 + (4 * mb + (ml >> 1)) * 128 + h * 64 + (ml & 1) * 32;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      uint32_t o[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        // two bytes under the exponent of 1024, less 1024 and the bias: exact in f16
        const uint32_t pair = __byte_perm(b[2 * e], b[2 * e + 1], a | (4 + a) << 8);
        const uint32_t bits = (pair & 0x00FF00FFu) | 0x64006400u;
        const __half2 bias = a == 3 ? __float2half2_rn(1024.0f) : __float2half2_rn(1152.0f);
        const __half2 f = __hsub2(*reinterpret_cast<const __half2 *>(&bits), bias);
        o[e] = *reinterpret_cast<const uint32_t *>(&f);
      }
      *reinterpret_cast<uint4 *>(dst + 8 * a) = make_uint4(o[0], o[1], o[2], o[3]);
    }
  }
}

uint32_t round16(uint32_t x) { return (x + 15u) & ~15u; }
uint32_t round64(uint32_t x) { return (x + 63u) & ~63u; }

}  // namespace

// Whole chunks while their digits stay within 1 GiB; longer ones in pieces whose digits
// fit the other tiles' bytes.  tight: the latter for every chunk of 32 rows or more.
uint32_t gemm_digit_rows(uint64_t nslots, uint32_t Kc, uint32_t Mp, bool tight) {
  if (!tight && Kc <= kDigitMaxRows && gemm_digit_query_bytes(nslots, Kc, Mp) <= ((size_t)1 << 30)) return Kc;
  const uint32_t r = Kc / 2 & ~63u;
  return r < 64 ? 64 : r > kDigitMaxRows ? kDigitMaxRows : r;
}

bool gemm_uses_digits(int layout, uint32_t tile, uint32_t M, uint32_t D2, uint32_t Kc, bool acc, bool maps) {
  if (layout == PIR_LAYOUT_TENSOR) return false;
  if (tile == (layout == PIR_LAYOUT_PLAIN ? kDigitTile : kLimbDigitTile)) return true;
  if (tile != 0 || !maps) return false;
  // INT8 mma.sync at its peak is 1.3 to 7 times slower at every size measured (32 to 512 rows
  // and columns, 1 to 32 queries).
  if (layout == PIR_LAYOUT_LIMB) return true;
  return gemm_plain_digits(M, D2, Kc, acc);
}

bool gemm_digit_available() { return tensor_maps_available(); }

size_t gemm_digit_query_bytes(uint64_t nslots, uint32_t Kc, uint32_t Mp) {
  return (size_t)nslots * round64(Kc) * Mp * 8;
}

cudaError_t launch_query_digits(const ParamCtx &c, int layout, const uint32_t *qhat, uint32_t B, uint32_t Ks,
                                uint32_t k0, uint32_t Kc, uint32_t Mp, uint16_t *qt, cudaStream_t s) {
  if (Mp % 4 != 0 || Kc == 0) return cudaErrorInvalidValue;
  dim3 grid((c.p.L << c.logn) / 32, round64(Kc) / 16, (Mp + 7) / 8);
  k_query_digits<<<grid, 256, 0, s>>>(qhat, 2 * B, Mp, Ks, k0, Kc, c.p.L, c.logn, layout == PIR_LAYOUT_LIMB, qt);
  return cudaGetLastError();
}

cudaError_t launch_gemm_digit(const ParamCtx &c, int layout, const void *db, uint32_t D1, uint32_t D2,
                              const uint16_t *qt, uint32_t M, uint32_t Mp, uint32_t i0, uint32_t Kc, uint32_t *out, int acc,
                              cudaStream_t s) {
  if (Kc == 0 || Kc > kDigitMaxRows || i0 + (uint64_t)Kc > D1 || Mp % 4 != 0 || Mp < M || D2 % 4 != 0)
    return cudaErrorInvalidValue;
  DigArgs a = {};
  cudaError_t e = device_error_word(&a.err);
  if (e != cudaSuccess) return e;
  a.out = out;
  a.M = M;
  a.D2 = D2;
  a.i0 = i0;
  a.Kc = Kc;
  a.Uc = round64(Kc) / 16;
  a.logn = c.logn;
  a.acc_in = acc;
  const uint32_t Ntot = 4 * Mp;
  a.mtiles = (Ntot + 255) / 256;
  const uint32_t NT = round16((Ntot + a.mtiles - 1) / a.mtiles);
  // Two accumulators of up to 192 columns leave the A ring 128 of the 512; wider units
  // take three of half their width.
  const uint32_t H = NT > 192 ? 2 : 1, SUB = 2 / H;
  a.NH = H == 2 ? round16(NT / 2) : NT;
  a.R = H == 2 ? 3 : 2;
  const uint32_t CG = H == 2 || (NT >= 128 && D2 > 32) ? 2 : 1;
  // column tiles per unit: as many as 128 accumulator columns hold, spread evenly.  The last unit
  // runs its tiles past D2 too (132 columns: two units of three tiles, 192 columns of work)
  const uint32_t tiles = (D2 + 32 * CG - 1) / (32 * CG);
  const uint32_t tmax = a.NH > 64 ? 1 : 128 / a.NH;
  a.cgroups = (tiles + tmax - 1) / tmax;
  a.T = (tiles + a.cgroups - 1) / a.cgroups;
  a.W = a.T * a.NH;
  a.a0 = a.R * a.W <= 256 ? 256 : 384;
  a.SA = (kTmem - a.a0) / (SUB * kBlockCols);
  const uint64_t nslots = (uint64_t)c.p.L << c.logn, nunits = nslots * a.cgroups * a.mtiles;
  if (nunits > 0x7fffffffull || nslots * a.Uc >= (1ull << 31)) return cudaErrorInvalidValue;
  a.nunits = (uint32_t)nunits;
  a.bstage = (SUB * kRows / 16) * (H * a.NH / CG) * 32;
  const size_t fixed = kBars * 8 + 16 + 8 * PIR_MAX_L * 4;
  a.SB = kMaxB;
  while (a.SB > 2 && a.SB * a.bstage > 100u << 10) --a.SB;
  a.SR = (uint32_t)((kSmemMax - fixed - a.SB * a.bstage) / kRawBytes);
  a.SR = a.SR >= kMaxRaw ? kMaxRaw : 8;  // whole rounds of the converter groups: a slot stays with one group
  size_t smem = a.SR * kRawBytes + a.SB * a.bstage + fixed;
  if (smem < kSmemMin) smem = kSmemMin;
  alignas(64) CUtensorMap tm_db = {}, tm_q = {};
  const bool limb = layout == PIR_LAYOUT_LIMB;
  if (!(limb ? limb_tensor_map(&tm_db, db, D1, D2, nslots, kRows) : word_tensor_map(&tm_db, db, D2, D1, nslots, kRows)) ||
      !digit_tensor_map(&tm_q, qt, Ntot / 8, nslots * a.Uc, a.NH / CG / 8, SUB * kRows / 16))
    return cudaErrorInvalidValue;
  auto launch = [&](auto which) {
    constexpr bool LIMB = decltype(which)::value;
    if (H == 2) return launch_persistent<k_gemm_digit<2, 1, LIMB>, 2>(nunits, kThreads, smem, s, a, c.mod, tm_db, tm_q);
    if (CG == 2) return launch_persistent<k_gemm_digit<2, 2, LIMB>, 2>(nunits, kThreads, smem, s, a, c.mod, tm_db, tm_q);
    return launch_persistent<k_gemm_digit<1, 2, LIMB>, 1>(nunits, kThreads, smem, s, a, c.mod, tm_db, tm_q);
  };
  return limb ? launch(std::true_type()) : launch(std::false_type());
}

}  // namespace gbpir
