// gadget.cu -- one level of query expansion or of folding: gadget decomposition (App. D.3)
// of ciphertexts in NTT form and the product with a key, over all ciphertexts of all queries.
//
// Three launches: (1) the inverse NTT of the polynomials, the CRT lift of every coefficient
// (Garner) and its ell digits of w bits; (2) the forward NTT of every digit row under every
// prime (ntt.cu); (3) the sums of digit times key row and the outputs:
//   expansion (expand.cu): one polynomial a of ciphertext (a, b); with p = perm(s)
//       S_c[s] = sum_d NTT(d)[p] K_d.c[s],
//       branch 0 -> (a + S_a, b + b[p] + S_b),
//       branch 1 -> ((a - S_a) m, (b - b[p] - S_b) m),   m = NTT(X^-2^j), m[p] = -m[s];
//   folding (fold.cu): both polynomials of c_1 - c_0,
//       c_0 + sum_r NTT(d_r) G_r,   r over the 2 ell digits.
//
// Four queries, n = 2^12, L = 2, ell = 4: nine levels of expansion 673 -> 440 us, eight of folding
// 620 -> 370 us against four and five launches with 64-bit divisions by n and L per element,
// 4-byte accesses and 64-bit reductions.  The last expansion level takes 32 + 75 + 68 us, bound by
// the transforms' multiply-adds, then by L2 and memory; a first one 3 x 7 us of latency.  A level as
// one launch (clusters of L CTAs, all in shared memory) took 182 us there and 193 instead of
// 135 us on the first folding level: its phases leave the multiply-add pipe idle more often
// than the arrays between the launches cost.
#include <atomic>
#include <type_traits>

#include "ntt_row.cuh"

namespace gbpir {
namespace {

// ldg4: of tables and keys only (chain_wait)
__device__ __forceinline__ void ldg4(uint32_t (&v)[4], const uint32_t *p) {
  const uint4 x = __ldg(reinterpret_cast<const uint4 *>(p));
  v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
}
__device__ __forceinline__ void ld4(uint32_t (&v)[4], const uint32_t *p) {
  const uint4 x = *reinterpret_cast<const uint4 *>(p);
  v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
}
__device__ __forceinline__ void st4(uint32_t *p, const uint32_t (&v)[4]) {
  *reinterpret_cast<uint4 *>(p) = make_uint4(v[0], v[1], v[2], v[3]);
}

// Coefficient from its residues (word k of stride `stride`: mod q_k).
template <uint32_t L>
__device__ __forceinline__ std::conditional_t<(L > 2), unsigned __int128, uint64_t> lift(
    const uint32_t *x, uint32_t stride, const NttConst &C, const GadgetConst &g) {
  uint32_t v[L];
#pragma unroll
  for (uint32_t k = 0; k < L; ++k) v[k] = x[k * stride];
  // Garner: X = v_0 + q_0 (v_1 + q_1 (v_2 + q_2 v_3)), v_k in [0, q_k)
#pragma unroll
  for (uint32_t k = 1; k < L; ++k) {
    const uint32_t qk = C.q[k];
    uint32_t r = v[k];
#pragma unroll
    for (uint32_t i = 0; i < k; ++i)
      r = csub(shoup_mul(r + qk - csub(v[i], qk), g.gc[k][i], g.gc_sh[k][i], qk), qk);
    v[k] = r;
  }
  std::conditional_t<(L > 2), unsigned __int128, uint64_t> X = v[L - 1];
#pragma unroll
  for (int k = (int)L - 2; k >= 0; --k) X = X * C.q[k] + v[k];
  return X;
}

// Rows inverted at once by a block (n/16 threads each).
template <int LOGN, uint32_t L>
constexpr uint32_t kGroups = L < (16384u >> LOGN) ? L : (16384u >> LOGN);

// Digits of one polynomial per block: dig [blocks][ell][n].  Expansion: block = ciphertext,
// its first polynomial; folding: block = 2 pair + component, of the pair's difference.
// Coefficients stay in shared memory between the inverse transform and the lift.
template <int LOGN, uint32_t L, bool FOLD>
__global__ void __launch_bounds__(kGroups<LOGN, L> << (LOGN - 4),
                                  (kGroups<LOGN, L> << (LOGN - 4)) > 768 ? 1 : 1536 / (kGroups<LOGN, L> << (LOGN - 4)))
    k_gadget_digits(const uint32_t *cur, uint32_t *dig, NttConst C, GadgetConst g, uint32_t ell, uint32_t w) {
  constexpr uint32_t N = 1u << LOGN, PADN = N + N / 16, T = N / 16, G = kGroups<LOGN, L>;
  extern __shared__ uint32_t sm[];
  const uint32_t grp = threadIdx.x / T, tid = threadIdx.x % T;
  const bool wide = wide_ok(cur);
  const uint64_t ctw = 2ull * L * N;
  chain_wait();
  const uint32_t *src = FOLD ? cur + (blockIdx.x >> 1) * 2 * ctw + (blockIdx.x & 1) * (L * N) : cur + blockIdx.x * ctw;
#pragma unroll 1
  for (uint32_t j0 = 0; j0 < L; j0 += G) {
    const uint32_t j = j0 + grp;
    const bool act = L % G == 0 || j < L;  // the barriers below are reached by all
    const uint32_t jj = act ? j : 0, q = pick(C.q, jj);
    const uint2 *tw = pick(C.inv, jj);
    uint32_t *row = sm + jj * PADN;
    if (act) {
      const uint32_t *p = src + jj * N + 16 * tid;
      uint32_t v[16];
      load16(p, v, wide);
      if (FOLD) {
        uint32_t u[16];
        load16(p + ctw, u, wide);
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = csub(u[e] + q - v[e], q);
      }
      inv_first<LOGN>(row, tw, q, tid, v);
      __syncwarp();
      mid_pass<LOGN, LOGN == 13 ? 5 : 4, false>(row, tw, q, tid);
    }
    __syncthreads();
    // (the last pass reads and writes the same elements of a thread)
    if (act)
      inv_last<LOGN>(row, tw, q, pick(C.ninv, jj), pick(C.ninv_sh, jj), tid,
                     [&](uint32_t i, uint32_t x) { row[padx<LOGN>(i)] = x; });
  }
  __syncthreads();
  uint32_t *out = dig + (uint64_t)blockIdx.x * ell * N;
  const uint32_t mask = (1u << w) - 1;
  for (uint32_t i = 4 * threadIdx.x; i < N; i += 4 * G * T) {
    const uint32_t pt = padx<LOGN>(i);  // four consecutive positions stay consecutive
    const auto X0 = lift<L>(sm + pt, PADN, C, g), X1 = lift<L>(sm + pt + 1, PADN, C, g),
               X2 = lift<L>(sm + pt + 2, PADN, C, g), X3 = lift<L>(sm + pt + 3, PADN, C, g);
    uint32_t *o = out + i;
    // (a shift past the lift's width leaves nothing: few bits over many digits)
    for (uint32_t k = 0, bit = 0; k < ell; ++k, bit += w, o += N) {
      uint32_t d[4] = {};
      if (bit < 8 * sizeof(X0))
        d[0] = (uint32_t)(X0 >> bit) & mask, d[1] = (uint32_t)(X1 >> bit) & mask, d[2] = (uint32_t)(X2 >> bit) & mask,
        d[3] = (uint32_t)(X3 >> bit) & mask;
      st4(o, d);
    }
  }
}

struct MacArgs {
  const uint32_t *cur, *dhat;  // cur [cts][2][L][n], folding [2 cts][2][L][n]; dhat [cts][rows][L][n]
  const uint32_t *key;         // [rows][2][L][n]; folding: of query 0 at this level
  const uint32_t *mon, *mon_sh, *perm;  // expansion: NTT(X^-2^j) [L][n], Shoup companions, [n]
  uint32_t *out;
  uint64_t key_query;          // folding: words from one query's keys to the next's
  uint32_t logn, rows;         // rows: digits per ciphertext
  uint32_t log2c;              // expansion: ciphertexts per query, folding: pairs per query (log2)
  uint32_t ostride, olimit;    // expansion: ciphertexts per query in out, and how many are wanted
  ModConst mod;
};

constexpr uint32_t kMacThreads = 128;

// Four neighbouring slots of one prime of C neighbouring ciphertexts (of one query, if C > 1) per
// thread: block = (C ciphertexts, prime, 512 slots).  Bound by L2: a key row is as long as a digit
// row and is read for both components, so C ciphertexts share one reading.
template <bool FOLD, int C>
__global__ void __launch_bounds__(kMacThreads) k_gadget_mac(const MacArgs a) {
  const uint32_t n = 1u << a.logn, L = gridDim.y, i = blockIdx.y, s = 4 * (blockIdx.z * kMacThreads + threadIdx.x);
  const uint32_t q = pick(a.mod.q, i), comp = L * n;
  const uint64_t mu = pick(a.mod.mu, i), k63 = pick(a.mod.k63, i), ctw = 2ull * comp;
  const uint64_t ct = (uint64_t)blockIdx.x * C, query = ct >> a.log2c;
  const uint32_t k0 = (uint32_t)ct & ((1u << a.log2c) - 1), at = i * n + s;
  chain_wait();
  if (!FOLD && k0 >= a.olimit) return;
  const uint32_t *in = a.cur + ct * (FOLD ? 2 : 1) * ctw + at;
  const uint64_t in_step = (FOLD ? 2 : 1) * ctw, dh_step = (uint64_t)a.rows * comp;
  uint64_t acc_a[C][4], acc_b[C][4];
  uint32_t va[C][4], vb[C][4], p[4];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    ld4(va[c], in + c * in_step);
    ld4(vb[c], in + c * in_step + comp);
#pragma unroll
    for (int e = 0; e < 4; ++e) acc_a[c][e] = FOLD ? va[c][e] : 0, acc_b[c][e] = FOLD ? vb[c][e] : 0;
  }
  if (!FOLD) ldg4(p, a.perm + s);
  const uint32_t *key = a.key + (FOLD ? query * a.key_query : 0) + at;
  const uint32_t *dh = a.dhat + ct * dh_step + i * n + (FOLD ? s : 0);
#pragma unroll 2
  for (uint32_t r = 0; r < a.rows; ++r) {
    uint32_t ka[4], kb[4];
    ldg4(ka, key);
    ldg4(kb, key + comp);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      uint32_t d[4];
      if (FOLD) {
        ld4(d, dh + c * dh_step);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) d[e] = dh[c * dh_step + p[e]];
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        mac_wide(acc_a[c][e], d[e], ka[e]);
        mac_wide(acc_b[c][e], d[e], kb[e]);
      }
    }
    key += ctw;
    dh += comp;
    if ((r & 7) == 7) {
#pragma unroll
      for (int c = 0; c < C; ++c)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc_a[c][e] = fold63(acc_a[c][e], k63), acc_b[c][e] = fold63(acc_b[c][e], k63);
    }
  }
  uint32_t m[4], msh[4], bp[C][4];  // bp: b[p] of all C, read before the first output is written
  if (!FOLD) {
    ldg4(m, a.mon + at);
    ldg4(msh, a.mon_sh + at);
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int e = 0; e < 4; ++e) bp[c][e] = a.cur[(ct + c) * ctw + comp + i * n + p[e]];
  }
#pragma unroll
  for (int c = 0; c < C; ++c) {
    uint32_t sa[4], sb[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) sa[e] = reduce64(acc_a[c][e], q, mu), sb[e] = reduce64(acc_b[c][e], q, mu);
    if (FOLD) {
      uint32_t *o = a.out + (ct + c) * ctw + at;
      st4(o, sa);
      st4(o + comp, sb);
    } else {
      if (k0 + c >= a.olimit) return;
      uint32_t *o = a.out + (query * a.ostride + k0 + c) * ctw + at;
      uint32_t o0[4], o1[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        sb[e] = csub(bp[c][e] + sb[e], q);  // b[p] + S_b
        o0[e] = csub(va[c][e] + sa[e], q);
        o1[e] = csub(vb[c][e] + sb[e], q);
      }
      st4(o, o0);
      st4(o + comp, o1);
      const uint32_t half = 1u << a.log2c;
      if (k0 + c + half < a.olimit) {
        // m[p] = -m[s]: the substitution takes X^-2^j to X^(-2^j - n) = -X^-2^j
        o += half * ctw;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          o0[e] = csub(shoup_mul(va[c][e] + q - sa[e], m[e], msh[e], q), q);
          o1[e] = csub(shoup_mul(vb[c][e] + q - sb[e], m[e], msh[e], q), q);
        }
        st4(o, o0);
        st4(o + comp, o1);
      }
    }
  }
}

template <int LOGN, uint32_t L, bool FOLD>
cudaError_t digits_launch(const ParamCtx &c, const GadgetConst &g, const uint32_t *cur, uint64_t polys, uint32_t ell,
                          uint32_t *dig, cudaStream_t s) {
  constexpr uint32_t N = 1u << LOGN;
  constexpr int smem = L * (N + N / 16) * 4;
  const auto kernel = k_gadget_digits<LOGN, L, FOLD>;
  if (smem > 48 * 1024) {
    static std::atomic<uint64_t> known{0};  // devices whose limit is raised
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 64 || !(known.load(std::memory_order_acquire) >> dev & 1)) {
      if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) return e;
      if (dev < 64) known.fetch_or(1ull << dev, std::memory_order_acq_rel);
    }
  }
  return launch_chained(kernel, (unsigned)polys, kGroups<LOGN, L> * N / 16, smem, s, cur, dig, c.ntt, g, ell,
                        gadget_bits(c.p, ell));
}

template <int LOGN, bool FOLD>
cudaError_t digits_ring(const ParamCtx &c, const GadgetConst &g, const uint32_t *cur, uint64_t polys, uint32_t ell,
                        uint32_t *dig, cudaStream_t s) {
  switch (c.p.L) {
    case 1: return digits_launch<LOGN, 1, FOLD>(c, g, cur, polys, ell, dig, s);
    case 2: return digits_launch<LOGN, 2, FOLD>(c, g, cur, polys, ell, dig, s);
    case 3: return digits_launch<LOGN, 3, FOLD>(c, g, cur, polys, ell, dig, s);
    case 4: return digits_launch<LOGN, 4, FOLD>(c, g, cur, polys, ell, dig, s);
  }
  return cudaErrorInvalidValue;
}

// cts ciphertexts (expansion) or pairs (folding) through the three launches.
template <bool FOLD>
cudaError_t level(const ParamCtx &c, const GadgetConst &g, MacArgs &a, uint64_t cts, uint32_t ell, uint32_t *dig,
                  uint32_t *dhat, cudaStream_t s) {
  if (cts == 0) return cudaSuccess;
  const uint32_t L = c.p.L, n = c.p.n;
  const uint64_t polys = FOLD ? 2 * cts : cts;
  if (polys > 0x7fffffffull) return cudaErrorInvalidValue;
  cudaError_t e = cudaErrorInvalidValue;
  switch (c.logn) {
    case 11: e = digits_ring<11, FOLD>(c, g, a.cur, polys, ell, dig, s); break;
    case 12: e = digits_ring<12, FOLD>(c, g, a.cur, polys, ell, dig, s); break;
    case 13: e = digits_ring<13, FOLD>(c, g, a.cur, polys, ell, dig, s); break;
  }
  if (e != cudaSuccess) return e;
  // local row r reads digit row r / L
  if ((e = launch_ntt_fwd_rows_t(c, dig, 0, L, 1, 0, dhat, polys * ell * L, s)) != cudaSuccess) return e;
  a.dhat = dhat;
  a.mod = c.mod;
  a.logn = c.logn;
  a.rows = FOLD ? 2 * ell : ell;
  // two ciphertexts a thread (the keys read once for both) once that still gives every SM sixteen
  // blocks; below, the level is bound by latency and wants the threads
  const dim3 grid((unsigned)cts, L, n / (4 * kMacThreads));
  if (a.log2c >= 1 && cts * L * grid.z >= 152 * 32)
    return launch_chained(k_gadget_mac<FOLD, 2>, dim3(grid.x / 2, grid.y, grid.z), kMacThreads, 0, s, a);
  return launch_chained(k_gadget_mac<FOLD, 1>, grid, kMacThreads, 0, s, a);
}

}  // namespace

cudaError_t launch_expand_level(const ParamCtx &c, const GadgetConst &g, const uint32_t *cur, const uint32_t *key,
                                const uint32_t *mon, const uint32_t *mon_sh, const uint32_t *perm, uint32_t queries,
                                uint32_t lev, uint32_t ell, uint32_t ostride, uint32_t olimit, uint32_t *dig,
                                uint32_t *dhat, uint32_t *out, cudaStream_t s) {
  MacArgs a = {};
  a.cur = cur, a.key = key, a.mon = mon, a.mon_sh = mon_sh, a.perm = perm, a.out = out;
  a.log2c = lev, a.ostride = ostride, a.olimit = olimit;
  return level<false>(c, g, a, (uint64_t)queries << lev, ell, dig, dhat, s);
}

cudaError_t launch_fold_level(const ParamCtx &c, const GadgetConst &g, const uint32_t *cur, const uint32_t *rgsw,
                              uint64_t query_words, uint32_t queries, uint32_t plog, uint32_t ell, uint32_t *dig,
                              uint32_t *dhat, uint32_t *out, cudaStream_t s) {
  MacArgs a = {};
  a.cur = cur, a.key = rgsw, a.key_query = query_words, a.out = out;
  a.log2c = plog;
  return level<true>(c, g, a, (uint64_t)queries << plog, ell, dig, dhat, s);
}

}  // namespace gbpir
