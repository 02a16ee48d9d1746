// expand.cu -- server-side query expansion (Sec. 3.5 "ExpPack" expansion; App. C.2:
// SealPIR's recursive expansion after pre-scaling by 2^-levels; App. D.3: expansion
// keys with a gadget of ell digits in base t = 2^ceil(log2 q / ell)).
//
// A client sends one ciphertext encrypting m = sum_i m_i X^i instead of D1
// ciphertexts; the server expands it into the D1 ciphertexts Enc(m_i).  Level j of
// the recursion turns each of its 2^j ciphertexts c (index k) into
//     c + Subs(c, g_j)                               at index k,
//     c X^-2^j + Subs(c X^-2^j, g_j)                 at index k + 2^j,
// with g_j = n / 2^j + 1 and Subs = substitution X -> X^g followed by key switching
// back to the secret s with level j's key.
//
// GPU design: ciphertexts stay in NTT form between levels.  In that form the
// substitution is a permutation of slots (NTT(tau_g a)[k] = NTT(a)[perm(k)], no
// arithmetic) and X^-2^j is a pointwise factor.  The gadget digits are those of the
// level's input a-part, moved by the same shift and substitution as the ciphertext
// (signed digits in (-t, t); sum_k t^k tau_g(d_k X^-C) = tau_g(a X^-C)).  Moved
// digits are permuted and scaled copies of NTT(d_k), so both branches share one
// key-switching sum S[s] = sum_k NTT(d_k)[perm(s)] K_k[s]; branch 1 multiplies it by
// NTT(X^-C)[perm(s)].  Each level is three launches over all its ciphertexts (gadget.cu).
#include <mutex>
#include <set>
#include <vector>

#include "common.cuh"

namespace gbpir {
namespace {

constexpr uint64_t kExpanderMagic = 0x4558504e44455231ull;  // "EXPNDER1"
constexpr uint32_t kMaxEll = 16;

// Pre-scaling constants of the ring.
struct ScaleConst {
  uint32_t q[PIR_MAX_L];
  uint32_t inv2l[PIR_MAX_L], inv2l_sh[PIR_MAX_L];  // 2^-levels mod q_i
};

// x * 2^-levels for every residue of rows [rows][n]: block = one row, row r under prime r % L.
__global__ void k_expand_scale(uint32_t *x, uint32_t n, uint32_t L, ScaleConst E) {
  const uint32_t i = blockIdx.x % L;
  uint32_t q = E.q[0], w = E.inv2l[0], wsh = E.inv2l_sh[0];
#pragma unroll
  for (uint32_t k = 1; k < PIR_MAX_L; ++k)
    if (i == k) q = E.q[k], w = E.inv2l[k], wsh = E.inv2l_sh[k];
  uint4 *row = reinterpret_cast<uint4 *>(x + (uint64_t)blockIdx.x * n);
  chain_wait();
  for (uint32_t e = threadIdx.x; e < n / 4; e += blockDim.x) {
    uint4 v = row[e];
    v.x = shoup_mul(v.x, w, wsh, q), v.x = min(v.x, v.x - q);
    v.y = shoup_mul(v.y, w, wsh, q), v.y = min(v.y, v.y - q);
    v.z = shoup_mul(v.z, w, wsh, q), v.z = min(v.z, v.z - q);
    v.w = shoup_mul(v.w, w, wsh, q), v.w = min(v.w, v.w - q);
    row[e] = v;
  }
}

uint64_t mul_mod64(uint64_t a, uint64_t b, uint64_t m) { return (uint64_t)((unsigned __int128)a * b % m); }
uint64_t pow_mod64(uint64_t b, uint64_t e, uint64_t m);
uint32_t shoup32(uint32_t w, uint32_t q);

ScaleConst make_scale_const(const pir_params_t &p, uint32_t levels) {
  ScaleConst E = {};
  for (uint32_t k = 0; k < p.L; ++k) {
    const uint32_t qk = p.q[k];
    E.q[k] = qk;
    E.inv2l[k] = (uint32_t)pow_mod64(pow_mod64(2, levels, qk), qk - 2, qk);
    E.inv2l_sh[k] = shoup32(E.inv2l[k], qk);
  }
  return E;
}
uint64_t pow_mod64(uint64_t b, uint64_t e, uint64_t m) {
  uint64_t r = 1 % m;
  b %= m;
  for (; e; e >>= 1) {
    if (e & 1) r = mul_mod64(r, b, m);
    b = mul_mod64(b, b, m);
  }
  return r;
}
uint32_t shoup32(uint32_t w, uint32_t q) { return (uint32_t)(((uint64_t)w << 32) / q); }
uint32_t brv32(uint32_t x, uint32_t bits) {
  uint32_t r = 0;
  for (uint32_t b = 0; b < bits; ++b) r |= ((x >> b) & 1u) << (bits - 1 - b);
  return r;
}

}  // namespace

struct pir_expander_impl {
  uint64_t magic;
  pir_params_t p;
  const ParamCtx *ctx;
  int device;
  uint32_t levels, ell, w;
  uint32_t *tables;  // one allocation: keys | mon | mon_sh | perm
  const uint32_t *keys, *mon, *mon_sh, *perm;
  ScaleConst scale;
  GadgetConst gadget;
};

namespace {
std::mutex g_ex_mu;
std::set<const void *> g_ex_live;

bool ex_live(const void *e) {
  std::lock_guard<std::mutex> lock(g_ex_mu);
  return e && g_ex_live.count(e) && static_cast<const pir_expander_impl *>(e)->magic == kExpanderMagic;
}

// ceil(log2 q) for q = prod q_j
uint32_t modulus_bits(const pir_params_t &p) {
  unsigned __int128 q = 1;
  for (uint32_t j = 0; j < p.L; ++j) q *= p.q[j];
  uint32_t bits = 0;
  while (bits < 128 && ((unsigned __int128)1 << bits) < q) ++bits;
  return bits;
}
}  // namespace

// Expansion of B packed ciphertexts (device, coefficient form [B][2][L][n]) into
// out [B][count][2][L][n] in NTT form.  Scratch from the stream-ordered allocator.
pir_status_t expand_device(const pir_expander_impl *ex, const uint32_t *packed, uint32_t B, uint32_t count,
                           uint32_t *out, cudaStream_t s, uint64_t *launch_count) {
  const ParamCtx &c = *ex->ctx;
  const uint32_t n = ex->p.n, L = ex->p.L, levels = ex->levels, ell = ex->ell;
  const uint64_t ctw = 2ull * L * n;             // words per ciphertext
  const uint64_t full = 1ull << levels;           // ciphertexts per query after the last level
  const uint64_t half = full >> 1 ? full >> 1 : 1;
  // per query: two ciphertext buffers of `full`, digits and their NTT
  const uint64_t per_q = (2 * full * ctw + half * ell * n + half * ell * L * n) * 4;
  size_t free_b = 0, total_b = 0;
  uint64_t budget = 1ull << 30;
  if (cudaMemGetInfo(&free_b, &total_b) == cudaSuccess && free_b / 4 > budget) budget = free_b / 4;
  uint32_t Bc = (uint32_t)(budget / per_q);
  if (Bc < 1) Bc = 1;
  if (Bc > B) Bc = B;
  void *scratch = nullptr;
  cudaError_t e = cudaMallocAsync(&scratch, per_q * Bc, s);
  if (e != cudaSuccess) return cuda_status(e);
  uint32_t *cur = static_cast<uint32_t *>(scratch);
  uint32_t *nxt = cur + Bc * full * ctw;
  uint32_t *dig = nxt + Bc * full * ctw;
  uint32_t *dhat = dig + Bc * half * ell * n;
  pir_status_t st = PIR_OK;
  auto ck = [&](cudaError_t err) {
    if (err != cudaSuccess && st == PIR_OK) st = cuda_status(err);
    return err == cudaSuccess;
  };
  uint64_t launches = 0;
  for (uint32_t b0 = 0; b0 < B && st == PIR_OK; b0 += Bc) {
    const uint32_t nb = B - b0 < Bc ? B - b0 : Bc;
    // level-0 input: NTT of the packed ciphertexts, times 2^-levels
    if (!ck(launch_ntt_fwd(c, packed + (uint64_t)b0 * ctw, cur, (uint64_t)nb * 2 * L, s))) break;
    if (!ck(launch_chained(k_expand_scale, nb * 2 * L, 256, 0, s, cur, n, L, ex->scale))) break;
    launches += 2;
    for (uint32_t lev = 0; lev < levels; ++lev) {
      const bool last = lev + 1 == levels;
      const uint32_t *mon = ex->mon + (uint64_t)lev * L * n, *msh = ex->mon_sh + (uint64_t)lev * L * n;
      const uint32_t width = last ? count : 2u << lev;  // ciphertexts per query after the level
      if (!ck(launch_expand_level(c, ex->gadget, cur, ex->keys + (uint64_t)lev * ell * ctw, mon, msh,
                                  ex->perm + (uint64_t)lev * n, nb, lev, ell, width, width, dig, dhat,
                                  last ? out + (uint64_t)b0 * count * ctw : nxt, s)))
        break;
      launches += 3;
      uint32_t *t = cur;
      cur = nxt;
      nxt = t;
    }
    if (levels == 0 && st == PIR_OK) {  // one ciphertext: the scaled input itself
      ck(cudaMemcpyAsync(out + (uint64_t)b0 * count * ctw, cur, (uint64_t)nb * ctw * 4, cudaMemcpyDeviceToDevice, s));
    }
  }
  cudaFreeAsync(scratch, s);
  *launch_count = launches;
  return st;
}

uint32_t gadget_bits(const pir_params_t &p, uint32_t ell) { return (modulus_bits(p) + ell - 1) / ell; }

GadgetConst gadget_const(const pir_params_t &p) {
  GadgetConst g = {};
  for (uint32_t k = 0; k < p.L; ++k)
    for (uint32_t i = 0; i < k; ++i) {
      g.gc[k][i] = (uint32_t)pow_mod64(p.q[i] % p.q[k], p.q[k] - 2, p.q[k]);
      g.gc_sh[k][i] = shoup32(g.gc[k][i], p.q[k]);
    }
  return g;
}

bool expander_view(pir_expander_t h, const pir_expander_impl **out) {
  if (!ex_live(h)) return false;
  *out = reinterpret_cast<const pir_expander_impl *>(h);
  return true;
}

bool expander_fits(const pir_expander_impl *ex, const pir_params_t &p) {
  if (ex->p.n != p.n || ex->p.L != p.L) return false;
  for (uint32_t j = 0; j < p.L; ++j)
    if (ex->p.q[j] != p.q[j] || ex->p.psi[j] != p.psi[j]) return false;
  return (1ull << ex->levels) >= p.D1;
}

}  // namespace gbpir

using namespace gbpir;

extern "C" {

pir_status_t pir_expander_create(const pir_params_t *params, uint32_t levels, uint32_t ell, const uint32_t *keys,
                                 int keys_on_device, void *stream, pir_expander_t *out) {
  if (!params || !keys || !out) return PIR_ERR_ARG;
  *out = nullptr;
  pir_status_t st = validate_params(params);
  if (st != PIR_OK) return st;
  const uint32_t n = params->n, L = params->L;
  if ((1u << levels) > n || levels > 31 || ell == 0 || ell > kMaxEll) return PIR_ERR_ARG;
  const uint32_t bits = modulus_bits(*params);
  const uint32_t w = (bits + ell - 1) / ell;
  if (w > 30 || w * (ell - 1) >= 128) return PIR_ERR_ARG;  // digits must stay below every prime's 2^30
  const ParamCtx *ctx = nullptr;
  if ((st = get_param_ctx(params, &ctx)) != PIR_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const uint32_t logn = ctx->logn;
  const uint64_t key_words = (uint64_t)levels * ell * 2 * L * n;
  const uint64_t mon_words = (uint64_t)levels * L * n;
  const uint64_t words = key_words + 2 * mon_words + (uint64_t)levels * n;

  auto *ex = new pir_expander_impl();
  ex->magic = kExpanderMagic;
  ex->p = *params;
  ex->p.D1 = ex->p.D2 = 0;
  ex->ctx = ctx;
  cudaGetDevice(&ex->device);
  ex->levels = levels;
  ex->ell = ell;
  ex->w = w;
  // host tables: NTT(X^-2^j) per prime (squares of NTT(X^-1)), slot permutations
  std::vector<uint32_t> host(2 * mon_words + (uint64_t)levels * n);
  uint32_t *hmon = host.data(), *hsh = hmon + mon_words, *hperm = hsh + mon_words;
  for (uint32_t i = 0; i < L; ++i) {
    const uint64_t q = params->q[i];
    const uint64_t psi_inv = pow_mod64(params->psi[i], q - 2, q);
    std::vector<uint64_t> v(n);
    for (uint32_t k = 0; k < n; ++k) v[k] = pow_mod64(psi_inv, 2ull * brv32(k, logn) + 1, q);  // X^-1 at slot k
    for (uint32_t j = 0; j < levels; ++j) {
      for (uint32_t k = 0; k < n; ++k) {
        const uint64_t o = ((uint64_t)j * L + i) * n + k;
        hmon[o] = (uint32_t)v[k];
        hsh[o] = shoup32((uint32_t)v[k], (uint32_t)q);
        v[k] = mul_mod64(v[k], v[k], q);  // X^-2^(j+1)
      }
    }
  }
  for (uint32_t j = 0; j < levels; ++j) {
    const uint64_t g = (n >> j) + 1, two_n = 2ull * n;
    for (uint32_t k = 0; k < n; ++k) {
      const uint64_t e = (2ull * brv32(k, logn) + 1) * g % two_n;
      hperm[(uint64_t)j * n + k] = brv32((uint32_t)((e - 1) / 2), logn);
    }
  }
  ex->scale = make_scale_const(*params, levels);
  ex->gadget = gadget_const(*params);
  cudaError_t e = cudaMalloc(&ex->tables, words * 4);
  if (e != cudaSuccess) {
    delete ex;
    return cuda_status(e);
  }
  ex->keys = ex->tables;
  ex->mon = ex->tables + key_words;
  ex->mon_sh = ex->mon + mon_words;
  ex->perm = ex->mon_sh + mon_words;
  auto fail = [&](cudaError_t err) {
    cudaFree(ex->tables);
    delete ex;
    return cuda_status(err);
  };
  if ((e = cudaMemcpyAsync(ex->tables, keys, key_words * 4,
                           keys_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s)) != cudaSuccess)
    return fail(e);
  if ((e = cudaMemcpyAsync(ex->tables + key_words, host.data(), host.size() * 4, cudaMemcpyHostToDevice, s)) !=
      cudaSuccess)
    return fail(e);
  // keys to NTT form: rows [levels][ell][2][L] with row r under prime r % L
  if ((e = launch_ntt_fwd(*ctx, ex->tables, ex->tables, key_words / n, s)) != cudaSuccess) return fail(e);
  count_launches(1);
  if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return fail(e);
  {
    std::lock_guard<std::mutex> lock(g_ex_mu);
    g_ex_live.insert(ex);
  }
  *out = reinterpret_cast<pir_expander_t>(ex);
  return PIR_OK;
}

pir_status_t pir_expander_free(pir_expander_t h) {
  if (!ex_live(h)) return PIR_ERR_HANDLE;
  auto *ex = reinterpret_cast<pir_expander_impl *>(h);
  {
    std::lock_guard<std::mutex> lock(g_ex_mu);
    g_ex_live.erase(ex);
  }
  cudaDeviceSynchronize();
  cudaFree(ex->tables);
  ex->magic = 0;
  delete ex;
  return PIR_OK;
}

pir_status_t pir_expand(pir_expander_t h, const uint32_t *packed, uint32_t B, uint32_t count, uint32_t *out,
                        void *stream) {
  const pir_expander_impl *ex = nullptr;
  if (!expander_view(h, &ex)) return PIR_ERR_HANDLE;
  if (!packed || !out || B == 0 || count == 0 || count > (1u << ex->levels)) return PIR_ERR_ARG;
  if (((uintptr_t)packed & 15u) || ((uintptr_t)out & 15u)) return PIR_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  uint64_t launches = 0;
  pir_status_t st = expand_device(ex, packed, B, count, out, s, &launches);
  count_launches(launches);
  if (st != PIR_OK) return st;
  // the public result is in coefficient form, like the queries pir_answer takes
  cudaError_t e = launch_ntt_inv(*ex->ctx, out, out, (uint64_t)B * count * 2 * ex->p.L, s);
  if (e != cudaSuccess) return cuda_status(e);
  count_launches(1);
  return PIR_OK;
}

}  // extern "C"
