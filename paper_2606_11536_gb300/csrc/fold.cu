// fold.cu -- the remaining dimensions of poly-HE folding: RGSW-RLWE external
// products (Sec. 3.2 and 3.6, OnionPIR's construction; gadget of App. D.3).
//
// After the first-dimension scan every query has 2^levels response ciphertexts.
// Level l pairs them, (c_2j, c_2j+1) -> c_2j + RGSW_l (x) (c_2j+1 - c_2j), where RGSW_l
// encrypts bit l of the wanted column, until one ciphertext is left.  The external
// product writes the difference in the gadget (ell digits of the CRT lift of every
// coefficient of both components) and sums digit x RGSW row products.
//
// GPU design: ciphertexts stay in NTT form between levels (the first-dimension result
// is handed over before its inverse NTT).  A level is three launches over all pairs of all
// queries (gadget.cu): the difference, its inverse NTT and gadget digits; their forward NTT
// under every prime; c_2j + sum_r NTT(d_r) RGSW[r].
#include "common.cuh"

namespace gbpir {

// Fold B queries' 2^levels ciphertexts (NTT form, cur [B][2^levels][2][L][n]) with
// their RGSW ciphertexts (NTT form, rgsw [B][levels][2 ell][2][L][n]) into out
// [B][2][L][n] (NTT form).  cur is overwritten.  Scratch from the stream-ordered allocator.
pir_status_t fold_device(const ParamCtx &c, uint32_t *cur, uint32_t B, uint32_t levels, uint32_t ell,
                         const uint32_t *rgsw, uint32_t *out, cudaStream_t s, uint64_t *launch_count) {
  const uint64_t ctw = 2ull * c.p.L * c.p.n;
  *launch_count = 0;
  if (levels == 0) {
    cudaError_t e = cudaMemcpyAsync(out, cur, (uint64_t)B * ctw * 4, cudaMemcpyDeviceToDevice, s);
    return e == cudaSuccess ? PIR_OK : cuda_status(e);
  }
  const uint64_t pairs0 = (uint64_t)B << (levels - 1);
  // scratch: next level | digits | their NTT
  const uint32_t n = c.p.n, L = c.p.L;
  void *scratch = nullptr;
  cudaError_t e = cudaMallocAsync(&scratch, (pairs0 * ctw + pairs0 * 2 * ell * n * (1 + L)) * 4, s);
  if (e != cudaSuccess) return cuda_status(e);
  uint32_t *nxt = static_cast<uint32_t *>(scratch);
  uint32_t *dig = nxt + pairs0 * ctw;
  uint32_t *dhat = dig + pairs0 * 2 * ell * n;
  const GadgetConst g = gadget_const(c.p);
  pir_status_t st = PIR_OK;
  auto ck = [&](cudaError_t err) {
    if (err != cudaSuccess && st == PIR_OK) st = cuda_status(err);
    return err == cudaSuccess;
  };
  for (uint32_t lev = 0; lev < levels; ++lev) {
    const uint32_t plog = levels - 1 - lev;  // pairs per query = 2^plog
    uint32_t *dst = lev + 1 == levels ? out : nxt;
    if (!ck(launch_fold_level(c, g, cur, rgsw + (uint64_t)lev * 2 * ell * ctw, (uint64_t)levels * 2 * ell * ctw, B, plog,
                              ell, dig, dhat, dst, s)))
      break;
    *launch_count += 3;
    // the level's output becomes the next input; the old input area takes the next output
    uint32_t *t = cur;
    cur = nxt;
    nxt = t;
  }
  cudaFreeAsync(scratch, s);
  return st;
}

}  // namespace gbpir

using namespace gbpir;

extern "C" pir_status_t pir_fold(const pir_params_t *params, const uint32_t *cts, uint32_t B, uint32_t levels,
                                 uint32_t ell, const uint32_t *rgsw, uint32_t *out, void *stream) {
  if (!params || !cts || !rgsw || !out || B == 0 || levels > 20 || ell == 0 || ell > 16) return PIR_ERR_ARG;
  if (((uintptr_t)cts & 15u) || ((uintptr_t)rgsw & 15u) || ((uintptr_t)out & 15u)) return PIR_ERR_ARG;
  const ParamCtx *ctx = nullptr;
  pir_status_t st = get_param_ctx(params, &ctx);
  if (st != PIR_OK) return st;
  if (gadget_bits(ctx->p, ell) > 30) return PIR_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const uint32_t L = params->L, n = params->n;
  const uint64_t ctw = 2ull * L * n, count = 1ull << levels;
  const uint64_t cur_words = (uint64_t)B * count * ctw, g_words = (uint64_t)B * levels * 2 * ell * ctw;
  void *scratch = nullptr;
  cudaError_t e = cudaMallocAsync(&scratch, (cur_words + g_words) * 4, s);
  if (e != cudaSuccess) return cuda_status(e);
  uint32_t *cur = static_cast<uint32_t *>(scratch), *g = cur + cur_words;
  // NTT form of the inputs and of the RGSW rows (rows [..][L][n], row r under prime r % L)
  if ((e = launch_ntt_fwd(*ctx, cts, cur, cur_words / n, s)) == cudaSuccess &&
      (e = launch_ntt_fwd(*ctx, rgsw, g, g_words / n, s)) == cudaSuccess) {
    uint64_t launches = 0;
    st = fold_device(*ctx, cur, B, levels, ell, g, out, s, &launches);
    count_launches(2 + launches);
    if (st == PIR_OK && (e = launch_ntt_inv(*ctx, out, out, (uint64_t)B * 2 * L, s)) != cudaSuccess)
      st = cuda_status(e);
    if (st == PIR_OK) count_launches(1);
  } else {
    st = cuda_status(e);
  }
  cudaFreeAsync(scratch, s);
  return st;
}
