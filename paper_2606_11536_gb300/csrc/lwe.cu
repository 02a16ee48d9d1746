// lwe.cu -- the scalar-HE (LWE) DB GEMM of SimplePIR's online step (Sec. 2.5) on the CUDA
// cores, and the choice between it and the tensor-core path (lwe_tc.cu):
//     out[b][i] = sum_j A[i][j] * Q[b][j]   (mod 2^32)
// with A the raw DB (D1 x D0 signed INT8 plaintexts, no NTT encoding, no bloating)
// and Q the B query vectors of Z_{2^32} entries.  As Sec. 4.1 decomposes it, every query
// word splits into four byte planes Q_p (Q = sum_p 2^(8p) Q_p); each A Q_p is an s8 x u8
// product with s32 accumulation, and out = sum_p (A Q_p) << 8p.  Wrapping 32-bit
// arithmetic is exactly arithmetic mod 2^32, so the accumulators need no K chunking.
//
// The products are dp4a: one DB row per thread, the query planes transposed once per
// stage in shared memory (eight prmt per 4 x 4 bytes) and read as broadcasts.
#include "common.cuh"
#include "tcgen.cuh"

namespace gbpir {
namespace {

constexpr int KS = 128;  // DB bytes of K per stage

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp16z(uint32_t saddr, const void *g, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(saddr), "l"(g), "r"(ok ? 16 : 0));
}

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}

// Byte planes of four words w0..w3: plane p = {w0.p, w1.p, w2.p, w3.p} (a 4 x 4 byte
// transpose in eight prmt).
__device__ __forceinline__ void byte_planes(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t (&p)[4]) {
  const uint32_t t0 = prmt(w0, w1, 0x5140), t1 = prmt(w0, w1, 0x7362);  // {w0.0 w1.0 w0.1 w1.1}, {.2 .2 .3 .3}
  const uint32_t t2 = prmt(w2, w3, 0x5140), t3 = prmt(w2, w3, 0x7362);
  p[0] = prmt(t0, t2, 0x5410);
  p[1] = prmt(t0, t2, 0x7632);
  p[2] = prmt(t1, t3, 0x5410);
  p[3] = prmt(t1, t3, 0x7632);
}

// A tile: rows of KS bytes, 16-byte chunks XOR-swizzled by row (16-byte reads without
// bank conflicts).
__device__ __forceinline__ uint32_t swz_a(uint32_t r, uint32_t ch) { return r * KS + ((ch ^ (r & 7)) << 4); }
// CUDA-core path: 256 rows per CTA (one per thread) x QB queries.  Per stage the raw
// query words are staged, then transposed once into planes [QB][KS/4][4] that every
// thread reads as broadcasts.  blockIdx.z takes K stages [z * kper, (z + 1) * kper):
// with more than one split the partial sums are added into the zeroed output with
// wrapping atomics, exact in any order because the result is taken mod 2^32.
template <int QB>
__global__ void __launch_bounds__(256) k_lwe_dp4a(const int8_t *__restrict__ A, uint32_t D1, uint32_t D0,
                                                  const uint32_t *__restrict__ Q, uint32_t B, uint32_t kper,
                                                  uint32_t *__restrict__ out) {
  constexpr int A_BYTES = 256 * KS, QR_BYTES = QB * KS * 4, STAGE = A_BYTES + QR_BYTES;
  extern __shared__ __align__(128) uint8_t smem[];
  uint4 *planes = reinterpret_cast<uint4 *>(smem + 2 * STAGE);  // [QB][KS/4] of {p0, p1, p2, p3}
  const uint32_t tid = threadIdx.x;
  const uint64_t m0 = (uint64_t)blockIdx.x * 256;
  const uint32_t q0 = blockIdx.y * QB;

  auto load_stage = [&](int buf, uint32_t k0) {
    const uint32_t sbase = smem_addr(smem + buf * STAGE);
    for (uint32_t t = tid; t < 256 * (KS / 16); t += 256) {  // 8 threads per 128-byte row segment
      const uint32_t ch = t & 7, r = t >> 3;
      const bool ok = (m0 + r < D1) && (k0 + ch * 16 < D0);
      const int8_t *g = A + (m0 + r) * D0 + k0 + ch * 16;
      cp16z(sbase + swz_a(r, ch), ok ? g : A, ok);
    }
    for (uint32_t t = tid; t < QB * (KS / 4); t += 256) {
      const uint32_t c = t % (KS / 4), n = t / (KS / 4);
      const bool ok = (q0 + n < B) && (k0 + c * 4 < D0);
      const uint32_t *g = Q + (uint64_t)(q0 + n) * D0 + k0 + c * 4;
      cp16z(sbase + A_BYTES + (n * (KS / 4) + c) * 16, ok ? g : Q, ok);
    }
    asm volatile("cp.async.commit_group;\n" ::);
  };

  int acc[QB][4];
#pragma unroll
  for (int b = 0; b < QB; ++b)
#pragma unroll
    for (int p = 0; p < 4; ++p) acc[b][p] = 0;

  const uint32_t nk_all = (D0 + KS - 1) / KS, kbeg = blockIdx.z * kper;
  const uint32_t nk = kbeg >= nk_all ? 0 : (nk_all - kbeg < kper ? nk_all - kbeg : kper);
  if (nk > 0) load_stage(0, kbeg * KS);
  for (uint32_t kt = 0; kt < nk; ++kt) {
    const int buf = kt & 1;
    asm volatile("cp.async.wait_group 0;\n" ::);
    __syncthreads();  // this stage landed; the previous stage's planes are no longer read
    const uint8_t *st = smem + buf * STAGE;
    for (uint32_t t = tid; t < QB * (KS / 4); t += 256) {
      const uint4 w = reinterpret_cast<const uint4 *>(st + A_BYTES)[t];
      uint32_t p[4];
      byte_planes(w.x, w.y, w.z, w.w, p);
      planes[t] = make_uint4(p[0], p[1], p[2], p[3]);
    }
    if (kt + 1 < nk) load_stage(buf ^ 1, (kbeg + kt + 1) * KS);
    __syncthreads();
#pragma unroll 2
    for (uint32_t ch = 0; ch < KS / 16; ++ch) {
      const uint4 a = *reinterpret_cast<const uint4 *>(st + swz_a(tid, ch));
      const uint32_t aw[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
      for (int b = 0; b < QB; ++b)
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const uint4 pl = planes[b * (KS / 4) + ch * 4 + w];  // the same address in every thread
          asm("dp4a.s32.u32 %0, %1, %2, %0;" : "+r"(acc[b][0]) : "r"(aw[w]), "r"(pl.x));
          asm("dp4a.s32.u32 %0, %1, %2, %0;" : "+r"(acc[b][1]) : "r"(aw[w]), "r"(pl.y));
          asm("dp4a.s32.u32 %0, %1, %2, %0;" : "+r"(acc[b][2]) : "r"(aw[w]), "r"(pl.z));
          asm("dp4a.s32.u32 %0, %1, %2, %0;" : "+r"(acc[b][3]) : "r"(aw[w]), "r"(pl.w));
        }
    }
  }
  const uint64_t i = m0 + tid;
  if (i >= D1) return;
#pragma unroll
  for (int b = 0; b < QB; ++b) {
    if (q0 + b >= B) break;
    uint32_t v = 0;
#pragma unroll
    for (int p = 0; p < 4; ++p) v += (uint32_t)acc[b][p] << (8 * p);
    if (gridDim.z > 1)
      atomicAdd(out + (uint64_t)(q0 + b) * D1 + i, v);
    else
      out[(uint64_t)(q0 + b) * D1 + i] = v;
  }
}

template <int QB>
cudaError_t dp4a_launch(const int8_t *A, uint32_t D1, uint32_t D0, const uint32_t *Q, uint32_t B, uint32_t *out,
                        cudaStream_t s, uint32_t *launches) {
  constexpr int smem = 2 * (256 * KS + QB * KS * 4) + QB * KS * 4;
  cudaError_t e = cudaFuncSetAttribute(k_lwe_dp4a<QB>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const uint64_t gx = (D1 + 255ull) / 256, gy = (B + QB - 1) / QB;
  if (gx > 0x7FFFFFFFull || gy > 65535) return cudaErrorInvalidConfiguration;
  // split K until the grid fills about four waves of resident CTAs
  int dev = 0, sms = 0, per_sm = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lwe_dp4a<QB>, 256, smem)) != cudaSuccess) return e;
  const uint32_t nk = (D0 + KS - 1) / KS;
  const uint64_t target = 4ull * sms * (per_sm > 0 ? per_sm : 1);
  uint64_t splits = (target + gx * gy - 1) / (gx * gy);
  const uint64_t max_splits = nk / 8 > 0 ? nk / 8 : 1;  // at least 8 stages per split
  if (splits > max_splits) splits = max_splits;
  if (splits > 64) splits = 64;
  if (splits < 1) splits = 1;
  const uint32_t kper = (uint32_t)((nk + splits - 1) / splits);
  splits = (nk + kper - 1) / kper;
  if (splits > 1) {
    if ((e = cudaMemsetAsync(out, 0, (size_t)B * D1 * sizeof(uint32_t), s)) != cudaSuccess) return e;
  }
  k_lwe_dp4a<QB><<<dim3((unsigned)gx, (unsigned)gy, (unsigned)splits), 256, smem, s>>>(A, D1, D0, Q, B, kper, out);
  *launches = 1;
  return cudaGetLastError();
}

}  // namespace

// PIR_LWE_AUTO: which path is the faster one.  The CUDA cores stream the DB once per four
// queries, at 5.5 TB/s with one or two queries, 4.2 with three, 3.4 with four; the tensor
// cores once per 32, at 6.5, with about 4 us more of fixed cost (a second kernel and
// scratch), and without the 2 us per query and K split that dp4a spends in its shortest
// rows.  Measured: 16384 x 16384, one query 57.8 (dp4a) against 51.8 us, eight 163 against
// 57; 1000 x 1024, four queries 16.5 against 13.0; 2000 x 512, 32 queries 10.4 against 13.2.
bool tensor_path_wins(uint32_t D1, uint32_t D0, uint32_t B) {
  const double mb = 1e-6 * D1 * D0, passes = (B + 3) / 4, tensor_passes = (B + 31) / 32;
  const double gain_us = mb * ((B <= 2 ? 1 / 5.5 : B == 3 ? 1 / 4.2 : passes / 3.4) - tensor_passes / 6.5);
  return gain_us >= 7 || (D0 >= 1024 && (B >= 4 || (B == 3 && gain_us >= 3)));
}

// The path that `path` stands for at these sizes: the tensor cores only where their tensor maps
// reach every row.
uint32_t lwe_path(uint32_t D1, uint32_t D0, uint32_t B, uint32_t path) {
  if (path == PIR_LWE_AUTO) path = tensor_path_wins(D1, D0, B) ? PIR_LWE_TENSOR : PIR_LWE_SIMT;
  return path == PIR_LWE_TENSOR && !lwe_tc_addresses(D1) ? PIR_LWE_SIMT : path;
}

// The tensor path takes scratch for the query digits; where there is none left, or the
// runtime offers no tensor maps, the CUDA cores answer.
cudaError_t launch_lwe_gemm(const int8_t *A, uint32_t D1, uint32_t D0, const uint32_t *Q, uint32_t B, uint32_t *out,
                            uint32_t path, cudaStream_t s, uint32_t *launches) {
  if (lwe_path(D1, D0, B, path) == PIR_LWE_TENSOR && tensor_maps_available()) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    keep_pool_memory(dev);  // scratch mapped anew after every synchronization costs 200 us a call
    void *qt = nullptr;
    e = cudaMallocAsync(&qt, lwe_tc_scratch_bytes(D0, B), s);
    if (e == cudaSuccess) {
      e = launch_lwe_tc(A, D1, D0, Q, B, out, static_cast<uint16_t *>(qt), s);
      cudaFreeAsync(qt, s);
      *launches = 2;
      return e;
    }
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
  }
  if (B >= 4) return dp4a_launch<4>(A, D1, D0, Q, B, out, s, launches);
  if (B == 3) return dp4a_launch<3>(A, D1, D0, Q, B, out, s, launches);
  if (B == 2) return dp4a_launch<2>(A, D1, D0, Q, B, out, s, launches);
  return dp4a_launch<1>(A, D1, D0, Q, B, out, s, launches);
}

}  // namespace gbpir

extern "C" pir_status_t pir_lwe_answer(const int8_t *db, uint32_t D1, uint32_t D0, const uint32_t *queries,
                                       uint32_t B, uint32_t *out, uint32_t path, void *stream) {
  using namespace gbpir;
  if (!db || !queries || !out || D1 == 0 || D0 == 0 || B == 0 || path > PIR_LWE_SIMT) return PIR_ERR_ARG;
  if (D0 % 16 != 0 || D0 > (1u << 24)) return PIR_ERR_ARG;
  if (((uintptr_t)db & 15u) || ((uintptr_t)queries & 15u) || ((uintptr_t)out & 15u)) return PIR_ERR_ARG;
  uint32_t launches = 0;
  cudaError_t e = launch_lwe_gemm(db, D1, D0, queries, B, out, path, static_cast<cudaStream_t>(stream), &launches);
  if (e != cudaSuccess) return cuda_status(e);
  count_launches(launches);
  return PIR_OK;
}

extern "C" pir_status_t pir_lwe_path(uint32_t D1, uint32_t D0, uint32_t B, uint32_t path, uint32_t *taken) {
  if (!taken || D1 == 0 || D0 == 0 || B == 0 || path > PIR_LWE_SIMT) return PIR_ERR_ARG;
  *taken = gbpir::lwe_path(D1, D0, B, path);
  return PIR_OK;
}
