// programs.cu -- multi-operation programs per instance (Sec. VI, Tables I and
// II), intermediates kept on chip or in scratch that stays in L2.
//
//   poly:       r = (a a + b) (b b + b) + a b  mod B^n  (Table II's Poly: four
//               multiplications and three additions, every value kept to n
//               limbs as the paper's same-width multiply and add do).
#include "divcore.cuh"

namespace bigint {

// Operands (limbs) from which Poly runs as batched products (the pipelined form
// takes every size from there up to the 10000 of a product).
constexpr int POLY_TC_MIN = 64;
int launch_mul_add(const uint64_t *a, const uint64_t *b, const uint64_t *c, uint64_t *out,
                   int64_t count, int n, cudaStream_t st);

// ---------------------------------------------------------------------------
// Poly: four launches of batched low products with an addend, the additions
// done as the products' limbs are formed,
//   T1 = a a + b,  T2 = b b + b,  r = a b,  r = T1 T2 + r,
// on chunks of the batch whose T1 and T2 stay in L2 (tcone.cuh, tcpipe.cuh:
// several CTAs per SM or the warp-specialised pipeline; as one persistent
// kernel a CTA at a time on each product, 16384 Polys of 1024 limbs took 7.9
// ms).  Below 64 limbs k_poly: persistent CTAs, per instance four low-part
// integer products (blk_mul) and three in-place additions through a per-CTA
// scratch of 3n limbs.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(512)
    k_poly(const uint64_t *__restrict__ A, const uint64_t *__restrict__ Bm,
           uint64_t *__restrict__ Out, int n, int64_t count, uint64_t *scratch) {
  extern __shared__ __align__(1024) uint32_t smem[];
  __shared__ uint32_t scr[BLK_SCRATCH_WORDS];
  uint64_t *T1 = scratch + (int64_t)blockIdx.x * 3 * n, *T2 = T1 + n, *T3 = T2 + n;
  auto prod = [&](const uint64_t *x, const uint64_t *y, uint64_t *out) {
    blk_mul_call<divc::DRB, divc::DQ, divc::DF>(x, n, y, n, out, n, smem, 0);
  };
  auto add_into = [&](uint64_t *t, const uint64_t *u) {  // t = t + u mod B^n
    auto load = [&](int j) { return make_ulonglong2(t[j], u[j]); };
    auto store = [&](int j, uint64_t v) { t[j] = v; };
    blk_addsub<false>(n, 0u, load, store, scr);
  };
  for (int64_t inst = blockIdx.x; inst < count; inst += gridDim.x) {
    const uint64_t *a = A + inst * (int64_t)n, *b = Bm + inst * (int64_t)n;
    uint64_t *o = Out + inst * (int64_t)n;
    prod(a, a, T1);
    add_into(T1, b);
    prod(b, b, T2);
    add_into(T2, b);
    prod(T1, T2, T3);
    prod(a, b, o);
    add_into(o, T3);
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
namespace {

// Instances per chunk of the batched form: whole rounds of the SMs (four CTAs
// each) whose T1 and T2 take at most POLY_CHUNK_BYTES, well inside the L2.
constexpr size_t POLY_CHUNK_BYTES = (size_t)80 << 20;
int64_t poly_chunk(int64_t count, int n, int sms) {
  const int64_t fit = (int64_t)(POLY_CHUNK_BYTES / (16 * (size_t)n)), round = 4 * (int64_t)sms;
  int64_t c = fit >= round ? fit / round * round : fit / sms * sms;
  if (c < sms) c = sms;
  return c < count ? c : count;
}

// CTAs of k_poly: one per SM.
int64_t poly_grid(int64_t count, int sms) { return count < sms ? count : sms; }

// T1 and T2 of a chunk, or 3n limbs per resident CTA (0: a CUDA error).
size_t poly_bytes(int64_t count, int n) {
  const int sms = sm_count();
  if (sms == 0) return 0;
  if (n >= POLY_TC_MIN) return (size_t)poly_chunk(count, n, sms) * 2 * (size_t)n * 8;
  return (size_t)poly_grid(count, sms) * 3 * (size_t)n * 8;
}

int launch_poly_batched(const uint64_t *a, const uint64_t *b, uint64_t *out, int64_t count, int n,
                        void *ws, cudaStream_t st) {
  int rc;
  const int64_t chunk = poly_chunk(count, n, sm_count());
  uint64_t *T1 = static_cast<uint64_t *>(ws), *T2 = T1 + chunk * n;
  for (int64_t i = 0; i < count; i += chunk) {
    const int64_t c = count - i < chunk ? count - i : chunk;
    const uint64_t *x = a + i * n, *y = b + i * n;
    uint64_t *o = out + i * n;
    if ((rc = launch_mul_add(x, x, y, T1, c, n, st)) != BIGINT_OK) return rc;
    if ((rc = launch_mul_add(y, y, y, T2, c, n, st)) != BIGINT_OK) return rc;
    if ((rc = launch_mul_add(x, y, nullptr, o, c, n, st)) != BIGINT_OK) return rc;
    if ((rc = launch_mul_add(T1, T2, o, o, c, n, st)) != BIGINT_OK) return rc;
  }
  return BIGINT_OK;
}

}  // namespace

size_t poly_workspace(int64_t count, int n) {
  if (n < 1) return 0;
  const size_t bytes = poly_bytes(count, n);
  return bytes ? bytes : 8;
}

int launch_poly(const uint64_t *a, const uint64_t *b, uint64_t *out, int64_t count, int n,
                void *ws, size_t bytes, cudaStream_t st) {
  if (count == 0) return BIGINT_OK;
  const size_t need = poly_bytes(count, n);
  if (need == 0) return BIGINT_ECUDA;
  if (bytes < need) return BIGINT_ENOMEM;
  if (n >= POLY_TC_MIN) return launch_poly_batched(a, b, out, count, n, ws, st);
  k_poly<<<(unsigned)poly_grid(count, sm_count()), 512,
           4 * (size_t)blk_mul_smem_words<divc::DRB, divc::DQ>(n, n), st>>>(
      a, b, out, n, count, static_cast<uint64_t *>(ws));
  return bigint_launch_status();
}

}  // namespace bigint
