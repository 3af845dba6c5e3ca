// programs.cu -- fused multi-operation programs per instance (Sec. VI,
// Tables I and II): the whole program runs in one launch, intermediates stay
// on chip (registers) or in a per-CTA scratch region that stays in L2, so
// global-memory traffic is that of one operation.
//
//   poly:       r = (a a + b) (b b + b) + a b  mod B^n  (Table II's Poly: four
//               multiplications and three additions, every value kept to n
//               limbs as the paper's same-width multiply and add do).
#include "divcore.cuh"

namespace bigint {

bool mul_add_ok(int n);
int launch_mul_add(const uint64_t *a, const uint64_t *b, const uint64_t *c, uint64_t *out,
                   int64_t count, int n, cudaStream_t st);

// ---------------------------------------------------------------------------
// Poly: four launches of batched low products with an addend, the additions
// done as the products' limbs are formed,
//   T1 = a a + b,  T2 = b b + b,  r = a b,  r = T1 T2 + r,
// on chunks of the batch whose T1 and T2 stay in L2 (tcone.cuh, tcpipe.cuh:
// several CTAs per SM or the warp-specialised pipeline; as one persistent
// kernel a CTA at a time on each product, 16384 Polys of 1024 limbs took 7.9
// ms).  Sizes those forms do not take run k_poly: persistent CTAs, per
// instance four low-part products (tensor cores for n beyond what the
// pipelined form holds, blk_mul below 64 limbs) and three in-place additions
// through a per-CTA scratch of 3n limbs.
// ---------------------------------------------------------------------------
template <bool TC, int NT, int G>
__global__ void __launch_bounds__(TC ? 2 * NT + 32 : 512, TC ? 256 / NT : 1)
    k_poly(const uint64_t *__restrict__ A, const uint64_t *__restrict__ Bm,
           uint64_t *__restrict__ Out, int n, int64_t count, uint64_t *scratch, int smem_words) {
  extern __shared__ __align__(1024) uint32_t smem[];
  __shared__ uint32_t scr[BLK_SCRATCH_WORDS];
  __shared__ tcm::TcShared tsh;
  tcm::TcCtx tcc;
  if constexpr (TC) tcm::tc_init<NT>(tcc, reinterpret_cast<uint8_t *>(smem), &tsh, scr);
  uint64_t *T1 = scratch + (int64_t)blockIdx.x * 3 * n, *T2 = T1 + n, *T3 = T2 + n;
  auto prod = [&](const uint64_t *x, const uint64_t *y, uint64_t *out) {
    if constexpr (TC) {
      tcm::tc_product<NT, G, true>(tcc, x, n, y, n, out, n, 0);
    } else {
      blk_mul_call<divc::DRB, divc::DQ, divc::DF>(x, n, y, n, out, n, smem, 0);
    }
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
    if constexpr (TC) {
      if (tcc.aborted) break;
    }
  }
  if constexpr (TC) tcm::tc_release<NT>(tcc);
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
namespace {

template <bool TC, int NT, int G>
int poly_dyn_max() {
  static int dyn = -1;
  if (dyn < 0) {
    int dev = 0, optin = 0;
    BIGINT_CUDA_TRY(cudaGetDevice(&dev));
    BIGINT_CUDA_TRY(
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    cudaFuncAttributes fa;
    BIGINT_CUDA_TRY(cudaFuncGetAttributes(&fa, k_poly<TC, NT, G>));
    const int d = optin - (int)fa.sharedSizeBytes;
    BIGINT_CUDA_TRY(cudaFuncSetAttribute(k_poly<TC, NT, G>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, d));
    dyn = d;
  }
  return dyn;
}

// CTAs of k_poly<TC, NT, G> resident on one SM with `smem` bytes of dynamic
// shared memory (the tensor memory allows 256 / NT of them), 0 on error.
template <bool TC, int NT, int G>
int poly_per_sm(size_t smem) {
  int dev = 0, smem_sm = 0, reserved = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) !=
          cudaSuccess)
    return 0;
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, k_poly<TC, NT, G>) != cudaSuccess) return 0;
  int per = smem_sm / (int)(smem + fa.sharedSizeBytes + reserved);
  const int cap = TC ? 256 / NT : 1;
  if (per > cap) per = cap;
  return per < 1 ? 1 : per;
}

int sm_count(int *sms) {
  int dev = 0;
  BIGINT_CUDA_TRY(cudaGetDevice(&dev));
  BIGINT_CUDA_TRY(cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev));
  return BIGINT_OK;
}

// The launch of Poly for n-limb operands: the form, and for k_poly its
// dynamic shared memory and CTAs per SM.
struct PolyPlan {
  int form;  // 0: k_poly, integer, 1: batched products, 3: k_poly NT 256 G 8, 4: NT 256 G 4
  size_t smem;
  int per_sm;
};

// Instances per chunk of the batched form: whole rounds of the SMs (four CTAs
// each) whose T1 and T2 take at most POLY_CHUNK_BYTES, well inside the L2.
constexpr size_t POLY_CHUNK_BYTES = (size_t)80 << 20;
int64_t poly_chunk(int64_t count, int n, int sms) {
  const int64_t fit = (int64_t)(POLY_CHUNK_BYTES / (16 * (size_t)n)), round = 4 * (int64_t)sms;
  int64_t c = fit >= round ? fit / round * round : fit / sms * sms;
  if (c < sms) c = sms;
  return c < count ? c : count;
}

template <bool TC, int NT, int G>
bool poly_try(int form, size_t smem, PolyPlan &P) {
  const int dyn = poly_dyn_max<TC, NT, G>();
  if (dyn <= 0 || smem > (size_t)dyn) return false;
  P.form = form;
  P.smem = smem;
  P.per_sm = poly_per_sm<TC, NT, G>(smem);
  return P.per_sm > 0;
}

bool poly_plan(int n, PolyPlan &P) {
  if (mul_add_ok(n)) {
    P = PolyPlan{1, 0, 0};
    return true;
  }
  if (n >= divc::TC_DIV_MIN) {
    if (poly_try<true, 256, 8>(3, tcm::layout<256, 8>(n, n).total, P)) return true;
    if (poly_try<true, 256, 4>(4, tcm::layout<256, 4>(n, n).total, P)) return true;
  }
  return poly_try<false, 256, 8>(0, 4 * (size_t)blk_mul_smem_words<divc::DRB, divc::DQ>(n, n),
                                 P);
}

int64_t poly_grid(const PolyPlan &P, int64_t count) {
  int sms = 0;
  if (sm_count(&sms) != BIGINT_OK) return 0;
  const int64_t slots = (int64_t)sms * P.per_sm;
  return count < slots ? count : slots;
}

// T1 and T2 of a chunk, or 3n limbs per resident CTA.
size_t poly_bytes(const PolyPlan &P, int64_t count, int n) {
  int sms = 0;
  if (sm_count(&sms) != BIGINT_OK) return 0;
  if (P.form == 1) return (size_t)poly_chunk(count, n, sms) * 2 * (size_t)n * 8;
  const int64_t slots = (int64_t)sms * P.per_sm;
  return (size_t)(count < slots ? count : slots) * 3 * (size_t)n * 8;
}

int launch_poly_batched(const uint64_t *a, const uint64_t *b, uint64_t *out, int64_t count, int n,
                        void *ws, cudaStream_t st) {
  int sms = 0;
  int rc = sm_count(&sms);
  if (rc != BIGINT_OK) return rc;
  const int64_t chunk = poly_chunk(count, n, sms);
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

template <bool TC, int NT, int G>
int launch_poly_variant(const uint64_t *a, const uint64_t *b, uint64_t *out, int64_t count, int n,
                        void *ws, int64_t grid, size_t smem, cudaStream_t st) {
  k_poly<TC, NT, G><<<(unsigned)grid, TC ? 2 * NT + 32 : 512, smem, st>>>(
      a, b, out, n, count, static_cast<uint64_t *>(ws), (int)(smem / 4));
  return bigint_launch_status();
}

}  // namespace

// BIGINT_ETIMEOUT if a Poly launch's tensor-core product hit a wait limit
// since the last call (synchronises the device), else BIGINT_OK.
int programs_take_timeout() { return tcm::take_timeout_here(); }
int programs_set_wait_limit(long long cycles) { return tcm::set_wait_limit_here(cycles); }

size_t poly_workspace(int64_t count, int n) {
  PolyPlan P;
  if (n < 1 || !poly_plan(n, P)) return 0;
  const size_t bytes = poly_bytes(P, count, n);
  return bytes ? bytes : 8;
}

int launch_poly(const uint64_t *a, const uint64_t *b, uint64_t *out, int64_t count, int n,
                void *ws, size_t bytes, cudaStream_t st) {
  if (count == 0) return BIGINT_OK;
  PolyPlan P;
  if (!poly_plan(n, P)) return BIGINT_EINVAL;
  const size_t need = poly_bytes(P, count, n);
  if (need == 0) return BIGINT_ECUDA;
  if (bytes < need) return BIGINT_ENOMEM;
  if (P.form == 1) return launch_poly_batched(a, b, out, count, n, ws, st);
  const int64_t grid = poly_grid(P, count);
  switch (P.form) {
    case 3: return launch_poly_variant<true, 256, 8>(a, b, out, count, n, ws, grid, P.smem, st);
    case 4: return launch_poly_variant<true, 256, 4>(a, b, out, count, n, ws, grid, P.smem, st);
    default: return launch_poly_variant<false, 256, 8>(a, b, out, count, n, ws, grid, P.smem, st);
  }
}

}  // namespace bigint
