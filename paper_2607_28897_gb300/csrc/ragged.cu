// ragged.cu -- the divisions and products of a ragged batch, grouped.
//
// The step-batched division (divstep.cu) for instances of different shapes:
// all divisions of a wave take each Newton step together.  The known limbs l
// run through the same sequence 3, 4, 6, 10, ... 130, 258, ... for every
// division, only a division's last step is shorter, so a step's products
// differ in size but not in kind: one launch per step, kind and product form
// (tile), each over the list of the operations that take it, largest first,
// every CTA reading its operation's sizes and offsets from a table.  The
// linear parts run one CTA per operation.  Operands are read from the input
// pool and results written to the output pool in place.  Multiplications of
// the batch run through the same product launches.
//
// Why: grouped by nearby shapes instead (padded classes of at least 8
// members, each class a chain of ~22 launches of its own), 20000 mixed
// operations made 199 classes of 30 members on average -- 4474 launches one
// after the other, each on a fraction of the SMs, 98 ms.  The grouped form
// takes some 70 launches over thousands of operations each, and the product
// launches of a step run side by side (below): 14.35 ms.
//
// Bound: the tensor-core products, whose floor is 10.5 ms at the cuBLAS rate;
// they run at about 0.8 of it, the linear parts take 0.9 ms and the
// persistent launch of the rest 0.3 ms.  In a batch of few operations each set of
// launches lasts as long as its largest product on one CTA.  The records of a
// wave (about 5.5 limbs per divisor limb) are kept to WAVE_BYTES.
#include "ragged.cuh"

#include <algorithm>
#include <unordered_map>

#include "divstep.cuh"
#include "tcpipe.cuh"

namespace bigint {

// The cheapest form of a product by the models of tcmul.cu, and whether its
// operands change roles (tcmul.cu).
int tc_choose(int nx, int ny, int nout, int lo, bool *swap);

namespace {

using namespace dstep;

// Bytes of records of one wave.
constexpr size_t WAVE_BYTES = (size_t)1 << 30;

// The steps up to this many known limbs run fused in one warp (every operand
// then has at most SMALL_STEP_LIMBS limbs).
constexpr int SMALL_L = 66;

struct RagArgs {
  const RagOp *ops;
  const int32_t *list;  // products: this launch's list
  int n;
  int kind, l, par;
  const uint64_t *in;
  uint64_t *out, *rec;
  int32_t *status;
  int *abort_flag;
};

__host__ __device__ inline int rag_L(int nu, int nv) { return nu - nv + 1; }

// Records of an operation: two iterates, low product, |d| (then r^), banded
// product (its top limbs become q^).
struct RagRec {
  uint64_t *w[2], *p, *d, *z;
};
__host__ __device__ inline int64_t rag_rec_limbs(int nu, int nv) {
  const int64_t L = rag_L(nu, nv);
  return 2 * (L + 4) + 2 * ((int64_t)nv + 2) + (nu + L + 6);
}
__device__ __forceinline__ RagRec rag_rec(const RagArgs &A, const RagOp &o) {
  const int L = rag_L(o.nu, o.nv);
  RagRec r;
  r.w[0] = A.rec + o.rec;
  r.w[1] = r.w[0] + L + 4;
  r.p = r.w[1] + L + 4;
  r.d = r.p + o.nv + 2;
  r.z = r.d + o.nv + 2;
  return r;
}

// Steps after the fused ones; the iterate they leave is w[parity of these].
__host__ __device__ inline int rag_big_steps(int L) {
  int n = 0;
  for (int l = 2 * (SMALL_L - 1); l < L; l += l - 2) n++;
  return n;
}

struct RagTask {
  const uint64_t *x, *y;
  uint64_t *out;
  int nx, ny, nout, lo;
};
// Sizes of the product of a kind (host and device).
__host__ __device__ inline void rag_sizes(int nu, int nv, int kind, int l, int &nx, int &ny,
                                          int &nout, int &lo) {
  const int k = nv - 1, L = rag_L(nu, nv);
  const Step S = newton_next(k, L, l);
  const int c = step_cut(S);
  switch (kind) {
    case RAG_P: nx = S.t + 1; ny = l + 2; nout = S.t + 2; lo = c > 0 ? c - 2 : 0; break;
    case RAG_P2: nx = l + 2; ny = S.t + 2 - c; nout = nx + ny; lo = S.t + l - S.m - c - 2; break;
    case RAG_UW: nx = nu; ny = L + 2; nout = nx + ny; lo = nu - 2; break;
    case RAG_QV: nx = L + 2; ny = nv; nout = nv + 1; lo = 0; break;
    default: nx = nu; ny = nv; nout = nu + nv; lo = 0; break;
  }
}
__device__ __forceinline__ RagTask rag_task(const RagArgs &A, const RagOp &o, bool swap) {
  RagTask T;
  rag_sizes(o.nu, o.nv, A.kind, A.l, T.nx, T.ny, T.nout, T.lo);
  const uint64_t *u = A.in + o.u, *v = A.in + o.v;
  if (A.kind == RAG_MUL) {
    T.x = u;
    T.y = v;
    T.out = A.out + o.q;
  } else {
    const RagRec r = rag_rec(A, o);
    switch (A.kind) {
      case RAG_P: T.x = v + (o.nv - T.nx); T.y = r.w[A.par]; T.out = r.p; break;
      case RAG_P2: T.x = r.w[A.par]; T.y = r.d; T.out = r.z; break;
      case RAG_UW: T.x = u; T.y = r.w[rag_big_steps(T.ny - 2) & 1]; T.out = r.z; break;
      default: T.x = r.z + o.nu; T.y = v; T.out = r.p; break;
    }
  }
  if (swap) {
    const uint64_t *t = T.x; T.x = T.y; T.y = t;
    const int n = T.nx; T.nx = T.ny; T.ny = n;
  }
  return T;
}

// ---- kernels ---------------------------------------------------------------
// One thread per division: the Newton start, or (zero top limb of the
// divisor) its index into the irregular list and a zero iterate, on which
// the steps stay within their buffers and whose results nobody reads.
__global__ void k_rag_start(RagArgs A, int32_t *irregular, int *nirr) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= A.n) return;
  const RagOp o = A.ops[i];
  const int L = rag_L(o.nu, o.nv), l = L < 3 ? L : 3;
  uint64_t *w = A.rec + o.rec;
  const uint64_t *v = A.in + o.v;
  if (v[o.nv - 1] == 0) {
    irregular[atomicAdd(nirr, 1)] = o.opi;
    for (int j = 0; j < l + 2; j++) w[j] = 0;
    return;
  }
  ds_start_one(v, o.nv, l, w);
}

// One warp per division: the steps from at most SMALL_L known limbs.
__global__ void __launch_bounds__(32 * SMALL_STEP_WARPS) k_rag_small(RagArgs A) {
  extern __shared__ __align__(16) uint64_t ssm[];
  constexpr int N = SMALL_STEP_LIMBS;
  const int wi = threadIdx.x >> 5, lane = (int)lane_id();
  const int i = blockIdx.x * SMALL_STEP_WARPS + wi;
  if (i >= A.n) return;  // the whole warp: no block barrier below
  const RagOp o = A.ops[i];
  uint64_t *base = ssm + (size_t)wi * small_step_warp_limbs(N);
  uint64_t *wb[2] = {base, base + N}, *vt = base + 2 * N, *d = base + 3 * N, *z = base + 4 * N;
  uint64_t *w = A.rec + o.rec;
  const int L = rag_L(o.nu, o.nv);
  int l = L < 3 ? L : 3, cur = 0, t = 0;
  if (l == L) return;  // no steps: the start value stands
  for (int ll = l; ll < L && ll <= SMALL_L;) {  // t of the last step: the largest
    const Step S = newton_next(o.nv - 1, L, ll);
    t = S.t;
    ll += S.m;
  }
  const uint64_t *v = A.in + o.v + (o.nv - 1 - t);
  for (int j = lane; j <= t; j += 32) vt[j] = v[j];
  for (int j = lane; j < l + 2; j += 32) wb[0][j] = w[j];
  __syncwarp();
  while (l < L && l <= SMALL_L) {
    const Step S = newton_next(o.nv - 1, L, l);
    ds_small_step(vt + (t - S.t), S, wb[cur], wb[cur ^ 1], d, z);
    cur ^= 1;
    l += S.m;
  }
  for (int j = lane; j < l + 2; j += 32) w[j] = wb[cur][j];
}

// One CTA per division: |d| and its sign (limb nv + 1 of the record's |d|).
__global__ void __launch_bounds__(LIN_THREADS) k_rag_mid(RagArgs A) {
  __shared__ uint32_t scr[BLK_SCRATCH_WORDS];
  const RagOp o = A.ops[blockIdx.x];
  const RagRec r = rag_rec(A, o);
  const Step S = newton_next(o.nv - 1, rag_L(o.nu, o.nv), A.l);
  const int c = step_cut(S);
  const bool ng = ds_mid_cta(r.p + c, r.d, S.t + 2 - c, scr);
  if (threadIdx.x == 0) r.p[0] = ng ? 1 : 0;  // the low product is used up
}

__global__ void __launch_bounds__(LIN_THREADS) k_rag_update(RagArgs A) {
  __shared__ uint32_t scr[BLK_SCRATCH_WORDS];
  const RagOp o = A.ops[blockIdx.x];
  const RagRec r = rag_rec(A, o);
  const Step S = newton_next(o.nv - 1, rag_L(o.nu, o.nv), A.l);
  const int nw = S.l + 2, c = step_cut(S), n2 = nw + S.t + 2 - c, s = S.t + S.l - S.m - c;
  ds_update_cta(r.w[A.par], nw, r.z + s, n2 - s, r.p[0] != 0, S.m, r.w[A.par ^ 1],
                S.l + S.m + 2, scr);
}

__global__ void __launch_bounds__(LIN_THREADS) k_rag_finish(RagArgs A) {
  __shared__ uint32_t scr[BLK_SCRATCH_WORDS];
  const RagOp o = A.ops[blockIdx.x];
  const uint64_t *u = A.in + o.u, *v = A.in + o.v;
  if (v[o.nv - 1] == 0) return;  // irregular
  const RagRec r = rag_rec(A, o);
  const int L = rag_L(o.nu, o.nv), nqh = L + 2;
  if (threadIdx.x == 0) r.z[o.nu + nqh] = 0;
  __syncthreads();
  int st = ds_finish_cta(u, o.nu, v, o.nv, r.p, r.d, r.z + o.nu, nqh + 1, A.out + o.q, L,
                         A.out + o.r, scr);
  if (*(volatile int *)A.abort_flag) st = BIGINT_ETIMEOUT;
  if (A.status != nullptr && threadIdx.x == 0) A.status[o.opi] = st;
}

// Entry k of this CTA: a list (largest first) is dealt to the CTAs in rounds,
// every second one backwards, so that no CTA gets the larger one each time
// (20000 mixed operations 16.67 -> 15.96 ms).
__device__ __forceinline__ int64_t rag_entry(int64_t k) {
  return k * gridDim.x + (k & 1 ? gridDim.x - 1 - blockIdx.x : blockIdx.x);
}

// The products of a list.  A CTA that gives up at a wait limit sets *abort_flag and reports
// BIGINT_ETIMEOUT for the rest of its multiplications.
template <class Product>
__device__ __forceinline__ void rag_products(const RagArgs &A, Product product) {
  bool ok = true;
  for (int64_t k = 0; rag_entry(k) < A.n; k++) {
    const int32_t e = A.list[rag_entry(k)];
    const RagOp o = A.ops[e & ~RAG_SWAP];
    if (ok) ok = product(rag_task(A, o, (e & RAG_SWAP) != 0));
    if (threadIdx.x == 0) {
      if (!ok) atomicExch(A.abort_flag, 1);
      if (A.kind == RAG_MUL && A.status != nullptr)
        A.status[o.opi] = ok ? BIGINT_OK : BIGINT_ETIMEOUT;
    }
  }
}

// Product launches of one set (one kind and step, one form each; also the
// batch's multiplications) depend on what came before the set but not on one
// another, and each may fill only some of the SMs.  So all but the first are
// launched as dependents (chain_launch) of the one before, which lets them
// start once all its CTAs have: every CTA triggers when it has its tensor
// memory, and CTA 0 waits for the launch before at its end, so that the last
// one's completion is the set's.  The first starts after everything before.
// Launches one after the other took 15.9 ms for 20000 mixed operations and
// 4.5 for 1500.
template <int NT, int G>
__global__ void __launch_bounds__(2 * NT + 32, 256 / NT) k_rag_tc(RagArgs A) {
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ tcm::TcShared sh;
  __shared__ uint32_t scr[BLK_SCRATCH_WORDS];
  tcm::TcCtx c;
  tcm::tc_init<NT>(c, sm, &sh, scr);
  pdl_trigger();
  rag_products(A, [&](const RagTask &T) {
    return tcm::tc_product<NT, G, true>(c, T.x, T.nx, T.y, T.ny, T.out, T.nout, T.lo);
  });
  tcm::tc_release<NT>(c);
  if (blockIdx.x == 0) pdl_wait();
}

template <int NT>
__global__ void __launch_bounds__(32 * tcm::one_warps<NT>(), 512 / NT) k_rag_one(RagArgs A) {
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ tcm::OneShared sh;
  tcm::OneCtx c;
  tcm::one_init<NT>(c, sm, &sh);
  pdl_trigger();
  rag_products(A, [&](const RagTask &T) {
    return tcm::one_product<NT, tcm::one_warps<NT>()>(c, T.x, T.nx, T.y, T.ny, T.out, T.nout,
                                                      T.lo);
  });
  tcm::one_release<NT>(c);
  if (blockIdx.x == 0) pdl_wait();
}

// The pipelined form.  The builders read an operation's table entries and
// hand the product to the other warps through a ring in shared memory, so
// that the issuing warp does not stall on two dependent loads per product.
constexpr int RING = 4;
struct RagRing {
  uint64_t full[RING], free[RING];
  tcm::PipeTask t[RING];
};

template <int KB, int NT>
__global__ void __launch_bounds__(tcm::PIPE_THREADS, 1) k_rag_pipe(RagArgs A, tcm::PipeLayout L) {
  using namespace tcm;
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ PipeShared sh;
  __shared__ RagRing ring;
  const int lane = (int)lane_id();
  const long long lim = wait_limit_here();
  if (threadIdx.x == 0) {
    for (int i = 0; i < RING; i++) {
      mbar_init(smem_u32(&ring.full[i]), 1);
      mbar_init(smem_u32(&ring.free[i]), PIPE_DRAIN / 32 + 1);
    }
  }
  auto next_b = [&](int64_t k, PipeTask &T) {
    const int64_t i = rag_entry(k), in = rag_entry(k + 1);
    const bool more = i < A.n;
    T.nx = 0;
    if (more) {
      const int32_t e = A.list[i];
      const RagTask t = rag_task(A, A.ops[e & ~RAG_SWAP], (e & RAG_SWAP) != 0);
      T = PipeTask{t.x, t.y, t.out, t.nx, t.ny, t.nout, t.lo, nullptr};
    }
    if (threadIdx.x == PIPE_DRAIN + 64 && in < A.n) {  // of the second warp
      const int32_t e = A.list[in];
      const RagTask t = rag_task(A, A.ops[e & ~RAG_SWAP], (e & RAG_SWAP) != 0);
      prefetch_l2(t.x, 8 * (size_t)t.nx);
      prefetch_l2(t.y, 8 * (size_t)t.ny);
    }
    if (threadIdx.x / 32 == PIPE_DRAIN / 32 + 1) {  // the first builder warp, as one
      const int r = (int)(k % RING);
      if (k >= RING && !pipe_wait_warp(&sh, &ring.free[r], (uint32_t)(k / RING - 1) & 1u, lim))
        return false;
      if (lane == 0) {
        ring.t[r] = T;
        mbar_arrive(smem_u32(&ring.full[r]));
      }
    }
    return more;
  };
  auto take = [&](int64_t k, PipeTask &T) {  // by a whole warp, once the slot is full
    T = ring.t[k % RING];
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&ring.free[k % RING]));
    return T.nx != 0;
  };
  auto next_i = [&](int64_t k, PipeTask &T) {
    if (!pipe_wait_warp(&sh, &ring.full[k % RING], (uint32_t)(k / RING) & 1u, lim)) return false;
    return take(k, T);
  };
  auto next_d = [&](int64_t k, PipeTask &T) {
    const bool bad = !pipe_wait(&sh, &ring.full[k % RING], (uint32_t)(k / RING) & 1u, lim);
    if (bar_or_drain<PIPE_DRAIN>(bad)) return false;  // all drain threads agree
    return take(k, T);
  };
  int64_t ndone = 0;
  auto status = [&](int64_t k, int32_t st) {
    if (A.kind == RAG_MUL && A.status != nullptr)
      A.status[A.ops[A.list[rag_entry(k)] & ~RAG_SWAP].opi] = st;
  };
  auto done = [&](int64_t k) {
    if (threadIdx.x == 0) status(k, BIGINT_OK);
    ndone = k + 1;
  };
  if (!pipe_run<KB, NT, false>(L, &sh, sm, next_b, next_i, next_d, done) && threadIdx.x == 0) {
    atomicExch(A.abort_flag, 1);
    for (int64_t k = ndone; rag_entry(k) < A.n; k++) status(k, BIGINT_ETIMEOUT);
  }
  if (blockIdx.x == 0) pdl_wait();
}

// ---- host ------------------------------------------------------------------
struct ShapeAttr {
  void (*kern)(RagArgs);                    // or, pipelined forms:
  void (*pipe)(RagArgs, tcm::PipeLayout);
  int threads, cap;    // CTAs per SM the tensor memory allows
  int dyn, overhead;   // largest dynamic shared memory; static and reserved
};

// The kernels of the product forms with their attributes on this device
// (dyn < 0 after an error).
struct Shapes {
  ShapeAttr a[RAG_NSHAPES];
  int sms = 0, smem_sm = 0;
  bool ok = false;
};
const Shapes &shapes() {
  static const Shapes S = [] {
    using tcm::one_warps;
    Shapes s;
    s.a[RAG_ONE128] = {k_rag_one<128>, nullptr, 32 * one_warps<128>(), 4, 0, 0};
    s.a[RAG_ONE256] = {k_rag_one<256>, nullptr, 32 * one_warps<256>(), 2, 0, 0};
    s.a[RAG_64] = {k_rag_tc<64, 7>, nullptr, 2 * 64 + 32, 4, 0, 0};
    s.a[RAG_128] = {k_rag_tc<128, 8>, nullptr, 2 * 128 + 32, 2, 0, 0};
    s.a[RAG_256] = {k_rag_tc<256, 8>, nullptr, 2 * 256 + 32, 1, 0, 0};
    s.a[RAG_PIPE128] = {nullptr, k_rag_pipe<128, 256>, tcm::PIPE_THREADS, 1, 0, 0};
    s.a[RAG_PIPE64] = {nullptr, k_rag_pipe<64, 256>, tcm::PIPE_THREADS, 1, 0, 0};
    s.a[RAG_PIPE128N] = {nullptr, k_rag_pipe<128, 128>, tcm::PIPE_THREADS, 1, 0, 0};
    s.a[RAG_PIPE64N] = {nullptr, k_rag_pipe<64, 128>, tcm::PIPE_THREADS, 1, 0, 0};
    int dev = 0, optin = 0, reserved = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&s.smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&s.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return s;
    for (ShapeAttr &x : s.a) {
      cudaFuncAttributes fa;
      const void *k = x.kern ? (const void *)x.kern : (const void *)x.pipe;
      if (cudaFuncGetAttributes(&fa, k) != cudaSuccess) return s;
      x.dyn = optin - (int)fa.sharedSizeBytes;
      x.overhead = (int)fa.sharedSizeBytes + reserved;
      if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, x.dyn) !=
          cudaSuccess)
        return s;
    }
    if (cudaFuncSetAttribute(k_rag_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             8 * SMALL_STEP_WARPS * small_step_warp_limbs(SMALL_STEP_LIMBS)) !=
        cudaSuccess)
      return s;
    s.ok = true;
    return s;
  }();
  return S;
}

// Shared memory of a pipelined launch for x of at most nx limbs (total = 0:
// does not fit).
tcm::PipeLayout pipe_layout_of(int shape, int nx) {
  const uint32_t dyn = (uint32_t)shapes().a[shape].dyn;
  return shape == RAG_PIPE128 || shape == RAG_PIPE128N ? tcm::pipe_layout<128>(nx, dyn)
                                                       : tcm::pipe_layout<64>(nx, dyn);
}

uint32_t shape_bytes(int shape, int nx, int ny, int nout, int lo) {
  using namespace tcm;
  switch (shape) {
    case RAG_ONE128: return one_bytes<128, one_warps<128>()>(nx, ny, nout, lo);
    case RAG_ONE256: return one_bytes<256, one_warps<256>()>(nx, ny, nout, lo);
    case RAG_64: return layout<64, 7>(nx, ny).total;
    case RAG_128: return layout<128, 8>(nx, ny).total;
    case RAG_PIPE128:
    case RAG_PIPE64:
    case RAG_PIPE128N:
    case RAG_PIPE64N: {
      const uint32_t t = pipe_layout_of(shape, nx).total;
      return t ? t : ~0u;
    }
    default: return layout<256, 8>(nx, ny).total;
  }
}

// The form of one product: shape (as an index), swap, shared memory and the
// CTAs per SM that leaves.  Sizes are rounded up to 1/16 of their highest
// power of two for the cost models, which a plan then evaluates a few
// hundred times, and a thread's next plan hardly at all: the choices (a
// function of the sizes alone) are kept per thread, MEMO_MAX of them at most.
// The shared memory is that of the actual sizes; a product that the chosen form
// does not hold takes the 256-column tile with its shorter operand whole in
// shared memory, and one that this does not hold either has no form
// (rag_takes).
struct Form {
  int shape, per_sm, group;  // products of one group share a launch
  int nx;                    // limbs of the operand stored whole
  bool swap;
  uint32_t bytes;
};
class Chooser {
 public:
  Form get(int nx, int ny, int nout, int lo) {
    // most operations of a step have the same sizes as the one before
    if (nx == last_[0] && ny == last_[1] && nout == last_[2] && lo == last_[3]) return last_form_;
    last_[0] = nx;
    last_[1] = ny;
    last_[2] = nout;
    last_[3] = lo;
    return last_form_ = choose(nx, ny, nout, lo);
  }

 private:
  static constexpr size_t MEMO_MAX = 1 << 15;
  Form choose(int nx, int ny, int nout, int lo) {
    static thread_local std::unordered_map<uint64_t, int> memo_;
    const int qx = up(nx), qy = up(ny);
    // a banded or low product keeps its kind: the same part of the result
    const int qo = std::min(qx + qy, nout == nx + ny ? qx + qy : up(nout));
    const int ql = std::min(lo > 0 ? down(lo) : 0, qo - 1);
    const uint64_t key = ((uint64_t)qx << 48) ^ ((uint64_t)qy << 32) ^ ((uint64_t)qo << 16) ^ ql;
    auto it = memo_.find(key);
    if (it == memo_.end()) {
      if (memo_.size() >= MEMO_MAX) memo_.clear();
      bool swap = false;
      const int sh = tc_choose(qx, qy, qo, ql, &swap);
      it = memo_.emplace(key, (sh << 1) | (swap ? 1 : 0)).first;
    }
    Form f;
    f.shape = it->second >> 1;
    f.swap = it->second & 1;
    int ax = f.swap ? ny : nx, ay = f.swap ? nx : ny;
    f.bytes = shape_bytes(f.shape, ax, ay, nout, lo);
    if (f.bytes > (uint32_t)shapes().a[f.shape].dyn) {
      f.swap = nx > ny;
      ax = std::min(nx, ny);
      ay = std::max(nx, ny);
      f.shape = RAG_256;
      f.bytes = shape_bytes(f.shape, ax, ay, nout, lo);
    }
    const ShapeAttr &a = shapes().a[f.shape];
    f.nx = ax;
    if (a.pipe) {  // one CTA per SM; those whose x is double buffered apart
      f.per_sm = 1;
      f.group = f.shape * 8 + pipe_layout_of(f.shape, ax).xbufs;
      return f;
    }
    f.per_sm = std::max(1, std::min(a.cap, shapes().smem_sm / ((int)f.bytes + a.overhead)));
    f.group = f.shape * 8 + f.per_sm;
    return f;
  }

  static int step(int n) {
    int s = 1;
    while (n >= 32 * s) s *= 2;
    return s;
  }
  static int up(int n) { return (n + step(n) - 1) / step(n) * step(n); }
  static int down(int n) { return n / step(n) * step(n); }
  int last_[4] = {-1, -1, -1, -1};
  Form last_form_{};
};

// Appends the launches of one kind of product over ops [first, first + n).
// joined: they belong to the set of launches appended last.
void plan_products(RagPlan &P, Chooser &C, int64_t first, int64_t n, int kind, int l, int par,
                   bool joined = false) {
  struct Item {
    Form f;
    double cost;
    int32_t entry;
  };
  std::vector<Item> items;
  items.reserve(n);
  for (int64_t i = 0; i < n; i++) {
    const RagOp &o = P.ops[first + i];
    int nx, ny, nout, lo;
    rag_sizes(o.nu, o.nv, kind, l, nx, ny, nout, lo);
    const Form f = C.get(nx, ny, nout, lo);
    items.push_back({f, (double)nx * ny, (int32_t)(first + i) | (f.swap ? RAG_SWAP : 0)});
  }
  std::stable_sort(items.begin(), items.end(), [](const Item &a, const Item &b) {
    return a.f.group != b.f.group ? a.f.group > b.f.group : a.cost > b.cost;
  });
  for (size_t i = 0; i < items.size();) {
    size_t j = i;
    RagLaunch R{};
    R.what = RAG_PROD;
    R.sibling = joined || i > 0;
    R.kind = kind;
    R.l = l;
    R.par = par;
    R.shape = items[i].f.shape;
    R.first = (int64_t)P.list.size();
    for (; j < items.size() && items[j].f.group == items[i].f.group; j++) {
      P.list.push_back(items[j].entry);
      R.smem = std::max(R.smem, items[j].f.bytes);
      R.nx = std::max(R.nx, items[j].f.nx);
    }
    R.n = (int64_t)(j - i);
    R.grid = (int)std::min<int64_t>(R.n, (int64_t)shapes().sms * items[i].f.per_sm);
    P.program.push_back(R);
    i = j;
  }
}

}  // namespace

bool rag_takes(int nu, int nv, bool mul) {
  if (!shapes().ok) return true;  // rag_plan reports the error
  // no product of a division has longer operands than u w, w of L + 2 limbs
  const int nx = mul ? nu : rag_L(nu, nv) + 2, ny = mul ? nv : nu + 1;
  return shape_bytes(RAG_256, std::min(nx, ny), std::max(nx, ny), nx + ny, 0) <=
         (uint32_t)shapes().a[RAG_256].dyn;
}

int rag_plan(std::vector<RagOp> divs, std::vector<RagOp> muls, RagPlan &P) {
  P = RagPlan();
  if (divs.empty() && muls.empty()) return BIGINT_OK;
  if (!shapes().ok) return BIGINT_ECUDA;
  Chooser C;
  auto linear = [&](int what, int64_t first, int64_t n, int l, int par) {
    RagLaunch R{};
    R.what = what;
    R.l = l;
    R.par = par;
    R.first = first;
    R.n = n;
    P.program.push_back(R);
  };
  // longest quotients first: the divisions still at work in a step are the
  // first ones of their wave
  std::stable_sort(divs.begin(), divs.end(), [](const RagOp &a, const RagOp &b) {
    return rag_L(a.nu, a.nv) > rag_L(b.nu, b.nv);
  });
  P.ndiv = (int64_t)divs.size();
  P.ops = divs;
  P.ops.insert(P.ops.end(), muls.begin(), muls.end());
  for (int64_t first = 0; first < P.ndiv;) {
    int64_t n = 0, limbs = 0;
    while (first + n < P.ndiv) {
      RagOp &o = P.ops[first + n];
      const int64_t r = rag_rec_limbs(o.nu, o.nv);
      if (n > 0 && 8 * (size_t)(limbs + r) > WAVE_BYTES) break;
      o.rec = limbs;
      limbs += r;
      n++;
    }
    P.rec_bytes = std::max(P.rec_bytes, 8 * (size_t)limbs);
    linear(RAG_START, first, n, 0, 0);
    linear(RAG_SMALL, first, n, 0, 0);
    int par = 0;
    for (int l = 2 * (SMALL_L - 1);; l += l - 2, par ^= 1) {
      int64_t act = 0;
      while (act < n && rag_L(P.ops[first + act].nu, P.ops[first + act].nv) > l) act++;
      if (act == 0) break;
      plan_products(P, C, first, act, RAG_P, l, par);
      linear(RAG_MID, first, act, l, par);
      plan_products(P, C, first, act, RAG_P2, l, par);
      linear(RAG_UPDATE, first, act, l, par);
    }
    plan_products(P, C, first, n, RAG_UW, 0, 0);
    if (first == 0) plan_products(P, C, P.ndiv, (int64_t)muls.size(), RAG_MUL, 0, 0, true);
    plan_products(P, C, first, n, RAG_QV, 0, 0);
    linear(RAG_FINISH, first, n, 0, 0);
    first += n;
  }
  if (P.ndiv == 0) plan_products(P, C, 0, (int64_t)muls.size(), RAG_MUL, 0, 0);
  return BIGINT_OK;
}

int rag_launch(const RagPlan &P, const RagBuffers &B, const uint64_t *in, uint64_t *out,
               int32_t *status, cudaStream_t st) {
  BIGINT_CUDA_TRY(cudaMemsetAsync(B.ctr, 0, 2 * sizeof(int), st));
  for (const RagLaunch &R : P.program) {
    RagArgs A;
    A.ops = R.what == RAG_PROD ? B.ops : B.ops + R.first;
    A.list = R.what == RAG_PROD ? B.list + R.first : nullptr;
    A.n = (int)R.n;
    A.kind = R.kind;
    A.l = R.l;
    A.par = R.par;
    A.in = in;
    A.out = out;
    A.rec = B.rec;
    A.status = status;
    A.abort_flag = B.ctr + 1;
    const unsigned n = (unsigned)R.n;
    switch (R.what) {
      case RAG_START: k_rag_start<<<(n + 127) / 128, 128, 0, st>>>(A, B.irregular, B.ctr); break;
      case RAG_SMALL:
        k_rag_small<<<(n + SMALL_STEP_WARPS - 1) / SMALL_STEP_WARPS, 32 * SMALL_STEP_WARPS,
                      8 * SMALL_STEP_WARPS * small_step_warp_limbs(SMALL_STEP_LIMBS), st>>>(A);
        break;
      case RAG_MID: k_rag_mid<<<n, LIN_THREADS, 0, st>>>(A); break;
      case RAG_UPDATE: k_rag_update<<<n, LIN_THREADS, 0, st>>>(A); break;
      case RAG_FINISH: k_rag_finish<<<n, LIN_THREADS, 0, st>>>(A); break;
      default: {
        const ShapeAttr &a = shapes().a[R.shape];
        int rc;
        if (a.pipe) {
          const tcm::PipeLayout L = pipe_layout_of(R.shape, R.nx);
          rc = chain_launch(R.sibling, a.pipe, (unsigned)R.grid, a.threads, L.total, st, A, L);
        } else {
          // no more CTAs on an SM than its tensor memory serves (one too many
          // would queue for it through all of another's products)
          const uint32_t least = (uint32_t)(shapes().smem_sm / (a.cap + 1) - a.overhead + 1);
          rc = chain_launch(R.sibling, a.kern, (unsigned)R.grid, a.threads,
                            std::max(R.smem, least), st, A);
        }
        if (rc != BIGINT_OK) return rc;
        continue;
      }
    }
    const int rc = bigint_launch_status();
    if (rc != BIGINT_OK) return rc;
  }
  return BIGINT_OK;
}

// This unit's record of products that gave up at a wait limit, and its wait
// limit (see tcm::take_timeout_here).
int rag_take_timeout() { return tcm::take_timeout_here(); }
int rag_set_wait_limit(long long cycles) { return tcm::set_wait_limit_here(cycles); }

}  // namespace bigint
