// tcmul.cu -- batched full (and low-part) products on the tensor cores.
//
// Persistent CTAs loop over the instances of a uniform batch, each product the
// digit convolution of tccore.cuh (tcgen05 fp16 MMAs with exact fp32
// accumulation, Sec. V-B's schoolbook product on the tensor cores) in the form
// the cost models below pick:
//   k_mul_one   one drain, two or four CTAs per SM (tcone.cuh): a shorter
//               operand of at most 512 limbs, with two accumulators of up to
//               about 640
//   k_mul_pipe  builder, issuing and drain warps, one CTA per SM
//               (tcpipe.cuh): most larger ones
//   k_mul_tc    all warps doing all of it in turn, one, two or four CTAs per
//               SM (tc_product): operands beyond the pipeline's shared memory,
//               some narrow products, and the forced shapes
//   k_mul_tc_sk, k_mul_tc_split  a few products, each over several CTAs
//
// Measured, 0.x of 1900 TFLOP/s: 512 limbs 0.55 (131072 products 4182 us,
// 6770 as tc_product), 1701 x 1103 limbs 0.73 (16384: 2815, 3860), 2048 limbs
// as Karatsuba leaves 0.87.
#include "tccore.cuh"
#include <cooperative_groups.h>

#include "ragged.cuh"
#include "tcone.cuh"
#include "tcpipe.cuh"

namespace bigint {
namespace tcm {

// 2 NT drain threads plus one issuer warp (tc_product<NT, G, true, XC, false,
// KB>).
// Instance i's operands start at X + i sx and Y + i sy, its result at
// Out + i so (limbs); lo > 0 is tc_product's band mode.  A CTA that gives up
// at a wait limit also sets *abort_flag (if given), so that a caller
// chaining products (the step-batched division) can report it per instance.
template <int NT, int G, bool XC, int KB = 128>
__global__ void __launch_bounds__(2 * NT + 32, 256 / NT)
    k_mul_tc(const uint64_t *X, const uint64_t *Y,
             uint64_t *Out, int nx, int ny, int nout, int64_t count, int64_t sx,
             int64_t sy, int64_t so, int lo, int *abort_flag) {
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ TcShared sh;
  __shared__ uint32_t scr[BLK_SCRATCH_WORDS];
  TcCtx c;
  tc_init<NT>(c, sm, &sh, scr);
  pdl_trigger();  // not before this CTA has its tensor memory
  pdl_wait();
  for (int64_t inst = blockIdx.x; inst < count; inst += gridDim.x) {
    const int64_t next = inst + gridDim.x;
    if (threadIdx.x == 0 && next < count) {
      prefetch_l2(X + next * sx, 8 * (size_t)nx);
      prefetch_l2(Y + next * sy, 8 * (size_t)ny);
    }
    if (!tc_product<NT, G, true, XC, false, KB>(c, X + inst * sx, nx, Y + inst * sy, ny,
                                                Out + inst * so, nout, lo))
      break;
  }
  if (c.aborted && abort_flag != nullptr && threadIdx.x == 0) atomicExch(abort_flag, 1);
  tc_release<NT>(c);
}

// The same for products whose shorter operand has at most ONE_MAX limbs
// (ONE_MAX2 with ACC = 2 accumulators; tcone.cuh): NT ACC tensor-memory columns
// and 32 W threads per CTA, 512 / (NT ACC) CTAs per SM.  add + i sadd: nout limbs added to product i (null: none).
template <int NT, int W, bool ADD, int ACC>
__global__ void __launch_bounds__(32 * W, 512 / (NT * ACC))
    k_mul_one(const uint64_t *X, const uint64_t *Y,
              uint64_t *Out, int nx, int ny, int nout, int64_t count, int64_t sx,
              int64_t sy, int64_t so, int lo, int *abort_flag, const uint64_t *add,
              int64_t sadd) {
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ OneShared sh;
  OneCtx c;
  one_init<NT * ACC>(c, sm, &sh);
  pdl_trigger();  // not before this CTA has its tensor memory
  pdl_wait();
  for (int64_t inst = blockIdx.x; inst < count; inst += gridDim.x) {
    const int64_t next = inst + gridDim.x;
    if (threadIdx.x == 0 && next < count) {
      prefetch_l2(X + next * sx, 8 * (size_t)nx);
      prefetch_l2(Y + next * sy, 8 * (size_t)ny);
    }
    if (!one_product<NT, W, ADD, ACC>(c, X + inst * sx, nx, Y + inst * sy, ny, Out + inst * so, nout,
                                 lo, ADD ? add + inst * sadd : nullptr))
      break;
  }
  if (c.aborted && abort_flag != nullptr && threadIdx.x == 0) atomicExch(abort_flag, 1);
  one_release<NT * ACC>(c);
}

// The same by the pipeline of tcpipe.cuh: one CTA per SM.
template <int KB, int NT>
__global__ void __launch_bounds__(PIPE_THREADS, 1)
    k_mul_pipe(const uint64_t *X, const uint64_t *Y,
               uint64_t *Out, int nx, int ny, int nout, int64_t count, int64_t sx,
               int64_t sy, int64_t so, int lo, int *abort_flag, const uint64_t *add, int64_t sadd,
               PipeLayout L) {
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ PipeShared sh;
  auto next = [&](int64_t k, PipeTask &T) {
    const int64_t i = blockIdx.x + k * gridDim.x;
    if (i >= count) return false;
    T = PipeTask{X + i * sx, Y + i * sy, Out + i * so, nx, ny, nout, lo,
                 add != nullptr ? add + i * sadd : nullptr};
    return true;
  };
  auto next_b = [&](int64_t k, PipeTask &T) {
    if (!next(k, T)) return false;
    const int64_t i = blockIdx.x + (k + 1) * gridDim.x;
    if (threadIdx.x == PIPE_DRAIN + 32 && i < count) {  // the first builder thread
      prefetch_l2(X + i * sx, 8 * (size_t)nx);
      prefetch_l2(Y + i * sy, 8 * (size_t)ny);
    }
    return true;
  };
  const bool ok = pipe_run<KB, NT>(L, &sh, sm, next_b, next, next, [](int64_t) {});
  if (!ok && abort_flag != nullptr && threadIdx.x == 0) atomicExch(abort_flag, 1);
}

// Split products: unit u is tile u % T of product u / T (tc_product's split
// mode), its outgoing (high word, carry) at tile_carry[2 u], [2 u + 1].
template <int NT, int G>
__global__ void __launch_bounds__(2 * NT + 32, 1)
    k_mul_tc_split(const uint64_t *__restrict__ X, const uint64_t *__restrict__ Y,
                   uint64_t *__restrict__ Out, int nx, int ny, int nout, int64_t count, int T,
                   uint64_t *tile_carry) {
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ TcShared sh;
  __shared__ uint32_t scr[BLK_SCRATCH_WORDS];
  TcCtx c;
  tc_init<NT>(c, sm, &sh, scr);
  const int64_t units = count * T;
  for (int64_t u = blockIdx.x; u < units; u += gridDim.x) {
    const int64_t inst = u / T;
    if (!tc_product<NT, G, true, true, true>(c, X + inst * (int64_t)nx, nx, Y + inst * (int64_t)ny,
                                             ny, Out + inst * (int64_t)nout, nout, 0,
                                             (int)(u - inst * T), tile_carry + 2 * u))
      break;
  }
  tc_release<NT>(c);
}

// ---- split-K products ---------------------------------------------------------
// A product cut into units of (tile, groups of Toeplitz blocks) so that even
// a single product keeps many SMs busy (tc_partial adds each unit's column
// sums into the product's buffer; k_tc_sk_finish turns them into limbs).
constexpr int SK_MAX_TILES = 8;
struct SkPlan {
  int T;                          // tiles
  int gpc;                        // groups per unit
  int cfirst;                     // first column of the first tile
  int c0[SK_MAX_TILES], W[SK_MAX_TILES];
  int first[SK_MAX_TILES + 1];    // first unit of each tile; first[T] units per product
};

template <int NT, int G>
__global__ void __launch_bounds__(2 * NT + 32, 1)
    k_mul_tc_sk(const uint64_t *X, const uint64_t *Y, int nx, int ny,
                int64_t sx, int64_t sy, int64_t count, SkPlan P, int *colsum, int64_t cs_stride,
                int *abort_flag) {
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ TcShared sh;
  __shared__ uint32_t scr[BLK_SCRATCH_WORDS];
  TcCtx c;
  tc_init<NT>(c, sm, &sh, scr);
  pdl_trigger();  // not before this CTA has its tensor memory
  pdl_wait();
  const int upi = P.first[P.T];
  for (int64_t u = blockIdx.x; u < count * upi; u += gridDim.x) {
    const int64_t inst = u / upi;
    const int r = (int)(u - inst * upi);
    int t = 0;
    while (t + 1 < P.T && P.first[t + 1] <= r) t++;
    const int g0 = (r - P.first[t]) * P.gpc;
    if (!tc_partial<NT, G>(c, X + inst * sx, nx, Y + inst * sy, ny, P.c0[t], P.W[t], g0,
                           g0 + P.gpc, colsum + inst * cs_stride + (P.c0[t] - P.cfirst) * 128))
      break;
  }
  if (c.aborted && abort_flag != nullptr && threadIdx.x == 0) atomicExch(abort_flag, 1);
  tc_release<NT>(c);
}

// A cluster of SKF_CLUSTER CTAs per product: its limbs [L0, nout) from its
// column sums (limb j from the coefficients 8 j .. 8 j + 7, biased, with
// `margin` in place of what limb L0 - 1 would carry; one carry scan, as in
// tcone.cuh), SKF_SPAN limbs per CTA and round; the CTAs exchange the high
// word of their last limb and their (generate, propagate) through distributed
// shared memory.  Bound by latency: 16384 limbs on one CTA, 512 threads and
// two scans took 27 us, 1024 threads and one scan 13.  CTAs past the products'
// clear `zero` ints of zbuf (the column sums of the product before).
constexpr int SKF_THREADS = 1024, SKF_R = 4, SKF_CLUSTER = 4, SKF_SPAN = SKF_R * SKF_THREADS;

__global__ void __launch_bounds__(SKF_THREADS)
    k_tc_sk_finish(const int *colsum, int64_t cs_stride, uint64_t *Out, int64_t so, int L0,
                   int nout, uint64_t margin, int64_t count, int *zbuf, int64_t zero) {
  constexpr int W = SKF_THREADS / 32;
  __shared__ uint32_t s_hi[SKF_R * W], s_g[SKF_R * W], s_p[SKF_R * W];
  __shared__ uint32_t c_hi[SKF_CLUSTER], c_g[SKF_CLUSTER], c_p[SKF_CLUSTER];
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  pdl_trigger();
  pdl_wait();
  const int64_t inst = blockIdx.x / SKF_CLUSTER;
  if (inst >= count) {  // the whole cluster
    const int64_t nz = gridDim.x - count * SKF_CLUSTER, z = blockIdx.x - count * SKF_CLUSTER;
    for (int64_t i = 4 * (z * SKF_THREADS + tid); i < zero; i += 4 * nz * SKF_THREADS)
      *reinterpret_cast<int4 *>(zbuf + i) = make_int4(0, 0, 0, 0);
    return;
  }
  const int rank = (int)(blockIdx.x % SKF_CLUSTER);
  const int *cs = colsum + inst * cs_stride;
  uint64_t *out = Out + inst * so + L0;
  const int n = nout - L0;
  uint32_t hprev = 0, cprev = 0;  // into the cluster's round
  cl.sync();                      // every CTA of the cluster runs: its shared memory is there
  for (int base = 0; base < n; base += SKF_CLUSTER * SKF_SPAN) {
    const int b = base + rank * SKF_SPAN;
    uint64_t low[SKF_R];
    uint32_t high[SKF_R];
#pragma unroll
    for (int r = 0; r < SKF_R; r++) {
      const int j = b + r * SKF_THREADS + tid;
      low[r] = 0;
      high[r] = 0;
      if (j < n) {
        // (the workspace of bigint_mul_split is 8-byte aligned)
        const int2 *p = reinterpret_cast<const int2 *>(cs + (size_t)j * 8);
        const int2 u0 = p[0], u1 = p[1], u2 = p[2], u3 = p[3];
        constexpr uint32_t B = 0x80000000u;
        const uint32_t w[8] = {u0.x + B, u0.y + B, u1.x + B, u1.y + B,
                               u2.x + B, u2.y + B, u3.x + B, u3.y + B};
        limb_of(w, 0ull, j == 0, low[r], high[r]);
      }
      if (lane == 31) s_hi[r * W + warp] = high[r];
    }
    if (tid == SKF_THREADS - 1)
      for (int i = 0; i < SKF_CLUSTER; i++) *cl.map_shared_rank(&c_hi[rank], i) = high[SKF_R - 1];
    cl.sync();
    const uint32_t hin = rank > 0 ? c_hi[rank - 1] : hprev;
    WarpCarry wc[SKF_R];
#pragma unroll
    for (int r = 0; r < SKF_R; r++) {
      const int j = b + r * SKF_THREADS + tid;
      uint32_t below = __shfl_up_sync(FULL, high[r], 1);
      if (lane == 0) below = r * W + warp > 0 ? s_hi[r * W + warp - 1] : hin;
      uint32_t g = 0, p = 1;
      if (j < n) {
        const uint64_t add = j == 0 ? margin : (uint64_t)below;
        low[r] += add;
        g = low[r] < add;
        p = low[r] == ~0ull;
      }
      wc[r] = warp_gp(g, p);
      if (lane == 0) {
        s_g[r * W + warp] = warp_carry_out(wc[r], 0);
        s_p[r * W + warp] = warp_all_propagate(wc[r]);
      }
    }
    hprev = c_hi[SKF_CLUSTER - 1];
    __syncthreads();
    WarpCarry bc[SKF_R];  // the CTA's warps, round by round
    uint32_t bg = 0, bp = 1;
#pragma unroll
    for (int r = 0; r < SKF_R; r++) {
      bc[r] = warp_gp(s_g[r * W + lane], s_p[r * W + lane]);
      bg = warp_carry_out(bc[r], 0) | (warp_all_propagate(bc[r]) & bg);
      bp &= warp_all_propagate(bc[r]);
    }
    if (tid < SKF_CLUSTER) {
      *cl.map_shared_rank(&c_g[rank], tid) = bg;
      *cl.map_shared_rank(&c_p[rank], tid) = bp;
    }
    cl.sync();
    uint32_t c = cprev;  // carry into this CTA's span, then through the cluster
#pragma unroll
    for (int i = 0; i < SKF_CLUSTER; i++) {
      if (i == rank) {
        uint32_t cc = c;
#pragma unroll
        for (int r = 0; r < SKF_R; r++) {
          const int j = b + r * SKF_THREADS + tid;
          const uint64_t cm = warp_carries(bc[r], cc);
          const uint64_t lc = warp_carries(wc[r], (uint32_t)(cm >> warp) & 1u);
          if (j < n) out[j] = low[r] + ((lc >> lane) & 1u);
          cc = (uint32_t)(cm >> 32);
        }
      }
      c = c_g[i] | (c_p[i] & c);
    }
    cprev = c;
    cl.sync();  // the exchange words are rewritten, or the CTA leaves
  }
}

// One CTA per product: tile t (limbs [t L, t L + L), L = tile_limbs) was
// computed without what flows in from tile t - 1, i.e. the high word H of
// that tile's last column sum and its carry out k.  So the product is the
// concatenated tiles plus sum_t (H_t + k_t) B^((t + 1) L), less the bias sum
// of the column sums (as in the unsplit product): two carry passes.
__global__ void __launch_bounds__(512)
    k_tc_split_finish(uint64_t *Out, int nout, int T, int tile_limbs, const uint64_t *tile_carry) {
  __shared__ uint32_t scr[BLK_SCRATCH_WORDS];
  uint64_t *o = Out + (int64_t)blockIdx.x * nout;
  const uint64_t *tc = tile_carry + 2 * (int64_t)blockIdx.x * T;
  auto st = [&](int j, uint64_t v) { o[j] = v; };
  auto ld_links = [&](int j) {
    uint64_t v = 0;
    if (j > 0 && j % tile_limbs == 0) {
      const int t = j / tile_limbs - 1;
      v = tc[2 * t] + tc[2 * t + 1];
    }
    return make_ulonglong2(o[j], v);
  };
  blk_addsub<false>(nout, 0u, ld_links, st, scr);
  auto ld_bias = [&](int j) {
    return make_ulonglong2(o[j], j == 0 ? 0x8080808080000000ull : 0x8080808080808080ull);
  };
  blk_addsub<true>(nout, 0u, ld_bias, st, scr);
}

}  // namespace tcm

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
template <int NT, int G, bool XC, int KB>
static int tc_dyn_max() {
  static int dyn = -1;
  if (dyn < 0) {
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
        cudaSuccess)
      return 0;
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, tcm::k_mul_tc<NT, G, XC, KB>) != cudaSuccess) return 0;
    const int d = optin - (int)fa.sharedSizeBytes;
    if (cudaFuncSetAttribute(tcm::k_mul_tc<NT, G, XC, KB>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, d) != cudaSuccess)
      return 0;
    dyn = d;
  }
  return dyn;
}

// The kernel shapes (tile columns NT, group G, x's carry digit XC, x block
// width KB).  128-digit blocks: the 256-column tile, one CTA per SM, for
// large products; the 128- and 64-column tiles (two and three CTAs per SM)
// for products whose columns fit one such tile, x's carry digit dropped
// (XC = false: one correction addition) where that makes them fit.  Narrow
// blocks (64 or 32 digits, 128-column tiles, two CTAs per SM) give each MMA
// 2 or 4 times the columns for the same 4 KB A operand, which bounds narrow
// MMAs; measured on GB300 they tie with 128-digit blocks at 512-limb
// products and lose from 1024 limbs on (4x the drains and column-sum rows
// per digit), so only the autotuner and the forced variants take them.
enum TcShape {
  TC_64_XC, TC_64_NOXC, TC_128_XC, TC_128_NOXC, TC_256,
  TC_N64_XC, TC_N64_NOXC, TC_N32_XC, TC_N32_NOXC, TC_NSHAPES
};
struct ShapeInfo {
  int nt, g, kb;
  bool xc;
};
static constexpr ShapeInfo SHAPES[TC_NSHAPES] = {
    {64, 7, 128, true},   {64, 7, 128, false},  {128, 8, 128, true}, {128, 8, 128, false},
    {256, 8, 128, true},  {128, 15, 64, true},  {128, 15, 64, false}, {128, 12, 32, true},
    {128, 12, 32, false}};

template <int NT, int G, bool XC, int KB>
static size_t tc_smem(int nx, int ny) {
  const tcm::Layout L = tcm::layout<NT, G, XC, KB>(nx, ny);
  const int d = tc_dyn_max<NT, G, XC, KB>();
  return d > 0 && L.total <= (uint32_t)d ? L.total : 0;
}

// Shared memory of a shape for x of nx and y of ny limbs, 0 if it does not fit.
static size_t shape_smem(TcShape sh, int nx, int ny) {
  switch (sh) {
    case TC_64_XC: return tc_smem<64, 7, true, 128>(nx, ny);
    case TC_64_NOXC: return tc_smem<64, 7, false, 128>(nx, ny);
    case TC_128_XC: return tc_smem<128, 8, true, 128>(nx, ny);
    case TC_128_NOXC: return tc_smem<128, 8, false, 128>(nx, ny);
    case TC_N64_XC: return tc_smem<128, 15, true, 64>(nx, ny);
    case TC_N64_NOXC: return tc_smem<128, 15, false, 64>(nx, ny);
    case TC_N32_XC: return tc_smem<128, 12, true, 32>(nx, ny);
    case TC_N32_NOXC: return tc_smem<128, 12, false, 32>(nx, ny);
    default: return tc_smem<256, 8, true, 128>(nx, ny);
  }
}

// Dynamic shared memory the tensor-core product of an na x nb product
// needs with the 256-column tile (which every product that fits any shape
// fits), or 0 if it does not fit (or the shapes are out of range).
size_t mul_tc_smem(int na, int nb) {
  const int nx = na < nb ? na : nb, ny = na < nb ? nb : na;
  if (nx < 1 || nx > 16383 || ny > 32768) return 0;
  return shape_smem(TC_256, nx, ny);
}

// Operands and results of one batched product launch: instance i's x at
// x + i sx, y at y + i sy, result at out + i so (limbs); band start lo (0:
// the low nout limbs exactly); abort_flag as for k_mul_tc (may be null).
struct TcArgs {
  const uint64_t *x, *y;
  uint64_t *out;
  int64_t sx, sy, so;
  int lo;
  int *abort_flag;
  const uint64_t *add = nullptr;  // one-drain and pipelined forms: added to the products
  int64_t sadd = 0;
};

// CTAs of a shape resident on one SM: TMEM allows 256 / NT, shared memory
// per SM / (dynamic + static + the per-block reservation).
template <int NT, int G, bool XC, int KB>
static int tc_per_sm(size_t smem) {
  static int smem_sm = 0, reserved = 0, static_smem = -1;
  if (static_smem < 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    if (cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) !=
            cudaSuccess)
      return 1;
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, tcm::k_mul_tc<NT, G, XC, KB>) != cudaSuccess) return 1;
    static_smem = (int)fa.sharedSizeBytes;
  }
  int per_sm = smem_sm / (int)(smem + static_smem + reserved);
  if (per_sm > 256 / NT) per_sm = 256 / NT;
  return per_sm < 1 ? 1 : per_sm;
}

template <int NT, int G, bool XC, int KB>
static int launch_tc(const TcArgs &A, int64_t count, int nx, int ny, int nout, cudaStream_t st) {
  const size_t smem = tc_smem<NT, G, XC, KB>(nx, ny);
  if (smem == 0) return BIGINT_EINVAL;
  if (count == 0) return BIGINT_OK;
  const int sms = sm_count();
  if (sms == 0) return BIGINT_ECUDA;
  const int64_t slots = (int64_t)sms * tc_per_sm<NT, G, XC, KB>(smem);
  const int64_t grid = count < slots ? count : slots;
  return chain_launch(grid <= sms, tcm::k_mul_tc<NT, G, XC, KB>, (unsigned)grid, 2 * NT + 32, smem, st, A.x,
                      A.y, A.out, nx, ny, nout, count, A.sx, A.sy, A.so, A.lo, A.abort_flag);
}

static int launch_shape(TcShape sh, const TcArgs &A, int64_t count, int nx, int ny, int nout,
                        cudaStream_t st) {
  switch (sh) {
    case TC_64_XC: return launch_tc<64, 7, true, 128>(A, count, nx, ny, nout, st);
    case TC_64_NOXC: return launch_tc<64, 7, false, 128>(A, count, nx, ny, nout, st);
    case TC_128_XC: return launch_tc<128, 8, true, 128>(A, count, nx, ny, nout, st);
    case TC_128_NOXC: return launch_tc<128, 8, false, 128>(A, count, nx, ny, nout, st);
    case TC_N64_XC: return launch_tc<128, 15, true, 64>(A, count, nx, ny, nout, st);
    case TC_N64_NOXC: return launch_tc<128, 15, false, 64>(A, count, nx, ny, nout, st);
    case TC_N32_XC: return launch_tc<128, 12, true, 32>(A, count, nx, ny, nout, st);
    case TC_N32_NOXC: return launch_tc<128, 12, false, 32>(A, count, nx, ny, nout, st);
    default: return launch_tc<256, 8, true, 128>(A, count, nx, ny, nout, st);
  }
}

// Modelled cycles of an MMA of N columns: the larger of its math (128 x N x
// 16 fp16 multiply-adds at ~6750 flop/cycle per SM) and its operand reads
// from shared memory (4 KB of A plus 32 N bytes of B at 128 bytes/cycle),
// and at least 46 (the tightest issue loop).
static double mma_cycles(int N) {
  const double math = 4096.0 * N / 6750.0, rd = 32.0 + N / 4.0;
  const double c = math > rd ? math : rd;
  return c > 46 ? c : 46;
}

// The models look at every st-th of n Toeplitz blocks (their widths change
// slowly), so that a choice costs a microsecond or two on the host.
static int sample_step(int n) { return n > 48 ? n / 24 : 1; }

// Modelled tensor-core cycles of one product of a shape (x of nx, y of ny
// limbs, low nout limbs, band start lo), following tc_product's tile loop;
// the tiles (each a fixed cost: its first Hankel build, last drain and column
// sums) count 4000 cycles.  tiles_out: the product's tiles.
static double tc_model(TcShape sh, int nx, int ny, int nout, int lo, int *tiles_out = nullptr) {
  const ShapeInfo &I = SHAPES[sh];
  const int KB = I.kb, S = 128 / KB, R = KB / 8, NT = I.nt;
  const int mx = (8 * nx + (I.xc ? 1 : 0) + KB - 1) / KB, ey = (8 * ny + KB - 1) / 128;
  const int ctot = mx + S * ey + S - 1;
  const int cfirst = lo > 0 ? (lo / R - (S - 1) > 0 ? lo / R - (S - 1) : 0) : 0;
  double cyc = 0;
  int tiles = 0;
  for (int c0 = cfirst; R * c0 < nout; c0 += NT) {
    int W = ctot - c0;
    if (W > NT) W = NT;
    const int need = (nout - R * c0 + R - 1) / R;
    if (W > need) W = need;
    W = (W + 15) & ~15;
    if (R * (c0 + W) <= lo) continue;
    tiles++;
    const int e_lo = c0 - mx + 1 > 0 ? (c0 - mx + S) / S : 0;
    const int e_hi = (c0 + W - 1) / S < ey ? (c0 + W - 1) / S : ey;
    const int st = sample_step(e_hi - e_lo + 1);
    for (int e = e_lo; e <= e_hi; e += st) {
      const int ca = (c0 > S * e ? c0 : S * e) - c0, cb = (c0 + W < S * e + mx ? c0 + W : S * e + mx) - c0;
      cyc += (KB / 16) * mma_cycles(((cb + 15) & ~15) - (ca & ~15)) *
             (e + st <= e_hi + 1 ? st : e_hi + 1 - e);
    }
  }
  if (tiles_out) *tiles_out = tiles;
  return cyc + 4000.0 * tiles;
}

// Whether a shape computes the product at all: the 64- and 128-column tiles
// of 128-digit blocks take products whose columns fit one tile; the others
// any number of tiles.
static bool shape_applies(TcShape sh, int nx, int ny, int nout, int lo) {
  const ShapeInfo &I = SHAPES[sh];
  if (I.kb != 128 || I.nt == 256) return true;
  int tiles = 0;
  tc_model(sh, nx, ny, nout, lo, &tiles);
  return tiles <= 1;
}

// Modelled time of a product on one SM: the tensor-core cycles times what the
// shape was measured to take of them (66 shapes of 8 to 9000 limbs, fitted
// together with the models of the other two forms so that the cheapest by
// model is the fastest within 1 % on average): several small-tile CTAs share
// the SM well (64 columns), two less so, and one alone does not cover its
// setup, drains and column sums.
static double shape_cost(TcShape sh, int nx, int ny, int nout, int lo) {
  if (!shape_applies(sh, nx, ny, nout, lo)) return -1;
  const size_t smem = shape_smem(sh, nx, ny);
  if (smem == 0) return -1;
  const double c = tc_model(sh, nx, ny, nout, lo);
  return c * (SHAPES[sh].nt == 256 ? 1.7 : (SHAPES[sh].nt == 128 ? 1.5 : 1.0));
}

// The cheapest shape by the model for x of nx, y of ny limbs (among those
// whose x block width is in kb_mask: bit 0 128, bit 1 64, bit 2 32, and
// whose tile is NT when nt > 0); cost_out its modelled cost.
static TcShape best_shape(int nx, int ny, int nout, int lo, int kb_mask, int nt,
                          double *cost_out) {
  TcShape best = TC_256;
  double bc = -1;
  for (int i = 0; i < TC_NSHAPES; i++) {
    const TcShape sh = (TcShape)i;
    const int kbit = SHAPES[i].kb == 128 ? 1 : (SHAPES[i].kb == 64 ? 2 : 4);
    if (!(kb_mask & kbit) || (nt > 0 && SHAPES[i].nt != nt)) continue;
    const double c = shape_cost(sh, nx, ny, nout, lo);
    if (c >= 0 && (bc < 0 || c < bc)) {
      bc = c;
      best = sh;
    }
  }
  *cost_out = bc;
  return best;
}

// ---- one-drain products (tcone.cuh) -------------------------------------------
using tcm::one_warps;

// Attributes of k_mul_one<NT>: its largest dynamic shared memory, and the
// CTAs of a given dynamic shared memory resident on one SM (TMEM allows
// 512 / NT).
struct OneAttr {
  int dyn = 0, smem_sm = 0, overhead = 0;
  bool ok = false;
};

template <int NT, int ACC, bool ADD = false>
static const OneAttr &one_attr() {
  static const OneAttr A = [] {
    OneAttr a;
    auto *kern = tcm::k_mul_one<NT, one_warps<NT, ACC>(), ADD, ACC>;
    int dev = 0, optin = 0, reserved = 0;
    cudaFuncAttributes fa;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&a.smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) !=
            cudaSuccess ||
        cudaFuncGetAttributes(&fa, kern) != cudaSuccess)
      return a;
    a.dyn = optin - (int)fa.sharedSizeBytes;
    a.overhead = (int)fa.sharedSizeBytes + reserved;
    a.ok = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, a.dyn) ==
           cudaSuccess;
    return a;
  }();
  return A;
}

template <int NT, int ACC>
static int one_per_sm(size_t smem) {
  const OneAttr &a = one_attr<NT, ACC>();
  const int per_sm = a.smem_sm / (int)(smem + a.overhead), cap = 512 / (NT * ACC);
  return per_sm > cap ? cap : (per_sm < 1 ? 1 : per_sm);
}

// At least so much shared memory that no SM takes more CTAs than its tensor
// memory serves: one too many queues for it through all of another CTA's
// products (65536 products of 64 limbs 390 us, 440 to 590 with five CTAs on
// some SMs).
template <int NT, int ACC>
static size_t one_smem_floor(size_t smem) {
  const OneAttr &a = one_attr<NT, ACC>();
  const size_t least = (size_t)(a.smem_sm / (512 / (NT * ACC) + 1) - a.overhead + 1);
  return smem > least ? smem : least;
}

// Shared memory of a product (x of nx, y of ny limbs, low nout limbs, band
// start lo) in the form with NT-column tiles (0: it does not take it), and
// its modelled time on one SM in tensor-core cycles, comparable with
// shape_cost: the MMAs (their math, their operands' reads, at least 46
// cycles each), the shared-memory cycles of a tile's Hankel matrices (16 per
// block) and transposes (8 per column), and the part of a tile's ~5000
// cycles of latency and limb work that the CTAs sharing the SM do not hide.
template <int NT, int ACC = 1>
static size_t one_plan(int nx, int ny, int nout, int lo, double *cost) {
  constexpr int S = tcm::ONE_S, W = one_warps<NT, ACC>();
  const int ns = nx < ny ? nx : ny;
  if (ns > (ACC == 2 ? tcm::ONE_MAX2 : tcm::ONE_MAX) || (ACC == 2 && ns <= tcm::ONE_MAX)) return 0;
  if (!one_attr<NT, ACC>().ok) return 0;
  const uint32_t total = tcm::one_bytes<NT, W>(nx, ny, nout, lo);
  if (total > (uint32_t)one_attr<NT, ACC>().dyn) return 0;
  if (cost != nullptr) {
    const int mx = tcm::one_layout<W>(nx, ny, 0).mx, per_sm = one_per_sm<NT, ACC>(total);
    double cyc = nx;
    tcm::one_tiles<NT>(nx, ny, nout, lo, [&](int c0, int Wd, int e_lo, int e_hi) {
      cyc += 8.0 * Wd + (per_sm == 1 ? 7400.0 : (NT == 128 ? 5000.0 : 4500.0) / per_sm);
      if (e_hi < e_lo) return;
      cyc += 16.0 * (e_hi - e_lo + 1);
      const int st = sample_step(e_hi - e_lo + 1);
      for (int e = e_lo; e <= e_hi; e += st) {
        const int ca = (c0 > S * e ? c0 : S * e) - c0;
        const int cb = (c0 + Wd < S * e + mx ? c0 + Wd : S * e + mx) - c0;
        cyc += 2 * mma_cycles(((cb + 15) & ~15) - (ca & ~15)) * (e + st <= e_hi + 1 ? st : e_hi + 1 - e);
      }
    });
    *cost = cyc;
  }
  return total;
}

template <int NT, int ACC = 1>
static int launch_one(const TcArgs &A, int64_t count, int nx, int ny, int nout, cudaStream_t st) {
  constexpr int W = one_warps<NT, ACC>();
  size_t smem = one_plan<NT, ACC>(nx, ny, nout, A.lo, nullptr);
  if (smem == 0) return BIGINT_EINVAL;
  if (count == 0) return BIGINT_OK;
  const int sms = sm_count();
  if (sms == 0) return BIGINT_ECUDA;
  const int64_t slots = (int64_t)sms * one_per_sm<NT, ACC>(smem);
  const int64_t grid = count < slots ? count : slots;
  smem = one_smem_floor<NT, ACC>(smem);
  auto *kern =
      A.add != nullptr ? tcm::k_mul_one<NT, W, true, ACC> : tcm::k_mul_one<NT, W, false, ACC>;
  if (A.add != nullptr && !one_attr<NT, ACC, true>().ok) return BIGINT_ECUDA;
  return chain_launch(grid <= sms, kern, (unsigned)grid, 32 * W, smem, st, A.x, A.y, A.out, nx, ny, nout, count,
                      A.sx, A.sy, A.so, A.lo, A.abort_flag, A.add, A.sadd);
}

// ---- pipelined products (tcpipe.cuh) --------------------------------------------
template <int KB, int NT>
static const OneAttr &pipe_attr() {
  static const OneAttr A = [] {
    OneAttr a;
    int dev = 0, optin = 0;
    cudaFuncAttributes fa;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
            cudaSuccess ||
        cudaFuncGetAttributes(&fa, tcm::k_mul_pipe<KB, NT>) != cudaSuccess)
      return a;
    a.dyn = optin - (int)fa.sharedSizeBytes;
    a.ok = cudaFuncSetAttribute(tcm::k_mul_pipe<KB, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                a.dyn) == cudaSuccess;
    return a;
  }();
  return A;
}

template <int KB, int NT>
static int launch_pipe(const TcArgs &A, int64_t count, int nx, int ny, int nout, cudaStream_t st) {
  if (!pipe_attr<KB, NT>().ok) return BIGINT_ECUDA;
  const tcm::PipeLayout L = tcm::pipe_layout<KB>(nx, (uint32_t)pipe_attr<KB, NT>().dyn);
  if (L.total == 0 || nx < 64) return BIGINT_EINVAL;
  if (count == 0) return BIGINT_OK;
  const int sms = sm_count();
  if (sms == 0) return BIGINT_ECUDA;
  return chain_launch(true, tcm::k_mul_pipe<KB, NT>, (unsigned)(count < sms ? count : sms),
                      tcm::PIPE_THREADS, L.total, st, A.x, A.y, A.out, nx, ny, nout, count, A.sx,
                      A.sy, A.so, A.lo, A.abort_flag, A.add, A.sadd, L);
}

// Modelled time of a product in the pipelined form (-1: x does not fit): its
// MMAs, at least 42 cycles each (warp-uniform issue), 10 % slower beside the
// drains and builds, 900 cycles a drain and 9000 (5000 with 128-column tiles)
// a tile, the part of its limbs that the groups ahead do not cover.  128-
// column tiles for products of one such tile only.
template <int KB, int NT>
static double pipe_cost(int nx, int ny, int nout, int lo) {
  constexpr int S = 128 / KB;
  if (nx < 64 || !pipe_attr<KB, NT>().ok ||
      tcm::pipe_layout<KB>(nx, (uint32_t)pipe_attr<KB, NT>().dyn).total == 0)
    return -1;
  const int mx = (8 * nx + KB - 1) / KB;
  double cyc = 0;
  int tiles = 0;
  tcm::pipe_tiles<KB, NT>(nx, ny, nout, lo, [&](int c0, int W, int e_lo, int e_hi) {
    tiles++;
    cyc += NT == 256 ? 9000 : 5000;
    if (e_hi < e_lo) return true;
    const int n = e_hi - e_lo + 1, st = sample_step(n);
    cyc += 900.0 * ((n * KB + 1023) / 1024);
    for (int e = e_lo; e <= e_hi; e += st) {
      const int ca = (c0 > S * e ? c0 : S * e) - c0;
      const int cb = (c0 + W < S * e + mx ? c0 + W : S * e + mx) - c0;
      const int N = ((cb + 15) & ~15) - (ca & ~15);
      const double math = N / 2.0, rd = 32.0 + N / 4.0, m = math > rd ? math : rd;
      cyc += 1.1 * (KB / 16) * (m > 42 ? m : 42) * (e + st <= e_hi + 1 ? st : e_hi + 1 - e);
    }
    return true;
  });
  return NT == 256 || tiles <= 1 ? cyc : -1;
}

// The pipeline with 32-digit blocks, for uniform batches only: a grouped
// launch per form more costs a step of a ragged batch more than it saves
// (20000 mixed operations 17.4 -> 17.8 ms).
constexpr int FORM_PIPE32 = RAG_NSHAPES;
// The one-drain form with two accumulators, likewise.
constexpr int FORM_ONE2 = RAG_NSHAPES + 1;

// The one-drain (RAG_ONE...) or pipelined (RAG_PIPE...) form, either operand as x (*swap), where its model is cheaper
// than `than` (< 0: anything); -1 where none is.
static int best_form(int nx, int ny, int nout, int lo, double than, bool *swap,
                     bool grouped = false) {
  int form = -1;
  auto offer = [&](double c, int f, int k) {
    if (c >= 0 && (than < 0 || c < than)) than = c, form = f, *swap = k != 0;
  };
  for (int k = 0; k < (nx == ny ? 1 : 2); k++) {
    const int mx = k ? ny : nx, my = k ? nx : ny;
    double c;
    if (one_plan<128>(mx, my, nout, lo, &c)) offer(c, RAG_ONE128, k);
    if (one_plan<256>(mx, my, nout, lo, &c)) offer(c, RAG_ONE256, k);
    offer(pipe_cost<128, 256>(mx, my, nout, lo), RAG_PIPE128, k);
    offer(pipe_cost<64, 256>(mx, my, nout, lo), RAG_PIPE64, k);
    offer(pipe_cost<128, 128>(mx, my, nout, lo), RAG_PIPE128N, k);
    offer(pipe_cost<64, 128>(mx, my, nout, lo), RAG_PIPE64N, k);
    if (grouped) continue;
    offer(pipe_cost<32, 256>(mx, my, nout, lo), FORM_PIPE32, k);
    if (one_plan<128, 2>(mx, my, nout, lo, &c)) offer(c, FORM_ONE2, k);
  }
  return form;
}

// Launches a form of best_form (sw: with the operands' roles exchanged).
static int launch_form(int form, TcArgs A, bool sw, int64_t count, int nx, int ny, int nout,
                       cudaStream_t st) {
  if (sw) {
    const uint64_t *t = A.x; A.x = A.y; A.y = t;
    const int64_t ts = A.sx; A.sx = A.sy; A.sy = ts;
    const int tn = nx; nx = ny; ny = tn;
  }
  switch (form) {
    case RAG_ONE128: return launch_one<128>(A, count, nx, ny, nout, st);
    case RAG_ONE256: return launch_one<256>(A, count, nx, ny, nout, st);
    case FORM_ONE2: return launch_one<128, 2>(A, count, nx, ny, nout, st);
    case RAG_PIPE128: return launch_pipe<128, 256>(A, count, nx, ny, nout, st);
    case RAG_PIPE64: return launch_pipe<64, 256>(A, count, nx, ny, nout, st);
    case RAG_PIPE128N: return launch_pipe<128, 128>(A, count, nx, ny, nout, st);
    case RAG_PIPE64N: return launch_pipe<64, 128>(A, count, nx, ny, nout, st);
    default: return launch_pipe<32, 256>(A, count, nx, ny, nout, st);
  }
}

// out = low n limbs of a b + c for a batch of n-limb operands (instance i at
// a + i sa, ...; c may be null or out), n >= 64, by a form that takes an addend.
int launch_mul_add(const uint64_t *a, const uint64_t *b, const uint64_t *c, uint64_t *out,
                   int64_t count, int n, cudaStream_t st) {
  bool sw = false;
  const int form = best_form(n, n, n, 0, -1, &sw);
  if (form < 0) return BIGINT_EINVAL;
  return launch_form(form, TcArgs{a, b, out, n, n, n, 0, nullptr, c, n}, sw, count, n, n, n, st);
}

// The same choice for a product of a grouped launch (ragged.cu): a RagShape,
// with x as the operand of nx limbs unless *swap.
int tc_choose(int nx, int ny, int nout, int lo, bool *swap) {
  int sh = RAG_256;
  double best = -1;
  *swap = nx > ny;
  for (int k = 0; k < (nx == ny ? 1 : 2); k++) {
    const int mx = k ? ny : nx, my = k ? nx : ny;
    if (mx > 16383) continue;
    static const struct { TcShape s; int r; } forms[3] = {
        {TC_64_XC, RAG_64}, {TC_128_XC, RAG_128}, {TC_256, RAG_256}};
    for (const auto &f : forms) {
      const double c = shape_cost(f.s, mx, my, nout, lo);
      if (c >= 0 && (best < 0 || c < best)) best = c, sh = f.r, *swap = k != 0;
    }
  }
  bool sw = false;
  const int form = best_form(nx, ny, nout, lo, best, &sw, true);
  if (form < 0) return sh;
  *swap = sw;
  return form;
}

// force: 0 (the one-drain, pipelined or 128-digit-block shape by the models
// above and below) or one of the autotuner's candidates -- TC_FORCE_64 / _128 / _256
// (128-digit blocks, that tile) and TC_FORCE_N64 / _N32 (narrow blocks).
int launch_mul_tc_ex(const uint64_t *a, int64_t sa, const uint64_t *b, int64_t sb, uint64_t *out,
                     int64_t so, int64_t count, int na, int nb, int nout, int lo, int *abort_flag,
                     cudaStream_t st, int force) {
  if (nout > na + nb) return BIGINT_EINVAL;
  if (lo == 0) {  // limbs at and above nout do not reach the low nout limbs
    if (na > nout) na = nout;
    if (nb > nout) nb = nout;
  }
  TcArgs A{a, b, out, sa, sb, so, lo, abort_flag};
  int nx = na, ny = nb;
  if (nb < na) {
    A.x = b; A.y = a; A.sx = sb; A.sy = sa;
    nx = nb; ny = na;
  }
  if (nx < 1 || nx > 16383 || ny > 32768 || nout < 1 || nout > na + nb || lo < 0 || lo >= nout)
    return BIGINT_EINVAL;
  if (shape_smem(TC_256, nx, ny) == 0) return BIGINT_EINVAL;
  int kb_mask = 1, nt = 0;
  switch (force) {
    case 0: break;
    case TC_FORCE_64: kb_mask = 1; nt = 64; break;
    case TC_FORCE_128: kb_mask = 1; nt = 128; break;
    case TC_FORCE_256: kb_mask = 1; nt = 256; break;
    case TC_FORCE_N64: kb_mask = 2; break;
    case TC_FORCE_N32: kb_mask = 4; break;
    default: return BIGINT_EINVAL;
  }
  // x is the operand stored whole in shared memory (the B side), y the one
  // whose Toeplitz blocks are the A side.  Either may be the shorter: the
  // model often prefers the shorter operand as y (fewer, wider MMAs for a
  // low product whose longer operand has most of the columns), as long as
  // the longer one fits shared memory as x and in a column sum's range.
  double keep = 0, swap = -1;
  TcShape sh = best_shape(nx, ny, nout, lo, kb_mask, nt, &keep);
  if (keep < 0 && force != 0) {  // the forced shape does not take this product
    kb_mask = 1;
    nt = 0;
    sh = best_shape(nx, ny, nout, lo, kb_mask, nt, &keep);
  }
  if (nx != ny && ny <= 16383) {
    const TcShape sw = best_shape(ny, nx, nout, lo, kb_mask, nt, &swap);
    if (swap >= 0 && (keep < 0 || swap < keep)) {
      const uint64_t *tp = A.x; A.x = A.y; A.y = tp;
      const int64_t ts = A.sx; A.sx = A.sy; A.sy = ts;
      const int tn = nx; nx = ny; ny = tn;
      sh = sw;
      keep = swap;
    }
  }
  if (force == 0) {
    bool sw = false;
    const int form = best_form(nx, ny, nout, lo, keep, &sw);
    if (form >= 0) return launch_form(form, A, sw, count, nx, ny, nout, st);
  }
  if (keep < 0) return BIGINT_EINVAL;
  return launch_shape(sh, A, count, nx, ny, nout, st);
}

int launch_mul_tc(const uint64_t *a, const uint64_t *b, uint64_t *out, int64_t count, int na,
                  int nb, int nout, cudaStream_t st, int force_nt) {
  return launch_mul_tc_ex(a, na, b, nb, out, nout, count, na, nb, nout, 0, nullptr, st, force_nt);
}

// ---- split-K products (host) --------------------------------------------------
namespace {

constexpr int SK_G = 8;  // Toeplitz blocks per group

int sk_dyn_max() {
  static int dyn = -1;
  if (dyn < 0) {
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
        cudaSuccess)
      return 0;
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, tcm::k_mul_tc_sk<256, SK_G>) != cudaSuccess) return 0;
    const int d = optin - (int)fa.sharedSizeBytes;
    if (cudaFuncSetAttribute(tcm::k_mul_tc_sk<256, SK_G>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, d) != cudaSuccess)
      return 0;
    dyn = d;
  }
  return dyn;
}

// Tiles of 256 columns of the low nout limbs of x * y (x with its carry
// digit) from the column of limb lo on, as tc_product computes them; groups
// of SK_G blocks per tile.  Returns false if there are more than SK_MAX_TILES.
bool sk_tiles(int nx, int ny, int nout, int lo, tcm::SkPlan &P, int *groups) {
  const int mx = (8 * nx + 1 + 127) / 128, ey = (8 * ny + 127) / 128, ctot = mx + ey;
  P.cfirst = lo > 0 ? lo / 16 : 0;
  P.T = 0;
  for (int c0 = P.cfirst; 16 * c0 < nout; c0 += 256) {
    if (P.T == tcm::SK_MAX_TILES) return false;
    int W = ctot - c0;
    if (W > 256) W = 256;
    const int need = (nout - 16 * c0 + 15) / 16;
    if (W > need) W = need;
    W = (W + 15) & ~15;
    const int e_lo = c0 - mx + 1 > 0 ? c0 - mx + 1 : 0, e_hi = c0 + W - 1 < ey ? c0 + W - 1 : ey;
    P.c0[P.T] = c0;
    P.W[P.T] = W;
    groups[P.T] = e_hi >= e_lo ? (e_hi - e_lo + SK_G) / SK_G : 0;
    P.T++;
  }
  return P.T > 0;
}

}  // namespace

// Column-sum buffer bytes of one split-K product (0: not splittable).
// (Shared memory bound as for the split products: the opt-in limit per block
// of sm_100 and sm_103 less room for the kernel's static shared memory, so
// that the size does not depend on querying a device.)
constexpr size_t SK_SMEM_CAP = 232448 - 2048;

size_t mul_sk_bytes_per_product(int na, int nb, int nout, int lo) {
  const int nx = na < nb ? na : nb, ny = na < nb ? nb : na;
  tcm::SkPlan P;
  int groups[tcm::SK_MAX_TILES];
  if (nx < 1 || nx > 16383 || ny > 32768 || nout < 1 || nout > na + nb || lo < 0 || lo >= nout)
    return 0;
  if (tcm::layout<256, SK_G>(nx, ny).total > SK_SMEM_CAP) return 0;
  if (!sk_tiles(nx, ny, nout, lo, P, groups)) return 0;
  return (size_t)P.T * 256 * 128 * sizeof(int);
}

// True if the split-K form would run more units than the ordinary launch
// has CTAs busy: few products (count x tiles well below the SMs).  Not for
// products the one-drain form takes: one of 512 limbs is 12 us there on one
// CTA, 18 us as units, sums and finish.
bool mul_sk_worth(int64_t count, int na, int nb, int nout, int lo) {
  const int nx = na < nb ? na : nb, ny = na < nb ? nb : na;
  if (nx <= tcm::ONE_MAX || mul_sk_bytes_per_product(na, nb, nout, lo) == 0) return false;
  tcm::SkPlan P;
  int groups[tcm::SK_MAX_TILES];
  if (!sk_tiles(nx, ny, nout, lo, P, groups)) return false;
  const int sms = sm_count();
  return sms > 0 && count * P.T * 2 <= sms;
}

// The low nout limbs (from limb lo: band mode, as tc_product) of a batch of
// products, each cut into units of (tile, groups) spread over the SMs; the
// units add their column sums into `colsum` (count x
// mul_sk_bytes_per_product bytes), zeroed here or, in a chain of products,
// by the finish of the product before, then a cluster per product forms the
// limbs.  Results are those of tc_product (bit-identical).
int launch_mul_tc_sk(const uint64_t *a, int64_t sa, const uint64_t *b, int64_t sb, uint64_t *out,
                     int64_t so, int64_t count, int na, int nb, int nout, int lo, void *colsum,
                     size_t colsum_bytes, SkBuffers *chain, int *abort_flag, cudaStream_t st) {
  const uint64_t *x = a, *y = b;
  int64_t sx = sa, sy = sb;
  int nx = na, ny = nb;
  if (nb < na) { x = b; y = a; sx = sb; sy = sa; nx = nb; ny = na; }
  if (count == 0) return BIGINT_OK;
  if (nx < 1 || nx > 16383 || ny > 32768 || nout < 1 || nout > na + nb || lo < 0 || lo >= nout)
    return BIGINT_EINVAL;
  const size_t per = mul_sk_bytes_per_product(na, nb, nout, lo);
  if (per == 0 || colsum == nullptr || colsum_bytes < per * (size_t)count) return BIGINT_EINVAL;
  const int sms = sm_count();
  if (sms == 0) return BIGINT_ECUDA;
  const size_t smem = tcm::layout<256, SK_G>(nx, ny).total;
  if (sk_dyn_max() <= 0 || smem > (size_t)sk_dyn_max()) return BIGINT_EINVAL;
  tcm::SkPlan P;
  int groups[tcm::SK_MAX_TILES];
  if (!sk_tiles(nx, ny, nout, lo, P, groups)) return BIGINT_EINVAL;
  // groups per unit: about one unit per SM over the whole launch (each unit
  // first stages x and its first Hankel buffer, so units are not cut finer)
  int64_t total = 0;
  for (int t = 0; t < P.T; t++) total += groups[t];
  total *= count;
  int64_t gpc = (total + sms - 1) / sms;
  if (gpc < 1) gpc = 1;
  P.gpc = (int)gpc;
  P.first[0] = 0;
  for (int t = 0; t < P.T; t++) P.first[t + 1] = P.first[t] + (int)((groups[t] + gpc - 1) / gpc);
  const int64_t units = count * P.first[P.T];
  int *zbuf = nullptr;
  int64_t zero = 0;
  if (chain != nullptr) {
    zbuf = static_cast<int *>(chain->buf[chain->cur ^ 1]);
    zero = (int64_t)(chain->used / sizeof(int));
    chain->used = per * (size_t)count;
    chain->cur ^= 1;
  } else {
    BIGINT_CUDA_TRY(cudaMemsetAsync(colsum, 0, per * (size_t)count, st));
  }
  const int64_t stride = (int64_t)(per / sizeof(int));
  const unsigned grid = (unsigned)(units < sms ? units : sms);
  int rc = chain_launch(true, tcm::k_mul_tc_sk<256, SK_G>, grid, 2 * 256 + 32, smem, st, x, y, nx, ny, sx, sy, count, P,
                        static_cast<int *>(colsum), stride, abort_flag);
  if (rc != BIGINT_OK) return rc;
  const int L0 = 16 * P.cfirst;
  // clearing CTAs: 16 KB each
  int64_t clear = (zero + 4095) / 4096;
  if (clear > 64) clear = 64;
  clear = (clear + tcm::SKF_CLUSTER - 1) / tcm::SKF_CLUSTER * tcm::SKF_CLUSTER;
  return chain_launch<tcm::SKF_CLUSTER>(
      true, tcm::k_tc_sk_finish, (unsigned)(count * tcm::SKF_CLUSTER + clear), tcm::SKF_THREADS, 0,
      st, static_cast<const int *>(colsum), stride, out, so, L0, nout,
      lo > 0 ? (1ull << 32) : 0ull, count, zbuf, zero);
}

// ---- split products ----------------------------------------------------------
int launch_mul(const uint64_t *a, const uint64_t *b, uint64_t *out, int64_t count, int na, int nb,
               int nout, cudaStream_t st);

namespace {

constexpr int SPLIT_NT = 256, SPLIT_G = 8, SPLIT_TILE_LIMBS = 16 * SPLIT_NT;

int split_dyn_max() {
  static int dyn = -1;
  if (dyn < 0) {
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
        cudaSuccess)
      return 0;
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, tcm::k_mul_tc_split<SPLIT_NT, SPLIT_G>) != cudaSuccess) return 0;
    const int d = optin - (int)fa.sharedSizeBytes;
    if (cudaFuncSetAttribute(tcm::k_mul_tc_split<SPLIT_NT, SPLIT_G>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, d) != cudaSuccess)
      return 0;
    dyn = d;
  }
  return dyn;
}

int launch_split(const uint64_t *x, const uint64_t *y, uint64_t *out, int64_t count, int nx, int ny,
                 int T, uint64_t *tile_carry, cudaStream_t st) {
  const size_t smem = tcm::layout<SPLIT_NT, SPLIT_G>(nx, ny).total;
  const int dyn = split_dyn_max();
  if (dyn <= 0 || smem > (size_t)dyn) return BIGINT_EINVAL;
  int dev = 0, sms = 0;
  BIGINT_CUDA_TRY(cudaGetDevice(&dev));
  BIGINT_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t units = count * T, grid = units < sms ? units : sms;
  const int nout = nx + ny;
  tcm::k_mul_tc_split<SPLIT_NT, SPLIT_G><<<(unsigned)grid, 2 * SPLIT_NT + 32, smem, st>>>(
      x, y, out, nx, ny, nout, count, T, tile_carry);
  int rc = bigint_launch_status();
  if (rc != BIGINT_OK) return rc;
  tcm::k_tc_split_finish<<<(unsigned)count, 512, 0, st>>>(out, nout, T, SPLIT_TILE_LIMBS,
                                                         tile_carry);
  return bigint_launch_status();
}

// Shared memory a split CTA may take (the opt-in limit per block of sm_100
// and sm_103, less room for the kernel's static shared memory).
constexpr size_t SPLIT_SMEM_CAP = 232448 - 2048;

// Tiles of an nx x ny split product, or 0 if it does not run split (columns
// of 128 digits that fit a 128-column tile, x too large for shared memory,
// or a single tile).
int split_tiles(int nx, int ny) {
  if (nx < 1 || ny > 16383 || (8 * nx + 127) / 128 + (8 * ny + 127) / 128 <= 128) return 0;
  if (tcm::layout<SPLIT_NT, SPLIT_G>(nx, ny).total > SPLIT_SMEM_CAP) return 0;
  const int T = (nx + ny + SPLIT_TILE_LIMBS - 1) / SPLIT_TILE_LIMBS;
  return T >= 2 ? T : 0;
}

}  // namespace

// Batches of at most this many products take the split-K form in
// bigint_mul_split (its column-sum buffers grow with the batch).
constexpr int64_t SPLIT_SK_MAX_COUNT = 16;

size_t mul_split_workspace(int64_t count, int na, int nb) {
  const int nx = na < nb ? na : nb, ny = na < nb ? nb : na;
  const size_t tiles = (size_t)16 * (size_t)count * (size_t)split_tiles(nx, ny);
  if (count > SPLIT_SK_MAX_COUNT || nx < 256) return tiles;
  const size_t sk = (size_t)count * mul_sk_bytes_per_product(na, nb, na + nb, 0);
  return sk > tiles ? sk : tiles;
}

// The full products of launch_mul spread over CTAs: up to SPLIT_SK_MAX_COUNT
// products in the split-K form (units of tile and groups, about one per SM),
// larger batches with each product's tiles on different CTAs (split_tiles),
// and launch_mul itself where the product has one tile or another shape.
int launch_mul_split(const uint64_t *a, const uint64_t *b, uint64_t *out, int64_t count, int na,
                     int nb, void *ws, size_t bytes, cudaStream_t st) {
  const size_t need = count > 0 ? mul_split_workspace(count, na, nb) : 0;
  if (need == 0) return launch_mul(a, b, out, count, na, nb, na + nb, st);
  if (bytes < need) return BIGINT_ENOMEM;
  if (!ws || (reinterpret_cast<uintptr_t>(ws) % 8) != 0) return BIGINT_EINVAL;
  // a few products: each cut into (tile, groups) units over the SMs
  if (count <= SPLIT_SK_MAX_COUNT && mul_sk_worth(count, na, nb, na + nb, 0))
    return launch_mul_tc_sk(a, na, b, nb, out, na + nb, count, na, nb, na + nb, 0, ws, bytes,
                            nullptr, nullptr, st);
  const uint64_t *x = a, *y = b;
  int nx = na, ny = nb;
  if (nb < na) { x = b; y = a; nx = nb; ny = na; }
  const int T = split_tiles(nx, ny);
  if (T == 0) return launch_mul(a, b, out, count, na, nb, na + nb, st);
  uint64_t *tcarry = static_cast<uint64_t *>(ws);
  return launch_split(x, y, out, count, nx, ny, T, tcarry, st);
}

// BIGINT_ETIMEOUT if a tensor-core product hit a wait limit since the last
// call (synchronises the device), else BIGINT_OK.
int tc_take_timeout() { return tcm::take_timeout_here(); }
int tc_set_wait_limit(long long cycles) { return tcm::set_wait_limit_here(cycles); }

}  // namespace bigint
