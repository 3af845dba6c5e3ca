// tcone.cuh -- tensor-core products whose column sums need a single drain.
//
// The digit convolution of tccore.cuh (signed base-256 digits as fp16,
// Toeplitz blocks of y times shifted blocks of x, exact fp32 accumulation),
// laid out for products whose shorter operand has at most ONE_MAX limbs:
//
//  * x in blocks of KB = 32 digits, S = 128 / KB = 4 rows per coefficient
//    (row u + 32 a of column c - a, a < 4, belongs to coefficient 32 c + u).
//    An MMA of a 512 x 512-limb product is then 128-144 columns wide instead
//    of 16-64 with 128-digit blocks, for the same 4 KB of A read from shared
//    memory: with at most 64 columns that read, not the arithmetic, is an
//    MMA's time (tccore.cuh: 32 + N / 4 cycles against N / 2).
//  * One accumulator, no drain before the end.  A row of a column sums at
//    most 32 ceil(n / 16) digit products, n the shorter operand's limbs, so
//    up to 512 limbs at most 1024 products of magnitude <= 2^14, plus one
//    with y's carry digit (0 or 1; x goes without one, below).  A partial
//    sum therefore is at most 2^24 -- exact in fp32 -- unless every one of
//    the 1024 products has magnitude 2^14; then it is a multiple of 128 below
//    2^25, exact as well.  (If one of them is not 128 * 128 it is at most
//    128 * 127 = 2^14 - 128, which makes room for the carry digit's 128.)
//  * Shorter operands of up to ONE_MAX2 limbs take two accumulators (ACC = 2):
//    even Toeplitz blocks add into one, odd ones into the other.  A column meets
//    at most ceil(n / 16) consecutive blocks, so each sums the products of at most
//    32 of them, within the same bound, and a column sum is the sum of two
//    drains at the end.  With 128-column tiles that is two CTAs per SM, as
//    long as the Hankel matrices of a tile's blocks (up to about 640 limbs) leave
//    room for two.  4096 products of 515 limbs by the top of 1024: 141 us, 192
//    in the pipeline; 6080 of 520 limbs 351, 399.
//  * So a CTA needs NT ACC tensor-memory columns and no registers for column
//    sums, and 512 / (NT ACC) CTAs share an SM: while one forms limbs, the others'
//    MMAs run.  The Hankel core matrices of all of y's blocks lie in shared
//    memory at once; the column sums are transposed through the same memory.
//  * Core matrices of A are 144 bytes apart instead of 128: a thread writes
//    the eight rows of one straight from its registers (no staging run), and
//    the warp's 16-byte stores then fall on different banks.
//  * Limbs.  A thread forms V_j = sum_k (coef(8 j + k) + 2^31) 2^(8 k) (plus
//    limb j - nx of y where x's top bit is set: x goes without its carry
//    digit), takes the bias word off the low 64 bits at once and the borrow
//    off the high word (never below 1: the bias puts more than 2^22 there),
//    so one carry scan of the low words plus the high words one limb up
//    finishes the tile; the words stay in registers until then.
//
// Bound: shared memory (the MMAs' operands, the transposes, the Hankel
// stores: 7K of 9.5K cycles a product at 512 limbs, tensor pipe 0.55 of the
// cuBLAS rate) and, below 200 limbs, latency: 16 warps an SM, all that the
// tensor memory admits, issue half the time.  131072 products of 512 limbs
// 4182 us (6770 as tc_product), 65536 of 160 limbs 662 us (2281 on the
// integer pipes), 72 of 512 limbs 10.6 us (24.6).
#pragma once
#include "tccore.cuh"

namespace bigint {
namespace tcm {

constexpr int ONE_KB = 32, ONE_S = 128 / ONE_KB, ONE_R = ONE_KB / 8;
constexpr int ONE_MAX = 1024 / ONE_KB * 16;  // limbs of the shorter operand
constexpr int ONE_MAX2 = 2 * ONE_MAX - 16;   // with two accumulators
constexpr int ONE_CM = 144;                  // bytes from core matrix to core matrix of A
constexpr int ONE_CS = 132;                  // words per transposed column

struct OneLayout {
  int mx, ey, cmma;  // x blocks, last Toeplitz block, columns the MMAs write
  int ptot;          // stored x blocks
  uint32_t xs, z, prev, hk, total;
};

// Dynamic shared memory: x, the zero A operand of the clearing MMA, the
// columns before a run of columns (three generations of S - 1), and the
// Hankel core matrices of at most `blocks` Toeplitz blocks, whose memory the
// column sums of one_bufs runs of 8 W columns reuse after the MMAs (W warps).
template <int W>
__host__ __device__ constexpr int one_bufs() { return W >= 16 ? 1 : 2; }
template <int W>
__host__ __device__ inline OneLayout one_layout(int nx, int ny, int blocks) {
  OneLayout L;
  L.mx = (8 * nx + ONE_KB - 1) / ONE_KB;
  L.ey = (8 * ny + ONE_KB - 1) / 128;
  L.cmma = L.mx + ONE_S * L.ey;
  L.ptot = (L.mx + 32 + 7) / 8 * 8 + 2;  // 2 mod 8: a warp's x stores hit distinct banks
  L.xs = 0;
  L.z = (uint32_t)L.ptot * 16u * ONE_R;
  L.prev = L.z + ZB * 128;
  L.hk = L.prev + 3 * (ONE_S - 1) * ONE_CS * 4;
  const uint32_t hb = (uint32_t)(16 * blocks + ONE_R - 1) * ONE_CM;
  const uint32_t cs = (uint32_t)one_bufs<W>() * 8 * W * ONE_CS * 4;
  L.total = L.hk + (hb > cs ? hb : cs);
  return L;
}

// Toeplitz blocks of the tile of columns [c0, c0 + W).
__host__ __device__ inline void one_blocks(int mx, int ey, int c0, int W, int &e_lo, int &e_hi) {
  e_lo = c0 - mx + 1 > 0 ? (c0 - mx + ONE_S) / ONE_S : 0;
  e_hi = (c0 + W - 1) / ONE_S < ey ? (c0 + W - 1) / ONE_S : ey;
}

// Warps per CTA.  More of them (8 / 16) shorten a lone product's phases by
// 15 % but not a batch, where the CTAs sharing the SM overlap anyway
// (512-limb products 2451 against 2167 us per 65536).
template <int NT, int ACC = 1>
__host__ __device__ constexpr int one_warps() { return NT * ACC == 128 ? 4 : 8; }

// The tiles of NT columns of a product (low nout limbs, band start lo):
// f(c0, W, e_lo, e_hi) for each.
template <int NT, class F>
inline void one_tiles(int nx, int ny, int nout, int lo, F f) {
  constexpr int R = ONE_R, S = ONE_S;
  const OneLayout L = one_layout<4>(nx, ny, 0);
  for (int c0 = lo > 0 ? (lo / R - (S - 1) > 0 ? lo / R - (S - 1) : 0) : 0; R * c0 < nout;
       c0 += NT) {
    int Wd = L.cmma + S - 1 - c0 < NT ? L.cmma + S - 1 - c0 : NT;
    const int need = (nout - R * c0 + R - 1) / R;
    if (Wd > need) Wd = need;
    Wd = (Wd + 15) & ~15;
    int e_lo, e_hi;
    one_blocks(L.mx, L.ey, c0, Wd, e_lo, e_hi);
    f(c0, Wd, e_lo, e_hi);
  }
}

// Dynamic shared memory of such a product with NT-column tiles.
template <int NT, int W>
inline uint32_t one_bytes(int nx, int ny, int nout, int lo) {
  int blocks = 0;
  one_tiles<NT>(nx, ny, nout, lo, [&](int, int, int e_lo, int e_hi) {
    if (e_hi - e_lo + 1 > blocks) blocks = e_hi - e_lo + 1;
  });
  return one_layout<W>(nx, ny, blocks).total;
}

// fp16 digits 7 .. 0 of limb v (below = the limb underneath), as four words.
__device__ __forceinline__ void digits_down(uint64_t v, uint64_t below, uint32_t *w) {
  const Digits16 d = recode16(v, below);
  const uint32_t el = (uint32_t)d.ev, eh = (uint32_t)(d.ev >> 32);
  const uint32_t ol = (uint32_t)d.od, oh = (uint32_t)(d.od >> 32);
  w[0] = unbias_h2(__byte_perm(oh, eh, 0x7632));
  w[1] = unbias_h2(__byte_perm(oh, eh, 0x5410));
  w[2] = unbias_h2(__byte_perm(ol, el, 0x7632));
  w[3] = unbias_h2(__byte_perm(ol, el, 0x5410));
}

// One Hankel core matrix: row r = the eight digits starting r places down the
// digits of the limbs v[0] and v[1] (v[2] underneath), at `row`.
__device__ __forceinline__ void hankel_rows(uint8_t *row, const uint64_t (&v)[3]) {
  uint32_t w[8], f[7];
  digits_down(v[0], v[1], w);
  digits_down(v[1], v[2], w + 4);
#pragma unroll
  for (int i = 0; i < 7; i++) f[i] = __byte_perm(w[i], w[i + 1], 0x5432);
  uint4 *o = reinterpret_cast<uint4 *>(row);
#pragma unroll
  for (int m = 0; m < 4; m++) {
    o[2 * m] = make_uint4(w[m], w[m + 1], w[m + 2], w[m + 3]);
    o[2 * m + 1] = make_uint4(f[m], f[m + 1], f[m + 2], f[m + 3]);
  }
}

// Limb of eight coefficients w (biased by 2^31): V = sum_k w_k 2^(8 k) + add,
// less the bias word of the limb (`first`: the lowest one kept), the borrow
// taken off the high word.
__device__ __forceinline__ void limb_of(const uint32_t (&w)[8], uint64_t add, bool first,
                                        uint64_t &low, uint32_t &high) {
  const uint64_t s0 = (uint64_t)w[0] + ((uint64_t)w[1] << 8) + ((uint64_t)w[2] << 16) +
                      ((uint64_t)w[3] << 24);
  const uint64_t s1 = (uint64_t)w[4] + ((uint64_t)w[5] << 8) + ((uint64_t)w[6] << 16) +
                      ((uint64_t)w[7] << 24);
  uint64_t l = s0 + (s1 << 32);
  uint32_t h = (uint32_t)(s1 >> 32) + (l < s0);
  l += add;
  h += l < add;
  const uint64_t b = first ? 0x8080808080000000ull : 0x8080808080808080ull;
  low = l - b;
  high = h - (l < b);
}

// Hankel core matrices 0 .. nb - 1 of the blocks ending with eb: row r of
// matrix j = recoded y digits 128 eb + 127 - 8 j - r - w, w < 8, i.e. the
// eight digits starting r places down the digits of the limbs 16 eb + 15 - j
// and the one below.
// A thread issues the loads of two matrices before it recodes either.
template <int THREADS>
__device__ __forceinline__ void one_hankel(uint8_t *hk, const uint64_t *__restrict__ y, int ny, int eb, int nb) {
  for (int j0 = threadIdx.x; j0 < nb; j0 += 2 * THREADS) {
    uint64_t v[2][3];
#pragma unroll
    for (int u = 0; u < 2; u++) {
      const int U = 16 * eb + 15 - (j0 + u * THREADS);
#pragma unroll
      for (int i = 0; i < 3; i++) v[u][i] = U >= i && U - i < ny ? y[U - i] : 0ull;
    }
#pragma unroll
    for (int u = 0; u < 2; u++) {
      const int j = j0 + u * THREADS;
      if (j >= nb) break;
      hankel_rows(hk + (uint32_t)j * ONE_CM, v[u]);
    }
  }
}

// The MMA and its commit by lane 0 of a warp that runs them converged, all
// lanes with the same operands: in straight-line warp-uniform code the
// descriptors are computed in and read from uniform registers, where a lone
// thread's code moves six registers per MMA over (an issue floor of ~46
// cycles an MMA, and ~64 cycles more per Toeplitz block).
__device__ __forceinline__ void mma_f16_warp(uint32_t d_tmem, uint64_t a, uint64_t b,
                                             uint32_t idesc, uint32_t accumulate,
                                             uint32_t leader) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(leader));
}
__device__ __forceinline__ void mma_commit_warp(uint32_t mbar, uint32_t leader) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}\n" ::
          "r"(mbar),
      "r"(leader)
      : "memory");
}

// One warp: the MMAs of the blocks e_lo .. e_hi into the columns
// [c0, c0 + W) at TMEM column dtm, then a commit to mbar.  The first block's
// columns are overwritten, those above it up to shi cleared by a zero A
// operand (ACC = 2: all W columns of both accumulators, NT apart).  A block has only two MMAs of some 70 cycles each, so the loop
// keeps a block's bookkeeping to a few independent integer operations
// (descriptor start addresses and the column count are low-word fields) and
// is unrolled so that they run ahead of the MMAs (otherwise ~105 cycles per
// MMA whatever its width).
template <int NT, int ACC>
__device__ __forceinline__ void one_issue(uint32_t dtm, uint32_t ha, uint32_t xs_a, uint32_t z_a,
                                          uint32_t lbo_b, int c0, int W, int e_lo, int e_hi,
                                          int mx, int shi, uint32_t mbar) {
  tc_fence_after();
  const uint32_t leader = lane_id() == 0;
  const uint64_t da0 = sdesc(ha, ONE_CM, ONE_CM), db0 = sdesc(xs_a, lbo_b, 128);
  const uint32_t a_hi = (uint32_t)(da0 >> 32), b_hi = (uint32_t)(db0 >> 32);
  const uint32_t step_b = (2u * lbo_b) >> 4;
  auto desc = [](uint32_t hi, uint32_t lo) { return (uint64_t)hi << 32 | lo; };
  if (ACC == 2) {  // every column of both accumulators
#pragma unroll
    for (int a = 0; a < 2; a++)
      mma_f16_warp(dtm + a * NT, sdesc(z_a, 128, 128), db0,
                   IDESC_M128 | ((uint32_t)(W >> 3) << 17), 0, leader);
  } else {
    const int hi =
        ((c0 + W < ONE_S * e_lo + mx ? c0 + W : ONE_S * e_lo + mx) - c0 + 15) & ~15;
    if (hi < shi)
      mma_f16_warp(dtm + (uint32_t)hi, sdesc(z_a, 128, 128), db0,
              IDESC_M128 | ((uint32_t)((shi - hi) >> 3) << 17), 0, leader);
  }
  uint32_t a_lo = (uint32_t)da0 + (uint32_t)(e_hi - e_lo) * ONE_CM;  // 16 matrices per block
  const uint32_t b0 = (uint32_t)db0 + 16;
  int sh = ONE_S * e_lo - c0;  // column of the block's x block 0
  uint32_t acc = ACC == 2;
#pragma unroll 4
  for (int e = e_lo; e <= e_hi; e++) {
    const int ca = sh > 0 ? sh >> 4 : 0, end = sh + mx < W ? sh + mx : W;
    const uint32_t id = IDESC_M128 | ((uint32_t)(((end + 15) >> 4) - ca) << 18);
    const uint32_t b_lo = b0 + (uint32_t)(16 * ca - sh);
    const uint32_t d = dtm + 16u * (uint32_t)ca + (ACC == 2 && (e & 1) ? NT : 0);
    mma_f16_warp(d, desc(a_hi, a_lo), desc(b_hi, b_lo), id, acc, leader);
    mma_f16_warp(d, desc(a_hi, a_lo + ((2 * ONE_CM) >> 4)), desc(b_hi, b_lo + step_b), id, 1, leader);
    acc = 1;
    sh += ONE_S;
    a_lo -= ONE_CM;
  }
  static_assert(ONE_KB == 32, "two MMAs per block");
  mma_commit_warp(mbar, leader);
}

struct OneShared {
  uint64_t bar;        // mbarrier: the tile's MMAs completed
  uint32_t tmem_slot;
  uint32_t hi[32];     // per warp and run: high word of its last limb
  uint32_t g[32], p[32];
};

struct OneCtx {
  uint8_t *sm;
  uint32_t sbase, tmem, phase;
  OneShared *sh;
  long long wlim;
  bool pending, aborted;
};

// All threads of the CTA: the mbarrier and NT TMEM columns.
template <int NT>
__device__ void one_init(OneCtx &c, uint8_t *sm, OneShared *sh) {
  c.sm = sm;
  c.sbase = smem_u32(sm);
  c.sh = sh;
  c.phase = 0;
  c.wlim = wait_limit_here();
  c.pending = c.aborted = false;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&sh->bar), 1);
    fence_mbar_init();
  }
  if (threadIdx.x < 32) {
    tmem_alloc(smem_u32(&sh->tmem_slot), NT);
    tmem_relinquish();
  }
  for (int i = threadIdx.x; i < 32; i += blockDim.x) sh->g[i] = 0, sh->p[i] = 1;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  c.tmem = sh->tmem_slot;
}

// All threads: after an abort waits (bounded) for the MMAs in flight and
// records the timeout; then frees the TMEM.
template <int NT>
__device__ void one_release(OneCtx &c) {
  if (c.aborted) {
    if (c.pending) mbar_wait(smem_u32(&c.sh->bar), c.phase, WAIT_LIMIT);
    if (threadIdx.x == 0) atomicExch(&g_timeout, 1);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (threadIdx.x < 32) tmem_dealloc(c.tmem, NT);
}

// out[0 .. nout) = low nout limbs of x y (+ add, nout limbs, which may be
// out itself: each limb is read by the thread that later writes it) by the
// whole CTA (32 W threads);
// band mode (lo > 0) as tc_product's: tiles anchored S - 1 columns before
// limb lo's, limbs below L0 = R floor(lo / R) untouched, out[L0 ..) with
// 2^32 added at L0.  The shorter operand has at most ONE_MAX limbs (ONE_MAX2
// with two accumulators); c.sm
// holds one_layout<W>(nx, ny, blocks of the widest tile).  Returns false
// (and sets c.aborted) if a wait hit its limit.
template <int NT, int W, bool ADD = false, int ACC = 1>
__device__ __forceinline__ bool one_product(OneCtx &c, const uint64_t *__restrict__ x, int nx,
                                            const uint64_t *__restrict__ y, int ny, uint64_t *out, int nout,
                                            int lo, const uint64_t *add = nullptr) {
  constexpr int THREADS = 32 * W, RUN = 8 * W, NRUN = NT / RUN, S = ONE_S, R = ONE_R;
  constexpr int BUFS = one_bufs<W>();
  static_assert(NRUN * W <= 32, "one warp resolves the carries of a tile");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const OneLayout Ly = one_layout<W>(nx, ny, 0);
  uint8_t *hk = c.sm + Ly.hk;
  uint32_t *Cs = reinterpret_cast<uint32_t *>(hk), *Pv = reinterpret_cast<uint32_t *>(c.sm + Ly.prev);
  const uint32_t xs_a = c.sbase + Ly.xs, z_a = c.sbase + Ly.z, lbo_b = (uint32_t)Ly.ptot * 16u;
  const uint32_t mb = smem_u32(&c.sh->bar);
  const int q = warp & 3, part = warp >> 2;  // TMEM lane quadrant, 32 columns of a run

  for (int i = tid; i < ZB * 128 / 16; i += THREADS)
    reinterpret_cast<uint4 *>(c.sm + Ly.z)[i] = make_uint4(0u, 0u, 0u, 0u);
  for (int i = tid; i < (S - 1) * ONE_CS; i += THREADS) Pv[i] = 0u;
  fill_x<false, ONE_KB>(c.sm + Ly.xs, x, nx, Ly.ptot);
  const bool tx = (x[nx - 1] >> 63) != 0;

  const int cfirst = lo > 0 ? (lo / R - (S - 1) > 0 ? lo / R - (S - 1) : 0) : 0;
  const int L0 = lo > 0 ? R * (lo / R) : 0;
  uint32_t hprev = 0, cprev = 0;  // high word and carry into the tile
  uint64_t margin = lo > 0 ? 1ull << 32 : 0ull;
  int gen = 0;                    // generation of the columns before a run
  for (int c0 = cfirst; R * c0 < nout; c0 += NT) {
    int Wd = Ly.cmma + S - 1 - c0;
    if (Wd > NT) Wd = NT;
    const int need = (nout - R * c0 + R - 1) / R;
    if (Wd > need) Wd = need;
    Wd = (Wd + 15) & ~15;
    int e_lo, e_hi;
    one_blocks(Ly.mx, Ly.ey, c0, Wd, e_lo, e_hi);
    // columns of the tile the MMAs write
    const int slo = ACC == 2 ? 0 : ((c0 > S * e_lo ? c0 : S * e_lo) - c0) & ~15;
    const int shi = e_hi >= e_lo
                        ? ACC == 2 ? Wd
                        : ((c0 + Wd < S * e_hi + Ly.mx ? c0 + Wd : S * e_hi + Ly.mx) - c0 + 15) & ~15
                        : 0;
    if (shi > 0) {
      one_hankel<THREADS>(hk, y, ny, e_hi, 16 * (e_hi - e_lo + 1) + R - 1);
      tc_fence_before();
      fence_async_smem();
      __syncthreads();
      if (__shfl_sync(FULL, warp, 0) == 0) {
        one_issue<NT, ACC>(c.tmem, c.sbase + Ly.hk, xs_a, z_a, lbo_b, c0, Wd, e_lo, e_hi, Ly.mx, shi, mb);
        c.pending = tid == 0;
      }
      bool bad = false;
      if (mbar_wait_lim(mb, c.phase, c.wlim)) {
        c.phase ^= 1u;
        c.pending = false;
      } else {
        bad = true;
      }
      if (__syncthreads_or(bad)) { c.aborted = true; return false; }
      tc_fence_after();
    } else {
      __syncthreads();
    }

    // ---- column sums -> limbs, a run of RUN columns at a time
    const int j0 = R * c0, nl = R * Wd < nout - j0 ? R * Wd : nout - j0;
    const int skip = L0 > j0 ? L0 - j0 : 0;  // band: limbs below L0 are not kept
    uint64_t low[NRUN];
    uint32_t high[NRUN];
#pragma unroll
    for (int r = 0; r < NRUN; r++) {
      low[r] = 0;
      high[r] = 0;
      if (RUN * r < Wd) {
        uint32_t *cs = Cs + (BUFS == 2 ? (r & 1) * RUN * ONE_CS : 0);
        const int gnext = gen == 2 ? 0 : gen + 1;
        const int t = 127 - (32 * q + lane);
        if (BUFS == 1 && r > 0) __syncthreads();  // the run before is read
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const int col0 = RUN * r + 32 * part + 16 * h;
          uint32_t v[16];
          if (col0 >= slo && col0 < shi) {
            tmem_ld16(c.tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)col0, v);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; i++)
              v[i] = (uint32_t)__float2int_rn(__uint_as_float(v[i]));
            if constexpr (ACC == 2) {
              uint32_t o[16];
              tmem_ld16(c.tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(NT + col0), o);
              tmem_ld_wait();
#pragma unroll
              for (int i = 0; i < 16; i++) v[i] += (uint32_t)__float2int_rn(__uint_as_float(o[i]));
            }
          } else {
#pragma unroll
            for (int i = 0; i < 16; i++) v[i] = 0u;
          }
          uint32_t *o = cs + (32 * part + 16 * h) * ONE_CS + t;
#pragma unroll
          for (int i = 0; i < 16; i++) o[i * ONE_CS] = v[i];
          if (h == 1 && part == W / 4 - 1) {
            uint32_t *pv = Pv + gnext * (S - 1) * ONE_CS + t;
#pragma unroll
            for (int i = 0; i < S - 1; i++) pv[i * ONE_CS] = v[16 - (S - 1) + i];
          }
        }
        __syncthreads();
        const int col = tid / R, jj = tid % R, lt = R * RUN * r + tid;
        if (lt < nl && lt >= skip) {
          uint32_t w[8];
#pragma unroll
          for (int a = 0; a < S; a++) {  // row 8 jj + 32 a of column col - a
            const uint32_t *p = col >= a ? cs + (col - a) * ONE_CS
                                         : Pv + (gen * (S - 1) + col - a + S - 1) * ONE_CS;
            const uint4 u0 = *reinterpret_cast<const uint4 *>(p + 8 * jj + ONE_KB * a);
            const uint4 u1 = *reinterpret_cast<const uint4 *>(p + 8 * jj + ONE_KB * a + 4);
            const uint32_t s[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
            for (int k = 0; k < 8; k++) w[k] = a == 0 ? s[k] + 0x80000000u : w[k] + s[k];
          }
          const int j = j0 + lt;
          limb_of(w, tx && j >= nx && j - nx < ny ? y[j - nx] : 0ull, j == L0, low[r], high[r]);
          if constexpr (ADD) {
            const uint64_t a = add[j];
            low[r] += a;
            high[r] += low[r] < a;
          }
        }
        if (lane == 31) c.sh->hi[r * W + warp] = high[r];
        gen = gnext;
      }
    }
    tc_fence_before();
    __syncthreads();
    // ---- low words plus the high words one limb up: one carry scan
    WarpCarry wc[NRUN];
#pragma unroll
    for (int r = 0; r < NRUN; r++) {
      const int lt = R * RUN * r + tid;
      uint32_t below = __shfl_up_sync(FULL, high[r], 1);
      if (lane == 0) below = r * W + warp > 0 ? c.sh->hi[r * W + warp - 1] : hprev;
      uint32_t g = 0, p = 1;
      if (lt < nl && lt >= skip) {
        const uint64_t add = j0 + lt == L0 ? margin : (uint64_t)below;
        low[r] += add;
        g = low[r] < add;
        p = low[r] == ~0ull;
      }
      wc[r] = warp_gp(g, p);
      if (lane == 0) {
        c.sh->g[r * W + warp] = warp_carry_out(wc[r], 0);
        c.sh->p[r * W + warp] = warp_all_propagate(wc[r]);
      }
    }
    const uint32_t hnext = c.sh->hi[NRUN * W - 1];
    __syncthreads();
    const uint64_t cm = warp_carries(warp_gp(c.sh->g[lane], c.sh->p[lane]), cprev);
#pragma unroll
    for (int r = 0; r < NRUN; r++) {
      const int lt = R * RUN * r + tid;
      const uint64_t lc = warp_carries(wc[r], (uint32_t)(cm >> (r * W + warp)) & 1u);
      if (lt < nl && lt >= skip) out[j0 + lt] = low[r] + ((lc >> lane) & 1u);
    }
    hprev = hnext;
    cprev = (uint32_t)(cm >> 32);
  }
  __syncthreads();
  return true;
}

}  // namespace tcm
}  // namespace bigint
