// tcpipe.cuh -- tensor-core products as a pipeline of three kinds of warps.
//
// The digit convolution of tccore.cuh for products that need several drains
// (operands from about 600 limbs), one CTA per SM, its work split by role so
// that the tensor core is fed across groups, tiles and products:
//
//   builders (3 warps)  x into the B layout (two buffers where they fit, so
//                       the next product's x is written during this one) and
//                       the Hankel core matrices of HS Toeplitz blocks a
//                       stage, straight from registers (tcone.cuh), two or
//                       three stages ahead;
//   issuer (1 warp)     the MMAs of a stage once it is full, a group of
//                       GS stages into one of 512 / NT accumulators of NT
//                       columns;
//   drains (16 warps)   a finished accumulator into int32 column sums in
//                       registers (NT / 4 per thread), and after a tile's last
//                       group the column sums into limbs, while the issuer is
//                       already at work on the next tile or product: with NT
//                       = 256 it may run two groups (~9K cycles) ahead, a
//                       tile's limbs taking ~13K beside them; with NT = 128
//                       (products of at most 128 columns: low and banded
//                       ones) four groups, and half the limbs per thread.
//
// Every hand-over is an mbarrier: stage full / free, accumulator full / free,
// x full / free (the "free" ones of operands are tcgen05.commit arrivals).
// All roles walk the same sequence of products, tiles and groups, so stage
// and accumulator numbers and mbarrier parities follow from counters.
//
// In the form with all warps doing all of it in turn (tc_product) the chain
// wait - drain - Hankel build of each group was as long as the group's MMAs
// and the ~20K cycles between products were not covered: 122K cycles for a
// 2048-limb product whose MMAs take 74K.
//
// Bound: the MMAs, whose operand reads take 94 % of the shared-memory
// bandwidth at 144 columns, at the clock the chip's power leaves (2048-limb
// products 1650 TFLOP/s, 94K cycles a product, 84K of them MMAs); for products
// of a single narrow tile the drain warps' serial work (515 limbs by the top
// 530, now a one-drain product: tensor pipe 20 % busy, issue slots 50 %).  16384 products of 1701 x
// 1103 limbs 3860 -> 2815 us, 8192 of 8192 limbs by Karatsuba 30.9 -> 25.4 ms.
//
// KB digits per x block: 128 (S = 1 row per coefficient), 64 (S = 2, MMAs
// twice as wide: operands below 2048 limbs) or 32 (S = 4, again twice: low and
// banded products of a few hundred columns).  KB * HS * GS = 1024 digit
// products per accumulated sum: exact (tccore.cuh).  x goes without its carry
// digit; where its top bit is set, limb j of the result takes limb j - nx of
// y more as its coefficients are summed.  Limbs, bias and the single carry
// scan are those of tcone.cuh, here for 64 columns at a time.
#pragma once
#include "tcone.cuh"

namespace bigint {
namespace tcm {

constexpr int PIPE_HS = 8, PIPE_BUILD = 3, PIPE_DRAIN = 512;
constexpr int PIPE_THREADS = PIPE_DRAIN + 32 + 32 * PIPE_BUILD;  // 20 warps: 96 registers
constexpr int PIPE_EX = 264;    // limbs per row of the S > 1 exchange (16 banks from row to row)
constexpr int PIPE_STAGES = 3;  // at most

template <int KB>
__host__ __device__ constexpr int pipe_matrices() { return 16 * PIPE_HS + KB / 8 - 1; }

// Shared memory of a launch: stages and x buffers as many as fit.
struct PipeLayout {
  uint32_t xs, xbytes, z, hk, hbytes, ex, total;
  int xbufs, stages;
};

// Rows of the exchange (limbs of a column times the row parts it collects).
template <int KB>
__host__ __device__ constexpr int pipe_ex_rows() { return KB == 128 ? 0 : (KB == 64 ? 8 : 12); }

template <int KB>
__host__ __device__ inline int pipe_ptot(int nx) {
  return ((8 * nx + KB - 1) / KB + 32) | 1;
}

// Layout for x of at most nx limbs within cap bytes (total = 0: does not fit).
template <int KB>
__host__ inline PipeLayout pipe_layout(int nx, uint32_t cap) {
  PipeLayout L{};
  constexpr int R = KB / 8;
  L.xbytes = ((uint32_t)pipe_ptot<KB>(nx) * 16u * R + 127) / 128 * 128;
  L.hbytes = (uint32_t)pipe_matrices<KB>() * ONE_CM;
  const uint32_t fixed = ZB * 128 + pipe_ex_rows<KB>() * PIPE_EX * 12;
  for (L.xbufs = 2; L.xbufs >= 1; L.xbufs--)
    for (L.stages = PIPE_STAGES; L.stages >= 2; L.stages--) {
      const uint32_t t = fixed + L.xbufs * L.xbytes + L.stages * L.hbytes;
      if (t > cap) continue;
      L.xs = 0;
      L.z = L.xbufs * L.xbytes;
      L.hk = L.z + ZB * 128;
      L.ex = L.hk + L.stages * L.hbytes;
      L.total = t;
      return L;
    }
  return L;
}

struct PipeShared {
  uint64_t hfull[PIPE_STAGES], hfree[PIPE_STAGES], afull[4], afree[4], xfull[2], xfree[2], done;
  uint32_t tmem_slot;
  int abort;
  uint32_t hx[4][256];    // high words of each warp's top limb of a column
  ulonglong2 gp[4][4];    // its columns' (generate, propagate)
};

// One product: x (the operand stored whole), y, the low nout limbs to out,
// band start lo (as tc_product's); add: nout limbs added to it (may be out
// itself), or null.
struct PipeTask {
  const uint64_t *x, *y;
  uint64_t *out;
  int nx, ny, nout, lo;
  const uint64_t *add;
};

// Tiles of a product and their Toeplitz blocks, as every role walks them:
// f(c0, W, e_lo, e_hi), e_hi < e_lo where no MMA writes the tile; f returns
// false to stop.
#pragma nv_exec_check_disable
template <int KB, int NT, class F>
__host__ __device__ __forceinline__ bool pipe_tiles(int nx, int ny, int nout, int lo, F f) {
  constexpr int S = 128 / KB, R = KB / 8;
  const int mx = (8 * nx + KB - 1) / KB, ey = (8 * ny + KB - 1) / 128;
  const int cols = mx + S * ey + S - 1;
  for (int c0 = lo > 0 ? (lo / R - (S - 1) > 0 ? lo / R - (S - 1) : 0) : 0; R * c0 < nout;
       c0 += NT) {
    int W = cols - c0 < NT ? cols - c0 : NT;
    const int need = (nout - R * c0 + R - 1) / R;
    if (W > need) W = need;
    W = (W + 15) & ~15;
    const int e_lo = c0 - mx + 1 > 0 ? (c0 - mx + S) / S : 0;
    const int e_hi = (c0 + W - 1) / S < ey ? (c0 + W - 1) / S : ey;
    if (!f(c0, W, e_lo, e_hi)) return false;
  }
  return true;
}

// Waits for the phase with this parity: false if the CTA gave up or the
// launch's limit passed (which makes the CTA give up), see mbar_wait_lim.
__device__ __forceinline__ bool pipe_wait(PipeShared *sh, uint64_t *bar, uint32_t parity,
                                          long long lim) {
  const uint32_t mb = smem_u32(bar);
  if (lim >= 0 && mbar_test_wait(mb, parity)) return true;
  volatile int *ab = &sh->abort;
  const long long t0 = clock64(), full = lim >= 0 ? lim : WAIT_LIMIT;
  bool ok = true;
  while (!(full < WAIT_LIMIT ? mbar_test_wait(mb, parity) : mbar_try_wait(mb, parity)))
    if (*ab != 0 || clock64() - t0 > full) { ok = false; break; }
  if (ok && lim >= 0) return true;
  if (ok) {  // the injected timeout of g_never_set
    const long long t1 = clock64();
    while (*(volatile int *)&g_never_set == 0)
      if (clock64() - t1 > -lim) { ok = false; break; }
    if (ok) return true;
  }
  *ab = 1;
  return false;
}

// The same by a converged warp: all lanes get the same answer.
__device__ __forceinline__ bool pipe_wait_warp(PipeShared *sh, uint64_t *bar, uint32_t parity,
                                               long long lim) {
  return __all_sync(FULL, pipe_wait(sh, bar, parity, lim));
}

// ---- builders -----------------------------------------------------------------
// Their waits are decided by whole warps (pipe_wait_warp): a lane that gave up
// alone would leave the others of its warp at the next __syncwarp for ever.
// x into the B layout (fill_x without the carry digit), by the builders.
template <int KB>
__device__ __forceinline__ void pipe_fill(uint8_t *xs, const uint64_t *__restrict__ x, int nx, int t) {
  constexpr int U = 4, R = KB / 8, LR = KB == 128 ? 4 : (KB == 64 ? 3 : 2), STEP = 32 * PIPE_BUILD;
  const int ptot = pipe_ptot<KB>(nx), total = R * ptot;
  for (int i0 = t; i0 < total; i0 += U * STEP) {
    uint64_t v[U], below[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int L = i0 + u * STEP - 16 * R;
      v[u] = L >= 0 && L < nx ? x[L] : 0ull;
      below[u] = L >= 1 && L < nx ? x[L - 1] : 0ull;
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int i = i0 + u * STEP;
      if (i < total) {
        const int pp = i >> LR, h = i & (R - 1);
        const Digits16 d = recode16(v[u], below[u]);
        const uint32_t el = (uint32_t)d.ev, eh = (uint32_t)(d.ev >> 32);
        const uint32_t ol = (uint32_t)d.od, oh = (uint32_t)(d.od >> 32);
        *reinterpret_cast<uint4 *>(xs + (size_t)(pp + h * ptot) * 16) = make_uint4(
            unbias_h2(__byte_perm(el, ol, 0x5410)), unbias_h2(__byte_perm(el, ol, 0x7632)),
            unbias_h2(__byte_perm(eh, oh, 0x5410)), unbias_h2(__byte_perm(eh, oh, 0x7632)));
      }
    }
  }
}

template <int KB, int NT, class Next>
__device__ __forceinline__ void pipe_builder(const PipeLayout &L, PipeShared *sh, uint8_t *sm,
                                             long long lim, int t, Next next) {
  constexpr int HS = PIPE_HS, NB = pipe_matrices<KB>(), STEP = 32 * PIPE_BUILD;
  static_assert(NB <= 2 * STEP, "two matrices per builder thread");
  const int lane = t & 31;
  auto post = [&](uint64_t *bar) {
    fence_async_smem();
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(bar));
  };
  uint32_t st = 0, sph = 0;  // stage, and bit s: stage s has been used before / parity
  uint32_t used = 0;
  uint32_t items = 0;
  PipeTask T;
  for (int64_t k = 0; next(k, T); k++) {
    const uint32_t xb = L.xbufs == 2 ? items & 1u : 0u, n = L.xbufs == 2 ? items >> 1 : items;
    if (n >= 1 && !pipe_wait_warp(sh, &sh->xfree[xb], (n - 1) & 1u, lim)) return;
    pipe_fill<KB>(sm + L.xs + xb * L.xbytes, T.x, T.nx, t);
    post(&sh->xfull[xb]);
    items++;
    const bool ok = pipe_tiles<KB, NT>(T.nx, T.ny, T.nout, T.lo, [&](int, int, int e_lo, int e_hi) {
      // AHEAD: the next stage's limbs are loaded while this one's rows are
      // written (32-digit blocks, whose stages are short: 16384 low products of
      // 1024 limbs 2 % faster; with the longer ones it only cost registers)
      constexpr bool AHEAD = KB == 32;
      uint64_t ahead[2][3];
      auto load = [&](int ea) {
        const int eb = ea + HS - 1 < e_hi ? ea + HS - 1 : e_hi;
        const int nb = 16 * (eb - ea + 1) + KB / 8 - 1;
#pragma unroll
        for (int u = 0; u < 2; u++) {
          const int Lm = 16 * eb + 15 - (t + u * STEP);
#pragma unroll
          for (int i = 0; i < 3; i++)
            ahead[u][i] = t + u * STEP < nb && Lm >= i && Lm - i < T.ny ? T.y[Lm - i] : 0ull;
        }
      };
      if (AHEAD && e_lo <= e_hi) load(e_lo);
      for (int ea = e_lo; ea <= e_hi; ea += HS) {
        const int eb = ea + HS - 1 < e_hi ? ea + HS - 1 : e_hi;
        const int nb = 16 * (eb - ea + 1) + KB / 8 - 1;
        if (!AHEAD) load(ea);
        uint64_t v[2][3];
#pragma unroll
        for (int u = 0; u < 2; u++)
#pragma unroll
          for (int i = 0; i < 3; i++) v[u][i] = ahead[u][i];
        if (AHEAD && ea + HS <= e_hi) load(ea + HS);
        if ((used >> st & 1u) && !pipe_wait_warp(sh, &sh->hfree[st], sph >> st & 1u, lim))
          return false;
        if (used >> st & 1u) sph ^= 1u << st;
        used |= 1u << st;
        uint8_t *hk = sm + L.hk + st * L.hbytes;
#pragma unroll
        for (int u = 0; u < 2; u++)
          if (t + u * STEP < nb) hankel_rows(hk + (uint32_t)(t + u * STEP) * ONE_CM, v[u]);
        post(&sh->hfull[st]);
        st = (int)st + 1 == L.stages ? 0 : st + 1;
      }
      return true;
    });
    if (!ok) return;
  }
}

// ---- issuer ---------------------------------------------------------------------
template <int KB, int NT, class Next>
__device__ __forceinline__ void pipe_issuer(const PipeLayout &L, PipeShared *sh, uint32_t sbase,
                                            uint32_t tmem, long long lim, Next next) {
  constexpr int HS = PIPE_HS, S = 128 / KB, GS = 1024 / (KB * HS), NACC = 512 / NT;
  uint32_t st = 0, sph = 0, items = 0, grp = 0;
  const uint32_t leader = lane_id() == 0;
  auto desc = [](uint32_t hi, uint32_t lo) { return (uint64_t)hi << 32 | lo; };
  const uint64_t zd = sdesc(sbase + L.z, 128, 128);
  const uint32_t a_hi = (uint32_t)(sdesc(0, ONE_CM, ONE_CM) >> 32);
  const uint32_t a_lo_fixed = (uint32_t)sdesc(0, ONE_CM, ONE_CM);
  PipeTask T;
  for (int64_t k = 0; next(k, T); k++) {
    const uint32_t xb = L.xbufs == 2 ? items & 1u : 0u, n = L.xbufs == 2 ? items >> 1 : items;
    if (!pipe_wait_warp(sh, &sh->xfull[xb], n & 1u, lim)) return;
    items++;
    const int mx = (8 * T.nx + KB - 1) / KB;
    const uint32_t lbo = (uint32_t)pipe_ptot<KB>(T.nx) * 16u;
    const uint64_t xd = sdesc(sbase + L.xs + xb * L.xbytes, lbo, 128);
    const uint32_t b_hi = (uint32_t)(xd >> 32), step_b = (2u * lbo) >> 4;
    const bool ok = pipe_tiles<KB, NT>(T.nx, T.ny, T.nout, T.lo, [&](int c0, int W, int e_lo,
                                                                int e_hi) {
      for (int eg = e_lo; eg <= e_hi; eg += HS * GS) {
        const int ee = eg + HS * GS - 1 < e_hi ? eg + HS * GS - 1 : e_hi;
        const uint32_t a = grp % NACC, gn = grp / NACC;
        if (gn >= 1 && !pipe_wait_warp(sh, &sh->afree[a], (gn - 1) & 1u, lim)) return false;
        const uint32_t dt = tmem + a * NT;
        const int shi = ((c0 + W < S * ee + mx ? c0 + W : S * ee + mx) - c0 + 15) & ~15;
        uint32_t acc = 0;
        for (int ea = eg; ea <= ee; ea += HS) {
          const int eb = ea + HS - 1 < ee ? ea + HS - 1 : ee;
          if (!pipe_wait_warp(sh, &sh->hfull[st], sph >> st & 1u, lim)) return false;
          sph ^= 1u << st;
          tc_fence_after();
          if (acc == 0) {  // columns above the first block's
            const int end = S * ea + mx - c0 < W ? S * ea + mx - c0 : W;
            const int hi = (end + 15) & ~15;
            if (hi < shi)
              mma_f16_warp(dt + (uint32_t)hi, zd, xd,
                      IDESC_M128 | ((uint32_t)((shi - hi) >> 3) << 17), 0, leader);
          }
          uint32_t a_lo = a_lo_fixed + ((sbase + L.hk + st * L.hbytes) >> 4) +
                          (uint32_t)(eb - ea) * ONE_CM;  // 16 matrices per block
          int sf = S * ea - c0;
#pragma unroll 2
          for (int e = ea; e <= eb; e++) {
            const int ca = sf > 0 ? sf >> 4 : 0, end = sf + mx < W ? sf + mx : W;
            const uint32_t id = IDESC_M128 | ((uint32_t)(((end + 15) >> 4) - ca) << 18);
            uint32_t b_lo = (uint32_t)xd + 16 + (uint32_t)(16 * ca - sf);
            const uint32_t d = dt + 16u * (uint32_t)ca;
#pragma unroll
            for (int s = 0; s < KB / 16; s++) {
              mma_f16_warp(d, desc(a_hi, a_lo + s * ((2 * ONE_CM) >> 4)), desc(b_hi, b_lo), id,
                      s == 0 ? acc : 1u, leader);
              b_lo += step_b;
            }
            acc = 1;
            sf += S;
            a_lo -= ONE_CM;
          }
          mma_commit_warp(smem_u32(&sh->hfree[st]), leader);
          st = (int)st + 1 == L.stages ? 0 : st + 1;
        }
        mma_commit_warp(smem_u32(&sh->afull[a]), leader);
        grp++;
      }
      return true;
    });
    if (!ok) return;
    mma_commit_warp(smem_u32(&sh->xfree[xb]), leader);
  }
}

// ---- drains ---------------------------------------------------------------------
__device__ __forceinline__ void bar_drain() {
  asm volatile("bar.sync 2, %0;" ::"n"(PIPE_DRAIN) : "memory");
}

// Column sums of a warp's 32 rows and 64 columns (row of lane i: t = 127 - 32
// q - i) to limbs, in registers: the eight coefficients of a limb are in
// eight lanes, so three exchanges (lanes 1, 2, 4 apart) halve the columns a
// lane holds and join the coefficients of those it keeps: afterwards lane i
// has for the columns 8 m + (i & 7), m < 8, the limb of its eight rows, as a
// signed value lo + hi 2^64.  80 shuffles, no barrier: through shared memory
// the same took 16K cycles beside the MMAs (whose operand reads leave little
// of its bandwidth), more than the two groups they may run ahead.
template <int CW>
__device__ __forceinline__ void pipe_limbs(int (&acc)[CW], uint64_t (&lo)[CW / 8],
                                           int (&hi)[CW / 8]) {
  const uint32_t lane = lane_id();
  const bool b0 = lane & 1u, b1 = lane & 2u, b2 = lane & 4u;
  // coefficient 7 - (lane & 7) of a limb; its weight within its half of the
  // limb, and that of the neighbour's coefficient
  const int wo = 1 << (8 * (3 - (lane & 3u))), wg = 1 << (8 * (3 - ((lane ^ 1u) & 3u)));
  int64_t v[CW / 4];
#pragma unroll
  for (int m = 0; m < CW / 4; m++) {
    int64_t u[2];
#pragma unroll
    for (int i = 0; i < 2; i++) {
      const int c0 = acc[4 * m + 2 * i], c1 = acc[4 * m + 2 * i + 1];
      const int got = __shfl_xor_sync(FULL, b0 ? c0 : c1, 1);
      u[i] = (int64_t)(b0 ? c1 : c0) * wo + (int64_t)got * wg;
    }
    v[m] = (b1 ? u[1] : u[0]) + __shfl_xor_sync(FULL, b1 ? u[0] : u[1], 2);
  }
#pragma unroll
  for (int m = 0; m < CW / 8; m++) {
    const int64_t own = b2 ? v[2 * m + 1] : v[2 * m];
    const int64_t got = __shfl_xor_sync(FULL, b2 ? v[2 * m] : v[2 * m + 1], 4);
    const int64_t l = b2 ? own : got, h = b2 ? got : own;
    lo[m] = (uint64_t)l + ((uint64_t)h << 32);
    hi[m] = (int)(h >> 32) + (int)(l >> 63) + (lo[m] < (uint64_t)l);
  }
}

// Byte b of four or eight words, as one.
template <int N>
__device__ __forceinline__ uint64_t pipe_bytes(const uint32_t (&w)[N], int b) {
  const uint32_t s = (uint32_t)b | (uint32_t)(4 + b) << 4;  // byte b of both
  const uint32_t a0 = __byte_perm(w[0], w[1], s), a1 = __byte_perm(w[2], w[3], s);
  const uint64_t low = __byte_perm(a0, a1, 0x5410);
  if constexpr (N == 4) {
    return low;
  } else {
    const uint32_t a2 = __byte_perm(w[4], w[5], s), a3 = __byte_perm(w[6], w[7], s);
    return (uint64_t)__byte_perm(a2, a3, 0x5410) << 32 | low;
  }
}

// Adds a warp's 32 lanes and CW columns of an accumulator (the group's
// columns [lo, hi)) to its column sums.
template <int CW>
__device__ __forceinline__ void pipe_drain_acc(uint32_t taddr, int cq, int lo, int hi,
                                               int (&acc)[CW]) {
#pragma unroll
  for (int k = 0; k < CW / 16; k++) {
    const int col = CW * cq + 16 * k;
    if (col >= lo && col < hi) {
      uint32_t r[16];
      tmem_ld16(taddr + (uint32_t)col, r);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 16; i++) acc[16 * k + i] += __float2int_rn(__uint_as_float(r[i]));
    }
  }
}

template <int KB, int NT, class Next, class Done>
__device__ __forceinline__ bool pipe_drain(const PipeLayout &L, PipeShared *sh, uint8_t *sm,
                                           uint32_t tmem, long long lim, Next next, Done done) {
  constexpr int HS = PIPE_HS, S = 128 / KB, R = KB / 8, GS = 1024 / (KB * HS);
  constexpr int NACC = 512 / NT, CW = NT / 4, CM = CW / 8;  // columns and limbs per lane
  constexpr int QTOP = S == 1 ? 0 : (S == 2 ? 2 : 3);  // lane quadrants 3 .. QTOP hold the limbs
  // added to a limb's signed high word to make it unsigned, and taken off the
  // next limb: |V_j| < 2^31 sum_k 2^(8 k), so the high word is at least -C
  constexpr uint32_t C = 0x808080u;
  static_assert(S <= 4, "one, two or four rows per coefficient");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q = warp & 3, cq = warp >> 2;  // TMEM lane quadrant, CW-column slice
  const uint32_t t_lane = tmem + ((uint32_t)(32 * q) << 16);
  const bool holds = q >= QTOP;
  const int jj = 4 * (3 - q) + 3 - (lane >> 3);  // limb of this lane within a column (holds)
  // S > 1: rows 128 / S and up are parts of limbs of later columns, exchanged
  // at the column they belong to: quadrant q's go `ahead` columns on, to the
  // holder with the same limbs, in exchange row xrow (limb, and part for S = 4)
  uint64_t *Xl = reinterpret_cast<uint64_t *>(sm + L.ex);
  int *Xh = reinterpret_cast<int *>(sm + L.ex + 8 * pipe_ex_rows<KB>() * PIPE_EX);
  const int ahead = S == 2 ? 1 : 3 - q;
  const int xrow = 3 - (lane >> 3) + 4 * (S == 2 ? 3 - (q | 2) : 2 - q);
  uint32_t grp = 0;
  int gen = 0;
  PipeTask T;
  for (int64_t k = 0; next(k, T); k++) {
    const int mx = (8 * T.nx + KB - 1) / KB;
    const int L0 = T.lo > 0 ? R * (T.lo / R) : 0;
    const bool tx = (T.x[T.nx - 1] >> 63) != 0;
    uint32_t hprev = 0, cprev = 0;  // high word and carry into the tile
    const uint64_t margin = T.lo > 0 ? 1ull << 32 : 0ull;
    if (S > 1 && tid < 4 * pipe_ex_rows<KB>()) {  // nothing before the first column
      const int at = (tid >> 2) * PIPE_EX + 256 + 4 * gen + (tid & 3);
      Xl[at] = 0ull;
      Xh[at] = 0;
    }
    const bool ok = pipe_tiles<KB, NT>(T.nx, T.ny, T.nout, T.lo, [&](int c0, int W, int e_lo,
                                                                int e_hi) {
      int acc[CW];
#pragma unroll
      for (int i = 0; i < CW; i++) acc[i] = 0;
      for (int eg = e_lo; eg <= e_hi; eg += HS * GS) {
        const int ee = eg + HS * GS - 1 < e_hi ? eg + HS * GS - 1 : e_hi;
        const uint32_t a = grp % NACC;
        const bool bad = !pipe_wait(sh, &sh->afull[a], (grp / NACC) & 1u, lim);
        if (bar_or_drain<PIPE_DRAIN>(bad)) return false;  // all drain threads agree
        grp++;
        tc_fence_after();
        const int slo = (S * eg > c0 ? S * eg - c0 : 0) & ~15;
        const int shi = ((c0 + W < S * ee + mx ? c0 + W : S * ee + mx) - c0 + 15) & ~15;
        pipe_drain_acc<CW>(t_lane + a * NT, cq, slo, shi, acc);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sh->afree[a]));
      }
      // ---- column sums -> limbs
      const int j0 = R * c0, nl = R * W < T.nout - j0 ? R * W : T.nout - j0;
      const int skip = L0 > j0 ? L0 - j0 : 0;  // band: limbs below L0 are not kept
      const int cb = CW * cq + (lane & 7);     // this lane's columns: cb + 8 m
      uint64_t low[CM];
      int high[CM];
      pipe_limbs<CW>(acc, low, high);
      if (S > 1) {
        // parts beyond the tile's last column wait for the next tile
        if (!holds) {
#pragma unroll
          for (int m = 0; m < CM; m++) {
            const int c = cb + 8 * m + ahead;
            const int at = xrow * PIPE_EX + (c < NT ? c : 256 + 4 * (gen ^ 1) + c - NT);
            Xl[at] = low[m];
            Xh[at] = high[m];
          }
        }
        bar_drain();
        if (holds) {
#pragma unroll
          for (int m = 0; m < CM; m++) {
#pragma unroll
            for (int a = 1; a < S; a++) {
              const int c = cb + 8 * m;
              const int row = S == 2 ? xrow : 3 - (lane >> 3) + 4 * (a - 1);
              const int at = row * PIPE_EX + (c >= a ? c : 256 + 4 * gen + c);
              const uint64_t l = Xl[at];
              low[m] += l;
              high[m] += Xh[at] + (int)(low[m] < l);
            }
          }
        }
        gen ^= 1;
      }
      // every limb of a whole tile is kept
      const bool whole = skip == 0 && nl == R * NT;
      if (holds) {
        if (tx) {
#pragma unroll
          for (int m = 0; m < CM; m++) {
            const int j = j0 + R * (cb + 8 * m) + jj - T.nx;
            const uint64_t add = j >= 0 && j < T.ny ? T.y[j] : 0ull;
            low[m] += add;
            high[m] += low[m] < add;
          }
        }
        if (T.add != nullptr) {
#pragma unroll
          for (int m = 0; m < CM; m++) {
            const int lt = R * (cb + 8 * m) + jj;
            const uint64_t a = lt < nl ? T.add[j0 + lt] : 0ull;
            low[m] += a;
            high[m] += low[m] < a;
          }
        }
#pragma unroll
        for (int m = 0; m < CM; m++) {
          const uint32_t off = j0 + R * (cb + 8 * m) + jj == L0 ? 0u : C;
          high[m] += (int)C - (int)(low[m] < off);
          low[m] -= off;
          if (lane < 8) sh->hx[q][cb + 8 * m] = (uint32_t)high[m];
        }
      }
      bar_drain();
      // ---- low words plus the high words one limb up.  Bit c of the 64-bit
      // words below stands for column CW cq + c (bits past CW pass carries
      // on); a warp's lanes 24-31 hold the
      // lowest of its four limbs of a column, quadrant 3 the lowest four.
      uint64_t Gs[4], Ps[4];  // of the limbs in lanes 8 i .. 8 i + 7
      if (holds) {
        uint32_t G[CM], P[CM];
#pragma unroll
        for (int m = 0; m < CM; m++) {
          const int c = cb + 8 * m, lt = R * c + jj;
          uint32_t below = __shfl_down_sync(FULL, (uint32_t)high[m], 8);
          if (lane >= 24)
            below = q < 3 ? sh->hx[q + 1][c] : (c > 0 ? sh->hx[QTOP][c - 1] : hprev);
          const uint64_t add = j0 + lt == L0 ? margin : (uint64_t)below;
          low[m] += add;
          const bool in = whole || (lt < nl && lt >= skip);
          G[m] = __ballot_sync(FULL, in && low[m] < add);
          P[m] = __ballot_sync(FULL, !in || low[m] == ~0ull);
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
          Gs[i] = pipe_bytes(G, i);
          Ps[i] = pipe_bytes(P, i);
        }
        const uint64_t g =
            Gs[0] | (Ps[0] & (Gs[1] | (Ps[1] & (Gs[2] | (Ps[2] & Gs[3])))));
        if (lane == 0)
          sh->gp[cq][q] = make_ulonglong2(
              g, (Ps[0] & Ps[1] & Ps[2] & Ps[3]) | (CW < 64 ? ~0ull << (CW & 63) : 0ull));
      }
      const uint32_t hnext = sh->hx[QTOP][NT - 1];
      bar_drain();
      uint64_t cin = 0;  // carries into this warp's limbs of its columns
      uint32_t c = cprev;
#pragma unroll
      for (int w = 0; w < 4; w++) {
        ulonglong2 x[4];
        uint64_t g = 0, p = ~0ull;
#pragma unroll
        for (int i = 3; i >= QTOP; i--) {
          x[i] = sh->gp[w][i];
          g = x[i].x | (x[i].y & g);
          p &= x[i].y;
        }
        const uint64_t X = g | p, s1 = X + g, s2 = s1 + c;
        const uint64_t into = s2 ^ X ^ g;
        c = (s1 < X) | (s2 < s1);
        if (w == cq) {
          cin = into;
#pragma unroll
          for (int i = 3; i > QTOP; i--)
            if (q < i) cin = x[i].x | (x[i].y & cin);
        }
      }
      cprev = c;
      hprev = hnext;
      if (holds) {
        if (lane < 24) cin = Gs[3] | (Ps[3] & cin);
        if (lane < 16) cin = Gs[2] | (Ps[2] & cin);
        if (lane < 8) cin = Gs[1] | (Ps[1] & cin);
        cin >>= lane & 7;
        uint64_t *o = T.out + j0 + R * cb + jj;
#pragma unroll
        for (int m = 0; m < CM; m++) {
          const int lt = R * (cb + 8 * m) + jj;
          if (whole || (lt < nl && lt >= skip)) o[8 * R * m] = low[m] + ((cin >> (8 * m)) & 1u);
        }
      }
      return true;
    });
    if (!ok) return false;
    done(k);
  }
  return true;
}

// ---- the CTA ----------------------------------------------------------------------
// Runs the products 0, 1, ... on PIPE_THREADS threads with 512 TMEM columns:
// next_b(k, T), next_i and next_d give product k (false: no more, the same
// answer for all lanes of a warp) to the builders, the issuing warp and the drain
// threads, which must all see the same sequence; done(k) is called by the drain threads after product k.
// Returns false if a wait hit its limit (the record for bigint_check_timeout
// is set).  WAIT: the products depend on the launch before (pdl_wait).
template <int KB, int NT, bool WAIT = true, class NextB, class NextI, class NextD, class Done>
__device__ __forceinline__ bool pipe_run(const PipeLayout &L, PipeShared *sh, uint8_t *sm,
                                         NextB next_b, NextI next_i, NextD next_d, Done done) {
  constexpr int ISSUER = PIPE_DRAIN / 32;
  const int tid = threadIdx.x, warp = __shfl_sync(FULL, tid >> 5, 0);
  const long long lim = wait_limit_here();
  if (tid == 0) {
    for (int i = 0; i < PIPE_STAGES; i++) {
      mbar_init(smem_u32(&sh->hfull[i]), PIPE_BUILD);
      mbar_init(smem_u32(&sh->hfree[i]), 1);
    }
    for (int i = 0; i < 4; i++) {
      mbar_init(smem_u32(&sh->afull[i]), 1);
      mbar_init(smem_u32(&sh->afree[i]), PIPE_DRAIN / 32);
    }
    for (int i = 0; i < 2; i++) {
      mbar_init(smem_u32(&sh->xfull[i]), PIPE_BUILD);
      mbar_init(smem_u32(&sh->xfree[i]), 1);
    }
    mbar_init(smem_u32(&sh->done), 1);
    fence_mbar_init();
    sh->abort = 0;
  }
  if (tid < 32) {
    tmem_alloc(smem_u32(&sh->tmem_slot), 512);
    tmem_relinquish();
  }
  for (int i = tid; i < ZB * 128 / 16; i += PIPE_THREADS)
    reinterpret_cast<uint4 *>(sm + L.z)[i] = make_uint4(0u, 0u, 0u, 0u);
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh->tmem_slot;
  pdl_trigger();  // not before this CTA has its tensor memory
  if constexpr (WAIT) pdl_wait();
  if (warp < ISSUER) {
    pipe_drain<KB, NT>(L, sh, sm, tmem, lim, next_d, done);
  } else if (warp == ISSUER) {
    pipe_issuer<KB, NT>(L, sh, smem_u32(sm), tmem, lim, next_i);
    // whatever was issued is finished before the tensor memory is freed
    mma_commit_warp(smem_u32(&sh->done), lane_id() == 0);
    mbar_wait(smem_u32(&sh->done), 0, WAIT_LIMIT);
  } else {
    pipe_builder<KB, NT>(L, sh, sm, lim, tid - 32 * (ISSUER + 1), next_b);
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const bool ok = sh->abort == 0;
  if (!ok && tid == 0) atomicExch(&g_timeout, 1);
  if (tid < 32) tmem_dealloc(tmem, 512);
  return ok;
}

}  // namespace tcm
}  // namespace bigint
