// addsub.cu -- batched addition and subtraction (Sec. V-A, Figs. 3 and 4).
//
// One CTA per instance (one warp, several to a CTA, for short ones).  The
// CTA's W warps split the instance into W contiguous segments per
// "super-round"; within its segment a warp reads R rounds of 32 lanes x LPL
// limbs with coalesced loads (16 bytes a lane where n is even and the
// buffers are aligned), straight into registers (step A1: no shared-memory
// staging is needed because each limb is used by exactly one lane).
//
// Carry propagation (step A2) is the exclusive (generate, propagate) scan of
// Fig. 3 evaluated in three levels:
//   lane   -- each lane folds its LPL limbs sequentially (Fig. 4, f1),
//   warp   -- two ballots per round resolve the carries of 32 lanes
//             (WarpCarry in common.cuh), and the rounds are folded in order,
//   block  -- warp aggregates go through shared memory and are resolved by
//             the same two-ballot trick (Fig. 4, the scan of carry_thds);
// then each lane applies its carry-in and ripples it through its limbs
// (Fig. 4, f2).  Subtraction is the same scan with generate = (a < b) and
// propagate = (a == b), applied as a borrow.
//
// The add chain a + b + ... + b (k additions, bigint_add_chain) is the same
// pass over a_j + k b_j: that sum's high word (at most 255) belongs to limb
// j + 1, so the low words and the high words one limb up are added with one
// carry scan, whatever k is.
//
// HBM traffic is the algorithmic minimum: 2 limbs read and 1 written per
// limb position (Table I's 3 x NumInsts x NumBits / 8 bytes).
#include "common.cuh"

namespace bigint {

// Operations of k_addsub: a + b, a - b, and a + k b (the add chain's k
// additions at once, k <= 255).
enum AddSubMode { ADD = 0, SUB = 1, CHAIN = 2 };

// WPI: one warp per instance (n at most one warp's segment), WPI_WARPS
// instances per CTA and no block barrier.
constexpr int WPI_WARPS = 8;

template <int MODE, int LPL, int R, bool WPI>
__global__ void __launch_bounds__(1024)
    k_addsub(const uint64_t *A, const uint64_t *B, uint64_t *Out,
             uint8_t *__restrict__ carry_out, int64_t count, int n, uint32_t k) {
  constexpr int SEG = 32 * LPL * R;  // limbs per warp per super-round
  __shared__ uint32_t s_g[32], s_p[32];
  __shared__ uint32_t s_hi;   // CHAIN: high word of the super-round's last limb
  __shared__ uint32_t s_top;  // CHAIN: high word of limb n - 1

  const uint32_t lane = lane_id();
  const int warp = WPI ? 0 : threadIdx.x >> 5;
  const int nwarps = WPI ? 1 : blockDim.x >> 5;
  const int64_t inst =
      WPI ? (int64_t)blockIdx.x * WPI_WARPS + (threadIdx.x >> 5) : (int64_t)blockIdx.x;
  if (WPI && inst >= count) return;  // the whole warp: no block barrier below
  const uint64_t *a = A + inst * (int64_t)n;
  const uint64_t *b = B + inst * (int64_t)n;
  uint64_t *out = Out + inst * (int64_t)n;
  uint32_t top = 0;  // CHAIN, WPI: high word of limb n - 1
  if (MODE == CHAIN && !WPI) {
    if (threadIdx.x == 0) s_hi = 0;
    __syncthreads();
  }

  uint32_t cin_block = 0;  // carry into the current super-round
  for (int base = 0; base < n; base += SEG * nwarps) {
    const int wbase = base + warp * SEG;
    uint64_t av[R][LPL], bv[R][LPL];
    // ---- A1: all loads of this super-round first (memory-level parallelism)
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int j = wbase + r * 32 * LPL + (int)lane * LPL;
      if constexpr (LPL == 2) {
        if (j + 1 < n) {
          ulonglong2 x = ld_stream2(a + j), y = ld_stream2(b + j);
          av[r][0] = x.x; av[r][1] = x.y; bv[r][0] = y.x; bv[r][1] = y.y;
        } else {
          av[r][0] = j < n ? a[j] : 0; av[r][1] = 0;
          bv[r][0] = j < n ? b[j] : 0; bv[r][1] = 0;
        }
      } else {
        av[r][0] = j < n ? __ldcs(a + j) : 0;
        bv[r][0] = j < n ? __ldcs(b + j) : 0;
      }
    }
    uint32_t hprev = 0;  // CHAIN: high word of the limb below this round's first
    if (MODE == CHAIN && !WPI) {
      // the warp's first limb takes the high word of the limb below it: from
      // the super-round before for warp 0, recomputed from memory otherwise
      // (this super-round stores nothing before its first barrier)
      if (lane == 0) {
        if (warp == 0) hprev = s_hi;
        else if (wbase <= n) {
          const uint64_t lo = (uint64_t)k * b[wbase - 1], t = a[wbase - 1] + lo;
          hprev = (uint32_t)__umul64hi(k, b[wbase - 1]) + (t < lo);
        }
      }
    }
    // ---- A2 level 1: per-limb sums and the lane's (g, p) per round
    uint64_t s[R][LPL];
    uint32_t gbits = 0, pbits = 0;  // per-limb generate/propagate, bit r*LPL+l
    WarpCarry wc[R];
    uint32_t hlast = 0;
#pragma unroll
    for (int r = 0; r < R; r++) {
      uint32_t g = 0, p = 1;
      uint32_t h[LPL];  // CHAIN: high words (at most 255) of the round's limbs
      if (MODE == CHAIN) {
#pragma unroll
        for (int l = 0; l < LPL; l++) {
          const uint64_t lo = (uint64_t)k * bv[r][l], t = av[r][l] + lo;
          h[l] = (uint32_t)__umul64hi(k, bv[r][l]) + (t < lo);
          av[r][l] = t;
          if (wbase + r * 32 * LPL + (int)lane * LPL + l == n - 1) {
            if (WPI) top = h[l]; else s_top = h[l];
          }
        }
        const uint32_t below = __shfl_up_sync(FULL, h[LPL - 1], 1);
        bv[r][0] = lane == 0 ? hprev : below;
        if constexpr (LPL == 2) bv[r][1] = h[0];
        hlast = h[LPL - 1];
        hprev = __shfl_sync(FULL, hlast, 31);
      }
#pragma unroll
      for (int l = 0; l < LPL; l++) {
        uint64_t x = av[r][l], y = bv[r][l];
        uint64_t t = MODE == SUB ? x - y : x + y;
        // positions past the end pass carries through, so the carry
        // out of the last limb reaches the end of the warp and of the block
        const int j = wbase + r * 32 * LPL + (int)lane * LPL + l;
        const bool in = j < n;
        uint32_t gl = in && (MODE == SUB ? (x < y) : (t < x));
        uint32_t pl = !in || (MODE == SUB ? (t == 0) : (t == ~0ull));
        s[r][l] = t;
        gbits |= gl << (r * LPL + l);
        pbits |= pl << (r * LPL + l);
        g = gl | (pl & g);  // limb l is more significant than the fold so far
        p = p & pl;
      }
      wc[r] = warp_gp(g, p);
    }
    uint32_t c = 0, cout_block;
    if (WPI) {
      cout_block = 0;  // known after the last round below
    } else {
      // ---- A2 level 2: fold the rounds into the warp's (g, p)
      uint32_t wg = 0, wp = 1;
#pragma unroll
      for (int r = 0; r < R; r++) {
        wg = warp_carry_out(wc[r], 0) | (warp_all_propagate(wc[r]) & wg);
        wp = wp & warp_all_propagate(wc[r]);
      }
      if (lane == 0) { s_g[warp] = wg; s_p[warp] = wp; }
      __syncthreads();
      // ---- A2 level 3: resolve the warps of the block
      const uint32_t gw = (int)lane < nwarps ? s_g[lane] : 0;
      const uint32_t pw = (int)lane < nwarps ? s_p[lane] : 0;
      const uint64_t cm = warp_carries(warp_gp(gw, pw), cin_block);
      c = (uint32_t)(cm >> warp) & 1u;
      cout_block = (uint32_t)(cm >> nwarps) & 1u;
      if (MODE == CHAIN && warp == nwarps - 1 && lane == 31) s_hi = hlast;
    }
    // ---- apply the carries (Fig. 4, f2) and store
#pragma unroll
    for (int r = 0; r < R; r++) {
      const uint64_t lc = warp_carries(wc[r], c);
      uint32_t cl = (uint32_t)(lc >> lane) & 1u;
      c = (uint32_t)(lc >> 32) & 1u;
      uint64_t res[LPL];
#pragma unroll
      for (int l = 0; l < LPL; l++) {
        res[l] = MODE == SUB ? s[r][l] - cl : s[r][l] + cl;
        const uint32_t gl = (gbits >> (r * LPL + l)) & 1u;
        const uint32_t pl = (pbits >> (r * LPL + l)) & 1u;
        cl = gl | (pl & cl);
      }
      const int j = wbase + r * 32 * LPL + (int)lane * LPL;
      if constexpr (LPL == 2) {
        if (j + 1 < n) {
          st_stream2(out + j, make_ulonglong2(res[0], res[1]));
        } else if (j < n) {
          out[j] = res[0];
        }
      } else {
        if (j < n) __stcs(out + j, res[0]);
      }
    }
    cin_block = WPI ? c : cout_block;
    if (!WPI) __syncthreads();  // s_g / s_p are rewritten by the next super-round
  }
  if (carry_out == nullptr) return;
  if (WPI) {
    if (MODE == CHAIN) top = __reduce_max_sync(FULL, top);  // one lane holds it
    if (lane == 0) carry_out[inst] = (uint8_t)(cin_block + top);
  } else if (threadIdx.x == 0) {
    carry_out[inst] = (uint8_t)(cin_block + (MODE == CHAIN ? s_top : 0u));
  }
}

// Launch shape: rounds per warp, and warps per CTA or (0) one warp per instance.
//
// A large batch is bound by HBM (24 bytes a limb), so what matters is loads in
// flight on every SM at every moment: one CTA that holds the SM alone reads,
// waits, then writes (operand arrays of 2^32 bits, 8192 limbs: 5.7 TB/s with 32
// warps of four rounds, 7.0 with 8).  A small one lasts as long as its last CTA,
// which wants less work per warp and more warps.  128 limbs a warp and up to 16
// warps serve both; where they do not:
//  * Batches of MANY instances per SM and MANY_LIMBS limbs take 8 warps of four
//    rounds for more than 4096 limbs (600 of 8192 limbs 16.9 us, 17.7 as 16 warps
//    of two) and for odd sizes (8-byte accesses: 2^26 limbs of 1025 234 us, 236
//    as 9 warps).
//  * Up to 1024 limbs, batches of at most HALF_LIMBS limbs per SM take 64 limbs a
//    warp (64 of 512 limbs 1.75 -> 1.66 us; 600 of 1024 limbs 2.90 -> 3.14, so
//    not there).
//  * At most one instance per SM (odd sizes: two) gets 32 warps (16 of 4096 limbs
//    2.9 us, 3.2 with 16), of four rounds above 4096 limbs (6000 limbs 3.6 us, 3.7
//    with two), and one of two 24 if that makes one super-round.
// Against 8 warps of four rounds (32 up to two instances per SM) at every size:
// 64 additions of 512 limbs 1.78 -> 1.45 us, 400 of 1024 limbs 2.77 -> 2.51, 600
// of 1536 limbs 3.70 -> 3.29, 304 of 8192 limbs 8.54 -> 7.09, 400 of 8193 limbs
// 15.4 -> 12.0, 2^26 limbs of 300 242 -> 224.
//
// The chain keeps 4 warps of four rounds (32 up to two instances per SM): its
// extra arithmetic wants more CTAs (8192 limbs: 6.8 against 6.5 TB/s with 8).
//
// Short operands go one warp per instance in larger batches, because a CTA each
// starts and ends too often (64 limbs, HBM-bound: 3.0 TB/s); a few instances are
// faster with several warps each (128 limbs x 152 1.77 -> 1.66 us, 256 limbs x 64
// 2.05 -> 1.56, x 400 2.08 -> 1.98).
struct Shape {
  int R, W;
};
constexpr int MANY = 3;
constexpr int64_t MANY_LIMBS = 3 << 20, HALF_LIMBS = 2048;

template <int MODE, int LPL>
static Shape shape_of(int64_t count, int n) {
  constexpr int ROUND = 32 * LPL;  // limbs of a warp's round
  const int sms = sm_count();
  const bool chain = MODE == CHAIN;
  if (n <= ROUND || (n <= 4 * ROUND && (chain || count > 2 * LPL * sms)))
    return Shape{n <= ROUND ? 1 : (n <= 2 * ROUND ? 2 : 4), 0};
  const bool many = count > MANY * sms && count * n > MANY_LIMBS && (LPL == 1 || n > 4096);
  const bool half = n <= 1024 && count * n <= HALF_LIMBS * sms;
  const bool four = chain || many || (n > 4096 && count <= sms);
  const int R = four ? 4 : (half ? 64 : 128) / ROUND;
  const int need = (n + R * ROUND - 1) / (R * ROUND);  // warps for one super-round
  int max_warps;
  if (chain)
    max_warps = count <= 2 * sms ? 32 : 4;
  else if (LPL == 1)
    max_warps = count <= 2 * sms ? 32 : (many ? 8 : 16);
  else
    max_warps = count <= sms ? 32 : (count <= 2 * sms && need <= 24 ? 24 : (many ? 8 : 16));
  const int rounds = (need + max_warps - 1) / max_warps;
  return Shape{R, (need + rounds - 1) / rounds};
}

template <int MODE, int LPL, int R>
static int launch_shape(const uint64_t *a, const uint64_t *b, uint64_t *out, uint8_t *carry,
                        int64_t count, int n, uint32_t k, int W, cudaStream_t st) {
  if (W == 0)
    k_addsub<MODE, LPL, R, true><<<(unsigned)((count + WPI_WARPS - 1) / WPI_WARPS), 32 * WPI_WARPS,
                                   0, st>>>(a, b, out, carry, count, n, k);
  else if constexpr (MODE != CHAIN || R == 4)
    k_addsub<MODE, LPL, R, false><<<(unsigned)count, 32 * W, 0, st>>>(a, b, out, carry, count, n,
                                                                      k);
  return bigint_launch_status();
}

template <int MODE, int LPL>
static int launch_lpl(const uint64_t *a, const uint64_t *b, uint64_t *out, uint8_t *carry,
                      int64_t count, int n, uint32_t k, cudaStream_t st) {
  const Shape S = shape_of<MODE, LPL>(count, n);
  switch (S.R) {
    case 1: return launch_shape<MODE, LPL, 1>(a, b, out, carry, count, n, k, S.W, st);
    case 2: return launch_shape<MODE, LPL, 2>(a, b, out, carry, count, n, k, S.W, st);
    default: return launch_shape<MODE, LPL, 4>(a, b, out, carry, count, n, k, S.W, st);
  }
}

template <int MODE>
static int launch_mode(const uint64_t *a, const uint64_t *b, uint64_t *out, uint8_t *carry,
                       int64_t count, int n, uint32_t k, cudaStream_t st) {
  const bool vec = (n % 2 == 0) && (((uintptr_t)a | (uintptr_t)b | (uintptr_t)out) % 16 == 0);
  return vec ? launch_lpl<MODE, 2>(a, b, out, carry, count, n, k, st)
             : launch_lpl<MODE, 1>(a, b, out, carry, count, n, k, st);
}

int launch_addsub(bool sub, const uint64_t *a, const uint64_t *b, uint64_t *out,
                  uint8_t *carry, int64_t count, int n, cudaStream_t st) {
  return sub ? launch_mode<SUB>(a, b, out, carry, count, n, 0, st)
             : launch_mode<ADD>(a, b, out, carry, count, n, 0, st);
}

int launch_add_chain(const uint64_t *a, const uint64_t *b, uint64_t *out, uint8_t *carry,
                     int64_t count, int n, int k, cudaStream_t st) {
  return launch_mode<CHAIN>(a, b, out, carry, count, n, (uint32_t)k, st);
}

}  // namespace bigint
