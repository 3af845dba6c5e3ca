// divstep.cu -- division of a uniform batch with every step batched across
// the instances (Sec. V-C, Fig. 6).
//
// The one-CTA-per-division kernel (divmod.cu) runs the whole algorithm of a
// division on one SM, as the paper's intragroup kernel does.  Its products
// are as fast as the SM allows, but the Newton loop is sequential: the early
// steps are tiny, every linear step waits at block barriers, and a batch
// smaller than a few waves of SMs leaves most of the GPU idle.  Here the
// division is instead cut at its steps, and each step runs for ALL instances
// of the batch at once: the products as batched launches of the multiply
// kernels (tensor-core products from a shorter operand of 64 limbs: tcmul.cu,
// each filling every SM), the linear steps as one small kernel with one warp
// or CTA per instance.  The arithmetic is that of divmod.cu; the schedule
// differs, and the products of a step are cut to the limbs it uses.
//
// Every instance of a batch has the same shape (nu, nv), and for the usual
// operands (top limb of v nonzero, "regular") the same precision k = nv - 1
// and the exponent h = nu, so the Newton schedule (l, m, t per step) is
// known on the host.  Instances whose divisor has a zero top limb
// (including v = 0) are listed and divided in a last launch, a warp each
// (k_ds_listed) or, longer ones, a CTA each (divmod.cu); the step kernels run
// over them too (their values are never used, and
// every size is fixed, so nothing reads out of bounds).
//
// Per step, with the iterate w ~ B^(k+l) / v kept to l + 2 limbs,
// m = min(l - 2, L - l), t = min(k, l + m + 2), vt = top t + 1 limbs of v:
//   P  = vt w mod B^(t+2)                    (banded from limb c - 2)
//   d  = B^(t+l) - vt w: |d| = P if P < B^(t+2)/2 (d <= 0), else B^(t+2) - P,
//        from limb c = t - m - 2 on (within a unit there, step_cut)
//   P2 = w |d|, banded from limb s - 2, s = t + l - m
//   w' = w B^m + floor(P2 / B^s)             (d >= 0)
//   w' = w B^m - floor(P2 / B^s) - 1         (d <  0; the ceiling of Fig. 6
//                                             rounded up by at most one)
// The band makes floor(P2 / B^s) exact or one unit high, and the unit of limb
// c by which |d| may be off moves it by less than 2 / B^2; so each step lands
// within a few units of B^(k+l+m) / v, and since m <= l - 2 the Newton error
// squared stays below a unit: the error does not grow from step to step.
// Then q^ = floor(u w / B^h) (banded from limb h - 2), r^ = u - q^ v modulo
// B^(nv+1), and the exact correction of divmod.cu settles q and r.  The
// leading steps whose operands all have at most SMALL_STEP_LIMBS limbs run in
// one launch, a warp per instance (k_ds_small), instead of four launches each.
//
// Measured: 4096 divisions of 1024 by 512 limbs 628 us, of which the products
// take 475 (their tensor-core floor is 145 us: low and banded triangles of
// small products, bound by the builds, drains and limb scans of tcone.cuh); one
// division of 16384 by 8192 limbs 282 us, a chain of 40 dependent launches of
// 4 to 27 us.
#include <algorithm>

#include "divstep.cuh"

namespace bigint {

using namespace divc;

int launch_mul_ex(const uint64_t *a, int64_t sa, const uint64_t *b, int64_t sb, uint64_t *out,
                  int64_t so, int64_t count, int na, int nb, int nout, int lo, int *abort_flag,
                  cudaStream_t st, int tc_min, SkBuffers *sk);
bool mul_ex_ok(int na, int nb, int tc_min);
int launch_divmod_cta(const uint64_t *u, const uint64_t *v, uint64_t *q, uint64_t *r,
                      int32_t *status, int64_t count, int nu, int nv, void *ws,
                      const int32_t *list, const int *nlist, cudaStream_t st);
size_t divmod_workspace(int64_t count, int nu, int nv);

namespace dstep {

// Shorter operand (limbs) from which a step's product runs on the tensor
// cores.  The steps' products are rectangular and come in batches of
// thousands; measured on 2n/n divisions at n = 512 the 132 x 262-limb and
// 68 x 134-limb products of the middle steps took 173 and 90 us on the
// integer pipes for 4096 instances, 39 and 30 us as one-drain products.
constexpr int STEP_TC_MIN = 64;

// The step schedule needs k = prec(v) - 1 = nv - 1.  The dividend may have
// leading zero limbs: with h = nu (not prec(u)) w ~ B^h / v still bounds the
// quotient estimate u w / B^h within a few units of u / v since u < B^h,
// and the banded u w + B^h < B^(nu + nw) still holds, so such instances
// stay on the step path at the cost of the product work above their
// precision.
__device__ __forceinline__ bool regular(const uint64_t *, int, const uint64_t *v, int nv) {
  return v[nv - 1] != 0;
}

// One thread per instance: lists the irregular instances and writes the
// Newton start w = floor(B^(2 l) / V), V = floor(v / B^(k-l)) + 1, into the
// first l + 2 limbs of the instance's iterate record (zero for irregular
// ones, whose divisor may have a zero top limb).  (Running the first,
// tiny Newton steps in this kernel too, one CTA per instance, was measured
// slower than their batched launches: 579 us for 4096 instances of 512
// limbs, the long chains of block barriers of the one-CTA form again.)
__global__ void k_ds_start(const uint64_t *U, const uint64_t *V, int nu,
                           int nv, int l, uint64_t *W, int64_t sw, int64_t count,
                           int32_t *irregular, int *nirr) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  pdl_trigger();
  pdl_wait();
  if (i >= count) return;
  const uint64_t *u = U + i * nu, *v = V + i * nv;
  uint64_t *w = W + i * sw;
  if (!regular(u, nu, v, nv)) {
    irregular[atomicAdd(nirr, 1)] = (int32_t)i;
    for (int j = 0; j < l + 2; j++) w[j] = 0;
    return;
  }
  ds_start_one(v, nv, l, w);
}

constexpr int WARP_CTA = 256;  // warp-per-instance kernels: 8 instances per CTA

// ---------------------------------------------------------------------------
// The early Newton steps, while every operand of a step has at most
// SMALL_STEP_LIMBS limbs, in one launch with one warp per instance: each
// such step is four small launches otherwise (P, |d|, P2, update), whose
// fixed costs are most of their time.  The warp keeps w, the divisor's top
// limbs, P / |d| and P2 in shared memory and runs the same arithmetic as the
// batched kernels (warp_mul's band makes floor(P2 / B^s) exact or one high).
// ---------------------------------------------------------------------------
constexpr int SMALL_STEP_MAX = 16;

// The steps the fused kernel runs; N bounds their operands (limbs, a
// multiple of 8).
struct SmallSteps {
  int n, N;
  Step s[SMALL_STEP_MAX];
};

// Steps S of every instance: the iterate from W0 (its first l + 2 limbs),
// the result (l + m + 2 limbs of the last step) to W0 or W1 as the batched
// steps would leave it (W0 after an even number of steps).
__global__ void __launch_bounds__(32 * SMALL_STEP_WARPS)
    k_ds_small(const uint64_t *V, int nv, uint64_t *W0, uint64_t *W1, int64_t sw,
               int64_t count, SmallSteps S) {
  extern __shared__ __align__(16) uint64_t ssm[];
  const int wi = threadIdx.x >> 5, lane = (int)lane_id();
  const int64_t i = (int64_t)blockIdx.x * SMALL_STEP_WARPS + wi;
  pdl_trigger();
  pdl_wait();
  if (i >= count) return;  // the whole warp: no block barrier below
  const int N = S.N;
  uint64_t *base = ssm + (size_t)wi * small_step_warp_limbs(N);
  uint64_t *wb[2] = {base, base + N}, *vt = base + 2 * N, *d = base + 3 * N, *z = base + 4 * N;
  const int t = S.s[S.n - 1].t;  // the largest
  const uint64_t *v = V + i * nv + (nv - 1 - t);
  for (int j = lane; j <= t; j += 32) vt[j] = v[j];
  for (int j = lane; j < S.s[0].l + 2; j += 32) wb[0][j] = W0[i * sw + j];
  __syncwarp();
  int cur = 0;
  for (int st = 0; st < S.n; st++) {
    ds_small_step(vt + (t - S.s[st].t), S.s[st], wb[cur], wb[cur ^ 1], d, z);
    cur ^= 1;
  }
  const int nlast = S.s[S.n - 1].l + S.s[S.n - 1].m + 2;
  uint64_t *out = (S.n & 1) ? W1 : W0;
  for (int j = lane; j < nlast; j += 32) out[i * sw + j] = wb[cur][j];
}

// One warp per instance: the sign of d from P = vt w mod B^nl and |d| (nl
// limbs): P itself if its top bit is clear (d <= 0), else B^nl - P.
__global__ void __launch_bounds__(WARP_CTA)
    k_ds_mid(const uint64_t *P, int64_t sp, uint64_t *D, int64_t sd,
             int nl, int32_t *neg, int64_t count) {
  const int64_t i = (int64_t)blockIdx.x * (WARP_CTA / 32) + (threadIdx.x >> 5);
  pdl_trigger();
  pdl_wait();
  if (i >= count) return;
  const bool ng = ds_mid_warp(P + i * sp, D + i * sd, nl);
  if (lane_id() == 0) neg[i] = ng ? 1 : 0;
}

// One warp per instance: w' = w B^m + Y (d >= 0) or w B^m - Y - 1 (d < 0),
// Y = floor(P2 / B^s) (ny limbs), into nout limbs of the next iterate record.
__global__ void __launch_bounds__(WARP_CTA)
    k_ds_update(const uint64_t *W, int64_t sw, int nw, const uint64_t *Z,
                int64_t sz, int s, int ny, const int32_t *neg, int m,
                uint64_t *Wn, int nout, int64_t count) {
  const int64_t i = (int64_t)blockIdx.x * (WARP_CTA / 32) + (threadIdx.x >> 5);
  pdl_trigger();
  pdl_wait();
  if (i >= count) return;
  ds_update_warp(W + i * sw, nw, Z + i * sz + s, ny, neg[i] != 0, m, Wn + i * sw, nout);
}

// The same two steps with one CTA per instance, for wide records (a warp
// takes its limbs 32 at a time, one round after the other).
__global__ void __launch_bounds__(LIN_THREADS_FEW)
    k_ds_mid_cta(const uint64_t *P, int64_t sp, uint64_t *D, int64_t sd,
                 int nl, int32_t *neg) {
  __shared__ uint32_t scr[BLK_SCRATCH_WORDS];
  pdl_trigger();
  pdl_wait();
  const int64_t i = blockIdx.x;
  const bool ng = ds_mid_cta(P + i * sp, D + i * sd, nl, scr);
  if (threadIdx.x == 0) neg[i] = ng ? 1 : 0;
}

__global__ void __launch_bounds__(LIN_THREADS_FEW)
    k_ds_update_cta(const uint64_t *W, int64_t sw, int nw,
                    const uint64_t *Z, int64_t sz, int s, int ny,
                    const int32_t *neg, int m, uint64_t *Wn, int nout) {
  __shared__ uint32_t scr[BLK_SCRATCH_WORDS];
  pdl_trigger();
  pdl_wait();
  const int64_t i = blockIdx.x;
  ds_update_cta(W + i * sw, nw, Z + i * sz + s, ny, neg[i] != 0, m, Wn + i * sw, nout, scr);
}

// Records up to this many limbs take the warp-per-instance kernels, except
// in batches of at most FEW instances (about the SMs).
constexpr int WARP_LIMBS = 1024;
constexpr int64_t FEW = 128;

// One CTA per regular instance: r^ = (u - R) mod B^(nv+1) with R the low
// nv + 1 limbs of q^ v, the exact correction of q^ (in place: the top limbs
// of the banded product) and r^ (divmod.cu), and the results.  Irregular
// instances are left to the last launch.  A tensor-core product of this division
// that gave up at a wait limit (*aborted) voids the results: BIGINT_ETIMEOUT.
__global__ void __launch_bounds__(LIN_THREADS_FEW)
    k_ds_finish(const uint64_t *U, int nu, const uint64_t *V, int nv,
                const uint64_t *R, int64_t sp, uint64_t *Rh, int64_t sd, uint64_t *Qh,
                int64_t sq, int nqh, uint64_t *Qo, int nq, uint64_t *Ro, int32_t *status,
                const int *aborted) {
  __shared__ uint32_t scr[BLK_SCRATCH_WORDS];
  pdl_trigger();
  pdl_wait();
  const int64_t i = blockIdx.x;
  const uint64_t *u = U + i * nu, *v = V + i * nv, *rr = R + i * sp;
  if (!regular(u, nu, v, nv)) return;
  uint64_t *qh = Qh + i * sq;
  if (threadIdx.x == 0) qh[nqh] = 0;  // room for a carry of the correction
  __syncthreads();
  int st = ds_finish_cta(u, nu, v, nv, rr, Rh + i * sd, qh, nqh + 1, Qo + i * nq, nq, Ro + i * nv,
                         scr);
  if (*(volatile const int *)aborted) st = BIGINT_ETIMEOUT;
  if (status != nullptr && threadIdx.x == 0) status[i] = st;
}

// ---------------------------------------------------------------------------
// The listed instances of short shapes: long division by 64-bit digits (Knuth's
// Algorithm D), one warp per instance, everything in shared memory.  Any divisor
// and quotient: v = 0, a quotient beyond nq limbs, u < v.
//
// Why: the one-CTA-per-division kernel takes the Newton steps again, one CTA's
// block barriers after the other, on top of the steps the batch has just been
// through.  Batches of divisors that all have a zero top limb (padded arrays):
// 300 of 144 by 96 limbs 149 -> 85 us, 20000 of 64 by 32 limbs 2736 -> 362 (99
// and 2450 without the step form).  Bound by latency: a quotient limb takes 0.3 us
// below 32 divisor limbs, 0.5 us at 127, so that the longest quotients taken
// here are no faster than a CTA's (one of 508 by 127 limbs 292 us, of which the
// steps 97; 341 with the CTA form in this place), and longer ones stay there.
// ---------------------------------------------------------------------------
constexpr int LIST_WARPS = 4, LIST_NV = 128, LIST_NU = 512;
constexpr int64_t LIST_CTAS = 2048;  // more than are ever resident; they loop over the list
__host__ __device__ inline bool list_warps_ok(int nu, int nv) {
  return nv < LIST_NV && nu <= LIST_NU;
}
__host__ __device__ inline int list_warp_limbs(int nu, int nv) { return nu + 1 + nv; }

// One warp: precision of x[0 .. n).
__device__ __forceinline__ int warp_prec(const uint64_t *x, int n) {
  for (int base = (n - 1) & ~31; base >= 0; base -= 32) {
    const int j = base + (int)lane_id();
    const uint32_t nz = __ballot_sync(FULL, j < n && x[j] != 0);
    if (nz) return base + 32 - __clz((int)nz);
  }
  return 0;
}

// One warp: x (nx limbs) shifted up by s bits (s < 64) into out, n >= nx limbs.
__device__ __forceinline__ void warp_shl(const uint64_t *x, int nx, int s, uint64_t *out, int n) {
  for (int j = lane_id(); j < n; j += 32) {
    const uint64_t a = j < nx ? x[j] : 0ull, b = j >= 1 && j - 1 < nx ? x[j - 1] : 0ull;
    out[j] = s ? a << s | b >> (64 - s) : a;
  }
}

// One warp: x[0 .. n] -= d y[0 .. n), n < 32 R, x in shared memory, lane i's R
// limbs of y from limb R i on in its registers (zero from n on); the borrow out
// of limb n (d one too large).  A lane subtracts the low R limbs of its product
// and the high word of the lane's below, then what that one borrowed (at most
// 2), and one scan settles the rest.
template <int R>
__device__ __forceinline__ bool warp_submul(uint64_t *x, const uint64_t (&y)[R], int n, uint64_t d) {
  const int lane = (int)lane_id(), j0 = R * lane;
  uint64_t t[R], hi = 0;
  uint32_t c = 0;
#pragma unroll
  for (int r = 0; r < R; r++) {
    const uint64_t lo = d * y[r] + hi;  // hi <= B - 2 before, so no overflow after
    hi = __umul64hi(d, y[r]) + (lo < hi);
    const uint64_t xv = j0 + r <= n ? x[j0 + r] : 0ull;
    const uint64_t u = xv - lo;
    t[r] = u - c;
    c = (uint32_t)(xv < lo) + (uint32_t)(u < c);
  }
  uint64_t in = __shfl_up_sync(FULL, hi, 1);
  if (lane == 0) in = 0;
  uint64_t b = in;
#pragma unroll
  for (int r = 0; r < R; r++) {
    const uint64_t u = t[r];
    t[r] = u - b;
    b = u < b;
  }
  c += (uint32_t)b;
  uint32_t cb = __shfl_up_sync(FULL, c, 1);
  if (lane == 0) cb = 0;
  b = cb;
  uint64_t any = 0;
#pragma unroll
  for (int r = 0; r < R; r++) {
    const uint64_t u = t[r];
    t[r] = u - b;
    b = u < b;
    any |= t[r];
  }
  const uint64_t bm = warp_carries(warp_gp((uint32_t)b, b == 0 && any == 0), 0);
  b = (bm >> lane) & 1u;
#pragma unroll
  for (int r = 0; r < R; r++) {
    const uint64_t u = t[r];
    if (j0 + r <= n) x[j0 + r] = u - b;
    b = u < b;
  }
  return __shfl_sync(FULL, c, 31) != 0 || (bm >> 32) != 0;
}

// One warp: the quotient digits of un / vn (normalised: vn of pv < 32 R limbs,
// bit 63 of the last set), L of them, into q (nq limbs); un becomes the
// remainder.  False if the quotient does not fit.
template <int R>
__device__ __forceinline__ bool warp_longdiv(uint64_t *un, const uint64_t *vn, int pv, int L,
                                             uint64_t *q, int nq) {
  typedef unsigned __int128 u128;
  const int lane = (int)lane_id();
  const uint64_t vt = vn[pv - 1], v2 = pv > 1 ? vn[pv - 2] : 0ull;
  const uint64_t rec = (uint64_t)((((u128)~vt << 64) | ~0ull) / vt);  // floor((B^2 - 1) / vt) - B
  uint64_t y[R];
#pragma unroll
  for (int r = 0; r < R; r++) y[r] = R * lane + r < pv ? vn[R * lane + r] : 0ull;
  bool fits = true;
  for (int j = L - 1; j >= 0; j--) {
    // the digit from the top limbs (Moeller and Granlund, as divcore.cuh's
    // small_div), at most one too large
    const uint64_t n1 = un[j + pv], n0 = un[j + pv - 1], n2 = pv > 1 ? un[j + pv - 2] : 0ull;
    uint64_t d = ~0ull;
    u128 rh = (u128)n0 + vt;
    if (n1 < vt) {
      const u128 f = (u128)rec * n1 + (((u128)n1 << 64) | n0);
      d = (uint64_t)(f >> 64) + 1;
      uint64_t r0 = n0 - d * vt;
      if (r0 > (uint64_t)f) {
        d--;
        r0 += vt;
      }
      if (r0 >= vt) {
        d++;
        r0 -= vt;
      }
      rh = r0;
    }
    for (int k = 0; k < 2 && (rh >> 64) == 0 && (u128)d * v2 > ((rh << 64) | n2); k++) {
      d--;
      rh += vt;
    }
    __syncwarp();
    if (warp_submul<R>(un + j, y, pv, d)) {
      d--;
      __syncwarp();
      warp_addsub<false>(pv, 0u, [&](int k) { return make_ulonglong2(un[j + k], vn[k]); },
                         [&](int k, uint64_t x) { un[j + k] = x; });
    }
    __syncwarp();
    if (j < nq) {
      if (lane == 0) q[j] = d;
    } else if (d != 0) {
      fits = false;
    }
  }
  return fits;
}

__global__ void __launch_bounds__(32 * LIST_WARPS)
    k_ds_listed(const uint64_t *U, int nu, const uint64_t *V, int nv, uint64_t *Qo, int nq,
                uint64_t *Ro, int32_t *status, const int32_t *list, const int *nlist) {
  extern __shared__ __align__(16) uint64_t lsm[];
  const int lane = (int)lane_id(), wi = (int)(threadIdx.x >> 5), n = *nlist;
  uint64_t *un = lsm + (size_t)wi * list_warp_limbs(nu, nv), *vn = un + nu + 1;
  for (int64_t e = (int64_t)blockIdx.x * LIST_WARPS + wi; e < n;
       e += (int64_t)gridDim.x * LIST_WARPS) {
    const int64_t i = list[e];
    const uint64_t *u = U + i * nu, *v = V + i * nv;
    uint64_t *q = Qo + i * nq, *r = Ro + i * nv;
    const int pv = warp_prec(v, nv), pu = warp_prec(u, nu);
    int st = pv == 0 ? BIGINT_EDIVZERO : BIGINT_OK;
    const int L = pv > 0 && pu >= pv ? pu - pv + 1 : 0;  // limbs the quotient may have
    for (int j = L + lane; j < nq; j += 32) q[j] = 0;
    if (L == 0) {  // v = 0: q = r = 0; u < v: r = u
      for (int j = lane; j < nv; j += 32) r[j] = pv > 0 && j < pu ? u[j] : 0ull;
    } else {
      const int s = __clzll((long long)v[pv - 1]);
      warp_shl(v, pv, s, vn, pv);
      warp_shl(u, pu, s, un, pu + 1);
      __syncwarp();
      const bool fits = pv < 32 ? warp_longdiv<1>(un, vn, pv, L, q, nq)
                                : (pv < 64 ? warp_longdiv<2>(un, vn, pv, L, q, nq)
                                           : warp_longdiv<4>(un, vn, pv, L, q, nq));
      if (!fits) st = BIGINT_ERANGE;
      for (int j = lane; j < nv; j += 32) {
        const uint64_t a = j < pv ? un[j] : 0ull, b = j + 1 < pv ? un[j + 1] : 0ull;
        r[j] = s ? a >> s | b << (64 - s) : a;
      }
    }
    if (status != nullptr && lane == 0) status[i] = st;
    __syncwarp();
  }
}

// The Newton schedule of a regular instance.
int schedule(int k, int h, int l0, Step *steps, int cap) {
  const int L = h - k;
  int l = l0, n = 0;
  while (l < L && n < cap) {
    steps[n] = newton_next(k, L, l);
    l += steps[n++].m;
  }
  return n;
}

// Limbs that a fused step takes per operand or result (w' too).
int small_step_need(const Step &S) {
  return std::max(std::max(S.l + 2, S.t + 2), S.l + S.m + 2);
}

// How many of the leading steps run fused in one launch.
int small_steps(const Step *steps, int ns) {
  int n = 0;
  while (n < ns && n < SMALL_STEP_MAX && small_step_need(steps[n]) <= SMALL_STEP_LIMBS) n++;
  return n;
}

// Per-instance record widths (limbs) and the workspace layout.
struct Layout {
  int64_t sw, sp, sd, sz;  // iterate, low product, |d| / r^, banded product (then q^)
  size_t w0, w1, p, d, z, neg, total;
};

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

Layout layout(int64_t count, int nu, int nv) {
  Layout Y;
  const int L = nu - nv + 1;
  Y.sw = L + 4;
  Y.sp = nv + 2;
  Y.sd = nv + 2;
  Y.sz = nu + L + 6;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = align256(o + bytes);
    return at;
  };
  Y.w0 = take(8 * count * Y.sw);
  Y.w1 = take(8 * count * Y.sw);
  Y.p = take(8 * count * Y.sp);
  Y.d = take(8 * count * Y.sd);
  Y.z = take(8 * count * Y.sz);
  Y.neg = take(4 * count);
  Y.total = o;
  return Y;
}

// The products of a division outside the fused steps, f(na, nb, nout, lo) for
// each: every step's two, then those of the tail.  f returns false to stop.
template <class F>
bool products(int nu, int nv, F f) {
  const int k = nv - 1, h = nu, L = h - k, l0 = L < 3 ? L : 3, nw = L + 2;
  Step steps[64];
  const int ns = schedule(k, h, l0, steps, 64);
  for (int i = small_steps(steps, ns); i < ns; i++) {
    const Step S = steps[i];
    const int c = step_cut(S), nl = S.t + 2 - c;
    if (!f(S.t + 1, S.l + 2, S.t + 2, c > 0 ? c - 2 : 0)) return false;
    if (!f(S.l + 2, nl, S.l + 2 + nl, S.t + S.l - S.m - c - 2)) return false;
  }
  return f(nu, nw, nu + nw, h - 2) && f(nw, nv, nv + 1, 0);
}

}  // namespace dstep

// True if divmod_steps can run this shape (with enough workspace): u w has a
// shorter operand of nu - nv + 3 limbs, and where that fits no product form
// (quotients of some 11000 limbs and more) the division is left to the
// one-CTA-per-division kernel, which slices its products.
bool divmod_steps_ok(int64_t count, int nu, int nv, size_t ws_bytes) {
  if (count < 1 || nv < 8 || nu < nv) return false;
  if (dstep::layout(count, nu, nv).total > ws_bytes) return false;
  return dstep::products(nu, nv, [](int na, int nb, int, int) {
    return mul_ex_ok(na, nb, dstep::STEP_TC_MIN);
  });
}

// Whether a uniform batch takes the step-batched form by default: all but
// few divisions with short quotients.  Up to four quotient limbs take one
// Newton step at most, and a CTA's two short products then end before the
// step form's eight launches (1 to 200 divisions of 67 by 64 limbs 32 us
// against 40, of 515 by 512 limbs 38 against 46), unless the batch fills the SMs
// (4096 of 66 by 64 limbs 94 against 58 us) or the divisor is long (one
// division of 4099 by 4096 limbs 110 against 65 us).  With longer quotients
// the step form is ahead from 8-limb divisors on: 16 by 8 limbs 47 : 37 us
// for up to 200 divisions and 1187 : 164 us for 20000, 192 by 96 limbs
// 142 : 66 us for 200 and 5093 : 714 us for 20000.
bool divmod_steps_default(int64_t count, int nu, int nv) {
  if (nv < 8 || nu < nv) return false;
  return !(nu - nv + 1 <= 4 && nv <= 1024 && count <= 1024 && count * nv <= (1 << 18));
}

// q = floor(u / v), r = u - q v for a uniform batch, step by step across the
// batch (see the top of this file); irregular instances at the end.
// ws: ws_bytes for the step records (the one-CTA-per-division kernel's
// per-instance regions, reused); list_and_counters: 4 count bytes rounded to
// 256, then two ints, OUTSIDE those regions (that kernel reads the list
// while it writes its regions); sk: sk_bytes for two sets of column sums of the
// split-K products of a small batch (null: none).
int launch_divmod_steps(const uint64_t *u, const uint64_t *v, uint64_t *q, uint64_t *r,
                        int32_t *status, int64_t count, int nu, int nv, void *ws, size_t ws_bytes,
                        void *list_and_counters, void *sk, size_t sk_bytes, cudaStream_t st) {
  using namespace dstep;
  if (!divmod_steps_ok(count, nu, nv, ws_bytes)) return BIGINT_EINVAL;
  const Layout Y = layout(count, nu, nv);
  char *base = static_cast<char *>(ws);
  uint64_t *W[2] = {reinterpret_cast<uint64_t *>(base + Y.w0),
                    reinterpret_cast<uint64_t *>(base + Y.w1)};
  uint64_t *P = reinterpret_cast<uint64_t *>(base + Y.p);
  uint64_t *D = reinterpret_cast<uint64_t *>(base + Y.d);
  uint64_t *Z = reinterpret_cast<uint64_t *>(base + Y.z);
  int32_t *neg = reinterpret_cast<int32_t *>(base + Y.neg);
  int32_t *list = static_cast<int32_t *>(list_and_counters);
  // [0] irregular instances listed, [1] a tensor-core product gave up
  int *ctr = reinterpret_cast<int *>(static_cast<char *>(list_and_counters) +
                                     ((size_t)4 * count + 255) / 256 * 256);
  const int k = nv - 1, h = nu, L = h - k;
  const int l0 = L < 3 ? L : 3;
  const int nq = nu - nv + 1;
  Step steps[64];
  const int ns = schedule(k, h, l0, steps, 64);
  BIGINT_CUDA_TRY(cudaMemsetAsync(ctr, 0, 8, st));
  SkBuffers skb, *skp = nullptr;
  if (sk != nullptr) {
    BIGINT_CUDA_TRY(cudaMemsetAsync(sk, 0, sk_bytes, st));
    skb.bytes = sk_bytes / 2;
    skb.buf[0] = sk;
    skb.buf[1] = static_cast<char *>(sk) + skb.bytes;
    skp = &skb;
  }
  const bool few = count <= FEW;
  const int lin = few ? LIN_THREADS_FEW : LIN_THREADS;
  int rc = chain_launch(few, k_ds_start, (unsigned)((count + 127) / 128), 128, 0, st, u, v, nu, nv,
                        l0, W[0], Y.sw, count, list, ctr);
  if (rc != BIGINT_OK) return rc;
  int cur = 0;
  const unsigned gw = (unsigned)((count + WARP_CTA / 32 - 1) / (WARP_CTA / 32));
  // the leading steps whose operands are all small, fused into one launch
  SmallSteps SS;
  SS.n = small_steps(steps, ns);
  SS.N = 8;
  for (int i = 0; i < SS.n; i++) {
    SS.N = std::max(SS.N, (small_step_need(steps[i]) + 7) / 8 * 8);
    SS.s[i] = steps[i];
  }
  if (SS.n > 0) {
    const size_t smem = (size_t)8 * SMALL_STEP_WARPS * small_step_warp_limbs(SS.N);
    static bool attr = false;
    if (!attr) {
      BIGINT_CUDA_TRY(cudaFuncSetAttribute(
          k_ds_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
          8 * SMALL_STEP_WARPS * small_step_warp_limbs(SMALL_STEP_LIMBS)));
      attr = true;
    }
    rc = chain_launch(few, k_ds_small,
                      (unsigned)((count + SMALL_STEP_WARPS - 1) / SMALL_STEP_WARPS),
                      32 * SMALL_STEP_WARPS, smem, st, v, nv, W[0], W[1], Y.sw, count, SS);
    if (rc != BIGINT_OK) return rc;
    cur = SS.n & 1;
  }
  for (int i = SS.n; i < ns; i++) {
    const Step S = steps[i];
    const int nw = S.l + 2, c = step_cut(S), nl = S.t + 2 - c;
    // P = vt w mod B^(t+2) from the cut on
    rc = launch_mul_ex(v + (k - S.t), nv, W[cur], Y.sw, P, Y.sp, count, S.t + 1, nw, S.t + 2,
                       c > 0 ? c - 2 : 0, ctr + 1, st, STEP_TC_MIN, skp);
    if (rc != BIGINT_OK) return rc;
    if (nl <= WARP_LIMBS && !few)
      rc = chain_launch(few, k_ds_mid, gw, WARP_CTA, 0, st, P + c, Y.sp, D, Y.sd, nl, neg, count);
    else
      rc = chain_launch(few, k_ds_mid_cta, (unsigned)count, lin, 0, st, P + c, Y.sp, D, Y.sd, nl, neg);
    if (rc != BIGINT_OK) return rc;
    // P2 = w |d|, its limbs from s on
    const int s = S.t + S.l - S.m - c, n2 = nw + nl;
    rc = launch_mul_ex(W[cur], Y.sw, D, Y.sd, Z, Y.sz, count, nw, nl, n2, s - 2, ctr + 1, st,
                       STEP_TC_MIN, skp);
    if (rc != BIGINT_OK) return rc;
    if (S.l + S.m + 2 <= WARP_LIMBS && !few)
      rc = chain_launch(few, k_ds_update, gw, WARP_CTA, 0, st, W[cur], Y.sw, nw, Z, Y.sz, s, n2 - s,
                        neg, S.m, W[cur ^ 1], S.l + S.m + 2, count);
    else
      rc = chain_launch(few, k_ds_update_cta, (unsigned)count, lin, 0, st, W[cur], Y.sw, nw, Z, Y.sz,
                        s, n2 - s, neg, S.m, W[cur ^ 1], S.l + S.m + 2);
    if (rc != BIGINT_OK) return rc;
    cur ^= 1;
  }
  // q^ = floor(u w / B^h), w of L + 2 limbs
  const int nw = L + 2, nz = nu + nw, nqh = nz - h;
  rc = launch_mul_ex(u, nu, W[cur], Y.sw, Z, Y.sz, count, nu, nw, nz, h - 2, ctr + 1, st,
                     STEP_TC_MIN, skp);
  if (rc != BIGINT_OK) return rc;
  // R = q^ v mod B^(nv+1)
  rc = launch_mul_ex(Z + h, Y.sz, v, nv, P, Y.sp, count, nqh, nv, nv + 1, 0, ctr + 1, st,
                     STEP_TC_MIN, skp);
  if (rc != BIGINT_OK) return rc;
  rc = chain_launch(few, k_ds_finish, (unsigned)count, lin, 0, st, u, nu, v, nv, P, Y.sp, D, Y.sd,
                    Z + h, Y.sz, nqh, q, nq, r, status, ctr + 1);
  if (rc != BIGINT_OK) return rc;
  // the irregular instances: a warp each, or one CTA per division (the workspace
  // is free again: everything above is stream-ordered before this launch)
  if (list_warps_ok(nu, nv)) {
    const int64_t ctas = (count + LIST_WARPS - 1) / LIST_WARPS;
    k_ds_listed<<<(unsigned)(ctas < LIST_CTAS ? ctas : LIST_CTAS), 32 * LIST_WARPS,
                  8 * LIST_WARPS * (size_t)list_warp_limbs(nu, nv), st>>>(u, nu, v, nv, q, nq, r,
                                                                          status, list, ctr);
    return bigint_launch_status();
  }
  return launch_divmod_cta(u, v, q, r, status, count, nu, nv, ws, list, ctr, st);
}

size_t divmod_steps_workspace(int64_t count, int nu, int nv) {
  return dstep::layout(count, nu, nv).total;
}

size_t mul_sk_bytes_per_product(int na, int nb, int nout, int lo);

// Batches of at most this many divisions cut their large products over the
// SMs (split-K): a handful of divisions would otherwise run each product on
// a handful of SMs.
constexpr int64_t DIV_SK_MAX_COUNT = 16;

// Column-sum bytes the split-K products of a batch of count 2n/n-shaped
// divisions need (0 for larger batches): the largest over the products of
// the step schedule and of the tail.
size_t divmod_sk_bytes(int64_t count, int nu, int nv) {
  if (count < 1 || count > DIV_SK_MAX_COUNT || nu < nv) return 0;
  size_t per = 0;
  dstep::products(nu, nv, [&](int na, int nb, int nout, int lo) {
    per = std::max(per, mul_sk_bytes_per_product(na, nb, nout, lo));
    return true;
  });
  return 2 * (size_t)count * per;  // two buffers in turn
}

}  // namespace bigint
