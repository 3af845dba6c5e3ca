// divstep.cuh -- device code of the step-batched division (divstep.cu for a
// uniform batch, ragged.cu for one of mixed shapes): the Newton start, the
// fused leading steps, the linear parts of a step and the final correction.
// The algorithm is described at the top of divstep.cu.
#pragma once
#include "divcore.cuh"

namespace bigint {
namespace dstep {
namespace {  // internal linkage: this header is included by several units

using namespace divc;

// CTA of the linear per-instance kernels: 256 threads keep every SM busy with
// several instances; a batch of fewer instances than SMs waits for one CTA's
// passes, which 1024 threads shorten (one division of 16384 by 8192 limbs:
// final correction 61 -> 20 us).
constexpr int LIN_THREADS = 256, LIN_THREADS_FEW = 1024;

// Fused leading steps: operands of at most SMALL_STEP_LIMBS limbs, i.e. up to
// 66 known limbs.  (Up to 34 only, the step from 66 as four launches: 3000
// divisions of 1024 by 512 limbs 522 us against 487, 40 of 200 by 100 limbs 66
// against 49, one of 16384 by 8192 limbs 294 against 290.)  A warp's
// shared memory holds, for steps of at most N limbs, two iterates (N each),
// the divisor's top limbs and |d| (N each) and P2 (2 N).
constexpr int SMALL_STEP_LIMBS = 136, SMALL_STEP_WARPS = 4;
__host__ __device__ constexpr int small_step_warp_limbs(int N) { return 6 * N; }

// One Newton step of an instance: l limbs of the inverse known, m new ones,
// the divisor truncated to its top t + 1 limbs.
struct Step {
  int l, m, t;
};
__host__ __device__ inline Step newton_next(int k, int L, int l) {
  Step s;
  s.l = l;
  s.m = l - 2 < L - l ? l - 2 : L - l;
  s.t = k < l + s.m + 2 ? k : l + s.m + 2;
  return s;
}

// The step's residue d = B^(t+l) - vt w is only needed from limb t - m - 2 on:
// what lies below, times w / B^s, is less than 2 / B^2 of a unit of the new
// iterate.  So vt w is a banded product from two limbs below this cut, and |d|
// starts at it: l x 2l and l x l limbs become two products of about l x l
// (4096 divisions of 1024 by 512 limbs 721 -> 675 us).  0: no cut.
__host__ __device__ inline int step_cut(Step S) {
  const int c = S.t - S.m - 2;
  return c > 2 ? c : 0;
}

// One thread: the Newton start w = floor(B^(2 l) / V), V = floor(v / B^(k-l))
// + 1, into w[0 .. l + 2) (the divisor's top limb is nonzero).
__device__ void ds_start_one(const uint64_t *v, int nv, int l, uint64_t *w) {
  const int k = nv - 1;
  if (l == 3 && start_div(v + k - 3, w)) return;
  uint64_t Vt[6] = {0, 0, 0, 0, 0, 0}, Un[8] = {0, 0, 0, 0, 0, 0, 0, 0}, Qt[8];
  for (int j = 0; j <= l; j++) Vt[j] = v[k - l + j];
  int j = 0;
  while (j <= l && ++Vt[j] == 0) j++;  // V + 1, which may carry into limb l + 1
  const int nV = j > l ? l + 2 : l + 1;
  if (j > l) Vt[l + 1] = 1;
  Un[2 * l] = 1;  // B^(2 l)
  small_div(Un, 2 * l + 1, Vt, nV, Qt);
  const int nq = 2 * l + 1 - nV + 1;
  for (int jj = 0; jj < l + 2; jj++) w[jj] = jj < nq ? Qt[jj] : 0;
}

// One warp: the step S on the iterate w (l + 2 limbs) into wn (l + m + 2),
// everything in shared memory (vt: the divisor's top t + 1 limbs, d: N limbs,
// z: 2 N).
__device__ __forceinline__ void ds_small_step(const uint64_t *vt, Step S, const uint64_t *w,
                                              uint64_t *wn, uint64_t *d, uint64_t *z) {
  const int l = S.l, m = S.m, t = S.t, nw = l + 2, c = step_cut(S), nl = t + 2 - c;
  // P = vt w mod B^(t+2) from the cut on; |d| = P (top bit clear: d <= 0) or
  // B^(t+2) - P
  warp_mul(vt, t + 1, w, nw, d, t + 2, c > 0 ? c - 1 : 0);
  d += c;
  const bool ng = (d[nl - 1] >> 63) == 0;
  if (!ng) {
    warp_addsub<true>(nl, 0u, [&](int j) { return make_ulonglong2(0ull, d[j]); },
                      [&](int j, uint64_t x) { d[j] = x; });
    __syncwarp();
  }
  // P2 = w |d| (band); w' = w B^m + floor(P2 / B^s) or w B^m - floor(P2 / B^s) - 1
  const int s = t + l - m - c, ny = nw + nl - s;
  warp_mul(w, nw, d, nl, z, nw + nl, s - 1);
  auto load = [&](int j) {
    const uint64_t x = (j >= m && j - m < nw) ? w[j - m] : 0ull;
    return make_ulonglong2(x, j < ny ? z[s + j] : 0ull);
  };
  auto store = [&](int j, uint64_t x) { wn[j] = x; };
  if (ng) warp_addsub<true>(l + m + 2, 1u, load, store);
  else warp_addsub<false>(l + m + 2, 0u, load, store);
  __syncwarp();
}

// One CTA: the sign of d from P = vt w mod B^nl and |d| (nl limbs): P itself
// if its top bit is clear (d <= 0; returns true), else B^nl - P.
__device__ __forceinline__ bool ds_mid_cta(const uint64_t *__restrict__ p,
                                           uint64_t *__restrict__ d, int nl, uint32_t *scr) {
  const bool ng = (p[nl - 1] >> 63) == 0;
  if (ng) {
    for (int j = threadIdx.x; j < nl; j += blockDim.x) d[j] = p[j];
  } else {
    blk_addsub<true>(nl, 0u, [&](int j) { return make_ulonglong2(0ull, p[j]); },
                     [&](int j, uint64_t x) { d[j] = x; }, scr);
  }
  return ng;
}

// One CTA: w' = w B^m + Y (d >= 0) or w B^m - Y - 1 (d < 0), Y (ny limbs) =
// floor(P2 / B^s), into nout limbs of the next iterate.
__device__ __forceinline__ void ds_update_cta(const uint64_t *__restrict__ w, int nw,
                                              const uint64_t *__restrict__ y, int ny, bool neg,
                                              int m, uint64_t *__restrict__ wn, int nout,
                                              uint32_t *scr) {
  auto load = [&](int j) {
    const uint64_t x = (j >= m && j - m < nw) ? w[j - m] : 0ull;
    return make_ulonglong2(x, j < ny ? y[j] : 0ull);
  };
  auto store = [&](int j, uint64_t x) { wn[j] = x; };
  if (neg) blk_addsub<true>(nout, 1u, load, store, scr);
  else blk_addsub<false>(nout, 0u, load, store, scr);
}

// The same two by one warp.
__device__ __forceinline__ bool ds_mid_warp(const uint64_t *__restrict__ p,
                                            uint64_t *__restrict__ d, int nl) {
  const bool ng = (p[nl - 1] >> 63) == 0;
  if (ng) {
    for (int j = lane_id(); j < nl; j += 32) d[j] = p[j];
  } else {
    warp_addsub<true>(nl, 0u, [&](int j) { return make_ulonglong2(0ull, p[j]); },
                      [&](int j, uint64_t x) { d[j] = x; });
  }
  return ng;
}
__device__ __forceinline__ void ds_update_warp(const uint64_t *__restrict__ w, int nw,
                                               const uint64_t *__restrict__ y, int ny, bool neg,
                                               int m, uint64_t *__restrict__ wn, int nout) {
  auto load = [&](int j) {
    const uint64_t x = (j >= m && j - m < nw) ? w[j - m] : 0ull;
    return make_ulonglong2(x, j < ny ? y[j] : 0ull);
  };
  auto store = [&](int j, uint64_t x) { wn[j] = x; };
  if (neg) warp_addsub<true>(nout, 1u, load, store);
  else warp_addsub<false>(nout, 0u, load, store);
}

// One CTA: r^ = (u - R) mod B^(nv+1) with R the low nv + 1 limbs of q^ v, the
// exact correction of q^ (nqcap limbs, in place) and r^, and the results q
// (nq limbs) and r (nv limbs).  Returns the status.
__device__ __forceinline__ int ds_finish_cta(const uint64_t *__restrict__ u, int nu,
                                             const uint64_t *__restrict__ v, int nv,
                                             const uint64_t *__restrict__ rr, uint64_t *rh,
                                             uint64_t *qh, int nqcap, uint64_t *q, int nq,
                                             uint64_t *r, uint32_t *scr) {
  {
    auto load = [&](int j) { return make_ulonglong2(j < nu ? u[j] : 0ull, rr[j]); };
    auto store = [&](int j, uint64_t x) { rh[j] = x; };
    blk_addsub<true>(nv + 1, 0u, load, store, scr);
  }
  int st = correct(v, nv, rh, qh, nqcap, scr);
  __syncthreads();
  const int pq = blk_prec(qh, nqcap, scr);
  if (pq > nq && st == BIGINT_OK) st = BIGINT_ERANGE;
  for (int j = threadIdx.x; j < nq; j += blockDim.x) q[j] = j < nqcap ? qh[j] : 0ull;
  for (int j = threadIdx.x; j < nv; j += blockDim.x) r[j] = rh[j];
  return st;
}

}  // namespace
}  // namespace dstep
}  // namespace bigint
