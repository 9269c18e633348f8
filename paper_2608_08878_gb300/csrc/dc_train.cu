// dc_train.cu -- the training-side kernels of App. C: the exact log-partition
// function of the Plackett-Luce distribution over size-B subsets, and
// Gumbel-top-B sampling with the log-probability of the sampled subset.
//
// log Z(s, B, tau) = log sum over subsets a of [L], |a| = B, of
// exp(sum_{i in a} y_i), y_i = s_i / tau: the log of the elementary symmetric
// polynomial e_B(exp y_1, ..., exp y_L). For any shift u, with p_i = 1 / (1 +
// exp(-(y_i + u))) and S the sum of independent Bernoulli(p_i) variables,
//
//   e_B = P(S = B) exp(-u B) prod_i (1 + exp(y_i + u))
//
// (expand the product: the subset a has probability prod_{a} p_i prod_{not a}
// (1 - p_i)). u is chosen so that E[S] is B to a tenth of a standard deviation
// (safeguarded Newton steps on the monotone E[S], see next_shift): P(S = B) is then of the order
// of 1 / (1 + sd), and an inverse discrete Fourier transform of the
// characteristic function phi(w) = prod_i (1 - p_i + p_i e^{iw}) gives it
// (Fernandez and Williams 2010; Hong 2013):
//
//   P(S = B) = 1/N sum_{j < N} phi(2 pi j / N) e^{-2 pi i j B / N}.
//
// With N = L + 1 that is exact. It is enough that P(|S - E[S]| >= N) is below
// the result's precision (Bernstein's inequality gives N: about 8.5 sd + 20),
// and that the terms kept reach |phi|^2 <= exp(-2 sd^2 (1 - cos w)) small
// enough: at most 22 of them, whatever L and B. So O(L) work in a few passes
// where the dynamic programme over e_k costs O(L B) exponentials (64 x 4096 x
// 1024: 255 us, bound by the exponentials of 268 M terms), and a smaller error:
// nothing of the size of log Z is added up term by term in fp32.
//
// Gumbel-top-B: perturbed scores s_i / tau + g_i (g_i ~ Gumbel(0, 1), given by
// the caller), the B largest kept (ties: lower index), their indices written
// in ascending order; log pi(a) = sum_{i in a} s_i / tau - log Z.
#include <cuda_runtime.h>

#include <cmath>
#include <string>

#include "../../include/distillcache.h"
#include "dc_common.cuh"
#include "dc_select.cuh"

namespace dc {
namespace {

constexpr int kLzMaxWarps = 16;      // 512 threads, 128 for short rows
constexpr int kRowSmem = 40 * 1024;  // values of a row kept in shared memory (160 KB)
constexpr int kTopThreads = 512;
constexpr int kTopWarps = kTopThreads / kWarp;
constexpr int kTopBins = 2048;
constexpr int kTopList = kTopThreads;  // keys of the threshold bin ranked directly

// A value held as an unevaluated sum hi + lo; (hi, lo) += x (Knuth's TwoSum).
__device__ __forceinline__ void add2(float& hi, float& lo, float x) {
  const float s = __fadd_rn(hi, x), bb = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb)));
  hi = s;
}

// The warp's sum of such pairs, in lane 0's (hi, lo).
__device__ __forceinline__ void warp_add2(float& hi, float& lo) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float h = __shfl_down_sync(0xffffffffu, hi, off), l = __shfl_down_sync(0xffffffffu, lo, off);
    add2(hi, lo, h);
    lo += l;
  }
}

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  return x;
}

// The larger of two, NaN if either is.
__device__ __forceinline__ float max_nan(float a, float b) { return a != a ? a : b <= a ? a : b; }

// p = sigma(x), q = 1 - p and e = exp(-|x|), each with its own relative precision.
__device__ __forceinline__ void logistic(float x, float& p, float& q, float& e) {
  e = expf(-fabsf(x));
  const float inv = __frcp_rn(1.f + e), small = e * inv;
  p = x > 0.f ? inv : small;
  q = x > 0.f ? small : inv;
}

// The search for the shift: E[S] < B at u = lo, > B at u = hi. Where equal values
// of 1e10 and more straddle the cut (a row padded with a large negative number, B
// beyond the items before the padding), no double near the root brings E[S] to B:
// fp32 values around -u are so far apart there that E[S] varies with one of them
// alone. Then that value is split off, u = tie + v with v in [lo, hi] instead
// (64 x 4096 x 1024, 500 items of each row live and 1e16 below them: 718 us in 400
// passes without an end -> 88; rows that need no tie: 20.6, as without it).
struct Search {
  double u, lo, hi;
  float tie;  // minus that value; 0 while u is a number of its own
};

constexpr int kNewtonSteps = 64;  // only halving after these
constexpr int kMaxSteps = 200;    // (147 at most: 64, 32 halvings between fp32 numbers, 31 below 2^20, 20 of v)

// A float's bits in the order of the numbers, as a signed integer, and back.
__device__ __forceinline__ int ordered(int bits) { return bits ^ ((bits >> 31) & 0x7fffffff); }

// The next shift, from d = B - E[S] and the variance at this one.
__device__ __forceinline__ void next_shift(Search& s, int step, float d, float var) {
  if (d > 0.f) s.lo = s.u;
  else s.hi = s.u;
  // From 2^33 on fp32 numbers are at least 2^-24 |u| >= 512 apart, and E[S] differs
  // from whole numbers by 0.05 only within ln(25599 / 0.05) < 14 of one.
  const double width = s.hi - s.lo, mag = fabs(s.u);
  if (s.tie == 0.f && mag >= 8589934592.0 && width <= fmax(256.0, mag * 0x1p-32)) {
    s.tie = (float)(0.5 * (s.lo + s.hi));
    s.lo = -64.0;
    s.hi = 64.0;
    s.u = 0.0;
    return;
  }
  // a Newton step where it stays inside the bracket, else its middle, counted in
  // fp32 numbers while it is wide (the values may span many orders of magnitude)
  double nu = s.u + (double)(d / var);
  if (!(step < kNewtonSteps && nu > s.lo && nu < s.hi)) {
    nu = 0.5 * (s.lo + s.hi);
    if (width > 1048576.0) {
      const long long a = ordered(__float_as_int((float)s.lo)), b = ordered(__float_as_int((float)s.hi));
      const double m = (double)__int_as_float(ordered((int)((a + b) >> 1)));
      if (m > s.lo && m < s.hi) nu = m;
    }
  }
  s.u = nu;
}

// One CTA per row. Bound by latency: a handful of block-wide reductions over a
// row held in shared memory, in short loops (unrolled over registers, the code
// ran once per row out of a cold instruction cache: 44 us against 22, caches
// flushed, at 64 x 4096 x 1024; the dynamic programme 255).
__global__ void __launch_bounds__(kLzMaxWarps* kWarp) pl_logz_kernel(const float* __restrict__ scores, int L, int B,
                                                                     float tau, float* __restrict__ out) {
  extern __shared__ float ys[];      // y_i, then p_i (rows of up to kRowSmem)
  __shared__ float rs[kLzMaxWarps][4];
  __shared__ float2 prod[kLzMaxWarps][kWarp];
  __shared__ double sh_u;
  __shared__ float sh_uh, sh_ul, sh_var;
  __shared__ int sh_state;
  // a kernel launched after this one may start (the sampler's selection)
  grid_dep_launch();
  const int row = blockIdx.x, tid = threadIdx.x, nt = blockDim.x, lane = tid % kWarp, warp = tid / kWarp;
  const int nw = nt / kWarp;
  const float* s = scores + (size_t)row * L;
  const bool in_smem = L <= kRowSmem;
  auto y_at = [&](int i) { return in_smem ? ys[i] : __fdiv_rn(s[i], tau); };
  // ---- range, mean and count of the finite items (-infinity takes no part);
  // +infinity and NaN make the result NaN (they have no finite partition function)
  float mx = -INFINITY, mn = INFINITY, sum = 0.f, cnt = 0.f;
#pragma unroll 2
  for (int i = tid; i < L; i += nt) {
    const float y = __fdiv_rn(s[i], tau);
    if (in_smem) ys[i] = y;
    mx = max_nan(mx, y);
    if (y > -INFINITY) {
      mn = fminf(mn, y);
      sum += y;
      cnt += 1.f;
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    mx = max_nan(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, off));
    sum += __shfl_xor_sync(0xffffffffu, sum, off);
    cnt += __shfl_xor_sync(0xffffffffu, cnt, off);
  }
  if (lane == 0) {
    rs[warp][0] = mx; rs[warp][1] = mn; rs[warp][2] = sum; rs[warp][3] = cnt;
  }
  __syncthreads();
  Search srch = {0.0, 0.0, 0.0, 0.f};  // (thread 0's)
  // u in three numbers for all threads: whole, and a float part with the rest
  auto publish = [&] {
    sh_uh = srch.tie != 0.f ? srch.tie : (float)srch.u;
    sh_ul = (float)(srch.tie != 0.f ? srch.u : srch.u - (double)sh_uh);
    sh_u = (double)srch.tie + srch.u;
  };
  if (tid == 0) {
    for (int w = 1; w < nw; ++w) {
      mx = max_nan(mx, rs[w][0]);
      mn = fminf(mn, rs[w][1]);
      sum += rs[w][2];
      cnt += rs[w][3];
    }
    // 0: search; 1: fewer finite items than B; 2: exactly B; 3: not finite
    const int st = !(mx < INFINITY) ? 3 : cnt < (float)B ? 1 : cnt == (float)B ? 2 : 0;
    if (st == 0) {
      const float rest = cnt - (float)B;
      srch.lo = (double)(logf((float)B / cnt) - 1.f) - (double)mx;
      srch.hi = (double)(1.f - logf(rest / cnt)) - (double)mn;
      const double u = (double)(logf((float)B / rest) - sum / cnt);
      srch.u = u < srch.lo ? srch.lo : u > srch.hi ? srch.hi : u;
      if (u != u) srch.u = 0.5 * (srch.lo + srch.hi);  // (partial sums of both infinities)
    }
    sh_state = st;
    publish();
  }
  __syncthreads();
  const int state = sh_state;
  if (state == 1 || state == 3) {
    if (tid == 0) out[row] = state == 1 ? -INFINITY : __int_as_float(0x7fc00000);
    return;
  }
  // ---- the shift: |E[S] - B| <= sd / 10 (or 1 / 20)
  for (int step = 0; state == 0 && step < kMaxSteps; ++step) {
    const float uh = sh_uh, ul = sh_ul;
    float fp = 0.f, fv = 0.f;
#pragma unroll 4
    for (int i = tid; i < L; i += nt) {
      const float y = y_at(i);
      float p, q, e;
      logistic(__fadd_rn(__fadd_rn(y, uh), ul), p, q, e);
      if (y == -INFINITY) p = 0.f;
      fp += p;
      fv = fmaf(p, q, fv);
    }
    fp = warp_sum(fp);
    fv = warp_sum(fv);
    if (lane == 0) {
      rs[warp][0] = fp;
      rs[warp][1] = fv;
    }
    __syncthreads();
    if (warp == 0) {
      fp = warp_sum(lane < nw ? rs[lane][0] : 0.f);
      fv = warp_sum(lane < nw ? rs[lane][1] : 0.f);
      if (lane == 0) {
        const float d = (float)B - fp;
        sh_var = fv;
        if (fabsf(d) <= 0.1f * fmaxf(sqrtf(fv), 0.5f)) {
          sh_state = 4;
        } else {
          next_shift(srch, step, d, fv);
          publish();
        }
      }
    }
    __syncthreads();
    if (sh_state == 4) break;
  }
  // ---- sum_i log(1 + exp(y_i + u)) = (sum of y_i + u over the positive ones)
  // + sum_i log1p(exp(-|y_i + u|)); all items when B of them are finite: the
  // sum of the y_i. The p_i take the y_i's place.
  const float uh = sh_uh, ul = sh_ul, var = sh_var;
  float ph = 0.f, pl = 0.f, np = 0.f;
#pragma unroll 2
  for (int i = tid; i < L; i += nt) {
    const float y = y_at(i);
    float p, q, e;
    const float x = __fadd_rn(__fadd_rn(y, uh), ul);
    logistic(x, p, q, e);
    if (y == -INFINITY) p = e = 0.f;
    if (y > -INFINITY && (state == 2 || x > 0.f)) {
      add2(ph, pl, y);
      np += 1.f;
    }
    if (state == 0) add2(ph, pl, log1pf(e));
    if (in_smem) ys[i] = p;
  }
  warp_add2(ph, pl);
  np = warp_sum(np);
  if (lane == 0) {
    rs[warp][0] = ph;
    rs[warp][1] = pl;
    rs[warp][2] = np;
  }
  __syncthreads();
  double A = 0.0;
  if (warp == 0) {
    ph = lane < nw ? rs[lane][0] : 0.f;
    pl = lane < nw ? rs[lane][1] : 0.f;
    warp_add2(ph, pl);
    np = warp_sum(lane < nw ? rs[lane][2] : 0.f);
    if (!(fabsf(ph) < INFINITY)) pl = 0.f;  // past the fp32 range: infinite, not NaN
    A = (double)ph + (double)pl + (double)(np - (float)B) * sh_u;
    if (state == 2 && lane == 0) out[row] = (float)A;  // (np = B: the shift takes no part)
  }
  if (state == 2) return;
  // ---- N points, of which j = 1 .. J count (j and N - j are conjugates)
  const float a = 30.f + log1pf(sqrtf(var)), t = a * (1.f / 3.f) + sqrtf(a * a * (1.f / 9.f) + 2.f * a * var) + 3.f;
  const int N = t < (float)L ? (int)t + 1 : L + 1;
  // point j counts while 2 j <= N and 2 var sin^2(pi j / N) <= 28; lane l tests
  // point l + 1 (at most 22 count: 32 lanes hold them)
  const float sl = sinpif((float)(lane + 1) / (float)N);
  const int J = __popc(__ballot_sync(0xffffffffu, 2 * (lane + 1) <= N && 2.f * var * sl * sl <= 28.f));
  // lanes [k J, (k + 1) J) of a warp multiply up the factors of points 1 .. J
  // over the k-th part of the warp's items
  const int parts = J ? kWarp / J : 1, k = J ? lane / J : 0, j = J ? lane % J + 1 : 1;
  const float sp = sinpif((float)j / (float)N), omc = 2.f * sp * sp, sn = sinpif((float)(2 * j) / (float)N);
  float R = 1.f, I = 0.f;
  if (J > 0 && k < parts) {
    const int slot = warp * parts + k, slots = nw * parts;
    const int i0 = (int)((long long)L * slot / slots), i1 = (int)((long long)L * (slot + 1) / slots);
#pragma unroll 4
    for (int i = i0; i < i1; ++i) {
      float p;
      if (in_smem) {
        p = ys[i];
      } else {
        float q, e;
        const float y = y_at(i);
        logistic(__fadd_rn(__fadd_rn(y, uh), ul), p, q, e);
        if (y == -INFINITY) p = 0.f;
      }
      const float ar = fmaf(-p, omc, 1.f), ai = p * sn;  // 1 - p (1 - cos w) + i p sin w
      const float nR = fmaf(R, ar, -(I * ai));
      I = fmaf(R, ai, I * ar);
      R = nR;
    }
  }
  prod[warp][lane] = make_float2(R, I);
  __syncthreads();
  if (warp == 0) {
    float term = 0.f;
    if (lane < J) {
      R = 1.f;
      I = 0.f;
      for (int w = 0; w < nw; ++w)
        for (int q = 0; q < parts; ++q) {
          const float2 z = prod[w][q * J + lane];
          const float nR = R * z.x - I * z.y;
          I = R * z.y + I * z.x;
          R = nR;
        }
      // the real part of phi e^{-2 pi i j B / N}, twice for the conjugate point
      const int at = (int)((unsigned)j * (unsigned)(B % N) % (unsigned)N);
      float c, d;
      sincospif(2.f * (float)at / (float)N, &d, &c);
      term = R * c + I * d;
      if (2 * j != N) term *= 2.f;
    }
    term = warp_sum(term);
    if (lane == 0) out[row] = (float)(A + log((double)((1.f + term) / (float)N)));
  }
}

// One CTA per row: top-B of the perturbed scores by (value desc, index asc),
// indices ascending into idx[row][0..B), and sum_{i in a} s_i / tau. Order keys
// into shared memory (where the row fits) with their range; a histogram of 2048
// equal-width bins over the range; the keys of the bin that holds the B-th
// largest listed and ranked by comparing each with all of them (a few, usually;
// more than 512, as with many equal scores, take a radix select over the row);
// the kept indices placed by ballots and one prefix sum over the warps. Bound by
// the latency of these passes: 64 x 4096 x 1024 in 25 us with flushed caches (33
// by four radix passes, one thread walking the bins, and a block-wide scan per
// 512 items); beside log Z, the whole call takes 24 us warm (285).
__global__ void __launch_bounds__(kTopThreads) gumbel_topb_kernel(const float* __restrict__ scores,
                                                                  const float* __restrict__ gumbel, int L,
                                                                  int B, float tau, int* __restrict__ idx,
                                                                  float* __restrict__ logp,
                                                                  const float* __restrict__ logz) {
  extern __shared__ uint32_t skeys[];
  __shared__ int hist[kTopBins];
  __shared__ int list[kTopList];
  __shared__ int sh[4];
  __shared__ int wsum[kTopWarps];
  __shared__ unsigned long long best[kTopWarps];
  __shared__ int best_slot[kTopWarps];
  __shared__ double dsum[kTopWarps];
  const SelectScratch scr{hist, sh, wsum, best, best_slot};
  auto sync = [] { __syncthreads(); };
  const int row = blockIdx.x, tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  const float* s = scores + (size_t)row * L;
  const float* g = gumbel + (size_t)row * L;
  const bool in_smem = L <= kRowSmem;
  auto compute = [&](int i) { return score_key(__fadd_rn(__fdiv_rn(s[i], tau), g[i])); };
  for (int b = tid; b < kTopBins; b += kTopThreads) hist[b] = 0;
  if (tid == 0) sh[2] = 0;
  uint32_t kmin = 0xFFFFFFFFu, kmax = 0u;
#pragma unroll 4
  for (int i = tid; i < L; i += kTopThreads) {
    const uint32_t k = compute(i);
    if (in_smem) skeys[i] = k;
    kmin = k < kmin ? k : kmin;
    kmax = k > kmax ? k : kmax;
  }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if (lane == 0) best[warp] = ((unsigned long long)kmax << 32) | kmin;
  __syncthreads();
  kmin = __reduce_min_sync(0xffffffffu, lane < kTopWarps ? (uint32_t)best[lane] : 0xFFFFFFFFu);
  kmax = __reduce_max_sync(0xffffffffu, lane < kTopWarps ? (uint32_t)(best[lane] >> 32) : 0u);
  auto key = [&](int i) { return in_smem ? skeys[i] : compute(i); };
  const int bits = kmax > kmin ? 32 - __clz(kmax - kmin) : 0, shift = bits > 11 ? bits - 11 : 0;
  auto bin = [&](uint32_t k) { return (k - kmin) >> shift; };  // < kTopBins
#pragma unroll 2
  for (int i = tid; i < L; i += kTopThreads) atomicAdd(&hist[bin(key(i))], 1);
  __syncthreads();
  // the threshold bin: thread t holds bins kTopBins - 1 - 4 t - (0..3), so that an
  // exclusive scan over the threads counts the keys of higher bins
  int c[4], tot4 = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    c[q] = hist[kTopBins - 1 - 4 * tid - q];
    tot4 += c[q];
  }
  int all_keys;
  int before = team_exclusive_scan<kTopThreads>(tot4, tid, wsum, &all_keys, sync);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (before < B && B <= before + c[q]) {
      sh[0] = kTopBins - 1 - 4 * tid - q;
      sh[1] = before;
    }
    before += c[q];
  }
  __syncthreads();
  const uint32_t dsel = (uint32_t)sh[0];
  const int above = sh[1], m = hist[dsel], need = B - above;
  // keys above (T, cut) are kept: key > T, or key == T and index <= cut
  uint32_t T = 0;
  int cut = -1;
  if (m <= kTopList) {
#pragma unroll 2
    for (int i = tid; i < L; i += kTopThreads)
      if (bin(key(i)) == dsel) list[atomicAdd(&sh[2], 1)] = i;
    __syncthreads();
    if (tid < m) {
      const int mine = list[tid];
      const uint32_t k = key(mine);
      int rank = 0;
      for (int o = 0; o < m; ++o) {
        const uint32_t ko = key(list[o]);
        rank += ko > k || (ko == k && list[o] < mine);
      }
      if (rank == need - 1) {
        sh[0] = (int)k;
        sh[1] = mine;
      }
    }
    __syncthreads();
    T = (uint32_t)sh[0];
    cut = sh[1];
  } else {
    __syncthreads();
    auto all = [](int) { return true; };
    int gt = 0;
    T = team_radix_select_wide<kTopThreads>(L, B, key, all, tid, scr, &gt, sync);
    // the (B - gt)-th lowest index among the keys equal to T
    auto tied = [&](int i) { return key(i) == T; };
    auto ikey = [](int i) { return ~(uint32_t)i; };
    int gt2 = 0;
    cut = (int)~team_radix_select_wide<kTopThreads>(L, B - gt, ikey, tied, tid, scr, &gt2, sync);
  }
  // each warp takes a contiguous run of 32-item groups: its kept items are
  // counted, the counts prefix-summed over the warps, and a second walk writes
  // the indices
  auto kept = [&](int i) {
    if (i >= L) return false;
    const uint32_t k = key(i);
    return k > T || (k == T && i <= cut);
  };
  const int ng = (L + kWarp - 1) / kWarp;
  const int g0 = (int)((long long)ng * warp / kTopWarps), g1 = (int)((long long)ng * (warp + 1) / kTopWarps);
  int n_kept = 0;
#pragma unroll 2
  for (int gi = g0; gi < g1; ++gi) n_kept += __popc(__ballot_sync(0xffffffffu, kept(gi * kWarp + lane)));
  if (lane == 0) wsum[warp] = n_kept;
  __syncthreads();
  int base = (int)__reduce_add_sync(0xffffffffu, lane < warp ? (unsigned)wsum[lane] : 0u);
  const unsigned lt = (1u << lane) - 1u;
  double part = 0.0;
  int* dst = idx + (size_t)row * B;
#pragma unroll 2
  for (int gi = g0; gi < g1; ++gi) {
    const int i = gi * kWarp + lane;
    const bool f = kept(i);
    const unsigned mk = __ballot_sync(0xffffffffu, f);
    if (f) {
      dst[base + __popc(mk & lt)] = i;
      if (logp) part += (double)__fdiv_rn(s[i], tau);
    }
    base += __popc(mk);
  }
  if (logp) {
    // sum_{i in a} s_i / tau in double, fixed reduction order
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
    if (lane == 0) dsum[warp] = part;
    __syncthreads();
    // log Z comes from the kernel before, beside which this one may have run
    grid_dep_wait();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < kTopWarps; ++w) t += dsum[w];
      logp[row] = (float)(t - (double)*reinterpret_cast<const volatile float*>(logz + row));
    }
  }
}

// Dynamic shared memory for a row of L 4-byte values (0: the row stays in
// global memory), allowed for `kernel` on the current device when it is more
// than every kernel may have.
template <class K>
cudaError_t row_smem(K kernel, int L, size_t* bytes) {
  *bytes = L <= kRowSmem ? (size_t)L * 4 : 0;
  if (*bytes <= 32 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmem * 4);
}

thread_local std::string g_train_error;

dc_status train_fail(dc_status s, const char* msg) {
  g_train_error = msg;
  return s;
}

}  // namespace
}  // namespace dc

extern "C" const char* dc_train_last_error(void) { return dc::g_train_error.c_str(); }

extern "C" dc_status dc_pl_log_partition(const float* scores, int rows, int L, int B, float tau, float* out,
                                         void* stream) {
  using namespace dc;
  if (!scores || !out) return train_fail(DC_ERR_INVALID_ARG, "NULL pointer");
  if (rows < 1 || rows > 65535 || L < 1 || B < 1 || B > L || !(tau > 0.f))
    return train_fail(DC_ERR_INVALID_ARG, "need 1 <= rows <= 65535, 1 <= B <= L and tau > 0");
  // (the limit of an earlier kernel that kept the B + 1 polynomials in shared memory)
  if (2 * (size_t)(B + 1) * sizeof(float) > 200 * 1024) return train_fail(DC_ERR_INVALID_ARG, "B too large (at most 25599)");
  size_t smem;
  cudaError_t e = row_smem(pl_logz_kernel, L, &smem);
  if (e == cudaSuccess) {
    pl_logz_kernel<<<rows, L <= 1024 ? 128 : kLzMaxWarps * kWarp, smem, static_cast<cudaStream_t>(stream)>>>(
        scores, L, B, tau, out);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return train_fail(DC_ERR_CUDA, cudaGetErrorString(e));
  return DC_OK;
}

extern "C" dc_status dc_gumbel_top_b(const float* scores, const float* gumbel, int rows, int L, int B, float tau,
                                     int* idx, float* logp, float* logz_scratch, void* stream) {
  using namespace dc;
  if (!scores || !gumbel || !idx || (logp && !logz_scratch)) return train_fail(DC_ERR_INVALID_ARG, "NULL pointer");
  if (rows < 1 || rows > 65535 || L < 1 || B < 1 || B > L || !(tau > 0.f))
    return train_fail(DC_ERR_INVALID_ARG, "need 1 <= rows <= 65535, 1 <= B <= L and tau > 0");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (logp) {
    dc_status st = dc_pl_log_partition(scores, rows, L, B, tau, logz_scratch, stream);
    if (st != DC_OK) return st;
  }
  size_t smem;
  cudaError_t e = row_smem(gumbel_topb_kernel, L, &smem);
  // with log Z, the selection may run beside its kernel and waits for it at the end
  if (e == cudaSuccess && logp)
    e = launch_pdl(gumbel_topb_kernel, dim3(rows), dim3(kTopThreads), smem, s, scores, gumbel, L, B, tau, idx, logp,
                   (const float*)logz_scratch);
  else if (e == cudaSuccess)
    gumbel_topb_kernel<<<rows, kTopThreads, smem, s>>>(scores, gumbel, L, B, tau, idx, logp, logz_scratch);
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) return train_fail(DC_ERR_CUDA, cudaGetErrorString(e));
  return DC_OK;
}
