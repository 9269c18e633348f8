// dc_full.cu -- full-cache decode attention on CUDA cores (the comparator of
// the paper's latency table, "Full" row, on the split engine; and
// dc_attend_noalloc): split-K flash-decode of the G query heads of each row over
// all n cached tokens, with no append, no features and no eviction.
//
// What bounds it: HBM (4 D bytes per token-row, each read once), as long as the
// arithmetic stays under it: 4 G D FLOP per token-row on the fp32 pipe, kept
// there (rather than on bf16 tensor cores) so that the weights stay 32-bit
// numbers. So: no staging of tiles in shared memory and no CTA barrier in the
// loop. A warp reads K and V with 16-byte loads straight into registers, D / 8
// lanes to a token, an iteration's values and the next one's keys in flight while its
// keys are computed; the dot products run on packed pairs (fma.rn.f32x2); the partial
// sums of U tokens x G heads are reduced over a token's lanes by a
// reduce-scatter (15 shuffles for 16 sums instead of 64), which leaves one
// (token, head) logit per lane, so that no exponential is computed twice; the
// weights go back to all lanes through shared memory. The splits of a row are a
// thread-block cluster and merge through distributed shared memory: no scratch
// in global memory, no second kernel.
// 64 rows x 8192 tokens, D 128, G 4: 182 -> 55 us (40 us at the copy
// bandwidth), and a smaller error against 64 bits (4.5e-7 -> 2.8e-7).
#include "dc_common.cuh"
#include "dc_device.h"
#include "dc_kernels.h"

namespace dc {
namespace {

// Threads per CTA and CTAs per SM: 12 warps of 168 registers, or 8 of 255 where
// eight heads' queries and accumulators take 128 of them.
template <int G>
constexpr int full_threads() { return G == 8 ? 256 : 192; }
constexpr int full_ctas(int G) { return G == 8 ? 1 : 2; }

__device__ __forceinline__ uint4 ld_once(const uint4* a) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(a));
  return v;
}

// Two fp32 values in one 64-bit register, and a fused multiply-add on both.
__device__ __forceinline__ uint64_t pair(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpair(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Shape of the warp's work: L lanes to a token (8 dims each), TPW tokens at a
// time, U of them per lane and iteration.
template <int D, int G>
struct FullShape {
  static constexpr int L = D / 8, TPW = kWarp / L;
  static constexpr int U = 4;
  static constexpr int V = U * G;                      // (token, head) sums of a lane group
  static constexpr int NV = V >= L ? V / L : 1;        // of which a lane ends up with NV,
  static constexpr int DUP = V >= L ? 1 : L / V;       // or DUP lanes with the same one
  static constexpr int TB = TPW * U;                   // tokens per warp and iteration
  static_assert(NV <= G, "a lane's sums belong to one token");
  // lane bits that tell heads apart (the others tell tokens, or copies, apart)
  static constexpr bool head_bit(int off) { return off >= DUP && off < DUP * (G / NV); }
  static constexpr bool token_bit(int off) { return off >= DUP && !head_bit(off); }
};

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// A float of the shared memory of CTA `rank` of the cluster, at this CTA's address of it.
__device__ __forceinline__ float ld_peer(const float* a, int rank) {
  uint32_t at;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(at)
               : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(a))), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
  return v;
}

// grid (nsplit, R), clusters (nsplit, 1), block full_threads. Split sp of row r
// covers tokens [sp chunk, (sp + 1) chunk). Its result (maximum, denominator and
// unnormalised output of every head) stays in shared memory; every CTA of the
// cluster merges a slice of the row's outputs, in split order.
template <int D, int G>
__global__ void __launch_bounds__(full_threads<G>(), full_ctas(G))
    full_kernel(Dev p, int n, int chunk, const __nv_bfloat16* __restrict__ q, float* __restrict__ out) {
  using S = FullShape<D, G>;
  constexpr int kFullThreads = full_threads<G>(), kFullWarps = kFullThreads / kWarp;
  __shared__ __align__(16) float sp_[kFullWarps][S::TPW * S::V];   // weights [token group][token][head]
  __shared__ float sf[kFullWarps][G];                              // rescale factors
  __shared__ float sml[kFullWarps][G][2];                          // a warp's maximum and denominator
  __shared__ float so[kFullWarps][G * D];                          // and its output
  __shared__ float cml[G][2], co[G * D];                           // the split's
  const int r = blockIdx.y, split = blockIdx.x, nsplit = gridDim.x;
  const int tid = threadIdx.x, lane = tid % kWarp, warp = tid / kWarp;
  const int li = lane % S::L, grp = lane / S::L;
  const int c0 = split * chunk, c1 = min(n, c0 + chunk), len = c1 - c0;
  const float c = p.c;
  const int qo = ((r / p.kvh) * p.qh + (r % p.kvh) * G) * D;
  uint64_t q2[G][4], acc[G][4];
#pragma unroll
  for (int h = 0; h < G; ++h) {
    const __nv_bfloat16* qh = q + qo + h * D + li * 8;  // (q needs no alignment beyond its type's)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      q2[h][e] = pair(__bfloat162float(qh[2 * e]), __bfloat162float(qh[2 * e + 1]));
      acc[h][e] = 0;
    }
  }
  // this lane's sums are (token vu, heads vh ..) of its group
  const int v0 = S::V >= S::L ? li * S::NV : li / S::DUP;
  const int vu = v0 / G, vh = v0 % G;
  float m[S::NV], l[S::NV];
#pragma unroll
  for (int i = 0; i < S::NV; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
  }
  const size_t row = (size_t)r * p.stride + c0;
  const uint4* K = reinterpret_cast<const uint4*>(p.K) + row * S::L + li;
  const uint4* Vp = reinterpret_cast<const uint4*>(p.V) + row * S::L + li;
  uint4 kr[S::U];
  auto load = [&](const uint4* src, int t0, uint4 (&k)[S::U]) {
#pragma unroll
    for (int u = 0; u < S::U; ++u)  // past the end: the last token again
      k[u] = ld_once(src + (size_t)min(t0 + u * S::TPW + grp, len - 1) * S::L);
  };
  constexpr int STEP = kFullWarps * S::TB;
  int t0 = warp * S::TB;
  if (t0 < len) load(K, t0, kr);
  for (; t0 < len; t0 += STEP) {
    // this iteration's values and the next one's keys on their way
    uint4 vr[S::U], kn[S::U];
    load(Vp, t0, vr);
    const bool more = t0 + STEP < len;
    if (more) load(K, t0 + STEP, kn);
    // dot products over this lane's 8 dims
    float x[S::V];
#pragma unroll
    for (int u = 0; u < S::U; ++u) {
      const uint32_t w[4] = {kr[u].x, kr[u].y, kr[u].z, kr[u].w};
      uint64_t k2[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) k2[e] = pair(bf16lo(w[e]), bf16hi(w[e]));
#pragma unroll
      for (int h = 0; h < G; ++h) {
        uint64_t s2 = mul2(q2[h][0], k2[0]);
#pragma unroll
        for (int e = 1; e < 4; ++e) s2 = fma2(q2[h][e], k2[e], s2);
        const float2 s = unpair(s2);
        x[u * G + h] = s.x + s.y;
      }
    }
    // summed over the token's lanes: half of the sums change sides at each
    // offset, until a lane holds its own
    int cnt = S::V;
#pragma unroll
    for (int off = S::L / 2; off > 0; off >>= 1) {
      if (cnt > S::NV) {
        const int half = cnt / 2;
        const bool up = (li & off) != 0;
#pragma unroll
        for (int i = 0; i < S::V / 2; ++i)
          if (i < half) {
            const float send = up ? x[i] : x[i + half], keep = up ? x[i + half] : x[i];
            x[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
          }
        cnt = half;
      } else {
#pragma unroll
        for (int i = 0; i < S::NV; ++i) x[i] += __shfl_xor_sync(0xffffffffu, x[i], off);
      }
    }
    const bool valid = t0 + vu * S::TPW + grp < len;
    // running maximum of every head over the warp's tokens
    float mn[S::NV];
    bool grew = false;
#pragma unroll
    for (int i = 0; i < S::NV; ++i) {
      float y = valid ? x[i] : -INFINITY;
#pragma unroll
      for (int off = 1; off < kWarp; off <<= 1)
        if (S::token_bit(off)) y = fmaxf(y, __shfl_xor_sync(0xffffffffu, y, off));
      mn[i] = fmaxf(m[i], y);
      grew |= mn[i] > m[i];
    }
    if (__any_sync(0xffffffffu, grew)) {
#pragma unroll
      for (int i = 0; i < S::NV; ++i) {
        const float f = m[i] == -INFINITY ? 0.f : ex2((m[i] - mn[i]) * c);
        l[i] *= f;
        m[i] = mn[i];
        if (vu == 0 && grp == 0) sf[warp][vh + i] = f;
      }
      __syncwarp();
#pragma unroll
      for (int h = 0; h < G; ++h) {
        const float f = sf[warp][h];
        const uint64_t f2 = pair(f, f);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[h][e] = mul2(acc[h][e], f2);
      }
    }
#pragma unroll
    for (int i = 0; i < S::NV; ++i) {
      // (a logit of -infinity has weight 0, also while the maximum is -infinity;
      // a NaN, which the maximum passes over, is its weight's and the output's)
      const float w = valid && x[i] != -INFINITY ? ex2((x[i] - m[i]) * c) : 0.f;
      l[i] += w;
      sp_[warp][grp * S::V + v0 + i] = w;
    }
    __syncwarp();
    // past the end: zero values, as a weight of 0 makes NaN of an infinity
    if (t0 + S::TB > len) {
#pragma unroll
      for (int u = 0; u < S::U; ++u)
        if (t0 + u * S::TPW + grp >= len) vr[u] = make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int u = 0; u < S::U; ++u) {
      const float* pw = &sp_[warp][grp * S::V + u * G];
      float w[G];
      if constexpr (G % 4 == 0) {
#pragma unroll
        for (int h = 0; h < G; h += 4) {
          const float4 f = *reinterpret_cast<const float4*>(pw + h);
          w[h] = f.x; w[h + 1] = f.y; w[h + 2] = f.z; w[h + 3] = f.w;
        }
      } else {
#pragma unroll
        for (int h = 0; h < G; ++h) w[h] = pw[h];
      }
      const uint32_t b[4] = {vr[u].x, vr[u].y, vr[u].z, vr[u].w};
      uint64_t b2[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) b2[e] = pair(bf16lo(b[e]), bf16hi(b[e]));
#pragma unroll
      for (int h = 0; h < G; ++h) {
        const uint64_t w2 = pair(w[h], w[h]);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[h][e] = fma2(w2, b2[e], acc[h][e]);
      }
    }
    __syncwarp();  // the weights have been read
    if (more) {
#pragma unroll
      for (int u = 0; u < S::U; ++u) kr[u] = kn[u];
    }
  }
  // the warp's denominator and output, summed over its tokens
#pragma unroll
  for (int i = 0; i < S::NV; ++i) {
#pragma unroll
    for (int off = 1; off < kWarp; off <<= 1)
      if (S::token_bit(off)) l[i] += __shfl_xor_sync(0xffffffffu, l[i], off);
    if (vu == 0 && grp == 0) {
      sml[warp][vh + i][0] = m[i];
      sml[warp][vh + i][1] = l[i];
    }
  }
#pragma unroll
  for (int h = 0; h < G; ++h)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float2 o = unpair(acc[h][e]);
#pragma unroll
      for (int off = S::L; off < kWarp; off <<= 1) {
        o.x += __shfl_xor_sync(0xffffffffu, o.x, off);
        o.y += __shfl_xor_sync(0xffffffffu, o.y, off);
      }
      if (grp == 0) *reinterpret_cast<float2*>(&so[warp][h * D + li * 8 + 2 * e]) = o;
    }
  __syncthreads();
  // the split's result over its warps. A maximum of -infinity (no tokens, or no
  // logit that is a number above it) counts 0 times: sums of 0 add nothing, NaN stays
  for (int e = tid; e < G * D; e += kFullThreads) {
    const int h = e / D;
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < kFullWarps; ++w) M = fmaxf(M, sml[w][h][0]);
    float num = 0.f, den = 0.f;
#pragma unroll
    for (int w = 0; w < kFullWarps; ++w) {
      const float f = sml[w][h][0] == -INFINITY ? 0.f : ex2((sml[w][h][0] - M) * c);
      den += sml[w][h][1] * f;
      num += so[w][e] * f;
    }
    if (nsplit == 1) {
      out[qo + e] = num / den;
    } else {
      co[e] = num;
      if (e % D == 0) {
        cml[h][0] = M;
        cml[h][1] = den;
      }
    }
  }
  if (nsplit == 1) return;
  cluster_sync();
  for (int e = split * kFullThreads + tid; e < G * D; e += nsplit * kFullThreads) {
    const int h = e / D;
    float M = -INFINITY;
    for (int s = 0; s < nsplit; ++s) M = fmaxf(M, ld_peer(&cml[h][0], s));
    float num = 0.f, den = 0.f;
    for (int s = 0; s < nsplit; ++s) {
      const float ms = ld_peer(&cml[h][0], s);
      const float f = ms == -INFINITY ? 0.f : ex2((ms - M) * c);
      den += ld_peer(&cml[h][1], s) * f;
      num += ld_peer(&co[e], s) * f;
    }
    out[qo + e] = num / den;
  }
  cluster_sync();  // no CTA leaves while its shared memory is read
}

// Splits per row = CTAs per cluster, 1 to 16 (above 8 where the device can place
// such clusters). A cluster sits within one group of SMs, so fewer fit at once
// than CTAs would (42 clusters of 7 do not: 42 x 11793 tokens took 90 us, 58 with
// 6); the device is asked how many of each size are resident, and the size
// with the least estimated time is taken: waves x (a split's tokens at an even
// share of the bandwidth + 3 us of launch, merge and exit). A split has at least
// 128 tokens.
constexpr int kMaxSplits = 16;

template <int D, int G>
void full_t(const Dev& p, int n, int num_sms, const void* q, float* out, cudaStream_t s) {
  const auto kernel = full_kernel<D, G>;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(full_threads<G>());
  cfg.stream = s;
  cudaLaunchAttribute la[1];
  la[0].id = cudaLaunchAttributeClusterDimension;
  cfg.attrs = la;
  cfg.numAttrs = 1;
  // resident clusters of each size, asked once per device
  struct Counts {
    int of[kMaxSplits + 1];
  };
  static PerDevice<Counts> resident;
  const Counts active = resident.get([&] {
    Counts r = {};
    const bool large = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    for (int k = 1; k <= kMaxSplits; ++k) {
      int m = 0;
      cfg.gridDim = dim3(k);
      la[0].val.clusterDim = {(unsigned)k, 1, 1};
      if ((k > 8 && !large) || cudaOccupancyMaxActiveClusters(&m, kernel, &cfg) != cudaSuccess) m = 0;
      r.of[k] = m;
    }
    cudaGetLastError();  // a size that the device refuses is not used
    if (r.of[1] == 0) r.of[1] = full_ctas(G) * num_sms;
    return r;
  });
  const int tiles = (n + 127) / 128;
  // ns per token of a CTA at its share of the bandwidth
  const double token_ns = 4.0 * D * full_ctas(G) * num_sms / 6787.0;
  int nsplit = 1, chunk = tiles * 128;
  double best = 0.0;
  for (int k = 1; k <= kMaxSplits && k <= tiles; ++k) {
    if (active.of[k] == 0) continue;
    const int c = (tiles + k - 1) / k * 128, waves = (p.R + active.of[k] - 1) / active.of[k];
    const double t = waves * (token_ns * c + 3000.0);
    if (best == 0.0 || t < best) {
      best = t;
      nsplit = (n + c - 1) / c;
      chunk = c;
    }
  }
  cfg.gridDim = dim3(nsplit, p.R);
  la[0].val.clusterDim = {(unsigned)nsplit, 1, 1};
  cudaLaunchKernelEx(&cfg, kernel, p, n, chunk, (const __nv_bfloat16*)q, out);
}

}  // namespace

bool launch_full_decode(const Dev& p, int n, int num_sms, const void* q, float* out, cudaStream_t s) {
#define DC_CASE(D_, G_) \
  if (p.d == D_ && p.G == G_) { full_t<D_, G_>(p, n, num_sms, q, out, s); return true; }
  DC_CASE(64, 1) DC_CASE(64, 2) DC_CASE(64, 4) DC_CASE(64, 8)
  DC_CASE(128, 1) DC_CASE(128, 2) DC_CASE(128, 4) DC_CASE(128, 8)
#undef DC_CASE
  return false;
}

}  // namespace dc
