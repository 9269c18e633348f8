// dc_batch_kernel.cuh -- the fused decode step on batches of short rows: one
// persistent kernel whose work item is a batch of rows, with three epilogue
// warpgroups.
//
// What bounds it: HBM for rows of a few tiles, the epilogue's arithmetic for
// rows of one. With one row per warpgroup and two warpgroups, short rows kept
// off the bandwidth (16384 rows of 411 tokens: 692 us a step, 80% of the copy
// bandwidth): (1) a row's serial parts (statistics merge, output, select: 3.7
// us) stopped the stage ring, as V tiles wait for weights and weights for the
// merged statistics; (2) the V pass is a chain of dependent arithmetic, some
// 4000 cycles a tile (clock64 stamps), which two warps a scheduler ran at a third
// of its issue rate. Here (1) the K passes of all rows of the batch run first,
// each row on one warpgroup, then all V passes, so that one row's merge or
// selection runs beside the tiles of the others; (2) three warpgroups take the
// V tiles in turn, whatever row they belong to, and a warp of its own makes the
// selections and moves. 623 us (89%; 256 rows: 19.7 -> 18.3); 641 (86%) since rows'
// sums keep whole rows' order (batch_dual). The V pass takes 1280 cycles a tile
// against 1200 of streaming; a fourth warpgroup would leave 96 registers a thread,
// and spills to an L1 that shared memory cut to 20 KB cost more than it gave (1380
// us).
//
// A row's arithmetic and its order do not depend on the batch or on the tiles'
// assignment: the statistics of a row come from one warpgroup in tile order
// (in the order of the schedule that the step had before, so that scores, and
// with them the tokens kept, are bit for bit what they were: one query head's
// softmax sum off by its last bit changed the token evicted in one row-step of
// 6000 to 25000), and the V pass works token by token.
//
// Warp roles (512 threads, 128 registers each):
//   warp 0      producer: takes items, loads each row's current, previous and
//               departing queries and their statistics (and its new pair, which
//               it appends) a row ahead of its tiles, streams K then V tiles
//               (TMA);
//   warp 1      MMA issuer (S = K Q^T, O^T += V^T P^T);
//   warp 2      policy-layer MMA issuer (Z = A W^T);
//   warp 3      mover: the one-eviction select of every row and its move;
//   warps 4-15  epilogue: row i of the batch has its K pass on warpgroup
//               i mod 3; tile j of row i has its V pass on warpgroup (i + j)
//               mod 3, and the one that gets the row's last tile also writes
//               the row's output.
//
// Barrier phases: a parity wait is sound only while its barrier can be neither
// two phases ahead of the waiter nor two behind. Every barrier has one waiter
// that waits its phases in order, and its next phase needs that waiter's
// release: what the tensor core finishes for a warpgroup is committed to the
// warpgroup's own barrier of the buffer it used (with one barrier for both S
// or both Z buffers, two tiles for one warpgroup could complete before it
// waits for the first).
//
// TMEM columns: S tiles [0, 2 NQ), O [2 NQ, 2 NQ + 64) (rows in turn; the even
// and the odd tiles of a row have an accumulator each, summed in fp32 at the
// end: the tensor core's accumulation loses a little at every tile), logits of
// heads 0..G-2 [2 NQ + 64, 256), policy layer [256, 512) (tiles in turn).
#pragma once
#include "dc_fused_kernel.cuh"

namespace dc {
namespace {

constexpr int kBatchWg = 3;                            // epilogue warpgroups
constexpr int kBatchEpi = kBatchWg * 128;
constexpr int kBatchThreads = 128 + kBatchEpi;         // 16 warps: 128 registers a thread
constexpr int kQSlots = 2;                             // query ring
constexpr int kBatchRows = 24;                         // rows of a batch at most (their statistics' slots)

// Tiles of a batch, whose logits wait on chip: heads 0..G-2 in TMEM (160
// columns with G <= 4, 128 with G = 8), head G-1 in shared memory (512 B a
// tile).
template <int G>
constexpr int batch_tiles() {
  return G == 8 ? 18 : 48;
}

template <int G>
struct BatchSmem {
  static constexpr int QBYTES = q_rows<G>() * 256;
  static constexpr int STAGE = 0;
  static constexpr int Q = STAGE + kStages * kStageBytes;
  static constexpr int P = Q + kQSlots * QBYTES;
  static constexpr int A = P + kBatchWg * 4096;                      // 128 tokens x [hi | lo] bf16 per warpgroup
  static constexpr int W = A + kBatchWg * 4096;
  static constexpr int AUX = W + 8192;
  static constexpr int SC = AUX + kStages * kAuxBytes;
  static constexpr int QST = SC + batch_tiles<G>() * kTok * 4;       // window queries' statistics: [slots][6][G] floats
  static constexpr int RST = QST + kQSlots * 6 * G * 4;              // rows' final statistics: [kBatchRows][3][G]
  static constexpr int RED = RST + kBatchRows * 3 * G * 4;           // merge scratch: [2 (row in turn)][warps x 2][G][3]
  static constexpr int CAND = RED + 2 * 8 * kBatchWg * G * 3 * 4;    // [kBatchRows][warps][4]: key, slot, position
  static constexpr int SEL = CAND + kBatchRows * 4 * kBatchWg * 16;   // select scratch per warpgroup: 288 ints
  static constexpr int MISC = (SEL + kBatchWg * 288 * 4 + 15) / 16 * 16;
  static constexpr int BYTES = MISC + 1024 + 1024;                   // misc area + alignment slack
  static_assert(BYTES <= 232448, "more shared memory than a CTA may have");
};

// barrier indices in the misc area
enum {
  C_FULL = 0, C_EMPTY = kStages, C_QFULL = 2 * kStages, C_QEMPTY = C_QFULL + kQSlots,
  C_SFULL = C_QEMPTY + kQSlots,        // [4][2] per warpgroup and buffer
  C_SEMPTY = C_SFULL + 2 * kBatchWg,   // [2] per buffer
  C_PFULL = C_SEMPTY + 2,              // [4] per warpgroup, as PEMPTY, AFULL, AEMPTY, OFULL
  C_PEMPTY = C_PFULL + kBatchWg, C_AFULL = C_PEMPTY + kBatchWg, C_AEMPTY = C_AFULL + kBatchWg,
  C_MFULL = C_AEMPTY + kBatchWg,       // [4][2] per warpgroup and buffer
  C_MEMPTY = C_MFULL + 2 * kBatchWg,   // [2] per buffer
  C_OFULL = C_MEMPTY + 2,
  C_OEMPTY = C_OFULL + kBatchWg,       // [2] per buffer
  C_CAND = C_OEMPTY + 2,               // [kBatchRows]
  C_DRAIN = C_CAND + kBatchRows, C_DRAIN2 = C_DRAIN + 1,
  C_XSTAT = C_DRAIN + 2, C_XO, C_XSEL,  // from the CTAs of a cluster: statistics, output, candidates
  C_COUNT
};

// A batch: rows [row, row + nr). The CTA's first one is its own block index
// (no round trip to the queue counter before the first load); the others come
// from the shared counter.
__device__ __forceinline__ Item take_batch(const FusedStep& fs, const Dev& p, bool first) {
  const unsigned w = first ? blockIdx.x : gridDim.x + atomicAdd(fs.work + (fs.epoch & 1u), 1u);
  const bool full = w < (unsigned)fs.batch_full;
  const int size = full ? fs.batch_rows : fs.batch_rest;
  const long long r0 = full ? (long long)w * size
                            : (long long)fs.batch_full * fs.batch_rows + (long long)(w - (unsigned)fs.batch_full) * size;
  if (r0 >= p.R) return Item{-1, 0, 0, 0};
  const int left = p.R - (int)r0;
  return Item{(int)r0, left < size ? left : size, 0, -1};
}

// HEUR, GLOB, GRAPH as in fused_kernel: a heuristic scorer instead of the
// policy; the global token mode's per-row partial sums; device-counted steps.
// CLUSTER: a row's tiles over the FusedStep::batch_cluster CTAs of a cluster,
// one row per cluster. Rank k streams and scores tiles [k nT / C, (k + 1) nT / C);
// through distributed shared memory the ranks exchange the row's softmax
// statistics between the passes (each merges them in rank order), slices of
// the output (rank k sums the k-th) and the lowest-ranked token (the last rank,
// which holds slot n - 1, moves it). Rank 0 publishes the row's query and
// statistics, once every rank has read the departing ones.
// Bound by latency: 8 rows x 2049 tokens took 23.4 us a step on one CTA each (a
// K and a V tile every 0.95 us, one after the other), 14.3 on clusters of 8: ~10
// of launch, set-up and the row's serial parts, ~2 of exchanges, two tiles a rank.
template <int D, int G, bool HEUR, bool GLOB, bool GRAPH, bool CLUSTER>
__global__ void __launch_bounds__(kBatchThreads, 1)
    batch_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                 const __grid_constant__ CUtensorMap tmK16, const __grid_constant__ CUtensorMap tmV16, Dev p, Step st,
                 FusedStep fs, FusedPolicy fp) {
  constexpr int GS = G - 1;
  constexpr int NQ = q_rows<G>();
  constexpr int kColO = 2 * NQ, kColStash = 2 * NQ + 64, kColZ = 256;
  static_assert(kColStash + GS * batch_tiles<G>() <= kColZ || GS == 0, "logits overlap the policy layer");
  static_assert(!GRAPH || (!HEUR && !GLOB), "device-counted steps: the plain step");
  static_assert(!CLUSTER || !GLOB, "rows over clusters: per-row selection");
  if constexpr (GRAPH) {
    grid_dep_wait();  // the counter is the previous launch's
    const int t = *reinterpret_cast<volatile int*>(p.gcount);
    st.p_newest += t;
    st.p_prev += t;
    st.p_dep += t;
    st.slot = (st.slot + t) % p.w;
    st.slot_prev = (st.slot_prev + t) % p.w;
    fs.epoch += (unsigned)t;
  }
  using L = BatchSmem<G>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + L::MISC);
  static_assert(8 * C_COUNT <= 640, "barriers overlap the misc fields");
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::MISC + 640);
  volatile int* abort = reinterpret_cast<volatile int*>(smem + L::MISC + 644);
  volatile int* items = reinterpret_cast<volatile int*>(smem + L::MISC + 656);  // [8][4] + seq [8]
  float* qst = reinterpret_cast<float*>(smem + L::QST);
  float* rst = reinterpret_cast<float*>(smem + L::RST);
  float* red = reinterpret_cast<float*>(smem + L::RED);

  const int warp = threadIdx.x / kWarp, lane = threadIdx.x % kWarp;
  // this CTA's tokens of a row: n from the row's token toff on
  const int csize = CLUSTER ? fs.batch_cluster : 1, crank = CLUSTER ? (int)(blockIdx.x % (unsigned)csize) : 0;
  const int tiles = (st.n + kTok - 1) / kTok, tile0 = CLUSTER ? crank * tiles / csize : 0;
  const int nT = CLUSTER ? (crank + 1) * tiles / csize - tile0 : tiles, toff = tile0 * kTok;
  const int n = CLUSTER && crank < csize - 1 ? nT * kTok : st.n - toff;
  // (rows on one CTA never use the second query slot's and the other rows'
  // candidates' memory)
  float* const xo = reinterpret_cast<float*>(smem + L::Q + L::QBYTES);                      // [csize][G D / csize]
  float* const xst = reinterpret_cast<float*>(smem + L::CAND + 1024);                       // [csize][G][3]
  unsigned* const xsel = reinterpret_cast<unsigned*>(smem + L::CAND + 2048);                // [csize][4]
  static_assert(G * D * 4 <= L::QBYTES && 8 * G * 12 <= 1024 && 2048 + 8 * 16 <= kBatchRows * 4 * kBatchWg * 16,
                "exchange areas");
  constexpr uint32_t kTileBytes = (uint32_t)D * kTok * 2;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&bar[C_FULL + s], 1);
      mbar_init(&bar[C_EMPTY + s], 5);
    }
    for (int s = 0; s < kQSlots; ++s) {
      mbar_init(&bar[C_QFULL + s], 1);
      mbar_init(&bar[C_QEMPTY + s], 5);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bar[C_SEMPTY + b], 4);
      mbar_init(&bar[C_MEMPTY + b], 4);
      mbar_init(&bar[C_OEMPTY + b], 4);
    }
    for (int w = 0; w < kBatchWg; ++w) {
      mbar_init(&bar[C_SFULL + 2 * w], 1);
      mbar_init(&bar[C_SFULL + 2 * w + 1], 1);
      mbar_init(&bar[C_PFULL + w], 4);
      mbar_init(&bar[C_PEMPTY + w], 1);
      mbar_init(&bar[C_AFULL + w], 4);
      mbar_init(&bar[C_AEMPTY + w], 1);
      mbar_init(&bar[C_MFULL + 2 * w], 1);
      mbar_init(&bar[C_MFULL + 2 * w + 1], 1);
      mbar_init(&bar[C_OFULL + w], 1);
    }
    // a row's candidates: one arrival per warp of the warpgroups with a tile of
    // it, and its last PV (no V tile of it is read after that)
    for (int s = 0; s < kBatchRows; ++s) mbar_init(&bar[C_CAND + s], 4 * (nT < kBatchWg ? nT : kBatchWg) + 1);
    mbar_init(&bar[C_DRAIN], 1);
    mbar_init(&bar[C_DRAIN2], 1);
    if constexpr (CLUSTER) {
      mbar_init(&bar[C_XSTAT], csize * G);
      mbar_init(&bar[C_XO], csize * 4);
      mbar_init(&bar[C_XSEL], csize);
    }
    *abort = 0;
    for (int e = 0; e < kItemRing; ++e) items[4 * kItemRing + e] = 0;
    fence_mbar_init();
  }
  // zero the stages, the query, weight and policy-input tiles and the
  // per-token areas (see fused_kernel), then write the policy's B operand
  for (int e = threadIdx.x; e < (L::W - L::STAGE) / 16; e += kBatchThreads)
    reinterpret_cast<uint4*>(smem + L::STAGE)[e] = make_uint4(0, 0, 0, 0);
  for (int e = threadIdx.x; e < kStages * kAuxBytes / 16; e += kBatchThreads)
    reinterpret_cast<uint4*>(smem + L::AUX)[e] = make_uint4(0, 0, 0, 0);
  if constexpr (!HEUR && !GLOB) {
    for (int e = threadIdx.x; e < 128 * 4; e += kBatchThreads) {
      const int row = e >> 2, c = e & 3;
      *reinterpret_cast<uint4*>(smem + L::W + sw64(row, c)) = reinterpret_cast<const uint4*>(fp.wtile)[row * 4 + c];
    }
  }
  fence_proxy_async();
  if (warp == 1) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  if (warp == 0 && lane == 0) {
    prefetch_tmap(&tmK);
    prefetch_tmap(&tmV);
    prefetch_tmap(&tmK16);
    prefetch_tmap(&tmV16);
  }
  grid_dep_wait();
  // the launch after this one may start its set-up (where an SM has room, at the
  // latest when a CTA leaves), one launch ahead at most
  if constexpr (!GRAPH) grid_dep_launch();
  // the next launch's queue counter (this launch uses the other one)
  if (blockIdx.x == 0 && threadIdx.x == 0) fs.work[(fs.epoch + 1u) & 1u] = 0u;
  __syncthreads();
  if constexpr (CLUSTER) cluster_sync();  // the ranks' barriers stand
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    // A row's queries are loaded into registers one row ahead of their tiles
    // (an item ahead at the end of an item), so that no tile waits for them.
    const uint64_t pol = l2_evict_first_policy();
    constexpr int QCH = G * (D / 8);                 // 16-byte chunks of a row's G query heads
    constexpr int QIT = (QCH + kWarp - 1) / kWarp;   // per lane
    uint4 qcur[QIT], qprev[QIT], qdep[QIT], kvn = make_uint4(0, 0, 0, 0);
    float4 rstat;
    constexpr int VPR = D / 8;  // 16-byte chunks of a K (or V) row
    const int sh = lane % G, sdep = lane / G;        // window statistics: lanes [0, 2G), head and query
    auto q_ok = [&](int rq) {
      return DC_INB(p, (long long)((rq / p.kvh) * p.qh + (rq % p.kvh) * G) * D + G * D - 1,
                    (long long)(p.R / p.kvh) * p.qh * D, 101) &&
             DC_INB(p, ((long long)rq * p.w + st.slot) * G * D + G * D - 1, (long long)p.R * p.w * G * D, 102) &&
             DC_INB(p, ((long long)rq * p.w + st.slot_prev) * G * D, (long long)p.R * p.w * G * D, 103);
    };
    const bool append = fs.k_new && crank == csize - 1;  // (the last rank holds slot st.n - 1)
    auto load_q = [&](int rq) {
      const uint4* cur = reinterpret_cast<const uint4*>(fs.q + ((rq / p.kvh) * p.qh + (rq % p.kvh) * G) * D);
      const uint4* prev = reinterpret_cast<const uint4*>(p.ring_q + ((size_t)rq * p.w + st.slot_prev) * G * D);
      const uint4* dep = reinterpret_cast<const uint4*>(p.ring_q + ((size_t)rq * p.w + st.slot) * G * D);
      const bool ok = q_ok(rq);
#pragma unroll
      for (int u = 0; u < QIT; ++u) {
        const int e = lane + u * kWarp;
        const bool ld = ok && e < QCH;
        qcur[u] = ld ? cur[e] : make_uint4(0, 0, 0, 0);
        qprev[u] = ld && st.has_prev ? prev[e] : make_uint4(0, 0, 0, 0);
        qdep[u] = ld && st.has_dep ? dep[e] : make_uint4(0, 0, 0, 0);
      }
      if (append && lane < 2 * VPR)
        kvn = (lane < VPR ? fs.k_new : fs.v_new)[(size_t)rq * VPR + lane % VPR];
      rstat = make_float4(0.f, 0.f, 0.f, 0.f);
      if (lane < 2 * G && ok)
        rstat = reinterpret_cast<const float4*>(p.ring_stats)[((size_t)rq * p.w + (sdep ? st.slot : st.slot_prev)) * G + sh];
    };
    // the loaded row's query tile and statistics into its slot; the current
    // query takes over the departing query's ring slot (read before)
    auto store_q = [&](int rq, int slot) {
      uint8_t* qt = smem + L::Q + slot * L::QBYTES;
      uint4* ring_slot = reinterpret_cast<uint4*>(p.ring_q + ((size_t)rq * p.w + st.slot) * G * D);
      const bool ok = q_ok(rq);
#pragma unroll
      for (int u = 0; u < QIT; ++u) {
        const int e = lane + u * kWarp;
        if (!ok || e >= QCH) continue;
        const int h = e / (D / 8), kc = e % (D / 8);
        uint8_t* qk = qt + (kc >> 3) * (NQ * 128);
        *reinterpret_cast<uint4*>(qk + sw128(h, kc & 7)) = qcur[u];
        *reinterpret_cast<uint4*>(qk + sw128(G + h, kc & 7)) = qprev[u];
        *reinterpret_cast<uint4*>(qk + sw128(2 * G + h, kc & 7)) = qdep[u];
        if constexpr (!CLUSTER) ring_slot[e] = qcur[u];
      }
      if (lane < 2 * G) {
        float* w = qst + slot * 6 * G + 3 * G * sdep;
        w[sh] = rstat.x;
        w[G + sh] = rstat.w;
        w[2 * G + sh] = rstat.z;
      }
      if (append && DC_INB(p, st.n - 1, p.cap, 301) && DC_INB(p, rq, p.R, 301)) {
        // the new pair into slot st.n - 1, with |v| and a clean state (as the append
        // kernel does it)
        const size_t at = (size_t)rq * p.stride + (st.n - 1);
        if (lane < VPR) reinterpret_cast<uint4*>(p.K)[at * VPR + lane] = kvn;
        else if (lane < 2 * VPR) reinterpret_cast<uint4*>(p.V)[at * VPR + lane - VPR] = kvn;
        const uint32_t w4[4] = {kvn.x, kvn.y, kvn.z, kvn.w};
        float ss = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float x0 = bf16lo(w4[e]), x1 = bf16hi(w4[e]);
          ss = fmaf(x0, x0, ss);
          ss = fmaf(x1, x1, ss);
        }
#pragma unroll
        for (int off = 1; off < VPR; off <<= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
        if (lane == VPR) {
          p.pos[at] = st.p_newest;
          p.vnorm[at] = sqrtf(ss);
          p.SZ[at] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (p.acc) p.acc[at] = 0.f;
        }
      }
      fence_proxy_async();
      __syncwarp();
    };
    auto take = [&](bool first) {
      int2 v = make_int2(-1, 0);
      if (lane == 0) {
        if constexpr (CLUSTER) {
          if (first) v = make_int2((int)(blockIdx.x / (unsigned)csize), 1);
        } else {
          const Item t = take_batch(fs, p, first);
          v = make_int2(t.row, t.t0);
        }
      }
      v.x = __shfl_sync(0xffffffffu, v.x, 0);
      v.y = __shfl_sync(0xffffffffu, v.y, 0);
      return v;
    };
    int g = 0, issued = 0, rs = 0;
    // one lane: K or V tiles [j0, j1) of row rt into the stage ring; false: winding down
    auto issue = [&](int rt, bool vpass, int j0, int j1) {
      const CUtensorMap* tm = vpass ? &tmV : &tmK;
      const CUtensorMap* tm16 = vpass ? &tmV16 : &tmK16;
      for (int j = j0; j < j1; ++j, ++g) {
        const int s = g % kStages;
        if (!mbar_wait(&bar[C_EMPTY + s], ((g / kStages) & 1) ^ 1, abort, p.dbg, 2u, (unsigned)g)) return false;
        const int valid = n - j * kTok < kTok ? n - j * kTok : kTok;
        const int nbox = valid < kTok ? (valid + 15) >> 4 : 0;
        const uint32_t kv_bytes = nbox ? (uint32_t)nbox * 16u * (uint32_t)D * 2u : kTileBytes;
        const uint32_t pos_bytes = ((uint32_t)valid * 4u + 15u) & ~15u, sz_bytes = (uint32_t)valid * 16u;
        const uint32_t aux_bytes = (vpass || GLOB) ? 0u : pos_bytes + sz_bytes;
        uint8_t* dst = smem + L::STAGE + s * kStageBytes;
        uint8_t* aux = smem + L::AUX + s * kAuxBytes;
        const int y = rt * p.stride + toff + j * kTok;
        issued = g + 1;
        if (!DC_INB(p, (long long)y + kTok - 1, (long long)p.R * p.stride, 104)) {
          mbar_arrive(&bar[C_FULL + s]);
          continue;
        }
        mbar_expect_tx(&bar[C_FULL + s], kv_bytes + aux_bytes);
        if (nbox == 0) {
          tma_load_2d(dst, tm, 0, y, &bar[C_FULL + s], pol);
          if (D == 128) tma_load_2d(dst + 16384, tm, 64, y, &bar[C_FULL + s], pol);
        } else {
          for (int b = 0; b < nbox; ++b) {
            tma_load_2d(dst + b * 2048, tm16, 0, y + 16 * b, &bar[C_FULL + s], pol);
            if (D == 128) tma_load_2d(dst + 16384 + b * 2048, tm16, 64, y + 16 * b, &bar[C_FULL + s], pol);
          }
        }
        if (aux_bytes) {
          bulk_load(aux + kAuxPos, p.pos + y, pos_bytes, &bar[C_FULL + s]);
          bulk_load(aux + kAuxSZ, p.SZ + y, sz_bytes, &bar[C_FULL + s]);
        }
      }
      return true;
    };
    int2 it = take(true);
    if (it.x >= 0) load_q(it.x);
    bool ok = true;
    for (int gr = 0; ok; ++gr) {
      if (lane == 0) publish_item(items, gr, Item{it.x, it.y, 0, -1});
      if (it.x < 0) break;
      for (int i = 0; i < it.y && ok; ++i, ++rs) {
        const int slot = rs % kQSlots;
        // (the warp leaves its loops together, also when the kernel winds down)
        ok = __all_sync(0xffffffffu, mbar_wait(&bar[C_QEMPTY + slot], ((rs / kQSlots) & 1) ^ 1, abort, p.dbg, 1u,
                                               (unsigned)rs));
        if (!ok) break;
        store_q(it.x + i, slot);
        if (lane == 0) mbar_arrive(&bar[C_QFULL + slot]);
        if (i + 1 < it.y) load_q(it.x + i + 1);
        // the last tile holds the new pair: its copies come after the writes of
        // it, whose latency the tiles before cover
        if (append) {
          if (elect_one()) ok = issue(it.x + i, false, 0, nT - 1);
          fence_proxy_async_global();
          __syncwarp();
          if (elect_one()) ok = ok && issue(it.x + i, false, nT - 1, nT);
        } else if (elect_one()) {
          ok = issue(it.x + i, false, 0, nT);
        }
        ok = __all_sync(0xffffffffu, ok);
      }
      if (!ok) break;
      const int2 nx = take(false);
      if (nx.x >= 0) load_q(nx.x);
      if (elect_one())
        for (int i = 0; i < it.y && ok; ++i) ok = issue(it.x + i, true, 0, nT);
      ok = __all_sync(0xffffffffu, ok);
      it = nx;
    }
    if constexpr (CLUSTER) {
      // every rank has read the departing query: the current one takes its slot
      const int rq = (int)(blockIdx.x / (unsigned)csize);
      if (crank == 0 && mbar_wait_cluster(&bar[C_XSTAT], 0, abort, p.dbg, 31u, (unsigned)rq) && q_ok(rq)) {
        uint4* ring_slot = reinterpret_cast<uint4*>(p.ring_q + ((size_t)rq * p.w + st.slot) * G * D);
#pragma unroll
        for (int u = 0; u < QIT; ++u)
          if (lane + u * kWarp < QCH) ring_slot[lane + u * kWarp] = qcur[u];
      }
      __syncwarp();
    }
    // every issued load must land before the CTA may exit
    if (elect_one())
      for (int t = issued - kStages < 0 ? 0 : issued - kStages; t < issued; ++t)
        mbar_wait_drain(&bar[C_FULL + t % kStages], (t / kStages) & 1);
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (elect_one()) {
      const uint32_t id_qk = idesc_bf16(128, NQ, 0, 0);
      const uint32_t id_pv = idesc_bf16(128, 16, 1, 1);
      const uint32_t stage_lo = sdesc_lo(smem_u32(smem + L::STAGE), 16), vstage_lo = sdesc_lo(smem_u32(smem + L::STAGE), 16384);
      const uint32_t p_lo = sdesc_lo(smem_u32(smem + L::P), 4096);
      int g = 0, gs = 0, rs = 0;
      unsigned tvp = 0;  // parity of each warpgroup's V tiles so far
      for (int gr = 0;; ++gr) {
        const Item it = read_item(items, gr, abort, p.dbg, 23u);
        if (it.row < 0) break;
        const int nr = it.t0;
        bool ok = true;
        for (int i = 0; i < nr && ok; ++i) {
          const int rq = rs + i, slot = rq % kQSlots;
          if (!(ok = mbar_wait(&bar[C_QFULL + slot], (rq / kQSlots) & 1, abort, p.dbg, 3u, (unsigned)rq))) break;
          const uint32_t qlo = sdesc_lo(smem_u32(smem + L::Q), 16) + (uint32_t)slot * (L::QBYTES >> 4);
          for (int j = 0; j < nT; ++j, ++g, ++gs) {
            const int s = g % kStages, b = gs & 1;
            if (!(ok = mbar_wait(&bar[C_FULL + s], (g / kStages) & 1, abort, p.dbg, 4u, (unsigned)g))) break;
            if (!(ok = mbar_wait(&bar[C_SEMPTY + b], ((gs >> 1) & 1) ^ 1, abort, p.dbg, 5u, (unsigned)gs))) break;
            tc_fence_after();
            const uint32_t klo = stage_lo + (uint32_t)s * (kStageBytes >> 4);
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
              const uint32_t off = (uint32_t)(ks >> 2) * 16384u + (uint32_t)(ks & 3) * 32u;
              const uint32_t qoff = (uint32_t)(ks >> 2) * (uint32_t)(NQ * 128) + (uint32_t)(ks & 3) * 32u;
              mma_bf16_lo(tmem + kColS + b * NQ, klo + (off >> 4), sdesc_hi(1024, 2), qlo + (qoff >> 4), sdesc_hi(1024, 2),
                          id_qk, ks > 0);
            }
            mma_commit(&bar[C_SFULL + 2 * (i % kBatchWg) + b]);
            mma_commit(&bar[C_EMPTY + s]);
          }
          mma_commit(&bar[C_QEMPTY + slot]);
        }
        for (int i = 0; i < nr && ok; ++i) {
          const int rq = rs + i, ob = rq & 1;
          for (int j = 0; j < nT; ++j, ++g) {
            const int s = g % kStages, w = (i + j) % kBatchWg;
            if (!(ok = mbar_wait(&bar[C_FULL + s], (g / kStages) & 1, abort, p.dbg, 13u, (unsigned)g))) break;
            // only these MMAs read a V stage: the four epilogue arrivals of the
            // stage's release are made here (its last one is the commit below)
            mbar_arrive_cnt(&bar[C_EMPTY + s], 4);
            if (!(ok = mbar_wait(&bar[C_PFULL + w], (tvp >> w) & 1, abort, p.dbg, 14u, (unsigned)g))) break;
            tvp ^= 1u << w;
            if (j == 0 && !(ok = mbar_wait(&bar[C_OEMPTY + ob], ((rq >> 1) & 1) ^ 1, abort, p.dbg, 15u, (unsigned)rq))) break;
            tc_fence_after();
            const uint32_t vlo = vstage_lo + (uint32_t)s * (kStageBytes >> 4);
            const uint32_t plo = p_lo + (uint32_t)w * (4096 >> 4);
#pragma unroll
            for (int ks = 0; ks < kTok / 16; ++ks)
              mma_bf16_lo(tmem + kColO + 32 * ob + 16 * (j & 1), vlo + ks * (2048u >> 4), sdesc_hi(1024, 2), plo + ks * (512u >> 4),
                          sdesc_hi(256, 6), id_pv, (j > 1 || ks > 0) ? 1u : 0u);
            mma_commit(&bar[C_PEMPTY + w]);
            mma_commit(&bar[C_EMPTY + s]);
            if (j == nT - 1) {
              mma_commit(&bar[C_OFULL + w]);
              mma_commit(&bar[C_CAND + i]);
            }
          }
        }
        rs += nr;
        if (!ok) break;
      }
      // all issued MMAs complete before TMEM is released
      mma_commit(&bar[C_DRAIN]);
      mbar_wait_drain(&bar[C_DRAIN], 0);
    }
    __syncwarp();
  } else if (warp == 2) {
    // ------------------------------------------------------------ policy-layer MMA issuer
    if (!HEUR && !GLOB && elect_one()) {
      const uint32_t id_m = idesc_bf16(128, 128, 0, 0);
      const uint32_t wlo = sdesc_lo(smem_u32(smem + L::W), 16), a_lo = sdesc_lo(smem_u32(smem + L::A), 16);
      unsigned gv = 0, tvp = 0;  // V tiles so far; their parity per warpgroup
      for (int gr = 0;; ++gr) {
        const Item it = read_item(items, gr, abort, p.dbg, 24u);
        if (it.row < 0) break;
        bool ok = true;
        for (int i = 0; i < it.t0 && ok; ++i) {
          for (int j = 0; j < nT; ++j, ++gv) {
            const int w = (i + j) % kBatchWg, b = (int)(gv & 1u);
            if (!(ok = mbar_wait(&bar[C_AFULL + w], (tvp >> w) & 1, abort, p.dbg, 16u, gv))) break;
            tvp ^= 1u << w;
            if (!(ok = mbar_wait(&bar[C_MEMPTY + b], ((gv >> 1) & 1) ^ 1, abort, p.dbg, 17u, gv))) break;
            tc_fence_after();
            const uint32_t alo = a_lo + (uint32_t)w * (4096 >> 4);
            // Z = [hi | lo] [W_hi | W_hi]^T + [hi | lo] [W_lo | 0]^T
#pragma unroll
            for (int ks = 0; ks < 2; ++ks)
              mma_bf16_lo(tmem + kColZ + b * 128, alo, sdesc_hi(256, 6), wlo + ks * (32u >> 4), sdesc_hi(512, 4), id_m,
                          ks > 0);
            mma_commit(&bar[C_MFULL + 2 * w + b]);
            mma_commit(&bar[C_AEMPTY + w]);
          }
        }
        if (!ok) break;
      }
      mma_commit(&bar[C_DRAIN2]);
      mbar_wait_drain(&bar[C_DRAIN2], 0);
    }
    __syncwarp();
  } else if (warp == 3) {
    // ------------------------------------------------------------ mover
    // one eviction (the steady state): slot B, the only mover, is loaded while
    // the row's V pass runs; once the row's candidates and its last PV are in,
    // their lowest-ranked token's slot takes its contents
    const unsigned* cand = reinterpret_cast<const unsigned*>(smem + L::CAND);
    const int Bsel = fs.B;
    for (int gr = 0;; ++gr) {
      int row0 = -1, nr = 0;
      if (lane == 0) {
        const Item t = read_item(items, gr, abort, p.dbg, 29u);
        row0 = t.row;
        nr = t.t0;
      }
      row0 = __shfl_sync(0xffffffffu, row0, 0);
      nr = __shfl_sync(0xffffffffu, nr, 0);
      if (named_bar_or(1, kBatchEpi + kWarp, *abort != 0 || row0 < 0)) break;
      named_bar(1, kBatchEpi + kWarp);
      for (int i = 0; !GLOB && fs.do_evict && st.n == Bsel + 1 && i < nr; ++i) {
        const int r = row0 + i;
        const size_t rbase = (size_t)r * (size_t)p.stride;
        const bool ok = crank == csize - 1 && DC_INB(p, Bsel, p.stride, 116) && DC_INB(p, (long long)rbase + Bsel, (long long)p.R * p.stride, 116);
        SlotCopy mv{};
        if (ok) slot_load_settled(p, rbase + Bsel, lane, fs.write_scores, mv);
        mbar_wait(&bar[C_CAND + i], gr & 1, abort, p.dbg, 28u, (unsigned)r);
        __syncwarp();
        if (ok) slot_load_late(p, rbase + Bsel, lane, fs.write_scores, mv);
        // warpgroup w (candidates 4 w .. 4 w + 3) has a tile of the row if one of
        // its first nT has index (w - i) mod kBatchWg; the order over the
        // candidates (lowest key, then the latest position) is total
        const unsigned* cd = cand + i * 4 * kBatchWg * 4;
        const bool in = lane < 4 * kBatchWg && ((lane >> 2) + kBatchRows * kBatchWg - i) % kBatchWg < nT;
        int cs = in ? (int)cd[lane * 4 + 1] : -1, cp = -1, fe = -1, pmax = -1;
        uint32_t ck = 0xFFFFFFFFu, kmin = 0xFFFFFFFFu;
        if (cs >= 0) {
          ck = cd[lane * 4];
          cp = (int)cd[lane * 4 + 2];
        }
        auto lowest = [&] {
          kmin = __reduce_min_sync(0xffffffffu, ck);
          pmax = __reduce_max_sync(0xffffffffu, ck == kmin ? cp : -1);
          const unsigned who = __ballot_sync(0xffffffffu, cs >= 0 && ck == kmin && cp == pmax);
          fe = who ? __shfl_sync(0xffffffffu, cs, __ffs(who) - 1) : -1;
        };
        lowest();
        if constexpr (CLUSTER) {
          // the ranks' candidates meet at the last rank, which moves; each rank
          // sends its own once its tiles have been read (C_CAND)
          if (lane == 0) {
            const uint32_t at = cluster_addr(xsel + crank * 4, (uint32_t)csize - 1);
            st_cluster(at, kmin);
            st_cluster(at + 4, (unsigned)fe);
            st_cluster(at + 8, (unsigned)pmax);
            mbar_arrive_cluster(cluster_addr(&bar[C_XSEL], (uint32_t)csize - 1));
          }
          if (!ok) continue;
          const bool all = mbar_wait_cluster(&bar[C_XSEL], 0, abort, p.dbg, 32u, (unsigned)r);
          __syncwarp();
          cs = all && lane < csize ? (int)xsel[lane * 4 + 1] : -1;
          ck = cs >= 0 ? xsel[lane * 4] : 0xFFFFFFFFu;
          cp = cs >= 0 ? (int)xsel[lane * 4 + 2] : -1;
          lowest();
        }
        if (ok && fe >= 0 && fe < Bsel && DC_INB(p, (long long)rbase + fe, (long long)p.R * p.stride, 117))
          slot_store(p, rbase + fe, lane, mv);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int ew = warp - 4, wg = ew >> 2, tw = ew & 3;   // tw: warp within the warpgroup
    const int quad = warp & 3;                            // TMEM lane quarter of this warp
    const int tok = quad * 32 + lane;                     // token (TMEM lane) within a tile
    constexpr int kTeam = 128;
    const int tid = tw * 32 + lane;                       // thread within the warpgroup
    const uint32_t lane_addr = tmem + ((uint32_t)(quad * 32) << 16);
    const float c = p.c;
    auto sync = [wg] { named_bar(2 + wg, kTeam); };
    // select scratch per warpgroup: [hist 256][sh 4][wsum 4][best 8][slots 4] ints
    int* scr_i = reinterpret_cast<int*>(smem + L::SEL) + wg * 288;
    const SelectScratch scr{scr_i, scr_i + 256, scr_i + 260,
                            reinterpret_cast<unsigned long long*>(scr_i + 264), scr_i + 272};
    unsigned* cand = reinterpret_cast<unsigned*>(smem + L::CAND);
    float* const scw = reinterpret_cast<float*>(smem + L::SC);
    const int Bsel = fs.B;
    const size_t stride = (size_t)p.stride;
    auto slot_ok = [&](int r, long long i, unsigned site) {
      return DC_INB(p, i, p.stride, site) && DC_INB(p, (long long)r * p.stride + i, (long long)p.R * p.stride, site);
    };
    int g = 0, gs = 0, rs0 = 0;
    unsigned tv = 0, ro = 0, gv = 0;  // this warpgroup's V tiles and finished rows; all V tiles
    unsigned sph = 0, zph = 0;        // parity of this warpgroup's uses of each S and each Z buffer
    for (int gr = 0;; ++gr) {
      int row0 = -1, nr = 0;
      if (lane == 0) {
        const Item t = read_item(items, gr, abort, p.dbg, 25u);
        row0 = t.row;
        nr = t.t0;
      }
      row0 = __shfl_sync(0xffffffffu, row0, 0);
      nr = __shfl_sync(0xffffffffu, nr, 0);
      // (all warpgroups: the rows' statistics, logits and scores of the batch
      // before have been read)
      tc_fence_before();
      if (named_bar_or(1, kBatchEpi + kWarp, *abort != 0 || row0 < 0)) break;
      tc_fence_after();
      // ---------------- K passes
      for (int i = wg; i < nr; i += kBatchWg) {
        const int r = row0 + i;
        const int rs = rs0 + i, slot = rs % kQSlots;
        const float* wq = qst + slot * 6 * G;
        const size_t rbase = (size_t)r * stride + toff;
        // online softmax state; with batch_dual, even and odd tiles apart, as on
        // whole rows, where each of two warpgroups takes every other tile
        float m[G], l[G], u[G], m2[G], l2[G], u2[G];
#pragma unroll
        for (int h = 0; h < G; ++h) {
          m[h] = m2[h] = kNoMax;
          l[h] = l2[h] = 0.f;
          u[h] = u2[h] = 0.f;
        }
        for (int j = 0; j < nT; ++j) {
          const int gj = g + i * nT + j, s = gj % kStages, b = (gs + i * nT + j) & 1;
          mbar_wait(&bar[C_SFULL + 2 * wg + b], (sph >> b) & 1, abort, p.dbg, 6u, (unsigned)gj);
          sph ^= 1u << b;
          if (j == 0) mbar_wait(&bar[C_QFULL + slot], (rs / kQSlots) & 1, abort, p.dbg, 27u, (unsigned)rs);
          mbar_wait(&bar[C_FULL + s], (gj / kStages) & 1, abort, p.dbg, 12u, (unsigned)gj);
          __syncwarp();
          tc_fence_after();
          float S16[NQ];  // the current, previous and departing queries' logits
          if constexpr (NQ == 32) tmem_ld32(lane_addr + kColS + b * NQ, S16);
          else tmem_ld16(lane_addr + kColS + b * NQ, S16);
          tmem_ld_wait();
          const uint8_t* aux = smem + L::AUX + s * kAuxBytes;
          const int pos = reinterpret_cast<const int*>(aux + kAuxPos)[tok];
          float4 sz = reinterpret_cast<const float4*>(aux + kAuxSZ)[tok];
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(&bar[C_SEMPTY + b]);
            mbar_arrive(&bar[C_EMPTY + s]);
          }
          const int ti = j * kTok + tok, lt = i * nT + j;
          if (ti < n) {
#pragma unroll
            for (int h = 0; h < G; ++h) {
              if (fs.batch_dual && (j & 1)) online_add(m2[h], l2[h], u2[h], S16[h], c);
              else online_add(m[h], l[h], u[h], S16[h], c);
            }
            if (!GLOB && (st.has_prev || st.has_dep)) {
              // terms of the previous and the departing query, masked (x 1 or x 0,
              // both exact) where the token was not yet in the cache at that step
              float zp, sp, zd, sd;
              window_terms<G>(S16 + G, wq, wq + G, wq + 2 * G, c, zp, sp);
              window_terms<G>(S16 + 2 * G, wq + 3 * G, wq + 4 * G, wq + 5 * G, c, zd, sd);
              const float mp = (st.has_prev && pos <= st.p_prev) ? 1.f : 0.f;
              const float md = (st.has_dep && pos <= st.p_dep) ? 1.f : 0.f;
              sz = window_update(sz, sp * mp, sd * md, zp * mp, zd * md);
              if (slot_ok(r, toff + ti, 105)) p.SZ[rbase + ti] = sz;
            }
          }
          scw[lt * kTok + tok] = S16[G - 1];
          __syncwarp();
          stash_store<GS>(lane_addr + kColStash + GS * lt, S16);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar[C_QEMPTY + slot]);
        // ---------------- row softmax statistics (deterministic merge order):
        // the maximum first, then every partial (l, u) rescaled to it and summed
        float* redp = red + ((i / kBatchWg) & 1) * 8 * kBatchWg * G * 3 + wg * 8 * G * 3;
        // (every operation rounded as written: a contracted first addition
        // would change the sums' last bits from one instantiation to another)
        auto partial = [&](const float (&pm)[G], const float (&pl)[G], const float (&pu)[G], int at) {
#pragma unroll
          for (int h = 0; h < G; ++h) {
            float mm = pm[h];
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) mm = fmaxf(mm, __shfl_xor_sync(0xffffffffu, mm, off));
            const float dm = __fmul_rn(__fsub_rn(pm[h], mm), c), f = ex2(dm);
            float ll = __fmul_rn(pl[h], f), uu = __fmul_rn(__fmaf_rn(pl[h], dm, pu[h]), f);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
              ll = __fadd_rn(ll, __shfl_xor_sync(0xffffffffu, ll, off));
              uu = __fadd_rn(uu, __shfl_xor_sync(0xffffffffu, uu, off));
            }
            if (lane == 0) {
              float* rw = redp + (at * G + h) * 3;
              rw[0] = mm;
              rw[1] = ll;
              rw[2] = uu;
            }
          }
        };
        // merged in the order of token quarters 2, 3, 0, 1; with batch_dual the
        // tiles of whole rows' warpgroup 0 first: the even ones, or on every
        // other item of a CTA with an odd tile count the odd ones
        const int flip = fs.batch_dual ? ((r / fs.batch_sms) * nT) & 1 : 0;
        partial(m, l, u, 4 * flip + (quad ^ 2));
        if (fs.batch_dual) partial(m2, l2, u2, 4 * (flip ^ 1) + (quad ^ 2));
        sync();  // (the scratch alternates between the warpgroup's rows: one barrier per row)
        // one lane per head merges the warps' partials, publishes the row's
        // statistics and pushes (m, l, H, -log2 l) into the ring slot of this
        // step (the query loader wrote the query there)
        if (tid < G) {
          const int h = tid, parts = fs.batch_dual ? 8 : 4;
          float mm = kNoMax;
#pragma unroll
          for (int w = 0; w < 8; ++w)
            if (w < parts) mm = fmaxf(mm, redp[(w * G + h) * 3 + 0]);
          float ll = 0.f, uu = 0.f;
#pragma unroll
          for (int w = 0; w < 8; ++w) {
            if (w >= parts) break;
            const float lw = redp[(w * G + h) * 3 + 1];
            const float dm = __fmul_rn(__fsub_rn(redp[(w * G + h) * 3 + 0], mm), c), f = ex2(dm);
            ll = __fmaf_rn(lw, f, ll);
            uu = __fmaf_rn(__fmaf_rn(lw, dm, redp[(w * G + h) * 3 + 2]), f, uu);
          }
          if constexpr (CLUSTER) {
            // to every rank, and the row's from all of them, in rank order
            for (int k = 0; k < csize; ++k) {
              const uint32_t at = cluster_addr(xst + (crank * G + h) * 3, (uint32_t)k);
              st_cluster(at, __float_as_uint(mm));
              st_cluster(at + 4, __float_as_uint(ll));
              st_cluster(at + 8, __float_as_uint(uu));
              mbar_arrive_cluster(cluster_addr(&bar[C_XSTAT], (uint32_t)k));
            }
            mbar_wait_cluster(&bar[C_XSTAT], 0, abort, p.dbg, 33u, (unsigned)r);
            mm = kNoMax;
            for (int k = 0; k < csize; ++k) mm = fmaxf(mm, xst[(k * G + h) * 3]);
            ll = uu = 0.f;
            for (int k = 0; k < csize; ++k) {
              const float lk = xst[(k * G + h) * 3 + 1];
              const float dm = __fmul_rn(__fsub_rn(xst[(k * G + h) * 3], mm), c), f = ex2(dm);
              ll = __fmaf_rn(lk, f, ll);
              uu = __fmaf_rn(__fmaf_rn(lk, dm, xst[(k * G + h) * 3 + 2]), f, uu);
            }
          }
          // H = ln l - ln 2 u / l
          float nl, hh;
          if (fs.batch_dual) {  // as whole rows do, from the hardware log2 and divide (l >= 1)
            const float lg = lg2_approx(ll);
            nl = -lg;
            hh = 0.69314718055994531f * (lg - __fdividef(uu, ll));
          } else {
            nl = -log2f(ll);
            hh = logf(ll) - 0.69314718055994531f * (uu / ll);
          }
          rst[(i * 3 + 0) * G + h] = mm;
          rst[(i * 3 + 1) * G + h] = nl;
          rst[(i * 3 + 2) * G + h] = hh;
          if (crank == 0 && DC_INB(p, (long long)r * p.w + st.slot, (long long)p.R * p.w, 109)) {
            reinterpret_cast<float4*>(p.ring_stats)[((size_t)r * p.w + st.slot) * G + h] = make_float4(mm, ll, hh, nl);
            p.hq[(size_t)r * G + h] = hh;
          }
        }
      }
      g += 2 * nr * nT;
      gs += nr * nT;
      if constexpr (GS > 0) tmem_st_wait();
      tc_fence_before();
      named_bar(1, kBatchEpi + kWarp);  // the rows' statistics, logits and window sums, for every warpgroup
      tc_fence_after();

      // ---------------- V passes: this warpgroup's tiles of every row; the
      // preparation of one tile overlaps the MMAs of the one before
      auto advance = [&](int& i, int& j) {  // the warpgroup's next tile; i = nr: none
        j += kBatchWg;
        while (j >= nT && i < nr) {
          ++i;
          j = (wg + kBatchRows * kBatchWg - i) % kBatchWg;
        }
      };
      // per-token state, loaded two tiles ahead: window sums, positions, |v|
      const float4 kZero4 = make_float4(0.f, 0.f, 0.f, 0.f);
      float4 szA = kZero4, szB = kZero4;
      int posA = 0, posB = 0;
      float vnA = 0.f, vnB = 0.f, acA = 0.f, acB = 0.f;
      const bool ac_ahead = HEUR && p.alpha_mode == 1;
      int fi = 0, fj = wg - kBatchWg;  // before the warpgroup's first tile
      auto fetch = [&](float4& sz, int& pos, float& vn, float& ac) {
        advance(fi, fj);
        const size_t at = (size_t)(row0 + fi) * stride + toff + fj * kTok + tok;
        if (fi < nr && DC_INB(p, (long long)at, (long long)p.R * p.stride, 107)) {
          if constexpr (!GLOB) {
            sz = p.SZ[at];
            pos = p.pos[at];
          }
          vn = p.vnorm[at];
          if (ac_ahead) ac = p.acc[at];
        }
      };
      fetch(szA, posA, vnA, acA);
      fetch(szB, posB, vnB, acB);
      const float pos_den = (float)max(st.p_newest, 1);
      auto prep = [&](int pi, int j, unsigned tvj) {
        const int r = row0 + pi, lt = pi * nT + j;
        const size_t rbase = (size_t)r * stride + toff;
        const float4 sz = szA;
        const int pos = posA;
        const float vn = vnA, ac = acA;
        szA = szB;
        posA = posB;
        vnA = vnB;
        acA = acB;
        if constexpr (HEUR || GLOB) fetch(szB, posB, vnB, acB);
        const int i = j * kTok + tok;
        const bool valid = i < n;
        const float* sr = rst + pi * 3 * G;  // M, -log2 l, H
        float sv[G];
        stash_load<GS>(lane_addr + kColStash + GS * lt, sv);
        if constexpr (GS > 0) tmem_ld_wait();
        sv[G - 1] = scw[lt * kTok + tok];
        float a[G], zc = 0.f, scur = 0.f;
#pragma unroll
        for (int h = 0; h < G; ++h) {
          a[h] = attn_weight(sv[h], sr[h], c, sr[G + h]);
          zc += a[h];
          scur = fmaf(a[h], sr[2 * G + h], scur);
        }
        // attention weights as the PV operand (see fused_kernel)
        auto put_weights = [&] {
          constexpr int NP = G == 8 ? 16 : 8;
          float pw[NP];
#pragma unroll
          for (int h = 0; h < NP; ++h) pw[h] = 0.f;
#pragma unroll
          for (int h = 0; h < G; ++h) {
            const float ah = valid ? a[h] : 0.f;
            const float hv = __bfloat162float(__float2bfloat16_rn(ah));
            pw[h] = hv;
            pw[G + h] = ah - hv;
          }
          mbar_wait(&bar[C_PEMPTY + wg], (tvj & 1) ^ 1, abort, p.dbg, 8u, tvj);
          uint8_t* prow = smem + L::P + wg * 4096 + (tok >> 3) * 256 + (tok & 7) * 32;
#pragma unroll
          for (int ck = 0; ck < NP / 8; ++ck)
            *reinterpret_cast<uint4*>(prow + ((ck ^ ((tok >> 2) & 1)) << 4)) =
                make_uint4(pack_bf16(pw[8 * ck + 0], pw[8 * ck + 1]), pack_bf16(pw[8 * ck + 2], pw[8 * ck + 3]),
                           pack_bf16(pw[8 * ck + 4], pw[8 * ck + 5]), pack_bf16(pw[8 * ck + 6], pw[8 * ck + 7]));
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bar[C_PFULL + wg]);
        };
        if constexpr (HEUR || GLOB) put_weights();
        if constexpr (GLOB) {
          // this row's share of the token's pooled sums
          if (valid && slot_ok(r, toff + i, 111)) {
            float a2 = 0.f;
#pragma unroll
            for (int h = 0; h < G; ++h) a2 = fmaf(a[h], a[h], a2);
            p.gpart[rbase + i] = make_float4(zc, a2, scur, vn);
          }
          return make_float2(0.f, 0.f);
        }
        const float mean = zc / (float)G;
        float var = 0.f;
#pragma unroll
        for (int h = 0; h < G; ++h) var = fmaf(a[h] - mean, a[h] - mean, var);
        var /= (float)G;
        const float Zt = __fadd_rn(__fadd_rn(sz.z, zc), sz.w);
        const float St = __fadd_rn(__fadd_rn(sz.x, scur), sz.y);
        float x[5] = {mean, vn, var, Zt > 0.f ? St / Zt : 0.f, (float)pos / pos_den};
        if (valid && slot_ok(r, toff + i, 112)) {
          const size_t at = rbase + i;
          if (p.alpha_mode == 1) {
            x[0] = (ac_ahead ? ac : p.acc[at]) + mean;
            p.acc[at] = x[0];
          }
          if (p.keep_features)
#pragma unroll
            for (int e = 0; e < 5; ++e) p.feat[at * 5 + e] = x[e];
        }
        if constexpr (HEUR) return make_float2(heuristic_score(p, x[0], pos, st.p_newest), __int_as_float(pos));
        // the policy layer's input row (see fused_kernel)
        float av[8];
        if (fp.layernorm) {
          const float xt[6] = {x[0], x[1], x[2], x[3], x[4], 1.f};
          float q2 = 0.f;
          int k = 0;
#pragma unroll
          for (int aa = 0; aa < 6; ++aa)
#pragma unroll
            for (int bb = aa; bb < 6; ++bb) q2 = fmaf(fp.M[k++] * xt[aa], xt[bb], q2);
          const float rn = rsqrtf(fmaxf(q2, 0.f) + 1e-5f);
#pragma unroll
          for (int e = 0; e < 6; ++e) av[e] = rn * xt[e];
          av[6] = 1.f;
          av[7] = 0.f;
        } else {
#pragma unroll
          for (int e = 0; e < 5; ++e) av[e] = x[e];
          av[5] = 1.f;
          av[6] = 0.f;
          av[7] = 0.f;
        }
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const __nv_bfloat16 h0 = __float2bfloat16_rn(av[2 * e]), h1 = __float2bfloat16_rn(av[2 * e + 1]);
          const float r0 = av[2 * e] - __bfloat162float(h0), r1 = av[2 * e + 1] - __bfloat162float(h1);
          hi[e] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
          lo[e] = pack_bf16(r0, r1);
        }
        mbar_wait(&bar[C_AEMPTY + wg], (tvj & 1) ^ 1, abort, p.dbg, 9u, tvj);
        // one 32-byte row [hi | lo] per token, 32-byte swizzle
        uint8_t* at = smem + L::A + wg * 4096 + (tok >> 3) * 256 + (tok & 7) * 32;
        const int sw = ((tok >> 2) & 1) << 4;
        *reinterpret_cast<uint4*>(at + sw) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<uint4*>(at + (sw ^ 16)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar[C_AFULL + wg]);
        // while the policy layer runs: the weights, the linear part of the score,
        // the state of the tile after next
        put_weights();
        fetch(szB, posB, vnB, acB);
        // the linear part of the score, sum_j sgn_j z_j, on the CUDA cores
        float lin = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) lin = fmaf(av[e], fp.u[e], lin);
        return make_float2(lin, __int_as_float(pos));
      };
      uint32_t ev_key = 0xFFFFFFFFu;
      int ev_slot = -1, ev_pos = -1;
      // records token j * 128 + tok's score and keeps this thread's
      // lowest-ranked token of the row so far (lower key, then later position)
      auto record = [&](int lt, int r, int j, float score, int pos) {
        const int i = j * kTok + tok;
        if (i < n && slot_ok(r, toff + i, 113)) {
          scw[lt * kTok + tok] = score;
          if (fs.write_scores) p.score[(size_t)r * stride + toff + i] = score;
          const uint32_t kk = score_key(score);
          if (ev_slot < 0 || kk < ev_key || (kk == ev_key && pos > ev_pos)) {
            ev_key = kk;
            ev_slot = toff + i;
            ev_pos = pos;
          }
        }
      };
      auto finish = [&](int lt, int r, int j, float lin, int pos) {
        const uint32_t zb = (gv + (unsigned)lt) & 1u;
        mbar_wait(&bar[C_MFULL + 2 * wg + zb], (zph >> zb) & 1, abort, p.dbg, 10u, tv);
        zph ^= 1u << zb;
        __syncwarp();
        tc_fence_after();
        // score = b2 + (lin + sum_j sgn_j |z_j|) / 2; eight independent partial sums
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c8 = 0; c8 < 2; ++c8) {
          float z2[2][32];
          tmem_ld32(lane_addr + kColZ + zb * 128 + c8 * 64, z2[0]);
          tmem_ld32(lane_addr + kColZ + zb * 128 + c8 * 64 + 32, z2[1]);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 64; ++e)
            acc[e & 7] = fmaf(fp.sgn[c8 * 64 + e], fabsf(z2[e >> 5][e & 31]), acc[e & 7]);
        }
        const float abs_sum = ((acc[0] + acc[1]) + (acc[2] + acc[3])) + ((acc[4] + acc[5]) + (acc[6] + acc[7]));
        const float relu_sum = 0.5f * (lin + abs_sum);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar[C_MEMPTY + zb]);
        record(lt, r, j, fp.b2 + relu_sum, pos);
      };
      int ci = 0, cj = wg - kBatchWg, ni, nj;
      advance(ci, cj);
      ni = ci;
      nj = cj;
      while (ci < nr) {
        advance(ni, nj);  // the tile after this one
        const float2 pf = prep(ci, cj, tv);
        {
          const int r = row0 + ci, lt = ci * nT + cj, rq = rs0 + ci;
          const bool last = cj == nT - 1;  // the row's last tile: this warpgroup finishes the row
          if constexpr (HEUR) record(lt, r, cj, pf.x, __float_as_int(pf.y));
          else if constexpr (!GLOB) finish(lt, r, cj, pf.x, __float_as_int(pf.y));
          ++tv;
          unsigned* cd = cand + ci * 4 * kBatchWg * 4;
          if (!GLOB && fs.do_evict && ni != ci) {
            // the warpgroup's last tile of the row: this warp's lowest-ranked
            // token (lowest key; among equal keys the latest position; no valid
            // key is 0xFFFFFFFF) for the mover
            const uint32_t kmin = __reduce_min_sync(0xffffffffu, ev_key);
            const bool mine = ev_key == kmin && ev_slot >= 0;
            const int pmax = __reduce_max_sync(0xffffffffu, mine ? ev_pos : -1);
            if (pmax < 0) {
              if (lane == 0) cd[ew * 4 + 1] = 0xFFFFFFFFu;  // no token of the row here
            } else if (mine && ev_pos == pmax) {
              cd[ew * 4 + 0] = ev_key;
              cd[ew * 4 + 1] = (unsigned)ev_slot;
              cd[ew * 4 + 2] = (unsigned)ev_pos;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar[C_CAND + ci]);
            ev_key = 0xFFFFFFFFu;
            ev_slot = -1;
            ev_pos = -1;
          }
          if (last) {
            // ---------------- attention output of the row
            const int ob = rq & 1;
            mbar_wait(&bar[C_OFULL + wg], ro & 1, abort, p.dbg, 11u, ro);
            ++ro;
            __syncwarp();
            tc_fence_after();
            float o16[16], odd[16];
            tmem_ld16(lane_addr + kColO + 32 * ob, o16);
            tmem_ld16(lane_addr + kColO + 32 * ob + 16, odd);  // (not written when the row has one tile)
            tmem_ld_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar[C_OEMPTY + ob]);
            if constexpr (CLUSTER) {
              // slice k of the row's outputs is rank k's to sum, in rank order
              const int sl = G * D / csize;
              if (tok < D)
#pragma unroll
                for (int h = 0; h < G; ++h) {
                  const int e = h * D + tok;
                  const float o = nT > 1 ? (o16[h] + odd[h]) + (o16[G + h] + odd[G + h]) : o16[h] + o16[G + h];
                  st_cluster(cluster_addr(xo + crank * sl + e % sl, (uint32_t)(e / sl)), __float_as_uint(o));
                }
              __syncwarp();
              if (lane < csize) mbar_arrive_cluster(cluster_addr(&bar[C_XO], (uint32_t)lane));
              const bool all = mbar_wait_cluster(&bar[C_XO], 0, abort, p.dbg, 34u, (unsigned)rq);
              __syncwarp();
              const long long o0 = (long long)((r / p.kvh) * p.qh + (r % p.kvh) * G) * D + crank * sl;
              if (all && DC_INB(p, o0 + sl - 1, (long long)(p.R / p.kvh) * p.qh * D, 115))
                for (int e = tid; e < sl; e += kTeam) {
                  float o = xo[e];
                  for (int k = 1; k < csize; ++k) o += xo[k * sl + e];
                  fs.out[o0 + e] = o;
                }
            } else if (tok < D && DC_INB(p, (long long)((r / p.kvh) * p.qh + (r % p.kvh) * G) * D + (G - 1) * D + tok,
                                  (long long)(p.R / p.kvh) * p.qh * D, 115)) {
              float* op = fs.out + ((r / p.kvh) * p.qh + (r % p.kvh) * G) * D;
#pragma unroll
              for (int h = 0; h < G; ++h)
                op[h * D + tok] = nT > 1 ? (o16[h] + odd[h]) + (o16[G + h] + odd[G + h]) : o16[h] + o16[G + h];
            }
            // ---------------- argtop_B and prune of the row: several evictions
            // here (radix select over its scores: every warp's are in), one by
            // the mover
            if (!GLOB && !CLUSTER && fs.do_evict && Bsel < n - 1) {
              mbar_wait(&bar[C_CAND + ci], gr & 1, abort, p.dbg, 30u, (unsigned)rq);
              __syncwarp();
              team_select_compact<kTeam>(p, r, n, Bsel, scw + ci * nT * kTok, tid, scr, sync);
            }
          }
        }
        ci = ni;
        cj = nj;
      }
      gv += (unsigned)(nr * nT);
      rs0 += nr;
    }
  }
  __syncthreads();
  if constexpr (CLUSTER) cluster_sync();  // no rank leaves while another may write to it
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
  if (threadIdx.x == 0 && *abort) atomicOr(p.status, kStatusTimeout);
  if constexpr (GRAPH) {
    // the last CTA to finish (every CTA has read the counter by then)
    // advances the step count for the next launch
    if (threadIdx.x == 0 && atomicAdd(p.gcount + 1, 1) == (int)gridDim.x - 1) {
      p.gcount[1] = 0;
      __threadfence();
      atomicAdd(p.gcount, 1);
    }
  }
}

template <int D, int G, bool HEUR = false, bool GLOB = false, bool GRAPH = false, bool CLUSTER = false>
static cudaError_t launch_batch_t(const FusedMaps& maps, const Dev& p, const Step& st, const FusedStep& fs,
                                  const FusedPolicy& fp, int num_sms, cudaStream_t s) {
  constexpr int kSmemBytes = BatchSmem<G>::BYTES;
  const auto kernel = batch_kernel<D, G, HEUR, GLOB, GRAPH, CLUSTER>;
  static SmemLimit limit;
  if (cudaError_t e = limit.raise(kernel, kSmemBytes); e != cudaSuccess) return e;
  const int rest = p.R - fs.batch_full * fs.batch_rows;
  const int items = fs.batch_full + (fs.batch_rest ? (rest + fs.batch_rest - 1) / fs.batch_rest : 0);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CLUSTER ? p.R * fs.batch_cluster : items < num_sms ? items : num_sms);
  cfg.blockDim = dim3(kBatchThreads);
  cfg.dynamicSmemBytes = kSmemBytes;
  cfg.stream = s;
  cudaLaunchAttribute la[2];
  cfg.attrs = la;
  if (!GRAPH) {
    la[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    la[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (CLUSTER) {
    la[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    la[cfg.numAttrs++].val.clusterDim = {(unsigned)fs.batch_cluster, 1, 1};
  }
  return cudaLaunchKernelEx(&cfg, kernel, maps.k, maps.v, maps.k16, maps.v16, p, st, fs, fp);
}

}  // namespace
}  // namespace dc
