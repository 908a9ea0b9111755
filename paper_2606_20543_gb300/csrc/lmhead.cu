// lmhead.cu — fused lm_head + acceptance (step a6).  Sec. 3.3, after Eq. 2:
// draft tokens are decoded through the base model's GenHead, a linear map
// from the (normalised) hidden state to vocabulary logits.  Verification
// needs it for the target hidden states H_t and the draft hidden states H_d:
//   l_p = H_t W_t,  l_q = H_d W_d   ([rows x K] x [K x V])
// followed by strategy (C) of Sec. 3.3 on every row (accept with probability
// min(p/q, 1), otherwise draw from [p - q]_+), exactly as accept.cu, but
// with the logits never written to memory.
//
// Design (GB300, tcgen05 + TMEM):
//  * one CTA per tile of 128 vocabulary entries, above 128 rows a pair of CTAs
//    (cta_group::2) per two tiles; draft rows on the MMA's M
//    dimension (TMEM lanes, padded to 128 per CTA), vocabulary on N, so
//    each epilogue thread owns 32 of one row's 128 logits of the tile;
//  * A = hidden states (K-major), B = weights (MN-major: the vocabulary is
//    contiguous in W[K][V]); both staged by TMA with the 128-byte swizzle
//    through an mbarrier ring of units of 64 or 128 K of one head, two warps
//    producing (hidden states; weights; one copy each per unit), one thread
//    issuing tcgen05.mma (bf16 x bf16 -> fp32) into two TMEM accumulators
//    (target, draft), tcgen05.commit releasing each stage;
//  * epilogue: tcgen05.ld of each row's tile, per-tile softmax partials to a
//    small workspace, a bounded grid barrier (the launch is cooperative, so
//    every CTA is resident), a warp-parallel combine of each row's partials
//    in a fixed order by one CTA (row r by CTA r mod the grid), which takes
//    the decision and publishes the row's normalisers; a second barrier; the
//    rows to draw (every rejected row, or, inside a one-round prefix-commit
//    step, only each sequence's first rejection: the one token the commit
//    keeps), their per-tile residual masses, a third barrier, and the CTA
//    holding the CDF crossing scans the chunk of 32 that holds it.  Logits stay
//    in TMEM throughout.
// Bound: the weights' bytes (each read once) in the main loop, then a chain of
// three grid barriers, each followed by one cold pass over a little code: 48 rows x
// 16384 x 4096 take 53.4 us (256 rows 69), 36 of them the loop (7.4 TB/s), 1.4 the
// partials, 2 to 4 each the combine, the masses and the search with their barriers,
// and 5 the launches.  Small rolled code over all 16 warps took the chain after the
// loop from 25 to 12 us.
#include "kernels.cuh"

namespace ssd {

namespace {

constexpr int kBM = 128;        // rows per MMA tile (TMEM lanes)
constexpr int kBN = 128;        // vocabulary entries per CTA
constexpr int kBK = 64;         // K of one 128-byte swizzle atom of bf16
constexpr int kMMAK = 16;       // K per tcgen05.mma (kind::f16)
constexpr int kThreadsL = 512;  // 16 warps: 4 TMEM lane quarters x 4 column chunks of a tile
constexpr int kCombWarps = kThreadsL / 32;
constexpr int kChunk = kBN / (kCombWarps / 4);  // columns of a tile per warp in the epilogues
constexpr int kMaxTilesPerLane = 8;  // vocabulary tiles per lane in the combines: V <= 32768
constexpr int kMaxRows = 2 * kBM;
constexpr size_t kMaxSmem = 232448;  // 227 KB
constexpr float kLog2eL = 1.4426950408889634f;
constexpr float kLn2L = 0.6931471805599453f;


struct LmPartial {  // one row, one vocabulary tile (32 bytes)
  float max_p, sum_p, max_q, sum_q;
  float xq_c, xp_c;  // logits at the tile's candidate (argmax of q, or the given token)
  int32_t cand;      // candidate index, -1 if none
  float pad;
};

// Instruction descriptors, kind::f16: fp32 D, bf16 A and B, A K-major,
// B MN-major; N = M = 128 in one CTA, 256 over a pair.
constexpr uint32_t kIdesc = idesc_bf16(kBM, kBN, false, true);
constexpr uint32_t kIdescPair = idesc_bf16(2 * kBM, 2 * kBN, false, true);

__device__ __forceinline__ bool better(float v, int32_t i, float bv, int32_t bi) {
  return v > bv || (v == bv && (uint32_t)i < (uint32_t)bi);
}

__device__ __forceinline__ void merge_ms(float& m, float& s, float m2, float s2, float c) {
  const float mn = fmaxf(m, m2);
  if (mn == -INFINITY) return;
  s = s * ex2_approx((m - mn) * c) + s2 * ex2_approx((m2 - mn) * c);
  m = mn;
}

__device__ __forceinline__ uint32_t ld_acquire(const unsigned int* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Bounded grid barrier over `ncta` co-resident CTAs (cooperative launch).
// *ctr counts arrivals over the kernel's barriers (cumulative targets) in its low 31
// bits; the top bit aborts the kernel: a CTA that gave up, here (after max_polls
// polls, SSD_ERR_TIMEOUT recorded) or before (good false: its partials are missing),
// raises it and arrives nowhere any more, so that no CTA goes on with missing
// partials.  (One word, so that a wait ends with the load that sees the count: a flag
// read after it cost ~0.6 us per barrier.)
// Returns false in every thread if this CTA gave up or the kernel was aborted.
constexpr unsigned int kAbort = 0x80000000u;
__device__ __noinline__ bool grid_barrier(unsigned int* ctr, unsigned int target, int32_t* status,
                             int32_t* flag, uint32_t max_polls, bool good) {
  __syncthreads();
  if (threadIdx.x == 0) {
    // (a release and an acquire, ordered with the block by its barriers, instead of
    // two full fences: ~1 us per grid barrier)
    if (good) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr) : "memory");
    else atomicOr(ctr, kAbort);
    bool ok = false, aborted = !good;
#pragma unroll 1
    for (uint32_t i = 0; i < max_polls && !ok && !aborted; ++i) {
      const uint32_t v = ld_acquire(ctr);
      aborted = (v & kAbort) != 0;
      ok = !aborted && v >= target;
      if (i > 256) __nanosleep(64);
    }
    if (!ok && !aborted) {
      atomicOr(ctr, kAbort);
      record_status(status, SSD_ERR_TIMEOUT);
    }
    *flag = ok ? 1 : 0;
  }
  __syncthreads();
  return *flag != 0;
}

// The 128 threads of one TMEM lane quarter (4 warps).
__device__ __forceinline__ void quarter_sync(int quarter) {
  asm volatile("bar.sync %0, 128;" ::"r"(quarter + 1) : "memory");
}

struct LmSmemRow {  // per-row results of the decision, broadcast inside the CTA
  float Cp, Cq;     // log2-domain normalisers max * c + log2(sum)
  float u_res;
  int32_t state;    // 0 skip (padding / accepted / invalid), 1 rejected: draw
  int32_t cstar;    // CTA holding the crossing for this row, -1 none
  float tc;         // remaining target inside that CTA's tile (INF: last positive)
  int32_t from_p;   // 1: zero residual mass, draw from p
  int32_t pad;
};

struct LmRowRec {   // one row's combine, for every CTA after the second barrier
  float Cp, Cq, u_res;
  int32_t state;    // 0: padding or accepted, 1: rejected (a draw candidate), 2: no draft token
};

struct LmLaunch {
  int32_t tiles, stages;   // vocabulary tiles; ring stages
  int32_t ku;           // K per stage (64 or 128)
  int32_t rpad;         // staged rows of a CTA: its rows in swizzle groups of 8
  LmPartial* part;      // [rows][tiles]
  float* mass;          // [rows][tiles]
  LmRowRec* rec;        // [rows] each row's decision, written by the CTA that combined it
  unsigned int* barrier;
  uint32_t max_polls;   // limit of every bounded wait of the kernel
  uint32_t shortfall;   // extra arrivals each grid barrier waits for (0; > 0 in tests)
};

// PAIR: rows above 128.  Two CTAs (a cluster) share two vocabulary tiles: each
// stages half of the rows and one tile of weights, the pair's MMAs (M = N = 256)
// read both CTAs' halves, and each CTA ends up with its rows' logits of both
// tiles.  A CTA staging all rows itself was bound by what an SM takes in: 240 rows
// and 128 columns bring 47 KB per 64 K, 49 us of copies at 64 B per clock for 4096 K
// of both heads, a pair 32 KB per CTA (256 rows x 16384 x 4096 84.9 -> 69.6 us, 136
// rows x 8192 x 1024 39.3 -> 34.8).
template <bool PAIR>
__global__ void __launch_bounds__(kThreadsL, 1)
lmhead_accept_kernel(const __grid_constant__ CUtensorMap tmHt, const __grid_constant__ CUtensorMap tmHd,
                     const __grid_constant__ CUtensorMap tmWt, const __grid_constant__ CUtensorMap tmWd,
                     LmHeadArgs a, LmLaunch L) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  if (a.early_dependents) pdl_launch_dependents();
  constexpr int kTiles = PAIR ? 2 : 1;  // vocabulary tiles with accumulators in this CTA
  const int S = L.stages;
  const int a_bytes = L.rpad * L.ku * 2, w_bytes = L.ku * kBN * 2;
  const int stage_bytes = a_bytes + w_bytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S * stage_bytes);
  uint64_t* empty = full + S;
  uint64_t* done = empty + S;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  int32_t* flag = reinterpret_cast<int32_t*>(tmem_slot + 1);
  int32_t* fail = flag + 1;
  LmSmemRow* rowinfo = reinterpret_cast<LmSmemRow*>(fail + 2);  // [128]: this CTA's rows

  const int tid = threadIdx.x, lane = tid & 31, warp = (int)warp_uniform(tid >> 5);
  const int cta = blockIdx.x, ncta = gridDim.x;
  const int rank = PAIR ? cta & 1 : 0;
  const int tile0 = cta - rank;              // the tiles of its accumulators: tile0, ...
  const int32_t row0 = rank * L.rpad;        // its rows: row0 .. row0 + nrows - 1
  const int32_t nrows = PAIR ? max(min(L.rpad, a.rows - row0), 0) : a.rows;
  // ring units: K step u / 2 of the target (even u) or draft head
  const int32_t nunits = 2 * (a.K / L.ku);
  constexpr uint32_t ncols = (uint32_t)(kTiles * 2 * kBN);  // target + draft accumulators

  // ---- set-up: barriers, TMEM
  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 2);  // the weight and the hidden-state producer
      mbar_init(&empty[s], 1);
    }
    mbar_init(done, 1);
    *fail = 0;
    fence_barrier_init();
  }
  if (warp == 0) {
    if constexpr (PAIR) {
      tmem_alloc_pair(tmem_slot, ncols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(tmem_slot, ncols);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  if constexpr (PAIR) cluster_sync_all();  // (the peer's barriers too are initialised)
  else __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // ---- main loop: warp 0 copies the weights, warp 2 the hidden states, warp 1
  // issues the MMAs (one elected lane of each, in warp-uniform loops); the other
  // threads wait at the block's barrier (not polling beside them).  A warp issues
  // a copy every ~0.3 us, so a unit of one head takes two copies of up to 32 KB,
  // from two warps.
  int issued = 0;  // units that this warp copied
  if (warp == 0 || warp == 2) {
    const bool w = warp == 0, leader = elect_one();
    const uint64_t pol = w ? policy_evict_first()   // weights: read once
                           : policy_evict_last();   // hidden states: read by every CTA
    int s = 0, u = 0;
    uint32_t ph = 1;
    // a pair's bytes are counted by its even CTA's barriers
    const uint32_t full0 = PAIR ? peer_addr(smem_u32(full), 0) : 0;
#pragma unroll 1
    for (; u < nunits; ++u) {
      const int k0 = (u >> 1) * L.ku;
      if (u >= S && !mbar_wait_warp(&empty[s], ph, a.status, L.max_polls)) {
        *fail = 1;
        break;
      }
      if (leader) {
        unsigned char* st = smem + s * stage_bytes;
        // weights: 3D view {64, K, V / 64}; hidden states: {64, rows, K / 64}
        const CUtensorMap* map = w ? ((u & 1) ? &tmWd : &tmWt) : ((u & 1) ? &tmHd : &tmHt);
        unsigned char* dst = w ? st + a_bytes : st;
        const int32_t c1 = w ? k0 : row0, c2 = w ? cta * (kBN / 64) : k0 / kBK;
        if (rank == 0)
          mbar_arrive_expect_tx(&full[s], (uint32_t)(kTiles * (w ? w_bytes : a_bytes)));
        if constexpr (PAIR) tma_load_3d_pair(dst, map, 0, c1, c2, full0 + 8 * s, pol);
        else tma_load_3d(dst, map, 0, c1, c2, &full[s], pol);
      }
      __syncwarp();
      if (++s == S) {
        s = 0;
        ph ^= 1u;
      }
    }
    issued = u;
  } else if (warp == 1 && rank == 0) {
    const uint32_t base = warp_uniform(smem_u32(smem)), tm = warp_uniform(tmem);
    const bool leader = elect_one();
    int s = 0;
    uint32_t ph = 0;
    bool good = true;
#pragma unroll 1
    for (int u = 0; u < nunits && good; ++u) {
      good = mbar_wait_warp(&full[s], ph, a.status, L.max_polls);
      if (!good) break;
      tc_fence_after();
      const uint32_t st = base + s * stage_bytes;
      // B (MN-major): 64-wide vocabulary atoms ku * 128 bytes apart (LBO), 8-row K
      // groups 1 KB apart (SBO); one MMA's K = 16 rows = 2 KB further per step.
      // A (K-major): 8-row groups 1 KB apart (SBO); K = 16 is 32 bytes along the
      // row, 64 K a [rpad][128 B] block.  (A row tile is read to 128 rows, past
      // the staged ones: those rows of the accumulators are never used.)
      const uint64_t db0 = smem_desc(st + a_bytes, L.ku * 128, 1024), da0 = smem_desc(st, 16, 1024);
      const uint32_t d = tm + (u & 1) * (kTiles * kBN);
      const uint32_t acc0 = u > 1 ? 1u : 0u;
      if (leader) {
#pragma unroll 1
        for (int sub = 0; sub < L.ku / kBK; ++sub) {
          const uint64_t da = smem_desc_at(da0, sub * L.rpad * 128), db = smem_desc_at(db0, sub * 8192);
#pragma unroll
          for (int kk = 0; kk < kBK / kMMAK; ++kk) {
            const uint64_t dak = smem_desc_at(da, kk * 32), dbk = smem_desc_at(db, kk * 2048);
            const uint32_t acc = kk > 0 || sub > 0 ? 1u : acc0;
            if constexpr (PAIR) mma_ss_pair(d, dak, dbk, kIdescPair, acc);
            else mma_ss(d, dak, dbk, kIdesc, acc);
          }
        }
        if constexpr (PAIR) mma_commit_pair(&empty[s]);
        else mma_commit(&empty[s]);
      }
      __syncwarp();
      if (++s == S) {
        s = 0;
        ph ^= 1u;
      }
    }
    if (leader) {
      if constexpr (PAIR) mma_commit_pair(done);
      else mma_commit(done);
    }
    // the accumulators, for every thread at the barrier below
    if (!good || !mbar_wait_warp(done, 0, a.status, L.max_polls)) *fail = 1;
    __syncwarp();
  }
  if (PAIR && warp == 1 && rank == 1) {  // (issued by the even CTA)
    if (!mbar_wait_warp(done, 0, a.status, L.max_polls)) *fail = 1;
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const bool main_ok = *fail == 0;
  bool ok = main_ok;

  const float c = kLog2eL / a.temperature;
  const int32_t rows = a.rows;
  // The epilogues over the accumulators use every warp: warp w reads the TMEM lane
  // quarter w % 4 (the lanes that the hardware gives it) and columns
  // [32 (w / 4), + 32) of the tile, and a quarter's four warps merge their
  // chunks through shared memory (the ring's, free now).
  const int quarter = warp & 3, chunk = warp >> 2;
  const int lrow = quarter * 32 + lane;  // of this CTA's rows
  const int32_t row_of = row0 + lrow;
  const bool live = lrow < nrows;
  const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
  float4* chunk_part = reinterpret_cast<float4*>(smem);  // [tiles][4 chunks][2][128 rows]
  // [tiles][4 chunks][128]
  float* chunk_mass = reinterpret_cast<float*>(chunk_part + kTiles * 8 * kBM);

  // ---- epilogue 1: per-tile softmax partials of every row (4 warps alone took
  // 1.7 us per tile)
#pragma unroll 1
  for (int m = 0; m < kTiles && ok; ++m) {
    const int32_t row = row_of, tile = tile0 + m;
    const uint32_t tp = tmem + lane_off + m * kBN + chunk * kChunk, tq = tp + kTiles * kBN;
    float xq_c = -INFINITY, xp_c = 0.f;
    int32_t cand = -1;
    const int32_t given = (a.draft_tok != nullptr && live) ? a.draft_tok[row] : -1;
    const int32_t c0 = tile * kBN + chunk * kChunk;
    float v[kChunk], w[kChunk];
    tmem_ld32(tp, v);
    tmem_ld32(tq, w);
    float cmp = -INFINITY, cmq = -INFINITY;
#pragma unroll
    for (int i = 0; i < kChunk; ++i) {
      cmp = fmaxf(cmp, v[i]);
      cmq = fmaxf(cmq, w[i]);
    }
    if (given < 0 && cmq > xq_c) {  // first maximum of q
#pragma unroll
      for (int i = kChunk - 1; i >= 0; --i)
        if (w[i] == cmq) { cand = c0 + i; xp_c = v[i]; }
      xq_c = cmq;
    }
    if (given >= c0 && given < c0 + kChunk) {
#pragma unroll
      for (int i = 0; i < kChunk; ++i)
        if (given == c0 + i) { cand = given; xp_c = v[i]; xq_c = w[i]; }
    }
    float lp = 0.f, lq = 0.f;
    const float cmpc = cmp * c, cmqc = cmq * c;
#pragma unroll
    for (int i = 0; i < kChunk; ++i) {
      lp += ex2_approx(fmaf(v[i], c, -cmpc));
      lq += ex2_approx(fmaf(w[i], c, -cmqc));
    }
    float4* part = chunk_part + m * 8 * kBM + lrow;
    part[(2 * chunk) * kBM] = make_float4(cmp, lp, cmq, lq);
    part[(2 * chunk + 1) * kBM] = make_float4(xq_c, xp_c, __int_as_float(cand), 0.f);
    quarter_sync(quarter);
    if (chunk == 0 && live && tile < L.tiles) {
      float mp = -INFINITY, sp = 0.f, mq = -INFINITY, sq = 0.f, xq = -INFINITY, xp = 0.f;
      int32_t t = -1;
#pragma unroll 1
      for (int k = 0; k < kCombWarps / 4; ++k) {  // ascending: the first maximum stays
        const float4 e0 = part[(2 * k) * kBM], e1 = part[(2 * k + 1) * kBM];
        merge_ms(mp, sp, e0.x, e0.y, c);
        merge_ms(mq, sq, e0.z, e0.w, c);
        if (__float_as_int(e1.z) >= 0 && (t < 0 || e1.x > xq)) {
          xq = e1.x;
          xp = e1.y;
          t = __float_as_int(e1.z);
        }
      }
      float4* out = reinterpret_cast<float4*>(L.part + (int64_t)row * L.tiles + tile);
      out[0] = make_float4(mp, sp, mq, sq);
      out[1] = make_float4(xq, xp, __int_as_float(t), 0.f);
    }
  }
  ok = grid_barrier(L.barrier, (unsigned)ncta + L.shortfall, a.status, flag, L.max_polls, ok);

  // ---- epilogue 2: combine the partials of each row and decide.  Row r is
  // combined by CTA r % ncta alone (one warp per row; lane l merges tiles l,
  // l + 32, ... in order, then a xor tree), which writes its outputs and its
  // record for the other CTAs.  All loads of a row are issued before any merge.
#pragma unroll 1
  for (int32_t row = cta + ncta * warp; row < rows && ok; row += ncta * kCombWarps) {
    const float4* prow = reinterpret_cast<const float4*>(L.part + (int64_t)row * L.tiles);
    float4 q0[kMaxTilesPerLane], q1[kMaxTilesPerLane];
#pragma unroll
    for (int j = 0; j < kMaxTilesPerLane; ++j) {
      const int k = lane + 32 * j;
      if (k < L.tiles) {
        q0[j] = __ldcg(prow + 2 * k);
        q1[j] = __ldcg(prow + 2 * k + 1);
      }
    }
    // (with the partials in flight)
    const int32_t given = a.draft_tok != nullptr ? a.draft_tok[row] : -1;
    const float2 u = row_uniforms(a.rng, row);
    bool pad = false;
    if (a.n_drafts != nullptr) {
      const int32_t b = row / a.D_max, j = row - b * a.D_max;
      pad = j >= a.n_drafts[b];
    }
    if (pad) {
      if (lane == 0) {
        L.rec[row].state = 0;
        a.out_tok[row] = -1;
        a.accepted[row] = 0;
        if (a.ratio) a.ratio[row] = 0.f;
        if (a.lse) { a.lse[2 * row] = 0.f; a.lse[2 * row + 1] = 0.f; }
      }
      continue;
    }
    float Mp = -INFINITY, Sp = 0.f, Mq = -INFINITY, Sq = 0.f, xq = -INFINITY, xp = 0.f;
    int32_t t = 0x7fffffff;
#pragma unroll
    for (int j = 0; j < kMaxTilesPerLane; ++j) {
      if (lane + 32 * j < L.tiles) {
        Mp = fmaxf(Mp, q0[j].x);
        Mq = fmaxf(Mq, q0[j].z);
        const int32_t ck = __float_as_int(q1[j].z);
        if (ck >= 0 && better(q1[j].x, ck, xq, t)) { xq = q1[j].x; xp = q1[j].y; t = ck; }
      }
    }
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) {
      Mp = fmaxf(Mp, __shfl_xor_sync(0xffffffffu, Mp, o));
      Mq = fmaxf(Mq, __shfl_xor_sync(0xffffffffu, Mq, o));
      const float oq = __shfl_xor_sync(0xffffffffu, xq, o);
      const float op = __shfl_xor_sync(0xffffffffu, xp, o);
      const int32_t ot = __shfl_xor_sync(0xffffffffu, t, o);
      if (better(oq, ot, xq, t)) { xq = oq; xp = op; t = ot; }
    }
#pragma unroll
    for (int j = 0; j < kMaxTilesPerLane; ++j) {
      if (lane + 32 * j < L.tiles) {  // (a tile of -inf alone has no sum)
        if (q0[j].x > -INFINITY) Sp = fmaf(q0[j].y, ex2_approx((q0[j].x - Mp) * c), Sp);
        if (q0[j].z > -INFINITY) Sq = fmaf(q0[j].w, ex2_approx((q0[j].z - Mq) * c), Sq);
      }
    }
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) {
      Sp += __shfl_xor_sync(0xffffffffu, Sp, o);
      Sq += __shfl_xor_sync(0xffffffffu, Sq, o);
    }
    if (lane == 0) {
      const bool valid_t = (t >= 0 && t < a.V) && (given < 0 || t == given);
      float ratio = 0.f;
      bool acc = false;
      if (valid_t) {
        const float l2p = (xp - Mp) * c - log2f(Sp);
        const float l2q = (xq - Mq) * c - log2f(Sq);
        ratio = exp2f(l2p - l2q);
        acc = u.x < fminf(ratio, 1.0f);
      }
      LmRowRec rr;
      rr.Cp = Mp * c + log2f(Sp);
      rr.Cq = Mq * c + log2f(Sq);
      rr.u_res = u.y;
      rr.state = acc ? 0 : valid_t ? 1 : 2;
      L.rec[row] = rr;
      if (!valid_t) record_status(a.status, SSD_ERR_DEVICE_BOUNDS);
      a.accepted[row] = acc ? 1 : 0;
      if (acc) a.out_tok[row] = t;
      else a.out_tok[row] = -1;  // a drawn row's token is written in epilogue 5
      if (a.ratio) a.ratio[row] = ratio;
      if (a.lse) {
        a.lse[2 * row] = Mp / a.temperature + log2f(Sp) * kLn2L;
        a.lse[2 * row + 1] = Mq / a.temperature + log2f(Sq) * kLn2L;
      }
    }
  }
  ok = grid_barrier(L.barrier, 2u * ((unsigned)ncta + L.shortfall), a.status, flag, L.max_polls, ok);

  // ---- the rows to draw, in every CTA: every valid rejected row, or (lazy)
  // the first rejected row of each sequence among its drafts
  int32_t* first = reinterpret_cast<int32_t*>(rowinfo + kBM);  // [rows / D_max]
  const bool lazy = a.lazy != 0 && a.n_drafts != nullptr;
  const int32_t ngroups = lazy ? rows / a.D_max : 0;
  int32_t* ndraw = first + kMaxRows;     // of this CTA's rows those to draw, in any order
  int32_t* drawn = ndraw + 1;            // [128]
  if (tid == 0) *ndraw = 0;
  if (tid < kBM) rowinfo[tid].state = 0;
  for (int32_t g = tid; g < ngroups; g += kThreadsL) first[g] = 0x7fffffff;
  // the record of a row, written by another CTA, read from L2 (at most one row
  // per thread; its state says all that the choice needs)
  static_assert(kMaxRows <= kThreadsL, "one row per thread");
  float4 rv = make_float4(0.f, 0.f, 0.f, 0.f);
  if (tid < rows && ok) rv = __ldcg(reinterpret_cast<const float4*>(L.rec + tid));
  const int32_t state = __float_as_int(rv.w);
  const int32_t group = lazy ? tid / a.D_max : 0;
  __syncthreads();
  if (lazy && state != 0) atomicMin(&first[group], tid - group * a.D_max);
  __syncthreads();
  if (tid >= row0 && tid < row0 + nrows) {
    LmSmemRow& ri = rowinfo[tid - row0];
    const bool pick = state == 1 && (!lazy || tid - group * a.D_max == first[group]);
    ri.Cp = rv.x;
    ri.Cq = rv.y;
    ri.u_res = rv.z;
    ri.state = pick ? 1 : 0;
    ri.from_p = 0;
    ri.cstar = -1;
    if (pick) drawn[atomicAdd(ndraw, 1)] = tid - row0;
  }
  __syncthreads();

  // ---- epilogue 3: residual mass of this tile for every row to draw: chunk sums
  // in vocabulary order, then their sum
#pragma unroll 1
  for (int m = 0; m < kTiles && ok; ++m) {
    const int32_t row = row_of, tile = tile0 + m;
    const LmSmemRow& ri = rowinfo[lrow];
    const uint32_t tp = tmem + lane_off + m * kBN + chunk * kChunk, tq = tp + kTiles * kBN;
    float mass = 0.f;
    // every lane of the warp takes part in tcgen05.ld; rows that do not draw
    // simply discard the values
    const bool draw = ri.state == 1;
    if (!__any_sync(0xffffffffu, draw)) continue;  // no row of this quarter draws
    const float Cp = ri.Cp, Cq = ri.Cq;
#pragma unroll 1
    for (int ch = 0; ch < kChunk; ch += 8) {
      float v[8], w[8];
      tmem_ld8(tp + ch, v);
      tmem_ld8(tq + ch, w);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        mass += fmaxf(ex2_approx(fmaf(v[i], c, -Cp)) - ex2_approx(fmaf(w[i], c, -Cq)), 0.f);
    }
    float* cm = chunk_mass + m * 4 * kBM + lrow;
    cm[chunk * kBM] = mass;
    quarter_sync(quarter);
    if (draw && chunk == 0 && tile < L.tiles)
      L.mass[(int64_t)row * L.tiles + tile] = mass + cm[kBM] + cm[2 * kBM] + cm[3 * kBM];
  }
  ok = grid_barrier(L.barrier, 3u * ((unsigned)ncta + L.shortfall), a.status, flag, L.max_polls, ok);

  // ---- epilogue 4: locate the tile holding u_res * Z: half a warp per row up to 128
  // tiles, else a warp; lane l of the row's lanes owns tiles [l*per, (l+1)*per) and
  // keeps their masses in registers; the same arithmetic in every CTA.  (The rows come
  // from the list: by row number the drawn rows of images of 48 rows fell to one
  // warp, 5 us.  The pass is bound by its instructions, ~1 us for 16 warps, so 47 drawn
  // rows took 3.4 us at a warp each.)
  if (ok) {
    const int32_t nd = *ndraw;
    const int W = L.tiles <= 16 * kMaxTilesPerLane ? 16 : 32;
    const int seg0 = lane & ~(W - 1), sl = lane & (W - 1);
    const uint32_t seg_mask = W == 32 ? 0xffffffffu : 0xffffu << seg0;
    const int32_t most = (L.tiles + W - 1) / W, per = most <= 2 ? most : most <= 4 ? 4 : 8;
    static_assert(kMaxTilesPerLane == 8, "two 16-byte loads per lane");
    const int32_t k0 = sl * per, own = min(per, L.tiles - k0);  // (own <= 0: none)
    const bool vec = per >= 4 && L.tiles % 4 == 0;
    auto tile_masses = [&](int32_t i, float* mk) {
      const int32_t n = i < nd ? own : 0;
      const float* m = L.mass + (int64_t)(row0 + (i < nd ? drawn[i] : 0)) * L.tiles + k0;
      if (vec) {
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 x = n > 0 ? __ldcg(reinterpret_cast<const float4*>(m)) : z;
        const float4 y = n > 4 ? __ldcg(reinterpret_cast<const float4*>(m) + 1) : z;
        mk[0] = x.x; mk[1] = x.y; mk[2] = x.z; mk[3] = x.w;
        mk[4] = y.x; mk[5] = y.y; mk[6] = y.z; mk[7] = y.w;
      } else {
#pragma unroll
        for (int q = 0; q < kMaxTilesPerLane; ++q) mk[q] = q < n ? __ldcg(m + q) : 0.f;
      }
    };
    const int32_t step = kCombWarps * (32 / W), i00 = warp * (32 / W);
    float mnext[kMaxTilesPerLane];  // of the lane's next row, in flight during this one
    tile_masses(i00 + seg0 / W, mnext);
#pragma unroll 1
    for (int32_t i0 = i00; i0 < nd; i0 += step) {  // warp-uniform
      const int32_t i = i0 + seg0 / W;
      const bool valid = i < nd;
      LmSmemRow& ri = rowinfo[drawn[valid ? i : i0]];
      float mk[kMaxTilesPerLane], ls, incl, Z;
#pragma unroll
      for (int q = 0; q < kMaxTilesPerLane; ++q) mk[q] = mnext[q];
      tile_masses(i + step, mnext);
      auto scan = [&]() {
        ls = 0.f;
#pragma unroll
        for (int q = 0; q < kMaxTilesPerLane; ++q) ls += mk[q];
        incl = ls;
#pragma unroll 1
        for (int o = 1; o < W; o <<= 1) {
          const float y = __shfl_up_sync(0xffffffffu, incl, o, W);
          if (sl >= o) incl += y;
        }
        Z = __shfl_sync(0xffffffffu, incl, W - 1, W);
      };
      scan();
      // zero residual mass: the draw is from p, whose tile masses are in the partials
      const bool empty = valid && !(Z > 0.f);
      if (__any_sync(0xffffffffu, empty)) {
        if (empty) {
          const float4* part = reinterpret_cast<const float4*>(
              L.part + (int64_t)(row0 + drawn[i]) * L.tiles + k0);
#pragma unroll
          for (int q = 0; q < kMaxTilesPerLane; ++q) {
            mk[q] = 0.f;
            if (q < own) {
              const float4 p0 = __ldcg(part + 2 * q);
              mk[q] = p0.y * ex2_approx(p0.x * c - ri.Cp);
            }
          }
        }
        __syncwarp();
        scan();
        if (empty && !(Z > 0.f) && sl == 0 && tile0 == 0) {
          a.out_tok[row0 + drawn[i]] = -1;
          record_status(a.status, SSD_ERR_DEVICE_BOUNDS);
        }
      }
      const float target = ri.u_res * Z;
      const uint32_t pos = __ballot_sync(0xffffffffu, ls > 0.f) & seg_mask;
      const uint32_t cross = __ballot_sync(0xffffffffu, ls > 0.f && incl > target) & seg_mask;
      const int32_t lstar = cross ? __ffs(cross) - 1 : pos ? 31 - __clz(pos) : lane;
      float t1 = __shfl_sync(0xffffffffu, incl - ls, lstar);
      t1 = cross ? target - t1 : INFINITY;
      if (valid && Z > 0.f && lane == lstar) {
        int32_t ks = -1, klast = -1;
        float tk = INFINITY, cum = 0.f;
#pragma unroll
        for (int q = 0; q < kMaxTilesPerLane; ++q) {
          if (mk[q] > 0.f) {  // (0 past the lane's tiles)
            klast = k0 + q;
            if (ks < 0 && cum + mk[q] > t1) { ks = klast; tk = t1 - cum; }
          }
          cum += mk[q];
        }
        if (ks < 0) { ks = klast; tk = INFINITY; }
        ri.cstar = ks;
        ri.tc = tk;
        ri.from_p = empty ? 1 : 0;
      }
      __syncwarp();
    }
  }
  __syncthreads();

  // ---- epilogue 5: the CTA holding the crossing scans the chunk that holds it
  // (its chunk masses say which) in order; a row drawn from p, whose chunk
  // masses are not kept, is scanned whole by the first chunk's warp
#pragma unroll 1
  for (int m = 0; m < kTiles && ok; ++m) {
    const int32_t row = row_of, tile = tile0 + m;
    const LmSmemRow& ri = rowinfo[lrow];
    bool mine = ri.state == 1 && ri.cstar == tile;
    if (!__any_sync(0xffffffffu, mine)) continue;  // warp-uniform
    const bool from_p = ri.from_p != 0;
    float target = ri.tc;
    if (mine && !from_p) {
      const float* cm = chunk_mass + m * 4 * kBM + lrow;
      int at = -1, last = -1;
      float before = 0.f, tk = INFINITY;
#pragma unroll
      for (int k = 0; k < kCombWarps / 4; ++k) {
        const float mk = cm[k * kBM];
        if (mk > 0.f) {
          last = k;
          if (at < 0 && before + mk > target) { at = k; tk = target - before; }
        }
        before += mk;
      }
      mine = chunk == (at >= 0 ? at : last);
      target = tk;
    } else {
      mine = mine && chunk == 0;
    }
    if (!__any_sync(0xffffffffu, mine)) continue;
    const uint32_t tp = tmem + lane_off + m * kBN + chunk * kChunk, tq = tp + kTiles * kBN;
    const float Cp = ri.Cp, Cq = ri.Cq;
    const int end = __any_sync(0xffffffffu, mine && from_p) ? kBN : kChunk;  // (then chunk is 0)
    const int end_row = from_p ? kBN : kChunk;
    float cum = 0.f;
    int32_t pick = -1, lastpos = -1;
    // (8 entries per rolled step: it runs once, and an unrolled tile was fetched
    // cold, 9.5 us in the CTAs that hold a crossing)
#pragma unroll 1
    for (int ch = 0; ch < end; ch += 8) {
      float v[8], w[8];
      tmem_ld8(tp + ch, v);
      tmem_ld8(tq + ch, w);
      if (ch < end_row) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float pv = ex2_approx(fmaf(v[i], c, -Cp));
          const float wt = from_p ? pv : fmaxf(pv - ex2_approx(fmaf(w[i], c, -Cq)), 0.f);
          cum += wt;
          if (wt > 0.f) {
            lastpos = tile * kBN + chunk * kChunk + ch + i;
            if (pick < 0 && cum > target) pick = lastpos;
          }
        }
      }
      __syncwarp();
    }
    if (mine) a.out_tok[row] = pick >= 0 ? pick : lastpos;
  }

  // ---- teardown.  After a failure in the main loop: the copies still in flight, among
  // each copying warp's last S units, and the products.  A pair's copies are counted
  // by its even CTA; after any failure the odd one waits its time out on a barrier that
  // nothing arrives at.
  if (rank == 1) {
    if (!ok && warp == 0) mbar_drain(&full[0], 0);
  } else if (!main_ok) {
    if (issued > 0) {
#pragma unroll 1
      for (int x = max(issued - S, 0); x < issued; ++x) mbar_drain(&full[x % S], (x / S) & 1);
    } else if (warp == 1) {
      mbar_drain(done, 0);
    }
  }
  // release TMEM (all MMAs have completed: `done` fired)
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync_all();  // (no copy or MMA of the pair is left)
  if (warp == 0) {
    tc_fence_after();
    if constexpr (PAIR) tmem_dealloc_pair(tmem, ncols);
    else tmem_dealloc(tmem, ncols);
  }
}

// bf16 [rows][K] hidden states as {64, rows, K / 64} (the last dimension steps
// 128 B along a row), box {64, rpad, ku / 64}: every row's next ku entries as
// [ku / 64][rpad][128 B] in one copy (rows past the matrix read as zero).
bool make_hidden_map(CUtensorMap* map, const void* base, uint64_t rows, uint64_t K, uint32_t rpad,
                     uint32_t ku) {
  const uint64_t dims[3] = {64, rows, K / 64}, strides[2] = {K * 2, 128};
  const uint32_t box[3] = {64, rpad, ku / 64};
  return bf16_tensor_map(map, base, 3, dims, strides, box);
}

// bf16 [K][V] weights as the 3D view {64 vocabulary entries, K rows, V / 64
// column blocks} (the last dimension steps 128 B along a row); a box
// {64, ku, 2} is one CTA's [2 blocks][ku rows][128 B] weight tile in one copy.
bool make_weight_map(CUtensorMap* map, const void* base, uint64_t V, uint64_t K, uint32_t ku) {
  const uint64_t dims[3] = {64, K, V / 64}, strides[2] = {V * 2, 128};
  const uint32_t box[3] = {64, ku, kBN / 64};
  return bf16_tensor_map(map, base, 3, dims, strides, box);
}

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

// Rows above one row tile run on CTA pairs, half of the rows (in swizzle groups of
// 8) in each CTA.
bool row_pairs(int32_t rows) { return rows > kBM; }
int staged_rows(int32_t rows) { return ((row_pairs(rows) ? (rows + 1) / 2 : rows) + 7) / 8 * 8; }
// CTAs of a launch: one per vocabulary tile, whole pairs.
int32_t lm_ctas(int32_t rows, int32_t V) {
  const int32_t tiles = V / kBN;
  return row_pairs(rows) ? (tiles + 1) / 2 * 2 : tiles;
}
size_t smem_bytes(int32_t rows, int ku, int stages) {
  // + the first rejected draft of each sequence (at most one per row), and the
  // list of the rows to draw
  return 1024 + (size_t)stages * (staged_rows(rows) + kBN) * ku * 2 + (2 * stages + 1) * 8 + 16 +
         (size_t)kBM * sizeof(LmSmemRow) + (size_t)(kMaxRows + 1 + kBM) * sizeof(int32_t);
}

// K per ring unit: 128 (fewer, larger copies) where it divides K and leaves four
// stages (up to 88 staged rows), else 64.  With three stages of 128 too little is
// in flight: 128 rows x 16384 x 4096 66.2 us against 64.1 with 64, 80 rows 59.7 and
// 59.3; 48 rows x 2048 x 4096 42.1 against 47.3.
int unit_k(int32_t rows, int32_t K) {
  return K % 128 == 0 && smem_bytes(rows, 128, 4) <= kMaxSmem ? 128 : kBK;
}

// As many stages as the shared memory holds, at most 8.
int stages_for(int32_t rows, int ku) {
  int s = 8;
  while (s > 2 && smem_bytes(rows, ku, s) > kMaxSmem) --s;
  return s;
}

// The launch: cooperative, above one row tile in clusters of two.
struct LmConfig {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  LmConfig(int32_t rows, int32_t V, size_t smem, cudaStream_t stream) {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)lm_ctas(rows, V), 1, 1);
    cfg.blockDim = dim3(kThreadsL, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = row_pairs(rows) ? 2 : 1;
  }
  LmConfig(const LmConfig&) = delete;  // (cfg points into it)
};

}  // namespace

size_t lmhead_workspace(int32_t rows, int32_t V) {
  const size_t ncta = (size_t)(V + kBN - 1) / kBN;
  return al256(2 * sizeof(unsigned int)) + al256((size_t)rows * ncta * sizeof(LmPartial)) +
         al256((size_t)rows * ncta * sizeof(float)) + al256((size_t)rows * sizeof(LmRowRec));
}

ssd_status lmhead_check(int32_t rows, int32_t V, int32_t K) {
  if (rows < 1 || rows > kMaxRows) return SSD_ERR_UNSUPPORTED;
  if (K <= 0 || K % kBK != 0) return SSD_ERR_UNSUPPORTED;
  if (V <= 0 || V % kBN != 0) return SSD_ERR_UNSUPPORTED;
  if (V / kBN > 32 * kMaxTilesPerLane) return SSD_ERR_UNSUPPORTED;
  // every CTA must be resident at once (one per SM: TMEM and shared memory), above one
  // row tile in pairs, fewer of which may fit than half of the SMs
  const int ku = unit_k(rows, K);
  const size_t smem = smem_bytes(rows, ku, stages_for(rows, ku));
  int n = 0;
  int64_t resident = 0;
  if (row_pairs(rows)) {
    LmConfig c(rows, V, smem, nullptr);
    if (cudaFuncSetAttribute(lmhead_accept_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, lmhead_accept_kernel<true>, &c.cfg) != cudaSuccess)
      return SSD_ERR_CUDA;
    resident = 2 * (int64_t)n;
  } else {
    if (cudaFuncSetAttribute(lmhead_accept_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, lmhead_accept_kernel<false>, kThreadsL,
                                                      smem) != cudaSuccess)
      return SSD_ERR_CUDA;
    resident = (int64_t)n * device_sm_count();
  }
  if (lm_ctas(rows, V) > resident) return SSD_ERR_UNSUPPORTED;
  return SSD_OK;
}

cudaError_t launch_lmhead(const LmHeadArgs& a, void* ws, size_t ws_bytes, cudaStream_t stream) {
  if (a.rows == 0) return cudaSuccess;
  LmLaunch L;
  L.tiles = a.V / kBN;
  L.ku = unit_k(a.rows, a.K);
  L.rpad = staged_rows(a.rows);
  L.stages = stages_for(a.rows, L.ku);
  L.max_polls = wait_poll_limit();
  L.shortfall = barrier_shortfall();
  unsigned char* w = static_cast<unsigned char*>(ws);
  L.barrier = reinterpret_cast<unsigned int*>(w);  // arrivals and the abort bit
  w += al256(2 * sizeof(unsigned int));
  L.part = reinterpret_cast<LmPartial*>(w);
  w += al256((size_t)a.rows * L.tiles * sizeof(LmPartial));
  L.mass = reinterpret_cast<float*>(w);
  w += al256((size_t)a.rows * L.tiles * sizeof(float));
  L.rec = reinterpret_cast<LmRowRec*>(w);
  CUtensorMap ht, hd, wt, wd;
  const uint32_t ku = (uint32_t)L.ku, rpad = (uint32_t)L.rpad;
  if (!make_hidden_map(&ht, a.h_tgt, (uint64_t)a.rows, (uint64_t)a.K, rpad, ku) ||
      !make_hidden_map(&hd, a.h_drf, (uint64_t)a.rows, (uint64_t)a.K, rpad, ku) ||
      !make_weight_map(&wt, a.w_tgt, (uint64_t)a.V, (uint64_t)a.K, ku) ||
      !make_weight_map(&wd, a.w_drf, (uint64_t)a.V, (uint64_t)a.K, ku))
    return cudaErrorInvalidValue;
  cudaError_t e = cudaSuccess;
  if (!a.counters_zeroed) {
    e = launch_zero(L.barrier, kLmheadCounters, stream);
    if (e != cudaSuccess) return e;
  }
  const size_t smem = smem_bytes(a.rows, L.ku, L.stages);
  auto launch = [&](auto kernel) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    LmConfig c(a.rows, a.V, smem, stream);
    return cudaLaunchKernelEx(&c.cfg, kernel, ht, hd, wt, wd, a, L);
  };
  return row_pairs(a.rows) ? launch(lmhead_accept_kernel<true>) : launch(lmhead_accept_kernel<false>);
}

}  // namespace ssd
