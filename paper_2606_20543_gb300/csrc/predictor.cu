// predictor.cu — the spatial draft predictor f_phi (Sec. 3.3 "Draft
// Prediction in Latent Space", Eq. 2) and the draft tokens it yields:
//
//   h_hat = W0 z + SwiGLU(RMSNorm(W0 z)),  z = [h ; e],
//   SwiGLU(x) = W2 (silu(W1 x) * W3 x),    t_hat = argmax GenHead(RMSNorm(h_hat)).
//
// Design (GB300): for one grid row of positions the predictor is a chain of
// skinny products — at most 128 rows against four weight matrices of 64 MB
// and the 128 MB GenHead at the paper's head size — so it is bound by reading
// the weights once from HBM.  One persistent cooperative kernel (one CTA per
// SM) runs the whole chain in four phases.  RMSNorm(x) g = s(x) (x * g) with
// the row scale s(x) = 1 / sqrt(mean(x^2) + eps), and s commutes with the
// products that follow, so every product input is an elementwise bf16 array
// that the previous phase writes tile by tile, and the row scale is applied
// to the product's output:
//   P0  A  = W0 z                        (features d, K = 2d);  Ag = bf16(A * g1)
//   P1  U  = s(A) W1 Ag, Vg = s(A) W3 Ag (features m, K = d);   G = bf16(silu(U) * Vg)
//   P2  h  = A + W2 G                    (features d, K = m);   Hg = bf16(h * g2)
//   P3  l  = W_head^T Hg                 (features V, K = d);   t = argmax l
// (the GenHead's row scale s(h) > 0 leaves the argmax unchanged; the lowest
// index wins ties).  Every product is D[rows x tile of features] += X[rows x
// 16] W[16 x features] on the tensor cores (tcgen05.mma kind::f16, fp32
// accumulation in tensor memory): the rows on M (64 or 128), the features on N.
// A phase's features are cut into about one tile per CTA (16 to 128 wide), and
// a tile's whole K runs in its CTA: no partial sums, so between the phases
// there is only the tile's epilogue, one counter and the next activations'
// copies, at the price of every CTA reading all of X from L2 (24 rows: 1.2 MB
// beside 3.1 MB of weights).  At d = 4096, m = 8192, V = 16384: 24 rows 79 us
// (0.76 of the rate of the measured copy), 64 rows 86, 128 rows 110; 92 rows at
// d = 896 33.  (In turn: with 4 epilogue warps of whole rows 89, 97, 120 and 42; 16
// warps that each polled for the products 86, 93, 123 and 41, one of them polling 85,
// 92, 117 and 38; started as a programmatic dependent's successor 82, 90, 114 and 37;
// then without the GPU-wide fences.)  Splitting each tile's K over CTAs instead, with the
// partials summed through L2 by the last contributor (~9 us per phase boundary,
// 254 KB of code), took 113, 135, 147 and 93 us.
//   * warp 0: weight producer, running ahead through all four phases into a
//     ring of units (up to 512 K of a tile; weights and activations of a unit
//     in one slot): the weights do not depend on the activations;
//   * warp 1: activation producer: once every tile of the previous phase is
//     final (a counter per phase), one copy per unit from z, Ag, G or Hg;
//   * warp 2: issues the MMAs of each unit into one of two TMEM accumulators
//     (a CTA's next tile overlaps the epilogue of the one before);
//   * warps 4-19: the epilogue, four warps per TMEM lane quarter.  Each TMEM lane is one row: A, Ag and the row's
//     sum of squares over the tile (P0); G (P1); h and Hg (P2); the tile's
//     argmax, raised into one 64-bit key per row by a max reduction (P3).  The
//     row scales s(A) are summed once per CTA, beside the P1 products; the last
//     tile of P3 to finish turns the keys into the tokens.
// Numerics: every product input is bf16 (z, the weights, Ag, G, Hg); A, U,
// Vg, h and the logits are fp32; every sum runs in a fixed order, so results
// do not depend on timing.
#include <algorithm>

#include "kernels.cuh"

namespace ssd {

namespace {

constexpr int kPThreads = 640;       // 20 warps
constexpr int kWarpW = 0;            // weight producer
constexpr int kWarpX = 1;            // activation producer
constexpr int kWarpMma = 2;
constexpr int kWarpTmem = 3;         // allocates / frees tensor memory
constexpr int kEpiWarp0 = 4;         // warps 4-19: TMEM lane quarter w % 4, column chunk (w - 4) / 4
constexpr int kEpiChunks = 4;
constexpr int kEpiThreads = 128 * kEpiChunks;
constexpr int kMaxRows = 128;
constexpr int kPhases = 4;
constexpr int kBarEpi = 1;           // named barrier of the epilogue warps
constexpr int kMaxN = 128;           // columns of one accumulator
constexpr int kSlotTarget = 57344;   // ring slots of at most 56 KB: four of them at 24 rows
// One 128-byte line per row's argmax key: every GenHead tile raises every
// row's key near the end of the kernel, and the rows' reductions go to
// separate lines.
constexpr int kKeyStride = 16;

struct PredPhase {
  int32_t F, K;     // features and contraction length
  int32_t tn;       // features per tile (P1: of each of W1 and W3)
  int32_t tiles;    // feature tiles
  int32_t ku;       // K per ring unit
  int32_t units;    // units per tile
};

struct PredLaunch {
  PredPhase ph[kPhases];
  int32_t ncta, rows, rpad;    // rpad: staged rows (swizzle groups of 8)
  int32_t stages, slot_bytes;  // ring
  int32_t d, m, V;
  uint32_t max_polls, shortfall;
  float eps;
  const float* gamma1;
  const float* gamma2;
  float* hid;                  // fp32 [rows][d]: A, then h_hat
  __nv_bfloat16* ag;           // bf16 [rows][d]: A * g1, then h_hat * g2
  __nv_bfloat16* g;            // bf16 [rows][m]: silu(U) * Vg
  float* ss;                   // fp32 [P0 tiles][128]: per-tile sums of squares of A's rows
  unsigned long long* best;    // [rows][kKeyStride]: the argmax key of row r at best[r * kKeyStride]
  unsigned int* ctr;           // done [4], abort, a 128-byte line each
  int32_t* out_tok;
  int32_t* status;
};

__device__ __forceinline__ void bar_named(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// Named barrier that also ORs a predicate over its `count` threads: every
// thread of the group leaves with the same answer from the same barrier.
__device__ __forceinline__ bool bar_or(int id, int count, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n"
      " bar.red.or.pred q, %2, %3, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"(pred ? 1u : 0u), "r"(id), "r"(count)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ uint32_t ld_acquire_u32(const unsigned int* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Order this thread's generic-proxy global accesses with async-proxy (TMA)
// accesses: after writing an array that other CTAs will load by TMA, and
// after learning that such an array is complete, before loading it.
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

// Counters, one per 128-byte line: tiles done per phase, abort.
constexpr int kCtrStride = 32;
__device__ __forceinline__ unsigned int* done_ctr(const PredLaunch& L, int p) {
  return L.ctr + p * kCtrStride;
}
__device__ __forceinline__ unsigned int* abort_flag(const PredLaunch& L) {
  return L.ctr + kPhases * kCtrStride;
}

// Bounded wait until *ctr >= target; false (SSD_ERR_TIMEOUT recorded, abort
// raised) if it gave up, or if another CTA aborted the kernel.
__device__ __noinline__ bool wait_count(const PredLaunch& L, const unsigned int* ctr, uint32_t target) {
#pragma unroll 1
  for (uint32_t i = 0; i < L.max_polls; ++i) {
    // (the count alone says that every tile is final: a CTA that gives up counts no
    // more of its own)
    if (ld_acquire_u32(ctr) >= target) return true;
    if ((i & 1023u) == 1023u && ld_acquire_u32(abort_flag(L)) != 0u) return false;
    if (i > 64) __nanosleep(128);
  }
  atomicExch(abort_flag(L), 1u);
  record_status(L.status, SSD_ERR_TIMEOUT);
  return false;
}

// The vocabulary argmax of each row is kept as one 64-bit key per row,
// raised by a max reduction from every finished GenHead tile: the logit in an
// order-preserving unsigned form (NaN as the lowest key) above the inverted
// index, so the largest logit wins and the lower index among equal ones
// (-0 is taken as +0, which compares equal to it).
__device__ __forceinline__ unsigned long long argmax_key(float v, int32_t i) {
  uint32_t u = v == 0.f ? 0u : __float_as_uint(v);
  u = (v != v) ? 0u : ((u & 0x80000000u) ? ~u : (u | 0x80000000u));
  return ((unsigned long long)u << 32) | (unsigned long long)(0xffffffffu - (uint32_t)i);
}
__device__ __forceinline__ int32_t argmax_index(unsigned long long key) {
  return (int32_t)(0xffffffffu - (uint32_t)(key & 0xffffffffull));
}

// The four warps of one TMEM lane quarter.
__device__ __forceinline__ void quarter_sync(int quarter) {
  bar_named(kBarEpi + 1 + quarter, 32 * kEpiChunks);
}

__device__ __forceinline__ uint4 pack8(const float* y) {
  return make_uint4(pack_bf16x2(y[0], y[1]), pack_bf16x2(y[2], y[3]), pack_bf16x2(y[4], y[5]),
                    pack_bf16x2(y[6], y[7]));
}

// The finishing step of tile t of phase p for one row (this thread's TMEM lane;
// live: the row exists), 8 features at a time, in one rolled loop per phase: it
// runs once per tile, so its instructions are fetched rather than reused.  The
// quarter's four warps take every fourth group of 8 (one warp per quarter took
// 1.3 us per tile, the gate 3.8) and combine sums and keys through `xch`
// (8 bytes per row: with 24 the ring lost a slot at 73 to 96 rows).
__device__ __forceinline__ void finish_hidden(const PredLaunch& L, int p, int32_t t, int32_t row,
                                              bool live, uint32_t acc, int chunk, int quarter,
                                              float2* xch, float* srow) {
  const PredPhase& ph = L.ph[p];
  const int32_t f0 = t * ph.tn, n = min(ph.tn, ph.F - f0);
  float* hid = L.hid + (int64_t)row * L.d + f0;
  __nv_bfloat16* ag = L.ag + (int64_t)row * L.d + f0;
  const float* gamma = (p == 0 ? L.gamma1 : L.gamma2) + f0;
  float sq = 0.f;
#pragma unroll 1
  for (int32_t c = 8 * chunk; c < n; c += 8 * kEpiChunks) {
    float y[8];
    tmem_ld8(acc + c, y);
    if (!live) continue;
    if (p == 2) {
      const float4 a0 = *reinterpret_cast<const float4*>(hid + c);
      const float4 a1 = *reinterpret_cast<const float4*>(hid + c + 4);
      y[0] = a0.x + y[0]; y[1] = a0.y + y[1]; y[2] = a0.z + y[2]; y[3] = a0.w + y[3];
      y[4] = a1.x + y[4]; y[5] = a1.y + y[5]; y[6] = a1.z + y[6]; y[7] = a1.w + y[7];
    }
    const float4 g0 = __ldg(reinterpret_cast<const float4*>(gamma + c));
    const float4 g1 = __ldg(reinterpret_cast<const float4*>(gamma + c + 4));
    *reinterpret_cast<float4*>(hid + c) = make_float4(y[0], y[1], y[2], y[3]);
    *reinterpret_cast<float4*>(hid + c + 4) = make_float4(y[4], y[5], y[6], y[7]);
    const float x[8] = {y[0] * g0.x, y[1] * g0.y, y[2] * g0.z, y[3] * g0.w,
                        y[4] * g1.x, y[5] * g1.y, y[6] * g1.z, y[7] * g1.w};
    *reinterpret_cast<uint4*>(ag + c) = pack8(x);
    sq += ((y[0] * y[0] + y[1] * y[1]) + (y[2] * y[2] + y[3] * y[3])) +
          ((y[4] * y[4] + y[5] * y[5]) + (y[6] * y[6] + y[7] * y[7]));
  }
  if (p == 0) {
    // (srow is free until P1)
    if (chunk > 0 && live) (chunk == 1 ? xch[row].x : chunk == 2 ? xch[row].y : srow[row]) = sq;
    quarter_sync(quarter);
    if (chunk == 0 && live)
      L.ss[(int64_t)t * kMaxRows + row] = sq + xch[row].x + xch[row].y + srow[row];
    quarter_sync(quarter);  // (the CTA's next tile writes them again)
  }
}
// P1: G = bf16(silu(U) * Vg) with U, Vg scaled by the row's s(A).
__device__ __forceinline__ void finish_gate(const PredLaunch& L, int32_t t, int32_t row, bool live,
                                            uint32_t acc, float sr, int chunk) {
  const PredPhase& ph = L.ph[1];
  const int32_t f0 = t * ph.tn, n = min(ph.tn, ph.F - f0);
  __nv_bfloat16* g = L.g + (int64_t)row * L.m + f0;
#pragma unroll 1
  for (int32_t c = 8 * chunk; c < n; c += 8 * kEpiChunks) {
    float u[8], v[8];
    tmem_ld8(acc + c, u);
    tmem_ld8(acc + kMaxN / 2 + c, v);
    if (!live) continue;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float x = u[i] * sr;
      u[i] = x / (1.0f + expf(-x)) * (v[i] * sr);
    }
    *reinterpret_cast<uint4*>(g + c) = pack8(u);
  }
}
// P3: the tile's argmax for the row (lowest index on ties) raised into the row's key.
__device__ __forceinline__ void finish_argmax(const PredLaunch& L, int32_t t, int32_t row, bool live,
                                              uint32_t acc, int chunk, int quarter,
                                              unsigned long long* xch) {
  const PredPhase& ph = L.ph[3];
  const int32_t f0 = t * ph.tn;
  unsigned long long key = 0;
#pragma unroll 1
  for (int32_t c = 8 * chunk; c < ph.tn; c += 8 * kEpiChunks) {
    float v[8];
    tmem_ld8(acc + c, v);
    float bv = v[0];
    int32_t bi = 0;
#pragma unroll
    for (int i = 1; i < 8; ++i)
      if (v[i] > bv) { bv = v[i]; bi = i; }
    const unsigned long long k = argmax_key(bv, f0 + c + bi);
    if (k > key) key = k;
  }
  if (chunk > 0 && live) atomicMax(&xch[row], key);
  quarter_sync(quarter);
  if (chunk > 0 || !live) return;
  key = max(key, xch[row]);
  xch[row] = 0;  // for the CTA's next tile
  asm volatile("red.relaxed.gpu.global.max.u64 [%0], %1;"
               ::"l"(L.best + (int64_t)row * kKeyStride), "l"(key) : "memory");
}

// The row scales s(A) = 1 / sqrt(mean(A^2) + eps) of every row from the P0
// tiles' sums of squares, into srow (shared): four threads per row, each
// summing every fourth tile, then combined in a fixed order.
__device__ __forceinline__ void row_scales(const PredLaunch& L, int et, float* srow) {
  const int k = et & 3;
  const int32_t nt = L.ph[0].tiles;
#pragma unroll 1
  for (int32_t r0 = 0; r0 < L.rows; r0 += kEpiThreads / 4) {
    const int32_t r = r0 + (et >> 2);
    float s = 0.f;
    if (r < L.rows)
#pragma unroll 8
      for (int32_t t = k; t < nt; t += 4) s += __ldcg(L.ss + (int64_t)t * kMaxRows + r);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if (r < L.rows && k == 0) srow[r] = 1.0f / sqrtf(s / (float)L.d + L.eps);
  }
}

// M: rows of the products (64 or 128).  M = 64: row m in TMEM lane
// 32 (m / 16) + m % 16; M = 128: in lane m.
template <int M>
__global__ void __launch_bounds__(kPThreads, 1)
predictor_kernel(const __grid_constant__ CUtensorMap tmW0, const __grid_constant__ CUtensorMap tmW1,
                 const __grid_constant__ CUtensorMap tmW3, const __grid_constant__ CUtensorMap tmW2,
                 const __grid_constant__ CUtensorMap tmWH, const __grid_constant__ CUtensorMap tmZ,
                 const __grid_constant__ CUtensorMap tmAg, const __grid_constant__ CUtensorMap tmG,
                 const __grid_constant__ CUtensorMap tmHg, PredLaunch L) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  // (the barriers before the ring: a row tile is read past its staged rows)
  uint64_t* full = reinterpret_cast<uint64_t*>(smem);  // [8]: the unit's weights and activations
  uint64_t* empty = full + 8;                          // [8]
  uint64_t* acc_full = empty + 8;      // [2]
  uint64_t* acc_empty = acc_full + 2;  // [2]
  uint64_t* mma_done = acc_empty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mma_done + 1);
  // a role that gives up raises `fail`; the epilogue warps decide to stop only
  // through a reducing named barrier (bar_or), so they leave their loop together
  volatile int32_t* fail = reinterpret_cast<volatile int32_t*>(tmem_slot + 1);
  uint32_t* bcast = reinterpret_cast<uint32_t*>(tmem_slot + 2);
  float* srow = reinterpret_cast<float*>(tmem_slot + 4);  // [128]
  unsigned char* ring = smem + 1024;
  const int S = L.stages;
  // past the ring: the epilogue's exchange, 8 bytes per row
  unsigned long long* xch = reinterpret_cast<unsigned long long*>(ring + (size_t)S * L.slot_bytes);

  const int tid = threadIdx.x, warp = (int)warp_uniform(threadIdx.x >> 5), lane = tid & 31;
  const int32_t cta = blockIdx.x;

  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 2);  // the weight producer's and the activation producer's arrivals
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&acc_full[s], 1);
      mbar_init(&acc_empty[s], kEpiThreads / 32);  // one arrival per epilogue warp
    }
    mbar_init(mma_done, 1);
    *fail = 0;
    fence_barrier_init();
  }
  if (warp == kWarpMma && lane < 9) {  // the descriptors of the first copies of every phase
    const CUtensorMap* map = lane == 0 ? &tmW0 : lane == 1 ? &tmW1 : lane == 2 ? &tmW3
                           : lane == 3 ? &tmW2 : lane == 4 ? &tmWH : lane == 5 ? &tmZ
                           : lane == 6 ? &tmAg : lane == 7 ? &tmG : &tmHg;
    prefetch_tensormap(map);
  }
  if (warp == kWarpTmem) {
    tmem_alloc(tmem_slot, 2 * kMaxN);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp <= kWarpX) {
    // ---- producers: the weights (warp 0) or the activations (warp 1) of every
    // unit, in the order of phases, tiles and K
    const bool w = warp == kWarpW, leader = elect_one();
    const uint64_t pol = w ? policy_evict_first()   // weights: read once
                           : policy_evict_last();   // activations: read by every CTA
    uint32_t gu = 0, ph = 1;  // units issued; the next phase of ring slot s
    int s = 0;
    bool ok = true;
#pragma unroll 1
    for (int p = 0; p < kPhases && ok; ++p) {
      const PredPhase& pp = L.ph[p];
      const uint32_t xb = (uint32_t)(L.rpad * pp.ku * 2), wb = (uint32_t)(pp.tn * pp.ku * 2);
      if (!w && p > 0 && cta < pp.tiles) {  // every tile of the previous phase final first
        ok = __all_sync(0xffffffffu,
                        lane != 0 || (*fail == 0 && wait_count(L, done_ctr(L, p - 1),
                                                               (uint32_t)L.ph[p - 1].tiles + L.shortfall))) != 0;
        if (!ok) break;
        __syncwarp();  // what the waiting lane acquired, for the lane that copies
        fence_proxy_async_global();  // written by generic stores, loaded by TMA
      }
      const CUtensorMap* map = w ? (p == 0 ? &tmW0 : p == 1 ? &tmW1 : p == 2 ? &tmW2 : &tmWH)
                                 : (p == 0 ? &tmZ : p == 1 ? &tmAg : p == 2 ? &tmG : &tmHg);
#pragma unroll 1
      for (int32_t t = cta; t < pp.tiles && ok; t += L.ncta) {
#pragma unroll 1
        for (int32_t u = 0; u < pp.units; ++u, ++gu) {
          ok = *fail == 0 && (gu < (uint32_t)S || mbar_wait(&empty[s], ph, L.status, L.max_polls));
          ok = __all_sync(0xffffffffu, ok) != 0;
          if (!ok) break;
          if (leader) {
            unsigned char* dst = ring + s * L.slot_bytes;
            if (!w) {  // {64, rows, K / 64}, box {64, rpad, ku / 64}
              mbar_arrive_expect_tx(&full[s], xb);
              tma_load_3d(dst, map, 0, 0, u * (pp.ku / 64), &full[s], pol);
            } else {
              // {64, features, K / 64}, box {64, tn, ku / 64}; the GenHead is
              // {64 vocabulary entries, K, V / 64}, box {64, ku, tn / 64}
              mbar_arrive_expect_tx(&full[s], p == 1 ? 2 * wb : wb);
              tma_load_3d(dst + xb, map, 0, p == 3 ? u * pp.ku : t * pp.tn,
                          p == 3 ? t * (pp.tn / 64) : u * (pp.ku / 64), &full[s], pol);
              if (p == 1)
                tma_load_3d(dst + xb + wb, &tmW3, 0, t * pp.tn, u * (pp.ku / 64), &full[s], pol);
            }
          }
          __syncwarp();
          if (++s == S) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
    }
    if (!ok) *fail = 1;
    // this warp's copies still in flight can only be among the last S units it
    // issued; each slot's barrier completes with the other warp's too, so after
    // a failure the wait is for this warp's own bytes at most max_polls long
#pragma unroll 1
    for (uint32_t x = gu > (uint32_t)S ? gu - S : 0; x < gu; ++x)
      mbar_wait(&full[x % S], (x / S) & 1, nullptr, L.max_polls);
    __syncwarp();
  } else if (warp == kWarpMma) {
    // ---- MMA issue (every lane in the loop, one elected around the products)
    const uint32_t tm = warp_uniform(tmem), ring0 = warp_uniform(smem_u32(ring));
    const bool leader = elect_one();
    uint32_t tc = 0, ph = 0;
    int s = 0;
    bool ok = true;
#pragma unroll 1
    for (int p = 0; p < kPhases && ok; ++p) {
      const PredPhase& pp = L.ph[p];
      const uint32_t xb = (uint32_t)(L.rpad * pp.ku * 2), wb = (uint32_t)(pp.tn * pp.ku * 2);
      const uint32_t idesc = idesc_bf16(M, pp.tn, false, p == 3);
      // per 64 K: the activations' and (K-major) the weights' next block; the
      // GenHead (vocabulary contiguous): 64 K rows further in every 64-wide block
      const uint32_t xstep = (uint32_t)L.rpad * 128u, wstep = p == 3 ? 8192u : (uint32_t)pp.tn * 128u;
      const uint32_t wk = p == 3 ? 2048u : 32u;  // per 16 K
#pragma unroll 1
      for (int32_t t = cta; t < pp.tiles && ok; t += L.ncta, ++tc) {
        const uint32_t buf = tc & 1u, dacc = tm + buf * kMaxN;
        if (tc >= 2)
          ok = mbar_wait_warp(&acc_empty[buf], ((tc >> 1) - 1) & 1, L.status, L.max_polls);
#pragma unroll 1
        for (int32_t u = 0; u < pp.units && ok; ++u) {
          ok = mbar_wait_warp(&full[s], ph, L.status, L.max_polls);
          if (!ok) break;
          tc_fence_after();
          const uint32_t x0 = ring0 + s * L.slot_bytes;
          const uint64_t dx = smem_desc(x0, 16, 1024);
          const uint64_t dw = smem_desc(x0 + xb, p == 3 ? pp.ku * 128 : 16, 1024);
          if (leader) {
#pragma unroll 1
            for (int32_t b = 0; b < pp.ku / 64; ++b) {
              const uint64_t bx = smem_desc_at(dx, b * xstep), bw = smem_desc_at(dw, b * wstep);
              const uint32_t a0 = (u > 0 || b > 0) ? 1u : 0u;
#pragma unroll
              for (int kk = 0; kk < 4; ++kk)
                mma_ss(dacc, smem_desc_at(bx, kk * 32), smem_desc_at(bw, kk * wk), idesc,
                       kk > 0 ? 1u : a0);
              if (p == 1) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                  mma_ss(dacc + kMaxN / 2, smem_desc_at(bx, kk * 32), smem_desc_at(bw, wb + kk * 32), idesc,
                         kk > 0 ? 1u : a0);
              }
            }
            mma_commit(&empty[s]);
            if (u == pp.units - 1) mma_commit(&acc_full[buf]);
          }
          __syncwarp();
          if (++s == S) {
            s = 0;
            ph ^= 1u;
          }
        }
      }
    }
    if (!ok) *fail = 1;
    if (leader) mma_commit(mma_done);  // arrives once every MMA issued above has completed
    __syncwarp();
  } else if (warp >= kEpiWarp0) {
    // ---- epilogue (warps 4-19): TMEM lane = row
    const int et = tid - kEpiWarp0 * 32, quarter = warp & 3, chunk = (warp - kEpiWarp0) >> 2;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    const int32_t row = quarter * (M / 4) + lane;
    const bool live = row < L.rows && (M == 128 || lane < 16);
    uint32_t tc = 0;
    bool ok = true;
#pragma unroll 1
    for (int p = 0; p < kPhases && ok; ++p) {
      const PredPhase& pp = L.ph[p];
      if (p == 3 && chunk == 0 && live) xch[row] = 0;  // (read again after P3's first barrier)
      if (p == 1 && cta < pp.tiles) {
        // the row scales, beside the first P1 products: once every P0 tile is
        // final (a bounded wait by one thread)
        bool stop = false;
        if (et == 0)
          stop = *fail != 0 ||
                 !wait_count(L, done_ctr(L, 0), (uint32_t)L.ph[0].tiles + L.shortfall);
        if (bar_or(kBarEpi, kEpiThreads, stop)) {
          ok = false;
          break;
        }
        row_scales(L, et, srow);
        bar_named(kBarEpi, kEpiThreads);
      }
#pragma unroll 1
      for (int32_t t = cta; t < pp.tiles; t += L.ncta, ++tc) {
        const uint32_t buf = tc & 1u, acc = tmem + lane_base + buf * kMaxN;
        bool stop = false;
        if (et == 0)  // (one thread polls; the others wait at the barrier)
          stop = *fail != 0 || !mbar_wait(&acc_full[buf], (tc >> 1) & 1, L.status, L.max_polls);
        if (bar_or(kBarEpi, kEpiThreads, stop)) {
          ok = false;
          break;
        }
        tc_fence_after();
        // (a quarter without rows has nothing to read)
        if (quarter * (M / 4) < L.rows) {
          if (p == 1)
            finish_gate(L, t, row, live, acc, live ? srow[row] : 0.f, chunk);
          else if (p == 3)
            finish_argmax(L, t, row, live, acc, chunk, quarter, xch);
          else
            finish_hidden(L, p, t, row, live, acc, chunk, quarter, reinterpret_cast<float2*>(xch), srow);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[buf]);
        fence_proxy_async_global();  // Ag, G, Hg are loaded by TMA in the next phase
        bar_named(kBarEpi, kEpiThreads);
        // One thread's release publishes the tile, ordered after the others' stores by
        // the barrier, and a wait's acquire load needs no fence behind it either: a
        // GPU-wide fence in every thread on both sides took 24 rows 81.4 us instead of
        // 79.2, 92 rows at d = 896 35.8 instead of 33.0.
        if (p < 3) {  // (a reduction: nothing waits for its result)
          if (et == 0)
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(done_ctr(L, p)) : "memory");
        } else {
          if (et == 0) *bcast = (uint32_t)atom_add_acq_rel(reinterpret_cast<int32_t*>(done_ctr(L, 3)), 1);
          bar_named(kBarEpi, kEpiThreads);
          if (*bcast == (uint32_t)(pp.tiles - 1)) {
            // the last tile of the vocabulary: every tile's key is in
            for (int32_t r = et; r < L.rows; r += kEpiThreads)
              L.out_tok[r] = argmax_index(__ldcg(L.best + (int64_t)r * kKeyStride));
          }
          bar_named(kBarEpi, kEpiThreads);  // (bcast is rewritten by the CTA's next tile)
        }
      }
    }
    if (!ok) *fail = 1;
  }

  // ---- teardown: every MMA complete before tensor memory is freed
  if (warp == kWarpTmem && lane == 0) mbar_wait(mma_done, 0, nullptr, L.max_polls);
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == kWarpTmem) {
    tc_fence_after();
    tmem_dealloc(tmem, 2 * kMaxN);
  }
}

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

struct PredPlan {
  PredPhase ph[kPhases];
  int32_t ncta, m_rows, rpad, stages;
  size_t slot, smem;
};

PredPlan make_plan(int32_t rows, int32_t d, int32_t m, int32_t V, int32_t sm_count) {
  PredPlan P;
  // P0: W0 [d][2d]; P1: W1, W3 [m][d]; P2: W2 [d][m]; P3: W_head [d][V]
  const int32_t F[kPhases] = {d, m, d, V}, K[kPhases] = {2 * d, d, m, d};
  P.m_rows = rows <= 64 ? 64 : 128;
  P.rpad = (rows + 7) / 8 * 8;
  P.ncta = 1;
  P.slot = 0;
  size_t over = 0;  // bytes that a row tile is read past the end of a slot
  for (int p = 0; p < kPhases; ++p) {
    PredPhase& q = P.ph[p];
    q.F = F[p];
    q.K = K[p];
    if (p == 3) {
      // 64-wide blocks of the vocabulary: tiles of 64, or of 128 where they take
      // no longer
      const int64_t r64 = (V / 64 + sm_count - 1) / sm_count, r128 = (V / 128 + sm_count - 1) / sm_count;
      q.tn = 128 * r128 <= 64 * r64 ? 128 : 64;
    } else {
      // about one tile per SM (or the fewest rounds of them), in steps of 16
      const int32_t cap = p == 1 ? kMaxN / 2 : kMaxN;
      const int32_t rounds = (q.F + sm_count * cap - 1) / (sm_count * cap);
      q.tn = std::min(cap, ((q.F + sm_count * rounds - 1) / (sm_count * rounds) + 15) / 16 * 16);
    }
    q.tiles = (q.F + q.tn - 1) / q.tn;
    P.ncta = std::max(P.ncta, std::min(q.tiles, sm_count));
    const int32_t wrows = p == 1 ? 2 * q.tn : q.tn;
    q.ku = 64;
    while (q.ku < (p == 3 ? 256 : 512) && q.ku * 2 <= (q.K + 63) / 64 * 64 &&
           (P.rpad + wrows) * q.ku * 2 * 2 <= kSlotTarget)
      q.ku *= 2;
    q.units = (q.K + q.ku - 1) / q.ku;
    const size_t unit = (size_t)(P.rpad + wrows) * q.ku * 2;
    P.slot = std::max(P.slot, unit);
    over = std::max(over, (size_t)(q.ku / 64 - 1) * P.rpad * 128 + (size_t)P.m_rows * 128);
  }
  over = over > P.slot ? over - P.slot : 0;
  over = std::max(over, (size_t)P.rpad * 8);  // (or the epilogue's exchange, in the same place)
  const size_t budget = 232448;  // 227 KB of dynamic shared memory per CTA
  P.stages = (int32_t)std::min<size_t>(8, (budget - 2048 - over) / P.slot);
  P.smem = 2048 + (size_t)P.stages * P.slot + over;
  return P;
}

struct PredWs {
  unsigned int* ctr;
  unsigned long long* best;  // after the counters: zeroed with them
  size_t zero_bytes;         // counters and keys
  float* ss;
  __nv_bfloat16* ag;
  __nv_bfloat16* g;
  float* hid;
  size_t bytes;
};

PredWs carve(const PredPlan& P, int32_t rows, int32_t d, int32_t m, bool own_hidden, void* base) {
  PredWs w;
  unsigned char* b = static_cast<unsigned char*>(base);
  size_t off = 0;
  auto take = [&](size_t n) {
    unsigned char* p = b + off;
    off += al256(n);
    return p;
  };
  const size_t ctr_bytes = al256((size_t)(kPhases + 1) * kCtrStride * 4);
  w.zero_bytes = ctr_bytes + (size_t)kMaxRows * kKeyStride * 8;
  w.ctr = reinterpret_cast<unsigned int*>(take(w.zero_bytes));
  w.best = reinterpret_cast<unsigned long long*>(reinterpret_cast<unsigned char*>(w.ctr) + ctr_bytes);
  w.ss = reinterpret_cast<float*>(take((size_t)P.ph[0].tiles * kMaxRows * 4));
  w.ag = reinterpret_cast<__nv_bfloat16*>(take((size_t)rows * d * 2));
  w.g = reinterpret_cast<__nv_bfloat16*>(take((size_t)rows * m * 2));
  w.hid = own_hidden ? reinterpret_cast<float*>(take((size_t)rows * d * 4)) : nullptr;
  w.bytes = off;
  return w;
}

bool shapes_ok(int32_t rows, int32_t d, int32_t m, int32_t V) {
  return rows >= 1 && rows <= kMaxRows && d >= 128 && m >= 128 && V >= 128 && d % 128 == 0 &&
         m % 128 == 0 && V % 128 == 0;
}

// One launch over at most kMaxRows rows.
cudaError_t launch_rows(const PredictorArgs& a, void* ws, size_t ws_bytes, int32_t* status,
                        cudaStream_t stream) {
  if (!shapes_ok(a.rows, a.d, a.m, a.V)) return cudaErrorInvalidValue;
  const PredPlan P = make_plan(a.rows, a.d, a.m, a.V, device_sm_count());
  const PredWs w = carve(P, a.rows, a.d, a.m, a.out_hidden == nullptr, ws);
  if (ws == nullptr || ws_bytes < w.bytes) return cudaErrorInvalidValue;

  PredLaunch L;
  for (int p = 0; p < kPhases; ++p) L.ph[p] = P.ph[p];
  L.ncta = P.ncta;
  L.rows = a.rows;
  L.rpad = P.rpad;
  L.stages = P.stages;
  L.slot_bytes = (int32_t)P.slot;
  L.d = a.d;
  L.m = a.m;
  L.V = a.V;
  L.max_polls = wait_poll_limit();
  L.shortfall = barrier_shortfall();
  L.eps = a.eps;
  L.gamma1 = a.gamma1;
  L.gamma2 = a.gamma2;
  L.hid = a.out_hidden != nullptr ? a.out_hidden : w.hid;
  L.ag = w.ag;
  L.g = w.g;
  L.ss = w.ss;
  L.best = w.best;
  L.ctr = w.ctr;
  L.out_tok = a.out_tok;
  L.status = status;

  const uint64_t d = (uint64_t)a.d, m = (uint64_t)a.m, V = (uint64_t)a.V, R = (uint64_t)a.rows;
  // a bf16 [outer][inner] matrix as {64, outer, inner / 64} (the last dimension
  // steps 128 B along a row), box {64, box_outer, box_blocks}
  auto map = [](CUtensorMap* t, const void* base, uint64_t outer, uint64_t inner, int32_t box_outer,
                int32_t box_blocks) {
    const uint64_t dims[3] = {64, outer, inner / 64}, strides[2] = {inner * 2, 128};
    const uint32_t box[3] = {64, (uint32_t)box_outer, (uint32_t)box_blocks};
    return bf16_tensor_map(t, base, 3, dims, strides, box);
  };
  CUtensorMap t0, t1, t3, t2, th, tz, tag, tg, thg;
  const PredPhase* q = P.ph;
  const bool ok =
      map(&t0, a.w0, d, 2 * d, q[0].tn, q[0].ku / 64) && map(&t1, a.w1, m, d, q[1].tn, q[1].ku / 64) &&
      map(&t3, a.w3, m, d, q[1].tn, q[1].ku / 64) && map(&t2, a.w2, d, m, q[2].tn, q[2].ku / 64) &&
      map(&th, a.w_head, d, V, q[3].ku, q[3].tn / 64) && map(&tz, a.z, R, 2 * d, P.rpad, q[0].ku / 64) &&
      map(&tag, w.ag, R, d, P.rpad, q[1].ku / 64) && map(&tg, w.g, R, m, P.rpad, q[2].ku / 64) &&
      map(&thg, w.ag, R, d, P.rpad, q[3].ku / 64);
  if (!ok) return cudaErrorInvalidValue;
  cudaError_t e = launch_zero(w.ctr, (int32_t)(w.zero_bytes / 4), stream);
  if (e != cudaSuccess) return e;
  auto launch = [&](auto kernel) {
    cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)P.smem);
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)P.ncta, 1, 1);
    cfg.blockDim = dim3(kPThreads, 1, 1);
    cfg.dynamicSmemBytes = P.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, t0, t1, t3, t2, th, tz, tag, tg, thg, L);
  };
  return P.m_rows == 64 ? launch(predictor_kernel<64>) : launch(predictor_kernel<128>);
}

}  // namespace

size_t predictor_workspace(int32_t rows, int32_t d, int32_t m, int32_t V, bool own_hidden) {
  // more rows run as several launches over one workspace, the first the largest
  const int32_t full = std::min(rows, kMaxRows);
  if (!shapes_ok(full, d, m, V)) return 0;
  return carve(make_plan(full, d, m, V, device_sm_count()), full, d, m, own_hidden, nullptr).bytes;
}

bool predictor_supported(int32_t d, int32_t m, int32_t V) { return shapes_ok(1, d, m, V); }

cudaError_t launch_predictor(const PredictorArgs& a, void* ws, size_t ws_bytes, int32_t* status,
                             cudaStream_t stream) {
  for (int32_t r0 = 0; r0 < a.rows; r0 += kMaxRows) {
    PredictorArgs c = a;
    c.rows = std::min(kMaxRows, a.rows - r0);
    c.z = static_cast<const __nv_bfloat16*>(a.z) + (int64_t)r0 * 2 * a.d;
    c.out_tok = a.out_tok + r0;
    c.out_hidden = a.out_hidden != nullptr ? a.out_hidden + (int64_t)r0 * a.d : nullptr;
    const cudaError_t e = launch_rows(c, ws, ws_bytes, status, stream);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace ssd
