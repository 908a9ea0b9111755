// attention_tc.cu — frontier attention (step a2) on the 5th-generation tensor
// cores.  Same contract as the mma.sync kernel in attention.cu (Sec. 3.3
// "Verification as Auto Correction": the drafted block passes through the
// backbone in parallel; every draft attends to the committed cache and to the
// drafts before it in raster order):
//   O[b][j][h] = softmax_s(scale * Q[b][j][h] . K[b][g][s] + M(s, j)) V[b][g][s]
//
// Design (GB300, tcgen05 + TMEM): a persistent kernel, two CTAs per SM in
// clusters of kCluster, that walks work items (sequence, KV head, tile of 128
// query rows = drafts x the Hq/Hkv heads sharing the KV head, up to 128 heads;
// 64-row tiles with M = 64 products when a KV head's query rows fit in 64).
// The horizontal stage's 6 rows per head run here too (20 images: 28.9 -> 17.8
// us per step, 20.7 of it with this kernel in the mma.sync one's place).  The kernel is
// bound by the K/V stream when its items fill the GPU and by the serial chain
// of one item (load, S, softmax, PV per tile) when they do not, hence:
//  * two CTAs per SM: one CTA's start-up, item boundaries and tile chain
//    overlap the other's (one 202 KB CTA per SM with 128-key tiles before: the
//    24x24 sweep's step 62.6 us, the 16 x 32x32 GQA step 51.6 us, 8 x 64x64 at
//    2300-3800 keys 75.5 us; now 46.4, 34.8 and 68.4 us, the last 6.15 TB/s);
//  * the producer warp alone sets up, plans and issues its first item's five
//    copies, a lane each in one instruction, before the block's barrier.  What
//    an SM waits for between that and the first P is instruction fetch once
//    other kernels ran in between: code is rolled wherever it runs once per
//    item (the kernel is 64 KB; at 107 KB the sweep's CTAs spent 2.4 us on
//    their first softmax tile instead of 0.4);
//  * every CTA computes the same plan from the cache lengths: the sequences
//    longest first, only the items that have drafts, dealt in snake order.
//    When the live items fit more than once into the CTAs (small batches, or
//    the last passes of a batch whose other images are complete, which only
//    the device knows), 2 or kCluster CTAs of a cluster share an item, each
//    streaming a part of its keys, and merge their partial rows through
//    distributed shared memory at the end: no partials in global memory and
//    no second kernel (one image left of 8 x 64x64: the attention 40 -> 27 us;
//    two rounds on 8 x 24x24: 86.5 -> 67.8 us at the time with no combine launch).
//  * warp 4 (producer): decodes the next item, checks and converts its draft
//    positions into an item slot (two slots), loads Q through a 3D tensor map
//    and the item's K tiles of 64 keys; warp 5 streams its V tiles (TMA,
//    128-byte swizzle, one copy per tile, issued by two threads because one
//    thread issues only a few million copies per second).  The producers run
//    ahead of the other warps, so the next item's loads overlap the current
//    item's last tiles and its epilogue;
//  * warp 6 issues S_t = Q K_t^T (N = 64 keys) into one of two TMEM S/P
//    buffers; warp 7, once the softmax has written P_t, O += P_t V_t with P
//    read from TMEM (the A operand of a tcgen05.mma may live in tensor
//    memory);
//  * warps 0-3 (softmax; query row = TMEM lane, warp w owns lane quarter w):
//    tcgen05.ld of the row of S_t, the spatial mask (a per-row bitmask of the
//    visible drafts, built once per item), the running max and sum, and P_t as
//    bf16 pairs stored with tcgen05.st over the first half of the same TMEM
//    buffer; then the item's epilogue.  Warps whose rows are all padding skip
//    the math.  The running max is only moved (and O in TMEM rescaled with
//    tcgen05.ld/st) when it grows by more than 2^8; otherwise the exponentials
//    use the stale max, which the final sum shares, so the result is exact.
// K stages, V stages and S/P buffers form rings of two indexed by tile t mod
// 2, and one barrier per ring slot covers several conditions: "K_t loaded and
// S/P buffer free (PV of tile t - 2 done)" and "V_t loaded and P_t written".
// An mbarrier poll costs a few hundred cycles even when the phase is complete
// and a tcgen05.mma tens of cycles to issue, so each issuing thread has one
// wait, one group of products and one commit per tile.  Code that runs once
// per item (mask, bitmask, epilogue) is kept small: unrolled cold paths cost
// instruction-cache misses of thousands of cycles.
// Every barrier a thread waits on is at most one phase ahead of it (tile
// barriers are per tile parity, item barriers per item slot), so parity
// waits are unambiguous.
#include <algorithm>
#include <atomic>

#include "kernels.cuh"

namespace ssd {

namespace {

constexpr int kBM = 128;          // most query rows per CTA (TMEM lanes)
constexpr int KTC = 64;           // keys per tile
constexpr int kNB = 2;            // ring depth: K stages, V stages, TMEM S/P buffers
constexpr uint32_t kTmemCols = 256;  // S/P x 2 (64 columns each), O (up to 128 columns) at 128
constexpr int kSoftWarps = 4;     // one per TMEM lane quarter
constexpr int kThreadsTC = (kSoftWarps + 4) * 32;  // + K/Q producer, V producer, S, PV
constexpr int kCtasPerSmTC = 2;   // 2 x 256 TMEM columns, 2 x ~107 KB of shared memory
constexpr int kCluster = 4;       // CTAs that can share one item
// (the plan's pairs of CTAs, and its groups of two or four, lie inside one cluster)
static_assert(kCluster == 2 || kCluster == 4, "cluster size");
// Fewest key tiles of a part of the longest item, with 4 and with 2 parts, while every
// part has an SM to itself (few) and beyond that (many): merging parts takes ~3 us
// and a tile 0.3-0.5 us, and the parts of items that fill the SMs anyway only share
// them.  With 8 throughout: one 32x32 GQA image (17 tiles, 16 items) 16.4 us per
// step in 2 parts, 13.2 in 4; six of them (96 items) 24.4 in 2 parts, 22.6 whole; one
// 48x48 image 16.0 and 13.0.  With 4 throughout two rounds on 8 x 24x24 (11 tiles,
// 128 items) took 55.8 us, whole 47.8, and one 24x24 image 11.9 and 11.7.
constexpr int kFew4 = 4, kMany4 = 8, kFew2 = 8, kMany2 = 12;
constexpr float kLog2eTC = 1.4426950408889634f;
constexpr float kRescale = 8.0f;  // log2 growth of the running max that forces a rescale

// 16-lane TMEM accesses of the M = 64 products, whose row m sits in lane
// 32 (m / 16) + m % 16.  .16x256b: thread t holds rows t/4 and t/4 + 8 of the
// 16 lanes, columns 8u + 2 (t % 4) + {0, 1} of unit u, as registers 4u + {0, 1}
// (row t/4) and 4u + {2, 3} (row t/4 + 8).  .16x128b: column 4u + t % 4 of
// unit u, register 2u (row t/4) and 2u + 1 (row t/4 + 8).
__device__ __forceinline__ void tld16x256_x8(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tld16x256_x4(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tst16x256_x4(uint32_t taddr, const float* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16};" ::"r"(taddr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
      "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
      "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])),
      "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
      "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
      "r"(__float_as_uint(v[15]))
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tst16x128_x8(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
      "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// kind::f16 instruction descriptor: fp32 D, bf16 A and B, A K-major, M = m (64 or 128).
__host__ __device__ constexpr uint32_t idesc_f16(int n, bool b_mn_major, int m = kBM) {
  return idesc_bf16(m, n, false, b_mn_major);
}

// 64 consecutive 32-bit columns of this thread's TMEM lane (warp-collective).
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, float* v) {
  uint32_t r[64];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x64.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32,%33,%34,%35,%36,"
      "%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,"
      "%59,%60,%61,%62,%63}, [%64];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
        "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
        "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
        "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]),
        "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]),
        "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]),
        "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]),
        "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]),
        "=r"(r[62]), "=r"(r[63])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 64; ++i) v[i] = __uint_as_float(r[i]);
}

// ------------------------------------------------ cluster (distributed smem)
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t n;
  asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(n));
  return n;
}
__device__ __forceinline__ float4 ld_peer4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a)
               : "memory");
  return v;
}
__device__ __forceinline__ float2 ld_peer2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];"
               : "=f"(v.x), "=f"(v.y)
               : "r"(a)
               : "memory");
  return v;
}

struct TcLaunch {
  int32_t mtiles;    // query tiles of a KV head with D_max drafts
  int32_t drafts;    // drafts per query tile (BM / G): its rows are drafts * G <= BM
  int32_t order;     // leading CTAs that only order the launches (programmatic launch), else 0
  int32_t sms;       // of the device
  int32_t q_copies;  // copies per Q tile: 1, or one per 64 columns if the tile has fewer than BM rows
};

// One work item (sequence, KV head, query tile, part of the keys) as the
// producer hands it to the MMA and softmax warps; ntiles < 0 ends the CTA's
// work.
struct TcItem {
  int32_t b, g, row0, row_end, cache, Lk, k_lo, k_hi, ntiles;  // query rows row0 .. row_end - 1
  int32_t order;       // kOrder*: how the drafts' positions are ordered
  int32_t pad[2];
  int32_t kflat[128];  // raster position of each draft of b
};

// The drafts' raster positions: in any order (kflat), strictly increasing
// (kflat; draft j sees draft j' iff j' <= j), or the flat positions right after
// the cache (the step's frontier: cache + j, kflat unused).
constexpr int32_t kOrderAny = 0, kOrderIncreasing = 1, kOrderFlat = 2;

// A sequence of the plan, in longest-first order; its items are off .. off +
// (items of the sequence) - 1.
struct TcSeq {
  int32_t b, cache, nd, off;
};

// Q buffers: the next item's Q loads while the current one is in use where
// two fit beside the rings (64-row tiles).
template <int BM>
constexpr int kQBufs = BM == 64 ? 2 : 1;
template <int D, int BM>
constexpr size_t tc_smem_bytes() {
  return 1024 + (size_t)kQBufs<BM> * BM * D * 2 + (size_t)2 * kNB * KTC * D * 2 + 256 +
         2 * sizeof(TcItem) + (size_t)kBM * 8;
}

// One Q, K or V tile in the MMA's layout [d / 64][rows][128 B] (128-byte
// swizzle) with one copy: every map is a 4D view whose dimension of extent d /
// 64 steps 128 B inside a row, so that one instruction (with a lane per tile)
// can issue the copies of all three.
__device__ __forceinline__ void load_tile(void* dst, const CUtensorMap* map, int32_t c1, int32_t c2,
                                          int32_t c3, uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3, %4, %5}], [%6], %7;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar)),
      "l"(policy)
      : "memory");
}

// Byte offset of 16-byte chunk ch of row r of a CTA's partial O [rows][D] fp32
// in shared memory: chunks permuted by the row so that a warp's stores of one
// column by 32 rows spread over the banks.
template <int D>
__device__ __forceinline__ uint32_t part_off(int32_t r, int32_t ch) {
  return (uint32_t)r * (D * 4) + (uint32_t)((ch ^ (r & 7)) << 4);
}

// Rows r0 .. r1 - 1 of a K or V tile set to zero, by one warp.
template <int D>
__device__ __forceinline__ void clear_rows(unsigned char* tile, int32_t r0, int32_t r1, int lane) {
#pragma unroll 1
  for (int32_t i = lane; i < (r1 - r0) * (D / 8); i += 32) {
    const int32_t r = r0 + i / (D / 8), ch = i % (D / 8);
    *reinterpret_cast<uint4*>(tile + (ch >> 3) * (KTC * 128) + r * 128 + (ch & 7) * 16) =
        make_uint4(0u, 0u, 0u, 0u);
  }
}

// The keys c0 .. c0 + 63 a row may see, as a bit mask: cache keys are a prefix
// of the window (visible up to qpos), draft keys come from the row's
// visibility bits (vhi:vlo), keys past the part are dropped.
__device__ __forceinline__ uint64_t keep_mask(int32_t c0, int32_t cache, int32_t k_hi, int32_t qpos,
                                              uint64_t vlo, uint64_t vhi) {
  auto low = [](int32_t n) -> uint64_t {
    return n <= 0 ? 0ull : (n >= 64 ? ~0ull : ((1ull << n) - 1ull));
  };
  const int32_t base = c0 - cache;  // draft index of column 0
  uint64_t win;                     // bit jj: draft base + jj is visible
  if (base >= 128 || base <= -64) win = 0;
  else if (base >= 64) win = vhi >> (base - 64);
  else if (base > 0) win = (vlo >> base) | (vhi << (64 - base));
  else if (base == 0) win = vlo;
  else win = vlo << (-base);
  const int32_t seen_end = qpos < cache ? qpos + 1 : cache;
  return (low(seen_end - c0) | (win & ~low(cache - c0))) & low(k_hi - c0);
}
// Visibility bits of drafts 0 .. n - 1.
__device__ __forceinline__ void first_bits(int32_t n, uint64_t& lo, uint64_t& hi) {  // 1 <= n <= 128
  lo = n >= 64 ? ~0ull : ((1ull << n) - 1ull);
  hi = n <= 64 ? 0ull : (n >= 128 ? ~0ull : ((1ull << (n - 64)) - 1ull));
}

// BM = 128: query tiles of 128 rows, row m in TMEM lane m.  BM = 64 (items of
// at most 64 query rows): M = 64 products, row m in lane 32 (m / 16) + m % 16,
// so the rows spread over the four lane quarters and their softmax over all
// four SM sub-partitions.
template <int D, int BM>
__global__ void __launch_bounds__(kThreadsTC, kCtasPerSmTC)
frontier_attn_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                        const __grid_constant__ CUtensorMap tmV, AttnArgs a, TcLaunch L) {
  static_assert(BM == 64 || BM == 128, "query tile");
  static_assert(kLptMax <= kThreadsTC, "one thread per planned sequence");
  constexpr int NQ = kQBufs<BM>;
  constexpr int Q_BYTES = BM * D * 2;
  constexpr int KV_BYTES = KTC * D * 2;      // one K (or V) tile
  constexpr uint32_t kIdescS = idesc_f16(KTC, false, BM);
  constexpr uint32_t kIdescO = idesc_f16(D, true, BM);
  static_assert(BM * D * 4 <= 2 * kNB * KV_BYTES, "a partial O fits in the K and V rings");

  // Launch ordering (programmatic dependent launch): launched as a dependent of
  // the step's acceptance pass, whose results it does not read, the kernel
  // starts as the acceptance's CTAs retire.  The first cluster has no items:
  // its block 0 waits for the acceptance to complete and only then lets the
  // kernel queued after this one (the counts and draws, which read them) be
  // scheduled beside this one; the other blocks let it be scheduled at once
  // (it is scheduled when every block has).  A thread of a working CTA holds up
  // its whole warp in that wait: with the wait in a V producer's idle lane the
  // CTA stood still until the acceptance's end (one image left of 8 x 64x64
  // 44.0 -> 36.9 us per step, GQA batch 41.1 -> 39.1 without it).
  if ((int32_t)blockIdx.x < L.order) {
    if (pdl_first_block()) pdl_wait();
    pdl_launch_dependents();
    return;
  }
  if (L.order == 0) pdl_wait();  // on its own: what precedes it is complete
  pdl_launch_dependents();
  const int32_t cta = (int32_t)blockIdx.x - L.order, ncta = (int32_t)gridDim.x - L.order;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ TcSeq s_seq[kLptMax];     // the plan: sequences longest first
  __shared__ int2 s_key[kLptMax];      // (keys, items) of each sequence
  __shared__ int32_t s_plan[3];        // live items, log2 of the CTAs per item, items shared by two
  __shared__ TcItem* s_merge;          // the item this CTA shares with its group (split mode)
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* sQ = smem;                         // [NQ][Q_BYTES]
  unsigned char* sK = sQ + NQ * Q_BYTES;            // [kNB][KV_BYTES]
  unsigned char* sV = sK + kNB * KV_BYTES;          // [kNB][KV_BYTES]
  uint64_t* bar = reinterpret_cast<uint64_t*>(sV + kNB * KV_BYTES);
  uint64_t* q_full = bar;                           // [NQ] per Q buffer
  uint64_t* q_empty = q_full + 2;                   // [NQ]
  uint64_t* it_full = q_empty + 2;                  // [2] per item slot
  uint64_t* it_empty = it_full + 2;                 // [2]
  uint64_t* o_empty = it_empty + 2;                 // O read by the epilogue
  // per ring slot t % kNB: k_ready = K_t loaded and the TMEM S/P buffer free
  // (PV_{t-kNB} done); s_full = S_t done (K stage free); v_ready = V_t loaded
  // and P_t written; pv_done = PV_t done (V stage free)
  uint64_t* k_ready = o_empty + 1;                  // [kNB]
  uint64_t* s_full = k_ready + kNB;                 // [kNB]
  uint64_t* v_ready = s_full + kNB;                 // [kNB]
  uint64_t* pv_done = v_ready + kNB;                // [kNB]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(pv_done + kNB);
  TcItem* items = reinterpret_cast<TcItem*>(bar + 32);  // [2]
  float2* s_ml = reinterpret_cast<float2*>(items + 2);  // [128] split mode: (max, sum) of each row

  const int32_t G = a.Hq / a.Hkv;
  const int32_t tid = threadIdx.x, lane = tid & 31, warp = (int32_t)warp_uniform(tid >> 5);
  const bool planned = a.B <= kLptMax;

  // ---- set-up.  The first copies are the start-up's critical path, so the
  // producer warp alone initialises the barriers, makes the plan (of up to 32
  // sequences, a lane each) and issues its first item's copies before the
  // block's barrier; larger batches are planned by the whole block.
  const float c2 = (a.scale != 0.f ? a.scale : rsqrtf((float)D)) * kLog2eTC;
  const uint64_t pol = policy_evict_first(), polq = policy_evict_last();
  const int32_t per_b = a.Hkv * L.mtiles;
  // this thread's sequence: (keys, items), cache length and drafts; a lane of
  // the producer warp each, or a thread of the block each for larger batches
  const bool small = a.B <= 32;
  const int32_t seq = small ? (warp == kSoftWarps ? lane : a.B) : tid;
  int2 key = make_int2(0, 0);
  int32_t c = 0, n = 0;
  if (planned && seq < a.B) {
    c = a.cache_len[seq];
    n = attn_drafts(a, seq);
    if (n < 0 || n > a.D_max || c < 0 || c > a.L_max - n) {
      if (cta == 0) record_status(a.status, SSD_ERR_DEVICE_BOUNDS);
    } else if (n > 0) {
      key = make_int2(c + n, a.Hkv * (L.mtiles == 1 ? 1 : (n + L.drafts - 1) / L.drafts));
    }
  }
  // CTAs per item: as many of a cluster (a power of two) as leave one item or none per
  // group of them, if the parts are long enough; by one thread, from the live items,
  // the longest item's keys and all items' tiles
  auto put_plan = [&](int32_t total, int32_t most, int32_t tiles) {
    const int32_t cs = (int32_t)cluster_size(), most_tiles = (most + KTC - 1) / KTC;
    auto fits = [&](int parts, int few, int many) {
      const int n = parts * total;
      return parts <= cs && n <= ncta && most_tiles >= parts * (n <= L.sms ? few : many);
    };
    int32_t log = 0, pairs = 0;
    if (fits(4, kFew4, kMany4)) log = 2;
    else if (fits(2, kFew2, kMany2)) log = 1;
    else if (total < ncta && most_tiles >= 2 * kMany2 && 4 * most_tiles * total >= 5 * tiles)
      // Whole items leave CTAs idle, fewer than a second one each, and the longest is
      // a quarter longer than their mean: the longest items take those CTAs, two per
      // item in the first clusters (five 64x64 sequences of 600 to 4100 keys 49.5
      // -> 41.8 us, seven 56.7 -> 53.9; with items of one length the merges cost
      // more: six of 3000 to 4000 61.1 -> 62.2).
      pairs = min(ncta - total, total) & ~1;
    s_plan[0] = total;
    s_plan[1] = log;
    s_plan[2] = pairs;
  };
  TcSeq mine{0, 0, 0, 0x7fffffff};  // producer warp: this lane's sequence and first item (B <= 32)
  if (warp == kSoftWarps) {
    if (lane == 0) {
      for (int i = 0; i < NQ; ++i) {
        mbar_init(&q_full[i], L.q_copies);
        mbar_init(&q_empty[i], 1);
      }
      for (int i = 0; i < 2; ++i) {
        mbar_init(&it_full[i], 1);
        mbar_init(&it_empty[i], kSoftWarps + 1);  // and the V producer
      }
      mbar_init(o_empty, kSoftWarps);
#pragma unroll 1
      for (int s = 0; s < kNB; ++s) {
        mbar_init(&k_ready[s], 2);
        mbar_init(&s_full[s], 1);
        mbar_init(&v_ready[s], 1 + kSoftWarps);
        mbar_init(&pv_done[s], 1);
      }
      fence_barrier_init();
      // every S/P buffer starts free: the PV arrivals of the first round
#pragma unroll 1
      for (int s = 0; s < kNB; ++s) mbar_arrive(&k_ready[s]);
      s_merge = nullptr;
    }
    if (small) {
      // sequences longest first (ties by index), those without drafts last
      int32_t off = 0;
#pragma unroll 2
      for (int32_t j = 0; j < a.B; ++j) {
        const int32_t kj = __shfl_sync(0xffffffffu, key.x, j), cj = __shfl_sync(0xffffffffu, key.y, j);
        off += (kj > key.x || (kj == key.x && j < lane)) ? cj : 0;
      }
      if (key.y > 0) mine = TcSeq{lane, c, n, off};
      const int32_t total = __reduce_add_sync(0xffffffffu, key.y);
      const int32_t most = __reduce_max_sync(0xffffffffu, key.x);
      const int32_t tiles = __reduce_add_sync(0xffffffffu, (key.x + KTC - 1) / KTC * key.y);
      if (lane == 0) put_plan(total, most, tiles);
    }
    __syncwarp();
  } else if (warp == kSoftWarps + 1) {
    if (lane < 3)  // the first copies need the descriptors
      prefetch_tensormap(lane == 0 ? &tmQ : (lane == 1 ? &tmK : &tmV));
  } else if (warp == kSoftWarps + 3) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  if (planned && !small) {
    if (tid < a.B) s_key[tid] = key;
    __syncthreads();
    if (tid < a.B) {
      int32_t r = 0, off = 0, total = 0, most = 0, tiles = 0;
#pragma unroll 1
      for (int32_t j = 0; j < a.B; ++j) {
        const int2 kj = s_key[j];
        const bool ahead = kj.x > key.x || (kj.x == key.x && j < tid);
        r += ahead ? 1 : 0;
        off += ahead ? kj.y : 0;
        total += kj.y;
        most = max(most, kj.x);
        tiles += (kj.x + KTC - 1) / KTC * kj.y;
      }
      s_seq[r] = TcSeq{tid, c, n, off};
      if (tid == 0) put_plan(total, most, tiles);
    }
    __syncthreads();
  }

  int32_t n_items = 0, ns_log = 0, shared = 0;
  auto read_plan = [&]() {
    n_items = planned ? s_plan[0] : a.B * per_b;
    if (planned) {
      shared = s_plan[2];
      ns_log = cta < 2 * shared ? 1 : s_plan[1];
    }
  };
  uint32_t tmem = 0, tS = 0, tO = 0;
  auto block_start = [&]() {  // every warp: the set-up is done
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    tmem = *tmem_slot;
    tS = tmem;          // [kNB] x KTC columns: S_t in fp32, then P_t in bf16
    tO = tmem + 128;    // up to 128 columns
  };
  if (warp != kSoftWarps) {
    block_start();
    read_plan();
  }

  if (warp == kSoftWarps) {
    // ------------------------------------------------------------ producer
    // Items in snake order over the longest-first list: round k takes items
    // k * ngroups + (group, or its mirror on odd rounds).
    const int32_t HW = a.grid.grid_h * a.grid.grid_w;
    bool ok = true, started = false;
    const bool leader = elect_one();
    int32_t k = 0;        // items handed out
    uint32_t T = 0;       // K tiles issued
    // per copy
    const uint32_t q_bytes = (uint32_t)(L.drafts * G * 128) * (L.q_copies == 1 ? D / 64 : 1);
    read_plan();
    const int32_t ns = 1 << ns_log;
    const int32_t part = cta & (ns - 1);
    // (shared items: one round, the pairs first)
    const int32_t group = ns_log > 0 || shared == 0 ? cta >> ns_log : cta - shared;
    const int32_t ngroups = shared > 0 ? n_items : ncta >> ns_log;
#pragma unroll 1
    for (int32_t round = 0; ok; ++round) {
      const int32_t base = round * ngroups;
      if (base >= n_items) break;
      const int32_t i = base + ((round & 1) ? (ngroups - 1 - group) : group);
      if (i >= n_items) continue;
      TcSeq q;
      int32_t mt = 1;
      if (small) {
        // the sequence with the last first item at or before i
        const int32_t first = __reduce_max_sync(0xffffffffu, mine.off <= i ? mine.off : -1);
        const int src = __ffs(__ballot_sync(0xffffffffu, mine.off == first)) - 1;
        q.b = src;
        q.cache = __shfl_sync(0xffffffffu, mine.cache, src);
        q.nd = __shfl_sync(0xffffffffu, mine.nd, src);
        q.off = first;
      } else if (planned) {
        // (sequences without items come last, at off == n_items)
        int32_t r = -1;
#pragma unroll 1
        for (int32_t r0 = 0; r0 < a.B; r0 += 32) {
          const bool le = r0 + lane < a.B && s_seq[r0 + lane].off <= i;
          const uint32_t m = __ballot_sync(0xffffffffu, le);
          if (m == 0) break;
          r = r0 + 31 - __clz(m);
        }
        q = s_seq[r];
      } else {
        q.b = i / per_b;
        q.off = q.b * per_b;
        q.cache = a.cache_len[q.b];
        q.nd = attn_drafts(a, q.b);
        mt = L.mtiles;
      }
      const int32_t b = q.b, cache = q.cache, nd = q.nd;
      if (planned && L.mtiles > 1) mt = (nd + L.drafts - 1) / L.drafts;
      int32_t g = i - q.off, mtile = 0;
      if (mt > 1) {
        const int32_t rem = g;
        g = rem / mt;
        mtile = rem - g * mt;
      }
      const int s = k & 1;
      TcItem& it = items[s];
      // (a slot is rewritten once the softmax is done with its item before)
      if (k >= 2 && lane == 0) ok = mbar_wait(&it_empty[s], ((k >> 1) - 1) & 1, a.status);
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
      bool valid = planned || (nd >= 0 && nd <= a.D_max && cache >= 0 && cache <= a.L_max - nd);
      int32_t order = kOrderFlat;
      if (!(a.raster && a.grid.row_stride == a.grid.grid_w) && valid) {
        // draft positions (validity is identical in every item of b); strictly
        // increasing ones?  (The draft before j is lane - 1's, or the last lane's
        // of the 32 before.)
        bool bad = false, dec = false;
        int32_t last = -1;
#pragma unroll 1
        for (int32_t j = lane; j - lane < nd; j += 32) {
          int32_t kf = 0x7fffffff;
          if (j < nd) {
            const int32_t gidx = attn_draft_pos(a, b, j);
            if (gidx < 0 || gidx >= HW) {
              bad = true;
            } else {
              const int32_t y = gidx / a.grid.grid_w, x = gidx - y * a.grid.grid_w;
              kf = a.grid.prefix_len + y * a.grid.row_stride + x;
            }
            it.kflat[j] = kf;
          }
          const int32_t up = __shfl_up_sync(0xffffffffu, kf, 1);
          if (j < nd && kf <= (lane > 0 ? up : last)) dec = true;
          last = __shfl_sync(0xffffffffu, kf, 31);
        }
        valid = !__any_sync(0xffffffffu, bad);
        order = __any_sync(0xffffffffu, dec) ? kOrderAny : kOrderIncreasing;
      }
      if (!valid && i == q.off && part == 0 && lane == 0)
        record_status(a.status, SSD_ERR_DEVICE_BOUNDS);
      const int32_t Lk = cache + nd, draft0 = mtile * L.drafts;
      if (!valid || draft0 >= nd) continue;
      const int32_t tiles = (Lk + KTC - 1) / KTC;
      const int32_t t_lo = (tiles * part) >> ns_log, t_hi = (tiles * (part + 1)) >> ns_log;
      const int32_t ntiles = t_hi - t_lo;
      const int32_t kvrow0 = (b * a.Hkv + g) * a.L_max + t_lo * KTC;  // 2D row of the first key
      const int32_t qrow = b * a.D_max + draft0;
      const int sq = k % NQ;
      int t = 0;
      if (lane == 0) {
        it.b = b;
        it.g = g;
        it.row0 = draft0 * G;
        it.row_end = min(nd, draft0 + L.drafts) * G;
        it.cache = cache;
        it.Lk = Lk;
        it.k_lo = t_lo * KTC;
        it.k_hi = min(Lk, t_hi * KTC);
        it.ntiles = ntiles;
        it.order = order;
        if (ns > 1) s_merge = &it;
      }
      if (ntiles == 0) continue;  // split mode: fewer tiles than CTAs in the group
      __syncwarp();
      if (k == 0) {
        // the CTA's first item: every ring slot is free, so its first K, Q and V
        // copies go out at once, one lane each
        t = min(ntiles, kNB);
        // lanes 0 K0, 1 Q, 2 V0, 3 K1, 4 V1, 5 (q_copies = 2) Q's second half
        const bool is_q = lane == 1 || lane == 5, is_k = lane == 0 || lane == 3;
        const int st = lane >= 3 ? 1 : 0;  // ring slot; Q: half
        if (is_q ? st < L.q_copies : (lane < 5 && st < ntiles)) {
          uint64_t* bar1 = is_q ? &q_full[0] : (is_k ? &k_ready[st] : &v_ready[st]);
          unsigned char* dst = is_q ? sQ + st * (BM * 128) : (is_k ? sK : sV) + st * KV_BYTES;
          mbar_arrive_expect_tx(bar1, is_q ? q_bytes : KV_BYTES);
          load_tile(dst, is_q ? &tmQ : (is_k ? &tmK : &tmV), is_q ? g * G : kvrow0 + st * KTC,
                    is_q ? qrow : 0, is_q ? st : 0, bar1, is_q ? polq : pol);
        }
        T = t;
        __syncwarp();
        if (lane == 0) mbar_arrive(&it_full[0]);
        block_start();
        started = true;
      } else if (lane == 0) {
        mbar_arrive(&it_full[s]);
        // Q of this item into its buffer once the S products of the item before
        // that used it are done
        if (k >= NQ) ok = mbar_wait(&q_empty[sq], ((k / NQ) - 1) & 1, a.status);
        if (ok) {
#pragma unroll 1
          for (int h = 0; h < L.q_copies; ++h) {
            mbar_arrive_expect_tx(&q_full[sq], q_bytes);
            load_tile(sQ + sq * Q_BYTES + h * (BM * 128), &tmQ, g * G, qrow, h, &q_full[sq], polq);
          }
        }
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
#pragma unroll 1
      for (; t < ntiles && ok; ++t, ++T) {
        const int sb = T % kNB;
        // K stage sb is free once S_{T-kNB} is done
        ok = T < (uint32_t)kNB || mbar_wait_warp(&s_full[sb], ((T / kNB) - 1) & 1, a.status);
        if (!ok) break;
        if (leader) {
          mbar_arrive_expect_tx(&k_ready[sb], KV_BYTES);
          load_tile(sK + sb * KV_BYTES, &tmK, kvrow0 + t * KTC, 0, 0, &k_ready[sb], pol);
        }
        __syncwarp();
      }
      ++k;
    }
    if (ok) {
      // end marker
      const int s = k & 1;
      if (k >= 2 && lane == 0) ok = mbar_wait(&it_empty[s], ((k >> 1) - 1) & 1, a.status);
      if (lane == 0 && ok) {
        // (split mode: at most one item, in slot 0, which the merge still reads)
        items[s].ntiles = -1;
        mbar_arrive(&it_full[s]);
      }
    }
    __syncwarp();
    if (!started) block_start();
  } else if (warp == kSoftWarps + 1) {
    // ---------------------------------------------------------- V producer
    // Follows the item slots like the MMA warp; a slot is not rewritten before
    // the softmax and this warp are done with its item (an item whose V tiles
    // are all among the first copies can finish without this warp).
    const bool leader = elect_one();
    uint32_t T = 0;
    bool ok = true;
#pragma unroll 1
    for (int32_t k = 0; ok; ++k) {
      const int s = k & 1;
      if (!mbar_wait_warp(&it_full[s], (k >> 1) & 1, a.status)) break;
      const TcItem& it = items[s];
      const int32_t ntiles = (int32_t)warp_uniform((uint32_t)it.ntiles);
      if (ntiles < 0) break;
      const int32_t kvrow0 =
          (int32_t)warp_uniform((uint32_t)((it.b * a.Hkv + it.g) * a.L_max + it.k_lo));
      int t = 0;
      if (k == 0) T = t = min(ntiles, kNB);  // issued by the producer with the first K tiles
#pragma unroll 1
      for (; t < ntiles; ++t, ++T) {
        const int sb = T % kNB;
        // V stage sb is free once PV_{T-kNB} is done
        ok = T < (uint32_t)kNB || mbar_wait_warp(&pv_done[sb], ((T / kNB) - 1) & 1, a.status);
        if (!ok) break;
        if (leader) {
          mbar_arrive_expect_tx(&v_ready[sb], KV_BYTES);
          load_tile(sV + sb * KV_BYTES, &tmV, kvrow0 + t * KTC, 0, 0, &v_ready[sb], pol);
        }
        __syncwarp();
      }
      if (ok && leader) mbar_arrive(&it_empty[s]);
    }
    __syncwarp();
  } else if (warp == kSoftWarps + 2) {
    // ----------------------------------------------------------- S products
    // (every lane in the loop, one elected around the products: elect_one())
    const uint32_t tSu = warp_uniform(tS), aQ = warp_uniform(smem_u32(sQ));
    const uint32_t aK = warp_uniform(smem_u32(sK));
    const bool leader = elect_one();
    bool ok = true;
    uint32_t T = 0;
#pragma unroll 1
    for (int32_t k = 0; ok; ++k) {
      const int s = k & 1, sq = k % NQ;
      if (!mbar_wait_warp(&it_full[s], (k >> 1) & 1, a.status)) break;
      const int32_t ntiles = (int32_t)warp_uniform((uint32_t)items[s].ntiles);
      if (ntiles < 0) break;
      if (!mbar_wait_warp(&q_full[sq], (k / NQ) & 1, a.status)) break;
      tc_fence_after();
      const uint64_t dq = smem_desc(aQ + sq * Q_BYTES, 16, 1024);
#pragma unroll 1
      for (int t = 0; t < ntiles; ++t, ++T) {
        const int sb = T % kNB;
        ok = mbar_wait_warp(&k_ready[sb], (T / kNB) & 1, a.status);
        if (!ok) break;
        tc_fence_after();
        const uint64_t dk = smem_desc(aK + sb * KV_BYTES, 16, 1024);
        if (leader) {
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) {
            const int sub = ks >> 2, kin = (ks & 3) * 32;
            mma_ss(tSu + sb * KTC, smem_desc_at(dq, sub * (BM * 128) + kin),
                 smem_desc_at(dk, sub * (KTC * 128) + kin), kIdescS, ks > 0 ? 1u : 0u);
          }
          mma_commit(&s_full[sb]);
          if (t == ntiles - 1) mma_commit(&q_empty[sq]);
        }
        __syncwarp();
      }
    }
    __syncwarp();
  } else if (warp == kSoftWarps + 3) {
    // ---------------------------------------------------------- PV products
    // Issued by a warp of its own: an mbarrier poll takes a few hundred cycles,
    // so one warp issuing both products would be the slowest stage of the tile
    // loop.
    const uint32_t tSu = warp_uniform(tS), tOu = warp_uniform(tO), aV = warp_uniform(smem_u32(sV));
    const bool leader = elect_one();
    bool ok = true;
    uint32_t T = 0;
#pragma unroll 1
    for (int32_t k = 0; ok; ++k) {
      const int s = k & 1;
      if (!mbar_wait_warp(&it_full[s], (k >> 1) & 1, a.status)) break;
      const int32_t ntiles = (int32_t)warp_uniform((uint32_t)items[s].ntiles);
      if (ntiles < 0) break;
      int32_t left = (int32_t)warp_uniform((uint32_t)(items[s].k_hi - items[s].k_lo));  // keys
      // the first product of the item overwrites O: the epilogue of the item before must be done
      if (k >= 1 && !mbar_wait_warp(o_empty, (k - 1) & 1, a.status)) break;
#pragma unroll 1
      for (int t = 0; t < ntiles; ++t, ++T, left -= KTC) {
        const int sb = T % kNB;
        ok = mbar_wait_warp(&v_ready[sb], (T / kNB) & 1, a.status);
        if (!ok) break;
        tc_fence_after();
        if (left < KTC) {
          // The sequence's last keys: the slots behind them hold whatever the cache
          // holds, and their P of 0 times a NaN or an infinity is a NaN in every row.
          // Steps of 16 keys past the last are left out, and the rest of its step is
          // cleared (whole rows of the tile, so the swizzle does not matter).
          clear_rows<D>(sV + sb * KV_BYTES, left, (left + 15) & ~15, lane);
          fence_proxy_async_shared();
          __syncwarp();
        }
        // A = P in TMEM (16 keys = 8 columns per step), B = V (MN-major: d
        // atoms KTC*128 bytes apart, 8-key groups 1 KB apart; 16 keys = 2 KB)
        const uint64_t dv = smem_desc(aV + sb * KV_BYTES, KTC * 128, 1024);
        if (leader) {
#pragma unroll
          for (int kk = 0; kk < KTC / 16; ++kk)
            if (16 * kk < left)
              mma_ts(tOu, tSu + sb * KTC + kk * 8, smem_desc_at(dv, kk * 2048), kIdescO,
                     (t == 0 && kk == 0) ? 0u : 1u);
          mma_commit(&pv_done[sb]);
          mma_commit(&k_ready[sb]);  // S_{T+kNB} may start: the S/P buffer is free again
        }
        __syncwarp();
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------- softmax
    // BM = 128: thread = query row = TMEM lane.  BM = 64: item row m sits in
    // TMEM lane 32 (m / 16) + m % 16, so lane quarter q holds item rows 16q ..
    // 16q + 15; with 16-lane accesses each thread holds two rows (t / 4 and
    // t / 4 + 8 of the quarter) x 16 of the 64 columns, and the four threads
    // t % 4 of a row finish its maxima and sums by shuffles.
    constexpr int NR = BM == 64 ? 2 : 1;      // rows per thread
    const bool split = ns_log > 0;
    if (split && tid < kBM) s_ml[tid] = make_float2(-INFINITY, 0.f);  // rows of a part without keys
    const uint32_t lane_off = (uint32_t)(warp * 32) << 16;
    const int cq = lane & 3;
    bool ok = true;
    uint32_t T = 0;
    for (int32_t k = 0; ok; ++k) {
      const int s = k & 1;
      if (!mbar_wait(&it_full[s], (k >> 1) & 1, a.status)) { ok = false; break; }
      const TcItem& it = items[s];
      const int32_t ntiles = it.ntiles;
      if (ntiles < 0) break;
      const int32_t row0 = it.row0, row_end = it.row_end, cache = it.cache, Lk = it.Lk;
      const int32_t k_lo = it.k_lo, k_hi = it.k_hi;
      const int32_t* kflat = it.kflat;
      const bool warp_live = row0 + warp * (BM / 4) < row_end;
      // this thread's query rows: item row, draft and position
      const int32_t order = it.order;
      int32_t rl[NR], jq[NR], qpos[NR];
#pragma unroll
      for (int e = 0; e < NR; ++e) {
        rl[e] = BM == 64 ? warp * 16 + (lane >> 2) + 8 * e : warp * 32 + lane;
        const int32_t r = row0 + rl[e];
        jq[e] = r < row_end ? r / G : 0;
        qpos[e] = r >= row_end ? 0x7fffffff : (order == kOrderFlat ? cache + jq[e] : kflat[jq[e]]);
      }
      // cache slots below every query position of this item are visible to all rows
      int32_t minq = 0x7fffffff;
      const int32_t j_lo = row0 / G;
      if (order == kOrderFlat) {
        minq = cache;
      } else if (order == kOrderIncreasing) {
        minq = kflat[j_lo];
      } else {
        const int32_t j_end = row_end / G;
#pragma unroll 1
        for (int32_t j = j_lo + lane; j < j_end; j += 32) minq = min(minq, kflat[j]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) minq = min(minq, __shfl_xor_sync(0xffffffffu, minq, o));
      }
      const int32_t mask_from = min(cache, minq + 1);
      // visibility of the item's drafts to each row: bit j of (vhi:vlo) is
      // kflat[j] <= qpos, that is j <= jq for increasing positions.  Runs once
      // per item, so the general loop is kept rolled (small code: a cold
      // unrolled path costs instruction-cache misses).
      uint64_t vlo[NR], vhi[NR];
#pragma unroll
      for (int e = 0; e < NR; ++e) vlo[e] = vhi[e] = 0;
      if (warp_live && order != kOrderAny) {
#pragma unroll
        for (int e = 0; e < NR; ++e) first_bits(jq[e] + 1, vlo[e], vhi[e]);
      } else if (warp_live) {
        const int32_t nd = Lk - cache;
#pragma unroll 1
        for (int j = 0; j < nd; j += 4) {
          const int4 kf = *reinterpret_cast<const int4*>(kflat + j);
#pragma unroll
          for (int e = 0; e < NR; ++e) {
            const uint64_t bits =
                (uint64_t)((uint32_t)(kf.x <= qpos[e]) | ((uint32_t)(kf.y <= qpos[e]) << 1) |
                           ((uint32_t)(kf.z <= qpos[e]) << 2) | ((uint32_t)(kf.w <= qpos[e]) << 3));
            if (j < 64) vlo[e] |= bits << j;
            else vhi[e] |= bits << (j - 64);
          }
        }
      }
      float m_run[NR], l_run[NR];  // l_run: BM = 64: this thread's columns only, until the epilogue
#pragma unroll
      for (int e = 0; e < NR; ++e) {
        m_run[e] = -INFINITY;
        l_run[e] = 0.f;
      }
#pragma unroll 1
      for (int t = 0; t < ntiles; ++t, ++T) {
        const int sb = T % kNB;
        if (!mbar_wait(&s_full[sb], (T / kNB) & 1, a.status)) ok = false;
        tc_fence_after();
        if (warp_live) {
          const int32_t c0 = k_lo + t * KTC;
          const bool masked = c0 + KTC > k_hi || c0 + KTC > mask_from;
          float alpha[NR];
          bool moved = false;
          // the running max moves only when it grows by more than 2^kRescale
          auto move_max = [&](int e, float mx) {
            alpha[e] = 1.f;
            if (mx != -INFINITY && (m_run[e] == -INFINITY || (mx - m_run[e]) * c2 > kRescale)) {
              alpha[e] = (m_run[e] == -INFINITY) ? 0.f : ex2_approx((m_run[e] - mx) * c2);
              m_run[e] = mx;
              moved = true;
            }
            return (m_run[e] == -INFINITY) ? 0.f : m_run[e] * c2;
          };
          uint32_t pk[32 / NR];
          if constexpr (BM == 128) {
            float sv[64];
            tmem_ld64(tS + lane_off + sb * KTC, sv);
            if (masked) {
              const uint64_t keep = keep_mask(c0, cache, k_hi, qpos[0], vlo[0], vhi[0]);
#pragma unroll
              for (int jj = 0; jj < 64; ++jj)
                if (!((keep >> jj) & 1ull)) sv[jj] = -INFINITY;
            }
            float m4[4];  // four chains of three-input maxima
#pragma unroll
            for (int w = 0; w < 4; ++w) {
              m4[w] = fmax3(sv[16 * w], sv[16 * w + 1], sv[16 * w + 2]);
#pragma unroll
              for (int i = 3; i < 15; i += 2) m4[w] = fmax3(m4[w], sv[16 * w + i], sv[16 * w + i + 1]);
              m4[w] = fmaxf(m4[w], sv[16 * w + 15]);
            }
            const float moff = move_max(0, fmaxf(fmax3(m4[0], m4[1], m4[2]), m4[3]));
            const float2 cc = make_float2(c2, c2), nm = make_float2(-moff, -moff);
            float2 s4[4];
#pragma unroll
            for (int i = 0; i < 32; ++i) {
              const float2 x = ffma2(make_float2(sv[2 * i], sv[2 * i + 1]), cc, nm);
              const float2 e = make_float2(ex2_approx(x.x), ex2_approx(x.y));
              s4[i & 3] = i < 4 ? e : fadd2(s4[i & 3], e);
              pk[i] = pack_bf16x2(e.x, e.y);
            }
            const float2 ss = fadd2(fadd2(s4[0], s4[1]), fadd2(s4[2], s4[3]));
            l_run[0] = l_run[0] * alpha[0] + (ss.x + ss.y);
          } else {
            float sv[32];
            tld16x256_x8(tS + lane_off + sb * KTC, sv);
            if (masked) {
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                const uint64_t keep = keep_mask(c0, cache, k_hi, qpos[e], vlo[e], vhi[e]) >> (2 * cq);
#pragma unroll
                for (int u = 0; u < 8; ++u)
#pragma unroll
                  for (int x = 0; x < 2; ++x)
                    if (!((keep >> (8 * u + x)) & 1ull)) sv[4 * u + 2 * e + x] = -INFINITY;
              }
            }
            float mx[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              float m0 = fmax3(sv[2 * e], sv[2 * e + 1], sv[4 + 2 * e]);
              float m1 = fmax3(sv[4 + 2 * e + 1], sv[8 + 2 * e], sv[8 + 2 * e + 1]);
              m0 = fmax3(m0, sv[12 + 2 * e], sv[12 + 2 * e + 1]);
              m1 = fmax3(m1, sv[16 + 2 * e], sv[16 + 2 * e + 1]);
              m0 = fmax3(m0, sv[20 + 2 * e], sv[20 + 2 * e + 1]);
              m1 = fmax3(m1, sv[24 + 2 * e], sv[24 + 2 * e + 1]);
              mx[e] = fmaxf(fmax3(m0, sv[28 + 2 * e], sv[28 + 2 * e + 1]), m1);
              mx[e] = fmaxf(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], 1));
              mx[e] = fmaxf(mx[e], __shfl_xor_sync(0xffffffffu, mx[e], 2));
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const float moff = move_max(e, mx[e]);
              const float2 cc = make_float2(c2, c2), nm = make_float2(-moff, -moff);
              float2 s2[2];
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                const float2 x = ffma2(make_float2(sv[4 * u + 2 * e], sv[4 * u + 2 * e + 1]), cc, nm);
                const float2 p = make_float2(ex2_approx(x.x), ex2_approx(x.y));
                s2[u & 1] = u < 2 ? p : fadd2(s2[u & 1], p);
                pk[2 * u + e] = pack_bf16x2(p.x, p.y);
              }
              const float2 ss = fadd2(s2[0], s2[1]);
              l_run[e] = l_run[e] * alpha[e] + (ss.x + ss.y);
            }
          }
          // O may be rescaled once PV_{T-1} is done
          if (__any_sync(0xffffffffu, moved && t > 0)) {
            if (!mbar_wait(&pv_done[(T - 1) % kNB], ((T - 1) / kNB) & 1, a.status)) ok = false;
            tc_fence_after();
#pragma unroll 1
            for (int cc = 0; cc < D / 32; ++cc) {
              const uint32_t ta = tO + lane_off + cc * 32;
              if constexpr (BM == 128) {
                float ov[32];
                tmem_ld32(ta, ov);
#pragma unroll
                for (int i = 0; i < 32; ++i) ov[i] *= alpha[0];
                tmem_st32(ta, ov);
              } else {
                float ov[16];
                tld16x256_x4(ta, ov);
#pragma unroll
                for (int i = 0; i < 16; ++i) ov[i] *= alpha[(i >> 1) & 1 ? NR - 1 : 0];
                tst16x256_x4(ta, ov);
              }
            }
          }
          // P_T as bf16 pairs over the first half of its S buffer
          if constexpr (BM == 128) tmem_st32(tS + lane_off + sb * KTC, pk);
          else tst16x128_x8(tS + lane_off + sb * KTC, pk);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&v_ready[sb]);
      }
      // ---- epilogue: wait for the item's last PV product; normalise and write
      // the rows, or (split mode) leave them for the merge
      const uint32_t Tl = T - 1;
      if (!mbar_wait(&pv_done[Tl % kNB], (Tl / kNB) & 1, a.status)) ok = false;
      tc_fence_after();
      if (warp_live) {
        if constexpr (BM == 64) {
#pragma unroll
          for (int e = 0; e < NR; ++e) {
            l_run[e] += __shfl_xor_sync(0xffffffffu, l_run[e], 1);
            l_run[e] += __shfl_xor_sync(0xffffffffu, l_run[e], 2);
          }
        }
        const int32_t b = it.b, g = it.g;
        bool live[NR];
        float inv[NR];
        int64_t orow[NR];
#pragma unroll
        for (int e = 0; e < NR; ++e) {
          const int32_t r = row0 + rl[e], h = g * G + r - jq[e] * G;
          orow[e] = ((int64_t)b * a.D_max + jq[e]) * a.Hq + h;
          // (debug builds: the row's store index against its buffer)
          live[e] = r < row_end && ok && dbg_in(orow[e], (int64_t)a.B * a.D_max * a.Hq, a.status);
          // fast reciprocal and logarithm: the epilogue runs once per item, and
          // its instruction count is its cost
          inv[e] = l_run[e] > 0.f ? __fdividef(1.0f, l_run[e]) : 0.f;
          if (live[e] && (BM == 128 || cq == 0)) {
            if (split)
              s_ml[rl[e]] = make_float2(m_run[e], l_run[e]);
            else if (a.lse != nullptr)
              a.lse[((int64_t)b * a.Hq + h) * a.D_max + jq[e]] =
                  l_run[e] > 0.f ? (m_run[e] * (c2 / kLog2eTC) + __logf(l_run[e])) : -INFINITY;
          }
        }
#pragma unroll 1
        for (int cc = 0; cc < D / 32; ++cc) {
          if constexpr (BM == 128) {
            float ov[32];
            tmem_ld32(tO + lane_off + cc * 32, ov);
            if (!live[0]) continue;
            if (split) {  // the partial row over the K and V rings, which are done
#pragma unroll
              for (int i = 0; i < 8; ++i)
                *reinterpret_cast<float4*>(sK + part_off<D>(rl[0], cc * 8 + i)) =
                    make_float4(ov[4 * i], ov[4 * i + 1], ov[4 * i + 2], ov[4 * i + 3]);
            } else {
              __nv_bfloat16* ob = reinterpret_cast<__nv_bfloat16*>(a.o) + orow[0] * D + cc * 32;
#pragma unroll
              for (int i = 0; i < 32; i += 8) {
                uint4 w;
                w.x = pack_bf16x2(ov[i] * inv[0], ov[i + 1] * inv[0]);
                w.y = pack_bf16x2(ov[i + 2] * inv[0], ov[i + 3] * inv[0]);
                w.z = pack_bf16x2(ov[i + 4] * inv[0], ov[i + 5] * inv[0]);
                w.w = pack_bf16x2(ov[i + 6] * inv[0], ov[i + 7] * inv[0]);
                *reinterpret_cast<uint4*>(ob + i) = w;
              }
            }
          } else {
            float ov[16];
            tld16x256_x4(tO + lane_off + cc * 32, ov);
#pragma unroll
            for (int e = 0; e < NR; ++e) {
              if (!live[e]) continue;
              // columns cc * 32 + 8 u + 2 cq + {0, 1}
              if (split) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                  *reinterpret_cast<float2*>(sK + part_off<D>(rl[e], cc * 8 + 2 * u + (cq >> 1)) +
                                             (cq & 1) * 8) =
                      make_float2(ov[4 * u + 2 * e], ov[4 * u + 2 * e + 1]);
              } else {
                __nv_bfloat16* ob =
                    reinterpret_cast<__nv_bfloat16*>(a.o) + orow[e] * D + cc * 32 + 2 * cq;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                  *reinterpret_cast<uint32_t*>(ob + 8 * u) =
                      pack_bf16x2(ov[4 * u + 2 * e] * inv[e], ov[4 * u + 2 * e + 1] * inv[e]);
              }
            }
          }
        }
      }
      // O and the item slot are free for the next items
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(o_empty);
        mbar_arrive(&it_empty[s]);
      }
    }
  }
  // ---- split mode: merge the group's partial rows.  Every CTA of the grid
  // takes the same branch (the plan is the same in all of them).
  if (ns_log > 0) {
    const int32_t ns = 1 << ns_log, part = cta & (ns - 1);
    __syncwarp();
    cluster_sync_all();  // every partial row and its (max, sum) written
    const TcItem* it = s_merge;
    if (it != nullptr) {
      const int32_t row0 = it->row0, rows = it->row_end - row0;
      const int32_t cs = (int32_t)cluster_size();
      const uint32_t rank0 = (uint32_t)(cta % cs - part);  // the group's first CTA
      const uint32_t base_o = smem_u32(sK), base_ml = smem_u32(s_ml);
      constexpr int LPR = D / 4;              // lanes per row (a float4 each)
      constexpr int RPW = 32 / LPR;           // rows per warp and step
      const int sub = lane / LPR, ch = lane % LPR;
      // the group's CTAs take every ns-th row, two rows of a lane at a time (both
      // rows' remote loads in flight)
      constexpr int RS = (kThreadsTC / 32) * RPW;  // rows per step of the block
#pragma unroll 1
      for (int32_t r0 = part + ns * (warp * RPW + sub); r0 < rows; r0 += 2 * ns * RS) {
        float2 ml[2][kCluster];
        float4 x[2][kCluster];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int32_t r = min(r0 + e * ns * RS, rows - 1);
#pragma unroll
          for (int p = 0; p < kCluster; ++p)
            if (p < ns) {
              ml[e][p] = ld_peer2(peer_addr(base_ml + r * 8, rank0 + p));
              x[e][p] = ld_peer4(peer_addr(base_o + part_off<D>(r, ch), rank0 + p));
            }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int32_t r = r0 + e * ns * RS;
          if (r >= rows) break;
          float M = -INFINITY;
#pragma unroll
          for (int p = 0; p < kCluster; ++p)
            if (p < ns && ml[e][p].y > 0.f) M = fmaxf(M, ml[e][p].x);
          float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
          float l = 0.f;
#pragma unroll
          for (int p = 0; p < kCluster; ++p)
            if (p < ns && ml[e][p].y > 0.f) {  // (a part whose keys the row does not see has no sum)
              const float w = ex2_approx((ml[e][p].x - M) * c2);
              l = fmaf(w, ml[e][p].y, l);
              acc.x = fmaf(w, x[e][p].x, acc.x);
              acc.y = fmaf(w, x[e][p].y, acc.y);
              acc.z = fmaf(w, x[e][p].z, acc.z);
              acc.w = fmaf(w, x[e][p].w, acc.w);
            }
          const int32_t jq = (row0 + r) / G, h = it->g * G + row0 + r - jq * G;
          const int64_t orow = ((int64_t)it->b * a.D_max + jq) * a.Hq + h;
          if (!dbg_in(orow, (int64_t)a.B * a.D_max * a.Hq, a.status)) continue;
          const float inv = l > 0.f ? __fdividef(1.0f, l) : 0.f;
          uint2 w;
          w.x = pack_bf16x2(acc.x * inv, acc.y * inv);
          w.y = pack_bf16x2(acc.z * inv, acc.w * inv);
          *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(a.o) + orow * D + 4 * ch) = w;
          if (a.lse != nullptr && ch == 0)
            a.lse[((int64_t)it->b * a.Hq + h) * a.D_max + jq] =
                l > 0.f ? (M * (c2 / kLog2eTC) + __logf(l)) : -INFINITY;
        }
      }
    }
    __syncwarp();
    cluster_sync_all();  // the peers have read this CTA's rows
  }
  // ---- teardown
  tc_fence_before();
  __syncthreads();
  if (warp == kSoftWarps + 3) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

}  // namespace

bool attention_tc_supported(int32_t Hq, int32_t Hkv, int32_t d) {
  const int32_t G = Hq / Hkv;
  return (d == 64 || d == 128) && G >= 1 && G <= kBM;
}

namespace {
// Query rows per tile: 64 when a KV group's rows under this grid's frontier fit
// (M = 64 products, their softmax spread over the four lane quarters), else
// 128.  Frontiers above the hint take more tiles.
int32_t tc_tile_rows(const AttnArgs& a) {
  return attention_rows_hint(a.grid, a.D_max) * (a.Hq / a.Hkv) <= 64 ? 64 : kBM;
}

// Clusters of the kernel <D, BM> that the current device can hold at once (a device
// constant, queried once per device and kernel), at least one.  The occupancy
// calculator counts one CTA per SM for any kernel that allocates tensor
// memory; kCtasPerSmTC of this kernel's CTAs, which share the 512 columns, do
// run on an SM (304 of 304 CTAs of a probe started at once).
constexpr int kMaxDevicesTC = 64;
template <int D, int BM>
int resident_clusters() {
  static std::atomic<int> known[kMaxDevicesTC];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  const bool slot = dev >= 0 && dev < kMaxDevicesTC;
  int n = slot ? known[dev].load(std::memory_order_relaxed) : 0;
  if (n > 0) return n;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kCluster);
  cfg.blockDim = dim3(kThreadsTC);
  cfg.dynamicSmemBytes = tc_smem_bytes<D, BM>();
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCluster;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaOccupancyMaxActiveClusters(&n, frontier_attn_tc_kernel<D, BM>, &cfg) != cudaSuccess ||
      n < 1) {
    cudaGetLastError();  // (not kept: the next launch asks again)
    return std::max(1, device_sm_count() / kCluster / 2) * kCtasPerSmTC;
  }
  n *= kCtasPerSmTC;
  if (slot) known[dev].store(n, std::memory_order_relaxed);
  return n;
}

// The launch of the kernel <D, BM>: persistent, whole clusters, as many as are
// resident, at most one per item.
template <int D, int BM>
cudaError_t launch_tiles(const AttnArgs& a, TcLaunch L, const CUtensorMap& tq, const CUtensorMap& tk,
                         const CUtensorMap& tv, cudaStream_t stream, bool pdl) {
  constexpr size_t smem = tc_smem_bytes<D, BM>();
  const cudaError_t e = cudaFuncSetAttribute(
      frontier_attn_tc_kernel<D, BM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t n_items = (int64_t)a.B * a.Hkv * L.mtiles;
  const int64_t clusters = std::min<int64_t>(n_items, resident_clusters<D, BM>());
  L.order = pdl ? kCluster : 0;
  return launch_clusters(frontier_attn_tc_kernel<D, BM>,
                         dim3((unsigned)(clusters * kCluster + L.order)), dim3(kThreadsTC), smem,
                         stream, /*pdl=*/true, kCluster, tq, tk, tv, a, L);
}
}  // namespace

cudaError_t launch_attention_tc(const AttnArgs& a, cudaStream_t stream, bool pdl) {
  const int32_t G = a.Hq / a.Hkv;
  const int32_t bm = tc_tile_rows(a);
  CUtensorMap tq, tk, tv;
  bool ok;
  const uint64_t row = (uint64_t)a.d * 2, halves = (uint64_t)a.d / 64;
  // Rows (draft, head of the group): a tile of bm / G drafts.  When G divides bm
  // its d / 64 column blocks of bm rows are one copy; a tile of fewer rows takes
  // a copy per block, so that every block starts on a swizzle atom (the rows
  // past it are never read back).
  TcLaunch L;
  L.sms = device_sm_count();
  L.drafts = bm / G;
  L.mtiles = (a.D_max + L.drafts - 1) / L.drafts;
  L.q_copies = bm % G == 0 ? 1 : (int32_t)halves;
  {  // {64 columns, Hq, B * D_max, d / 64}, box {64, G, bm / G, d / 64 or 1}
    const uint64_t dims[4] = {64, (uint64_t)a.Hq, (uint64_t)a.B * a.D_max, halves};
    const uint64_t strides[3] = {row, (uint64_t)a.Hq * row, 128};
    const uint32_t box[4] = {64, (uint32_t)G, (uint32_t)L.drafts,
                             L.q_copies == 1 ? (uint32_t)halves : 1u};
    ok = bf16_tensor_map(&tq, a.q, 4, dims, strides, box);
  }
  {  // {64 columns, rows, 1, d / 64}, box {64, KTC, 1, d / 64}
    const uint64_t dims[4] = {64, (uint64_t)a.B * a.Hkv * a.L_max, 1, halves};
    const uint64_t strides[3] = {row, row, 128};
    const uint32_t box[4] = {64, KTC, 1, (uint32_t)halves};
    ok = ok && bf16_tensor_map(&tk, a.k, 4, dims, strides, box) &&
         bf16_tensor_map(&tv, a.v, 4, dims, strides, box);
  }
  if (!ok) return cudaErrorInvalidValue;
  if (a.d == 128)
    return bm == 64 ? launch_tiles<128, 64>(a, L, tq, tk, tv, stream, pdl)
                    : launch_tiles<128, 128>(a, L, tq, tk, tv, stream, pdl);
  return bm == 64 ? launch_tiles<64, 64>(a, L, tq, tk, tv, stream, pdl)
                  : launch_tiles<64, 128>(a, L, tq, tk, tv, stream, pdl);
}

}  // namespace ssd
