// Eq. 1 of Sec. 3.1 on the 5th-generation tensor cores: per (vehicle, head, key split) a CTA
// computes softmax(Q [K_vlm ; K_ae]^T / sqrt(128)) [V_vlm ; V_ae] for the
// expert's queries (at most 48, padded to an M = 64 tile) with a bf16 or fp32 backbone
// cache, fp32 accumulation. S = Q K^T in fp16: the cache K rows are
// converted in shared memory (exact for bf16 |x| in [2^-14, 65504]) by the warps that
// stage them. P V keeps bf16 cache V rows in bf16 and splits P into bf16 P_hi + P_lo
// (16 significant bits, more than fp16's 11); the own chunk (fp16 V) and fp32 cache rows
// (converted to fp16) split P into fp16 P_hi + P_lo instead.
//
// Data path ("slot" = 64 keys; shared-memory operands 128-byte swizzled; kSlots = 3, 2 for fp32):
//   Q                [64 q][128 d] fp16   smem, A of S          (K-major)
//   K slot (xkSlots) [64 keys][128 d]     smem, B of S          (K-major)
//   V slot (xkSlots) [64 keys][128 d]     smem, B of P V        (N = d contiguous, MN-major;
//                                         bf16 cache rows, fp16 own rows and fp32 caches)
//   raw (x2, fp32)   [16 keys][128 d] fp32 smem, rows as they lie in the cache, per tensor
//   S (x2)           [64 q][64 keys] fp32 tensor memory, 64 columns each
//   P_hi, P_lo       [64 q][64 keys]      tensor memory, A of P V, written over the
//                                         S buffer they were computed from (32 columns each)
//   O                [64 q][128 d] fp32   tensor memory, 128 columns
//   Row q of an M = 64 tile lives in lane (q mod 16) + 32 (q / 16).
// The vehicle's cache keys are cut into 64-key chunks and the chunks into near-equal runs, one
// per split; split 0 (never the longest run) takes the expert's own keys (fp16 as produced) as
// its chunk 0 before its cache chunks. The g-th chunk of a CTA sits in K / V slot g mod kSlots.
//
// Items: without splits a CTA works through up to 32 (vehicle, head) items, two CTAs per SM, one wave.
// The chunks of its items are one stream for every warp role: the next item's first loads, queries and
// S run under the softmax and the output of the one before. A CTA per item paid for start-up, output
// and launch 4.9 of the 9.2 us of a 3-chunk item; with the smaller code below, 8 layers, before -> now:
// a 40-frame clip (64-224 rows) 812 -> 730 us, 128 vehicles with 64-2048 rows 3996 -> 3800 (3985 where
// such long items kept a CTA each), 16 with 96-480 rows 483 -> 480.
//
// Warp roles: warps 0-2 run the online softmax for query rows
// 16 w .. 16 w + 15, two rows per thread; warp 3 lane 0 loads the queries and issues S and P V as their
// inputs become ready; warps 4-5 stage and convert the K rows, warps 6-7 the V rows, two
// chunks ahead. Queries, own rows and whole bf16 chunks come by TMA; a short last bf16 chunk by 16-byte
// copies; fp32 rows in 16-key stages by 16-byte copies, two in flight per tensor (32 KB a CTA), converted
// into the slot by the warp that copied the rows.
// Code size: the kernel is cold when a layer starts, its instructions come through a memory system
// that the first chunks' loads keep busy, and every CTA waits for the same lines: at 92 KB the first
// softmax chunk took 4.5 us on every SM at once (40-frame clip 769 us), at 43 KB 0.7 us (728).
// Splits: the CTAs of one (vehicle, head) form a thread-block cluster and merge
// (log-sum-exp weights) by pushing each split's normalised fp32 rows to the rank that owns them
// through distributed shared memory. Split and fp32 launches check every cache value they stage
// against the fp16 range and go on with it clipped to +-65504 (bf16 values of V to +-65536, the
// nearest bf16).
// Measured against the mma.sync kernel of attention.cu, which split and fp32 launches ran before: a
// tick of 4 vehicles with 0-700 bf16 rows, 8 layers, 2 splits: 740 -> 452 us; one vehicle with 2048
// rows, 8 splits, Eq. 1 alone: 34 -> 27 us a call; 24 vehicles with 16-1000 fp32 rows, Eq. 1
// alone: 104 -> 66 us a call (5.0 TB/s) with the order below.
// Launches of more than one wave without a plan take the longest caches first (each CTA sorts at most
// 128 vehicles by counting; the 24 fp32 vehicles: 76.8 -> 67.7 us). A tick's plan is sorted already.
// Every wait is bounded; a timeout raises the status word and the CTA drains its
// MMAs before it frees the tensor memory.
#include <cuda.h>
#include <math_constants.h>

#include "device_util.cuh"
#include "gemm_tc.h"
#include "kernels.h"
#include "tcgen05.cuh"

namespace fsx {

namespace {

constexpr int kD = kHeadDim;           // 128
constexpr int kSlotKeys = 64;          // keys per chunk
constexpr int kSoftmaxWarps = 3;       // rows 0..47
constexpr int kMmaWarp = 3;
constexpr int kProdWarp0 = 4;          // then the K staging warps, then the V staging warps
constexpr int kTmemCols = 256;         // S[2] x 64 + O 128
constexpr uint32_t kColS = 0;    // S / P buffers at columns 0 and 64
constexpr uint32_t kColO = 128;
constexpr int kMaxClusterSplits = 8;
constexpr int kMaxRounds = 32;     // items a CTA works on, at most (one lane prepares each)
// vehicles a launch without a plan sorts: each of its CTAs compares every pair, and 128 is the largest
// batch that was measured; larger ones run in the given order
constexpr int kMaxByLength = 128;
constexpr int kBoxBytes = kSlotKeys * 64 * 2;  // a TMA box: 64 rows of 64 values

// shared-memory layout (bytes from the 1024-aligned base)
constexpr int kQBytes = 64 * kD * 2;            // 16 KB
constexpr int kSlotBytes = kSlotKeys * kD * 2;  // 16 KB
constexpr int kRawKeys = 16;                     // keys of a raw fp32 stage
constexpr int kRawBytes = kRawKeys * kD * 4;
constexpr int kRawPerChunk = kSlotKeys / kRawKeys;
constexpr int kProdWarps = 2;                    // per tensor
constexpr int kProdThreads = 32 * kProdWarps;
constexpr int kThreadsTc = 32 * (kProdWarp0 + 2 * kProdWarps);
constexpr int kCtasPerSm = kAttentionCtasPerSm;
// barriers: kfull[3], kempty[3], vfull[3], vempty[3], sfull[2], pfull[2], pvdone[2], drain, ktma[3], vtma[3],
// qfull, qempty, oread
constexpr int kNumBars = 28;
template <bool F32>
struct CacheType {
  using T = __nv_bfloat16;
};
template <>
struct CacheType<true> {
  using T = float;
};
template <bool F32>
struct Shape {
  static constexpr int kSlots = F32 ? 2 : 3;           // per tensor
  static constexpr int kOffQ = 0;
  static constexpr int kOffK = kOffQ + kQBytes;
  static constexpr int kOffV = kOffK + kSlots * kSlotBytes;
  static constexpr int kOffRaw = kOffV + kSlots * kSlotBytes;  // [K, V][2]
  static constexpr int kOffBar = kOffRaw + (F32 ? 4 * kRawBytes : 0);
  static constexpr int kOffItems = kOffBar + kNumBars * 8 + 16 /*tmem slot, abort, items*/;
  static constexpr int kSmem = kOffItems + kMaxRounds * 16;
};
static_assert(kCtasPerSm * (Shape<false>::kSmem + 1024) <= 228 * 1024, "two CTAs per SM");
static_assert(kCtasPerSm * (Shape<true>::kSmem + 1024) <= 228 * 1024, "two CTAs per SM");
// merge buffers at the start of the K slots: at most (48 + 7) rows of 128 fp32 values, then their log-sum-exps
static_assert((48 + kMaxClusterSplits - 1) * (kD + 1) * 4 <= Shape<true>::kSlots * kSlotBytes, "merge buffers");

// byte offset of 16-byte unit u (8 elements) of row r in a [rows][128] tile made of
// 64-element swizzled column blocks (1024-byte atoms of 8 rows; blocks 8 KB apart
// for 64-row tiles)
__device__ __forceinline__ uint32_t tile128_off(int r, int u) {
  return (u >> 3) * 8192 + (r >> 3) * 1024 + (r & 7) * 128 + ((((u & 7) ^ (r & 7))) << 4);
}

// MN-major 128-byte-swizzled descriptor: LBO = distance between 64-element blocks
// along N, SBO = distance between 8-row groups along K
__device__ __forceinline__ uint64_t sw128_desc_mn(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>((lbo >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>((sbo >> 4) & 0x3FFFu) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}

// kind::f16 instruction descriptor, fp16 A and B, fp32 D; b_mn: B is N-contiguous
__host__ __device__ constexpr uint32_t idesc_f16_mn(int m, int n, bool b_mn) {
  return (1u << 4) | (b_mn ? (1u << 16) : 0u) | (static_cast<uint32_t>(n >> 3) << 17) |
         (static_cast<uint32_t>(m >> 4) << 24);
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// two fp32 -> bf16x2 (round to nearest even), lo in the low half
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// D[tmem] (+)= A[tmem] * B[smem]^T, one K = 16 step (A: M rows in the D lane layout,
// two 16-bit values per column)
__device__ __forceinline__ void umma_f16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(tmem_d),
      "r"(tmem_a), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// bounded wait that also gives up once another thread of the CTA gave up. Written for size, as the
// rest of the kernel is: its code is cold when a layer starts and arrives through a memory system
// that the first chunks' loads keep busy. The timer's low word wraps after 4.3 s.
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, int* status, volatile int* abort) {
  const uint32_t addr = smem_addr(bar);
  uint32_t t0 = 0;
  for (;;) {
    uint32_t done, now;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
    if (*abort) return false;
    asm volatile("mov.u32 %0, %%globaltimer_lo;" : "=r"(now));
    if (t0 == 0) t0 = now | 1u;
    if (now - t0 > kWaitLimitNs && now - t0 < 0x80000000u) {
      set_status(status, kStatusTimeout);
      *abort = 1;
      return false;
    }
  }
}

// non-blocking test of the phase of `parity`
__device__ __forceinline__ bool test_bar(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(done)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return done != 0;
}

// 16 lanes x 256 bits, 8 repetitions along the columns: thread t gets, per 8-column
// group g, lane t / 4 columns 8 g + 2 (t mod 4) + {0, 1}, then lane t / 4 + 8 the same
__device__ __forceinline__ void tmem_ld_16x256b_x8(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  tmem_wait_ld32(r);
}
__device__ __forceinline__ void tmem_st_16x256b_x8(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
      "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
      "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
// 16 lanes x 128 bits, 8 repetitions: thread t gets, per 4-column group j, column
// 4 j + (t mod 4) of lane t / 4, then of lane t / 4 + 8
__device__ __forceinline__ void tmem_st_16x128b_x8(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}

constexpr float kLazyRescale = 8.f;  // log2 units; P <= 2^8 between rescales

// bits 15 / 31 set where a bf16 value lies outside the fp16 range (magnitude bits >= 0x4780)
__device__ __forceinline__ uint32_t bf16x2_out_of_range(uint32_t v) {
  return ((v & 0x7fff7fffu) + 0x38803880u) & 0x80008000u;
}

// the same values clipped to +-65536 (0x4780, the smallest bf16 magnitude out of range); a NaN stays
__device__ __forceinline__ uint32_t clip_bf16x2(uint32_t v) {
  const uint32_t lo = v & 0x7fffu, hi = v & 0x7fff0000u;
  if (lo > 0x4780u && lo <= 0x7f80u) v = (v & 0xffff8000u) | 0x4780u;
  if (hi > 0x47800000u && hi <= 0x7f800000u) v = (v & 0x8000ffffu) | 0x47800000u;
  return v;
}
// a finite value clipped to the fp16 range
__device__ __forceinline__ float clip_finite(float x) {
  return fabsf(x) < CUDART_INF_F ? fminf(fmaxf(x, -65504.f), 65504.f) : x;
}

// arrive at and wait for the cluster's barrier (threads of a warp may come apart)
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t peer_addr(const void* local, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(local)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_peer2(uint32_t addr, float a, float b) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(a), "f"(b) : "memory");
}
__device__ __forceinline__ void st_peer(uint32_t addr, float a) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(a) : "memory");
}

// one 64-token x 64-dim box of a head of the cache (3-D map [rows, heads, 128], 128-byte swizzle)
__device__ __forceinline__ void tma_load_cache(void* dst, const CUtensorMap* map, int x, int head, int row,
                                               uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(smem_addr(dst)),
      "l"(map), "r"(x), "r"(head), "r"(row), "r"(smem_addr(bar))
      : "memory");
}

// one 64-row x 64-dim box of a vehicle's queries or own rows (4-D map [B, rows, heads, 128]; rows past the
// vehicle's are filled with zeros)
__device__ __forceinline__ void tma_load_rows(void* dst, const CUtensorMap* map, int x, int head, int b,
                                              uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];" ::"r"(smem_addr(dst)),
      "l"(map), "r"(x), "r"(head), "r"(0), "r"(b), "r"(smem_addr(bar))
      : "memory");
}
__device__ __forceinline__ void tma_load_rows_pair(void* dst, const CUtensorMap* map, int head, int b, uint64_t* bar) {
  mbar_arrive_expect_tx(bar, 2 * kBoxBytes);
  tma_load_rows(dst, map, 0, head, b, bar);
  tma_load_rows(static_cast<unsigned char*>(dst) + kBoxBytes, map, 64, head, b, bar);
}

__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

// maps.k, maps.v: maps of the one layer's caches when p.cache_maps is NULL and p.param_maps is set
struct AttnMaps {
  CUtensorMap q, k_own, v_own, k, v;
};
template <bool F32, bool SPLIT>
__global__ void __launch_bounds__(kThreadsTc, kCtasPerSm)
    attn_tc_kernel(const AttnArgs p, const int n_vehicles, const __grid_constant__ AttnMaps maps) {
  using SH = Shape<F32>;
  using CT = typename CacheType<F32>::T;
  constexpr int kSlots = SH::kSlots;
  constexpr bool kCheck = F32 || SPLIT;  // every staged cache value against the fp16 range
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int lane = tid & 31;
  const int H = p.n_heads;
  const int S = SPLIT ? static_cast<int>(gridDim.x) : 1;     // the cluster spans the grid's x extent
  const int rank = SPLIT ? static_cast<int>(blockIdx.x) : 0;
  const int has_own = rank == 0 ? 1 : 0;                     // an item's chunk 0 holds the own keys

  pdl_launch_dependents();
  if (tid == kMmaWarp * 32) prefetch_map(&maps.q);
  if (tid == kProdWarp0 * 32) prefetch_map(&maps.k_own);
  if (tid == (kProdWarp0 + kProdWarps) * 32) prefetch_map(&maps.v_own);
  pdl_wait();
  if ((smem_addr(smem) & 1023u) != 0u) {  // the swizzled operands need a 1024-byte aligned base
    if (tid == 0) set_status(p.status, kStatusDeviceArg);
    return;
  }
  const CT* kc;
  const CT* vc;
  if (p.targs != nullptr) {
    kc = static_cast<const CT*>(p.targs->k_cache[p.layer]);
    vc = static_cast<const CT*>(p.targs->v_cache[p.layer]);
  } else {
    kc = static_cast<const CT*>(p.k_cache);
    vc = static_cast<const CT*>(p.v_cache);
  }

  unsigned char* qt = smem + SH::kOffQ;
  unsigned char* kslot = smem + SH::kOffK;
  unsigned char* vslot = smem + SH::kOffV;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SH::kOffBar);
  uint64_t* kfull = bars + 0;    // [3] K rows of a chunk staged
  uint64_t* kempty = bars + 3;   // [3] S done with a K slot
  uint64_t* vfull = bars + 6;    // [3] V rows staged
  uint64_t* vempty = bars + 9;   // [3] P V done with a V slot
  uint64_t* sfull = bars + 12;   // [2] S of a chunk in tensor memory
  uint64_t* pfull = bars + 14;   // [2] P of a chunk written over its S
  uint64_t* pvdone = bars + 16;  // [2] P V of a chunk done (one per buffer)
  uint64_t* drain = bars + 18;   // every MMA of the CTA done
  uint64_t* ktma = bars + 19;    // [3] a chunk's K rows landed by TMA
  uint64_t* vtma = bars + 22;    // [3] the same for V
  uint64_t* qfull = bars + 25;   // an item's queries landed
  uint64_t* qempty = bars + 26;  // every S of an item done with them
  uint64_t* oread = bars + 27;   // an item's O read
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kNumBars);
  volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* n_work = reinterpret_cast<volatile int*>(tmem_slot + 2);
  struct Packed {  // an item as it lies in the table
    long long row0;
    int L;
    uint32_t bh;
  };
  struct Item {
    long long row0;  // this CTA's first cache row of the vehicle
    int L, b, h, n;  // its number of cache keys; vehicle; head; chunks
    int last;        // rows of the last cache chunk
  };
  Packed* table = reinterpret_cast<Packed*>(smem + SH::kOffItems);
  static_assert(sizeof(Packed) == 16, "item table");
  auto item = [&](int k) {
    const Packed w = table[k];
    const int n_cc = (w.L + kSlotKeys - 1) / kSlotKeys;
    return Item{w.row0, w.L, static_cast<int>(w.bh >> 16), static_cast<int>(w.bh & 0xffffu), has_own + n_cc,
                w.L - (n_cc - 1) * kSlotKeys};
  };

  // ---- items: (vehicle, head) pairs, the vehicle's place in the schedule major. A CTA works on item
  // k gridDim + (k even ? its index : its mirror image), k = 0, 1, ...: with the longest caches
  // first the CTA of the longest item of a round gets the shortest of the next.
  int* order = reinterpret_cast<int*>(smem + SH::kOffK);  // before a slot is staged into
  if (p.by_length) {  // order[z]: the vehicle with z longer caches before it (ties by index)
    long long* len = reinterpret_cast<long long*>(order + kMaxByLength);
    if (tid < n_vehicles) len[tid] = p.offsets[tid + 1] - p.offsets[tid];
    __syncthreads();
    if (tid < n_vehicles) {
      const long long mine = len[tid];
      int before = 0;
#pragma unroll 1
      for (int j = 0; j < n_vehicles; ++j) before += len[j] > mine || (len[j] == mine && j < tid) ? 1 : 0;
      order[before] = tid;
    }
    __syncthreads();
  }
  if (warp == 0) {  // lane k: the k-th item
    const long long n_items = static_cast<long long>(n_vehicles) * H;
    const int G = static_cast<int>(gridDim.x), c = static_cast<int>(blockIdx.x);
    long long j = static_cast<long long>(lane) * G + ((lane & 1) ? G - 1 - c : c);
    if (SPLIT) j = lane == 0 ? static_cast<long long>(blockIdx.z) * H + blockIdx.y : n_items;
    bool valid = lane < kMaxRounds && j < n_items;
    long long row0 = 0, len = 0;
    int b = 0, h = 0;
    if (valid) {
      const int z = static_cast<int>(j) / H;
      h = static_cast<int>(j) % H;
      if (p.plan != nullptr) {  // written by the tick's first kernel: one 16-byte entry
        const AttnPlan w = p.plan[z];
        b = w.b;
        row0 = w.lo;
        len = w.len;
      } else {
        b = p.by_length ? order[z] : z;
        row0 = p.offsets[b];
        len = p.offsets[b + 1] - row0;
      }
      // never read outside the caller's cache: such a vehicle is reported and passed over
      valid = row0 >= 0 && len >= 0 && row0 <= p.max_total && len <= p.max_total - row0 &&
              len <= INT32_MAX - kSlotKeys && (len == 0 || (kc != nullptr && vc != nullptr));
      if (!valid) set_status(p.status, kStatusDeviceArg);
    }
    if (SPLIT) {  // this split's run of whole chunks
      const uint32_t n_cc = static_cast<uint32_t>((len + kSlotKeys - 1) / kSlotKeys);
      const long long k_lo = n_cc * rank / S * static_cast<long long>(kSlotKeys);
      const long long k_hi = min(len, n_cc * (rank + 1) / S * static_cast<long long>(kSlotKeys));
      row0 += k_lo;
      len = k_hi > k_lo ? k_hi - k_lo : 0;
    }
    const uint32_t mask = __ballot_sync(0xffffffffu, valid);
    if (valid)
      table[__popc(mask & ((1u << lane) - 1u))] =
          Packed{row0, static_cast<int>(len), static_cast<uint32_t>(b) << 16 | static_cast<uint32_t>(h)};
    if (lane == 0) *n_work = __popc(mask);
  }
  if (p.by_length) fence_proxy_async();  // the order lies where a slot is staged into

  // ---- producers' staging
  const bool is_prod = warp >= kProdWarp0;
  const bool is_v = warp >= kProdWarp0 + kProdWarps;
  const int pw = warp & (kProdWarps - 1);  // warp within the tensor's staging warps
  const int pt = pw * 32 + lane;           // thread within them
  const int pu = pt & 15;                  // 16-byte unit of a 256-byte row
  const int pr0 = pt >> 4;                 // rows pr0, pr0 + kRowStep, ...
  constexpr int kRowStep = kProdThreads / 16;
  const size_t tok = static_cast<size_t>(H) * kD;
  unsigned char* pslots = is_v ? vslot : kslot;
  uint64_t* tbar = is_v ? vtma : ktma;
  const CUtensorMap* omap = is_v ? &maps.v_own : &maps.k_own;
  // Own keys and whole cache chunks (every cache chunk but a short last one) come by two TMA box
  // loads issued by one thread of the tensor's warps; a short last chunk by 16-byte copies of every
  // thread, zeros behind it.
  const CUtensorMap* tmap = nullptr;
  if (!F32) {
    if (p.cache_maps != nullptr && p.targs != nullptr) {
      tmap = p.cache_maps + 2 * p.layer + (is_v ? 1 : 0);
      if (is_prod && pt == 0) tensormap_acquire(tmap);  // the thread that issues this tensor's loads
    } else if (p.param_maps)
      tmap = is_v ? &maps.v : &maps.k;
  }
  // the producers' next chunk to issue: chunk ci of item ck
  int ci = 0, ck = 0;
  // bf16: stage chunk g of the CTA; returns its rows, bit 8 own keys, bit 9 by TMA
  auto issue = [&](int g) {
    unsigned char* slot = pslots + (g % kSlots) * kSlotBytes;
    uint64_t* bar = tbar + g % kSlots;
    const Item cur = item(ck);
    int desc;
    if (ci < has_own) {
      desc = p.n_own | 0x300;
      if (pt == 0) tma_load_rows_pair(slot, omap, cur.h, cur.b, bar);
    } else {
      const long long c0 = (ci - has_own) * static_cast<long long>(kSlotKeys);
      const int rows = ci + 1 < cur.n ? kSlotKeys : cur.last;
      desc = rows;
      if (tmap != nullptr && rows == kSlotKeys) {
        desc |= 0x200;
        if (pt == 0) {
          const int y = static_cast<int>(cur.row0 + c0);
          mbar_arrive_expect_tx(bar, kSlotBytes);
          tma_load_cache(slot, tmap, 0, cur.h, y, bar);
          tma_load_cache(slot + kSlotBytes / 2, tmap, 64, cur.h, y, bar);
        }
      } else {
        const CT* src = (is_v ? vc : kc) + (static_cast<size_t>(cur.row0 + c0) * H + cur.h) * kD + pu * 8;
#pragma unroll 2
        for (int m = 0; m < kSlotKeys / kRowStep; ++m) {
          const int r = pr0 + kRowStep * m;
          unsigned char* dst = slot + tile128_off(r, pu);
          if (r < rows)
            cp_async_16(smem_addr(dst), src + static_cast<size_t>(r) * tok);
          else
            *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);  // keys past the range: finite zeros
        }
      }
    }
    cp_async_commit();  // one group per chunk, empty behind a TMA load
    if (++ci == cur.n) {
      ci = 0;
      ++ck;
    }
    return desc;
  };
  // fp32: raw stage t of an item (keys 16 t .. of its cache rows), one warp instruction a row; row r of a
  // stage is the warp's that has r mod kProdWarps == pw. Past the item's end an empty group.
  auto issue_raw = [&](const Item& cur, int t) {
    const int rows = static_cast<int>(
        min(static_cast<long long>(kRawKeys), cur.L - static_cast<long long>(t) * kRawKeys));
    const uint32_t raw = smem_addr(smem + SH::kOffRaw + ((is_v ? 2 : 0) + (t & 1)) * kRawBytes) + lane * 16;
    const size_t row = static_cast<size_t>(cur.row0 + t * static_cast<long long>(kRawKeys));
    const CT* src = (is_v ? vc : kc) + (row * H + cur.h) * kD + lane * 4;
#pragma unroll
    for (int r = pw; r < kRawKeys; r += kProdWarps)
      if (r < rows) cp_async_16(raw + r * (kD * 4), src + static_cast<size_t>(r) * tok);
    cp_async_commit();
  };

  if (tid == 0) {
    for (int i = 0; i < kSlots; ++i) {
      mbar_init(kfull + i, kProdThreads);
      mbar_init(kempty + i, 1);
      mbar_init(vfull + i, kProdThreads);
      mbar_init(vempty + i, 1);
      mbar_arrive(kempty + i);  // release 0 of every slot: free from the start
      mbar_arrive(vempty + i);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(sfull + i, 1);
      mbar_init(pfull + i, kSoftmaxWarps * 32);
      mbar_init(pvdone + i, 1);
    }
    mbar_init(drain, 1);
    mbar_init(qempty, 1);
    mbar_init(oread, kSoftmaxWarps * 32);
    // a kernel before this one has already abandoned the tick: this CTA stops below (outside a tick only
    // this launch sets the word, and the other vehicles' rows are still written)
    *abort = p.targs != nullptr && *reinterpret_cast<volatile int*>(p.status) != 0 ? 1 : 0;
  }
  if (warp == kMmaWarp) {
    if (lane == 0) mbar_init(qfull, 1);
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  } else if (is_prod && pt < kSlots) {
    mbar_init(tbar + pt, 1);
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(tmem_slot);
  const int n_my = *n_work;
  if (*abort || n_my == 0) {  // the tick was abandoned before this kernel, or no vehicle is valid: nothing was issued
    if (SPLIT) {  // the other splits may not have seen the status yet: they push their rows here
      cluster_barrier();
      cluster_barrier();
    }
    if (warp == kMmaWarp) {
      __syncwarp();
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
    return;
  }

  if (warp == kMmaWarp) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      const uint32_t id_s = idesc_f16_mn(64, kSlotKeys, false);
      const uint32_t id_pv_own = idesc_f16_mn(64, kD, true);       // fp16 P, fp16 own V
      const uint32_t id_pv = idesc_f16_mn(64, kD, true) | (1u << 7) | (1u << 10);  // bf16 P, bf16 cache V
      const uint32_t aq = smem_addr(qt);
      auto issue_s = [&](int g) {  // S of chunk g of the CTA into buffer g & 1
        const uint32_t d = tmem + kColS + (g & 1) * kSlotKeys;
        const uint32_t kb = smem_addr(kslot + (g % kSlots) * kSlotBytes);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t off = (kk >> 2) * 8192 + (kk & 3) * 32;
          umma_f16(d, sw128_desc(aq + off), sw128_desc(kb + off), id_s, kk > 0 ? 1u : 0u);
        }
        umma_commit(kempty + (g % kSlots));
        umma_commit(sfull + (g & 1));
      };
      auto issue_pv = [&](int g, bool first) {  // O (+)= P V of chunk g, P from tensor memory
        const uint32_t pa = tmem + kColS + (g & 1) * kSlotKeys;
        const uint32_t vb = smem_addr(vslot + (g % kSlots) * kSlotBytes);
        const uint32_t idv = F32 || (first && has_own != 0) ? id_pv_own : id_pv;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {  // 16 keys = 8 columns of packed fp16 pairs
          const uint64_t bd = sw128_desc_mn(vb + kk * 2048, 8192, 1024);
          umma_f16_ta(tmem + kColO, pa + kk * 8, bd, idv, (!first || kk > 0) ? 1u : 0u);  // P_hi
          umma_f16_ta(tmem + kColO, pa + kSlotKeys / 2 + kk * 8, bd, idv, 1u);            // P_lo
        }
        umma_commit(vempty + (g % kSlots));
        umma_commit(pvdone + (g & 1));
      };
      // S(gs) and P V(gp) are issued as soon as their inputs are ready: S(gs) needs its item's
      // queries, its K rows and P V(gs - 2) done with the buffer it overwrites; P V(gp) needs P(gp),
      // its V rows and, as an item's first, the O of the item before read. An item's queries are
      // loaded once the last S of the item before is done with theirs. Each test is at most one
      // phase behind its barrier.
      int k = 0, i = 0, kq = -1;        // S(gs) is chunk i of item k; queries loaded up to item kq
      int n = item(0).n;
      int gs = 0, gp = 0, kp = -1;      // P V(gp - 1) is of item kp
      uint32_t firsts = 0;              // bit g & 31: chunk g is an item's first
      unsigned long long t_idle = 0;
      for (uint32_t spin = 0; i < n || gp < gs; ++spin) {
        bool progressed = false;
        if (kq < k && i < n && (k == 0 || test_bar(qempty, (k - 1) & 1))) {
          tma_load_rows_pair(qt, &maps.q, item(k).h, item(k).b, qfull);
          kq = k;
          progressed = true;
        }
        if (i < n && kq == k && (gs < 2 || gp >= gs - 1) && test_bar(kfull + (gs % kSlots), (gs / kSlots) & 1) &&
            (gs < 2 || test_bar(pvdone + (gs & 1), ((gs - 2) >> 1) & 1)) && (i > 0 || test_bar(qfull, k & 1))) {
          tc_fence_after();
          issue_s(gs);
          firsts = (firsts & ~(1u << (gs & 31))) | ((i == 0 ? 1u : 0u) << (gs & 31));
          ++gs;
          if (++i == n) {
            umma_commit(qempty);
            i = 0;
            n = ++k < n_my ? item(k).n : 0;
          }
          progressed = true;
        }
        if (gp < gs && test_bar(pfull + (gp & 1), (gp >> 1) & 1) &&
            test_bar(vfull + (gp % kSlots), (gp / kSlots) & 1)) {
          const bool first = ((firsts >> (gp & 31)) & 1u) != 0u;
          if (!first || kp < 0 || test_bar(oread, kp & 1)) {
            tc_fence_after();
            issue_pv(gp, first);
            kp += first ? 1 : 0;
            ++gp;
            progressed = true;
          }
        }
        if (progressed) {
          t_idle = 0;
        } else if ((spin & 63u) == 63u) {
          if (*abort) break;
          const unsigned long long now = global_timer_ns();
          if (t_idle == 0) {
            t_idle = now;
          } else if (now - t_idle > kWaitLimitNs) {
            set_status(p.status, kStatusTimeout);
            *abort = 1;
            break;
          }
        }
      }
      umma_commit(drain);  // completes once every MMA issued above has (waited on even after an abort)
      mbar_wait(drain, 0, p.status);
      if (kq >= 0) mbar_wait(qfull, kq & 1, p.status);  // after an abort the last queries may still be on their way
    }
    __syncwarp();
  } else if (is_prod) {
    // ---------------------------------------------------------------- producers
    uint64_t* full = is_v ? vfull : kfull;
    uint64_t* empty = is_v ? vempty : kempty;
    bool ok = true;
    uint32_t range = 0;    // fp32: largest magnitudes of the staged values; bf16: bits set by out-of-range ones
    uint32_t tphase = 0;   // bit s: parity of slot s's next TMA chunk
    if (F32) {
      // per item: own keys by TMA, then per cache chunk four raw stages converted into the slot
      int g = 0;
      for (int k = 0; k < n_my; ++k) {
        const Item cur = item(k);
#pragma unroll 1
        for (int t = 0; t < 2; ++t) issue_raw(cur, t);
        if (has_own != 0) {
          ok = wait_bar(empty + g % kSlots, (g / kSlots) & 1, p.status, abort);
          if (!ok) break;
          if (pt == 0) tma_load_rows_pair(pslots + (g % kSlots) * kSlotBytes, omap, cur.h, cur.b, tbar + g % kSlots);
          ok = wait_bar(tbar + g % kSlots, (tphase >> (g % kSlots)) & 1u, p.status, abort);
          if (!ok) {
            if (pt == 0) mbar_wait(tbar + g % kSlots, (tphase >> (g % kSlots)) & 1u, p.status);
            break;
          }
          tphase ^= 1u << (g % kSlots);
          mbar_arrive(full + (g % kSlots));
          ++g;
        }
        const int n_cc = cur.n - has_own;
        for (int c = 0; c < n_cc; ++c, ++g) {  // raw rows -> fp16 slot, once its previous chunk is consumed
          unsigned char* slot = pslots + (g % kSlots) * kSlotBytes;
          ok = wait_bar(empty + g % kSlots, (g / kSlots) & 1, p.status, abort);
          if (!ok) break;
          const int rows = c + 1 < n_cc ? kSlotKeys : cur.last;
          const int u = lane & 15;
          const int sw = (lane >> 2) & 1;  // the two 16-byte reads of a unit in an order that spreads the banks
#pragma unroll 1
          for (int st = 0; st < kRawPerChunk; ++st) {
            const int t = c * kRawPerChunk + st;
            cp_async_wait<1>();  // stage t landed, t + 1 in flight
            __syncwarp();        // the warp's copies of its rows
            const unsigned char* raw = smem + SH::kOffRaw + ((is_v ? 2 : 0) + (t & 1)) * kRawBytes;
#pragma unroll
            for (int m = 0; m < kRawKeys / kProdWarps; m += 2) {
              const int r = pw + kProdWarps * (m + (lane >> 4));
              uint4 out = make_uint4(0u, 0u, 0u, 0u);  // keys past the range: finite zeros
              if (st * kRawKeys + r < rows) {
                const float4 x = *reinterpret_cast<const float4*>(raw + r * (kD * 4) + u * 32 + sw * 16);
                const float4 y = *reinterpret_cast<const float4*>(raw + r * (kD * 4) + u * 32 + (sw ^ 1) * 16);
                const uint32_t x0 = f32x2_to_half2_peak(x.x, x.y, range), x1 = f32x2_to_half2_peak(x.z, x.w, range);
                const uint32_t y0 = f32x2_to_half2_peak(y.x, y.y, range), y1 = f32x2_to_half2_peak(y.z, y.w, range);
                out = sw == 0 ? make_uint4(x0, x1, y0, y1) : make_uint4(y0, y1, x0, x1);
                if (out_of_range(range)) out = saturate_half8(out);
              }
              *reinterpret_cast<uint4*>(slot + tile128_off(st * kRawKeys + r, u)) = out;
            }
            __syncwarp();  // the raw rows are read before they are refilled
            issue_raw(cur, t + 2);
          }
          fence_proxy_async();
          mbar_arrive(full + (g % kSlots));
        }
        if (!ok) break;
      }
      flag_range(p.status, range);
      cp_async_wait<0>();
    } else {
      // per chunk g: wait for its rows, convert cache K rows bf16 -> fp16 in place (each thread the
      // units it copied), signal. Up to two chunks behind it, of this item or the next, are staged:
      // g + 1 before g is waited for, g + 2 once the MMAs have released the slot of g - 1.
      int g = 0, staged = 0;
      int d0 = -1, d1 = -1, d2 = -1;  // chunks g, g + 1, g + 2 as staged; -1: not staged
      for (;;) {
        if (ck < n_my && item(ck).n > 0 && staged < g + 3) {
          uint64_t* bar = empty + staged % kSlots;
          const uint32_t parity = (staged / kSlots) & 1;
          bool free;
          if (staged < g + 2) {
            free = ok = wait_bar(bar, parity, p.status, abort);
            if (!ok) break;
          } else {
            free = __all_sync(0xffffffffu, test_bar(bar, parity));
          }
          if (free) {
            const int d = issue(staged);
            if (staged == g) d0 = d;
            else if (staged == g + 1) d1 = d;
            else d2 = d;
            ++staged;
            if (staged < g + 3) continue;
          }
        }
        if (d0 < 0) break;
        if (d2 >= 0) cp_async_wait<2>();
        else if (d1 >= 0) cp_async_wait<1>();
        else cp_async_wait<0>();
        unsigned char* slot = pslots + (g % kSlots) * kSlotBytes;
        if (d0 & 0x200) {
          ok = wait_bar(tbar + g % kSlots, (tphase >> (g % kSlots)) & 1u, p.status, abort);
          if (!ok) break;
          tphase ^= 1u << (g % kSlots);
        }
        if (!(d0 & 0x100) && (!is_v || kCheck)) {  // a cache chunk: K rows -> fp16 (V stays bf16)
#pragma unroll 1
          for (int m0 = 0; m0 < kSlotKeys / kRowStep; m0 += 8) {
            uint4 v[8];
#pragma unroll
            for (int m = 0; m < 8; ++m)
              v[m] = *reinterpret_cast<const uint4*>(slot + tile128_off(pr0 + kRowStep * (m0 + m), pu));
            if (kCheck) {
#pragma unroll
              for (int m = 0; m < 8; ++m)
                range |= bf16x2_out_of_range(v[m].x) | bf16x2_out_of_range(v[m].y) | bf16x2_out_of_range(v[m].z) |
                         bf16x2_out_of_range(v[m].w);
            }
            if (!is_v) {
#pragma unroll
              for (int m = 0; m < 8; ++m)
                *reinterpret_cast<uint4*>(slot + tile128_off(pr0 + kRowStep * (m0 + m), pu)) =
                    make_uint4(bf16x2_to_half2(v[m].x), bf16x2_to_half2(v[m].y), bf16x2_to_half2(v[m].z),
                               bf16x2_to_half2(v[m].w));
            }
            if (kCheck && range != 0) {  // an error: this thread's units in place, clipped
#pragma unroll 1
              for (int m = m0; m < m0 + 8; ++m) {
                uint4* u = reinterpret_cast<uint4*>(slot + tile128_off(pr0 + kRowStep * m, pu));
                const uint4 w = *u;
                *u = is_v ? make_uint4(clip_bf16x2(w.x), clip_bf16x2(w.y), clip_bf16x2(w.z), clip_bf16x2(w.w))
                          : saturate_half8(w);
              }
            }
          }
        }
        fence_proxy_async();
        mbar_arrive(full + (g % kSlots));
        d0 = d1;
        d1 = d2;
        d2 = -1;
        ++g;
      }
      if (!ok && pt == 0) {  // after an abort: the TMA chunks issued but not consumed land before the CTA leaves
#pragma unroll 1
        for (int j = 0; j < 3; ++j) {
          const int d = j == 0 ? d0 : (j == 1 ? d1 : d2);
          const int sl = (g + j) % kSlots;
          if (d >= 0 && (d & 0x200)) mbar_wait(tbar + sl, (tphase >> sl) & 1u, p.status);
        }
      }
      if (SPLIT && range != 0) set_status(p.status, kStatusRange);
      cp_async_wait<0>();
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------------- softmax rows
    // Warp w owns query rows 16 w .. 16 w + 15 (tensor-memory lanes 32 w .. + 15).
    // With the 16x256b load shape each thread holds rows ra = 16 w + t / 4 and
    // rb = ra + 8, and the key pairs 8 g + 2 (t mod 4) + {0, 1} of every 8-key group
    // g; a row's maximum and sum are completed across the 4 threads of a quad. Its
    // P pairs are exactly the packed columns 4 g + (t mod 4) that the 16x128b store
    // shape gives the same thread.
    const int t4 = lane & 3;
    const int ra = warp * 16 + (lane >> 2);
    const int rbw = ra + 8;
    const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;
    const float scale_log2 = 1.4426950408889634f * rsqrtf(static_cast<float>(kD));
    const bool va = ra < p.n_q;
    const bool vb = rbw < p.n_q;
    bool ok = true;
    int g0 = 0;  // item k starts with chunk g0 of the CTA
#pragma unroll 1
    for (int k = 0; k < n_my; ++k) {
    const int n = item(k).n;
    float m_run[2] = {-CUDART_INF_F, -CUDART_INF_F};
    float l_run[2] = {0.f, 0.f};
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      const int g = g0 + i;
      const bool own = i < has_own;
      const int valid = own ? p.n_own : (i + 1 < n ? kSlotKeys : item(k).last);
      ok = wait_bar(sfull + (g & 1), (g >> 1) & 1, p.status, abort);
      if (!ok) break;
      tc_fence_after();
      const uint32_t sbuf = tmem + lane_base + kColS + (g & 1) * kSlotKeys;
      uint32_t sv[32];  // [g][row a: 2 keys, row b: 2 keys]
      tmem_ld_16x256b_x8(sbuf, sv);
      float s[2][16];   // [row][g * 2 + e] for key 8 g + 2 t4 + e
#pragma unroll
      for (int g = 0; g < 8; ++g)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          s[0][2 * g + e] = __uint_as_float(sv[4 * g + e]);
          s[1][2 * g + e] = __uint_as_float(sv[4 * g + 2 + e]);
        }
      if (valid < kSlotKeys) {
#pragma unroll
        for (int g = 0; g < 8; ++g)
#pragma unroll
          for (int e = 0; e < 2; ++e)
            if (8 * g + 2 * t4 + e >= valid) {
              s[0][2 * g + e] = -CUDART_INF_F;
              s[1][2 * g + e] = -CUDART_INF_F;
            }
      }
      float mx[2], alpha[2] = {1.f, 1.f};
      bool grow = false;
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float m4[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) m4[e] = fmaxf(fmaxf(s[r][e], s[r][e + 4]), fmaxf(s[r][e + 8], s[r][e + 12]));
        mx[r] = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
        mx[r] *= scale_log2;
        grow = grow || mx[r] > m_run[r] + kLazyRescale;
      }
      const bool any_grow = __any_sync(0xffffffffu, grow);
      if (any_grow) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const float m_new = fmaxf(m_run[r], mx[r]);
          alpha[r] = ex2_approx(m_run[r] - m_new);  // 0 for the first chunk
          m_run[r] = m_new;
        }
      }
      uint32_t ph[16], pl[16];  // 16x128b order: [g][row a, row b]
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float nm = -m_run[r];
        float r4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          s[r][2 * g] = ex2_approx(fmaf(s[r][2 * g], scale_log2, nm));
          s[r][2 * g + 1] = ex2_approx(fmaf(s[r][2 * g + 1], scale_log2, nm));
          r4[g & 3] += s[r][2 * g] + s[r][2 * g + 1];
        }
        float rs = (r4[0] + r4[1]) + (r4[2] + r4[3]);
        rs += __shfl_xor_sync(0xffffffffu, rs, 1);
        rs += __shfl_xor_sync(0xffffffffu, rs, 2);
        l_run[r] = l_run[r] * alpha[r] + rs;
      }
      if (F32 || own) {  // fp16 like the V rows
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const float p0 = s[e & 1][e & ~1], p1 = s[e & 1][e | 1];
          ph[e] = pack_half2(p0, p1);
          const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&ph[e]));
          pl[e] = pack_half2(p0 - f.x, p1 - f.y);
        }
      } else {  // bf16 cache chunks: bf16 like the V rows
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const float p0 = s[e & 1][e & ~1], p1 = s[e & 1][e | 1];
          ph[e] = pack_bf16x2(p0, p1);
          pl[e] = pack_bf16x2(p0 - __uint_as_float(ph[e] << 16), p1 - __uint_as_float(ph[e] & 0xffff0000u));
        }
      }
      if (any_grow && i > 0) {
        // rescale this warp's O rows once P V of the previous chunk is done
        ok = wait_bar(pvdone + ((g - 1) & 1), ((g - 1) >> 1) & 1, p.status, abort);
        if (!ok) break;
        tc_fence_after();
#pragma unroll 1
        for (int c = 0; c < kD; c += 64) {
          uint32_t o[32];
          tmem_ld_16x256b_x8(tmem + lane_base + kColO + c, o);
#pragma unroll
          for (int g = 0; g < 8; ++g)
#pragma unroll
            for (int e = 0; e < 4; ++e) o[4 * g + e] = __float_as_uint(__uint_as_float(o[4 * g + e]) * alpha[e >> 1]);
          tmem_st_16x256b_x8(tmem + lane_base + kColO + c, o);
        }
      }
      // P = P_hi + P_lo over the S it came from: P_hi in columns 0..31, P_lo in 32..63
      tmem_st_16x128b_x8(sbuf, ph);
      tmem_st_16x128b_x8(sbuf + kSlotKeys / 2, pl);
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      tc_fence_before();
      mbar_arrive(pfull + (g & 1));
    }
    if (!ok) break;
    g0 += n;
    // the item's last P V done, and with it those before
    if (n > 0) ok = wait_bar(pvdone + ((g0 - 1) & 1), ((g0 - 1) >> 1) & 1, p.status, abort);
    if (!ok) break;
    tc_fence_after();
    const float inv[2] = {l_run[0] > 0.f ? 1.f / l_run[0] : 0.f, l_run[1] > 0.f ? 1.f / l_run[1] : 0.f};
    // A cache key beyond the fp16 range became an infinity here; where it raised a
    // score to +inf (or NaN) the row's sum is NaN: report it, the tick is abandoned.
    // (A key whose scores all fell to -inf carries weight 0, as the exact value would.)
    if (((va && !(l_run[0] == l_run[0])) || (vb && !(l_run[1] == l_run[1])))) set_status(p.status, kStatusRange);
    if (SPLIT) {
      // every CTA of the cluster is done with its slots; rows go to their owners' K slots
      __syncwarp();
      cluster_barrier();
      const int rows_per = (p.n_q + S - 1) / S;
      const int own_a = ra / rows_per, own_b = rbw / rows_per;
      float* rows_o = reinterpret_cast<float*>(smem + SH::kOffK);  // [S][rows_per][128]
      float* rows_l = rows_o + S * rows_per * kD;                  // [S][rows_per] log2-domain log-sum-exp
      const int ia = rank * rows_per + ra - own_a * rows_per, ib = rank * rows_per + rbw - own_b * rows_per;
      const uint32_t da = peer_addr(rows_o + ia * kD + 2 * t4, va ? own_a : 0);
      const uint32_t db = peer_addr(rows_o + ib * kD + 2 * t4, vb ? own_b : 0);
#pragma unroll 1
      for (int c = 0; c < kD; c += 64) {
        uint32_t o[32];
        __syncwarp();
        tmem_ld_16x256b_x8(tmem + lane_base + kColO + c, o);
        const bool any = n > 0;  // a split without keys pushes zeros (its accumulator was never written)
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          if (va) st_peer2(da + (c + 8 * g) * 4, any ? __uint_as_float(o[4 * g]) * inv[0] : 0.f,
                           any ? __uint_as_float(o[4 * g + 1]) * inv[0] : 0.f);
          if (vb) st_peer2(db + (c + 8 * g) * 4, any ? __uint_as_float(o[4 * g + 2]) * inv[1] : 0.f,
                           any ? __uint_as_float(o[4 * g + 3]) * inv[1] : 0.f);
        }
      }
      if (t4 == 0) {
        if (va) st_peer(peer_addr(rows_l + ia, own_a), l_run[0] > 0.f ? m_run[0] + log2f(l_run[0]) : -CUDART_INF_F);
        if (vb) st_peer(peer_addr(rows_l + ib, own_b), l_run[1] > 0.f ? m_run[1] + log2f(l_run[1]) : -CUDART_INF_F);
      }
      __syncwarp();
      break;
    }
    const int b = item(k).b, h = item(k).h;
    __half* oa = p.out + (static_cast<size_t>(b) * p.n_q + (va ? ra : 0)) * p.out_stride + h * kD + 2 * t4;
    __half* ob = p.out + (static_cast<size_t>(b) * p.n_q + (vb ? rbw : 0)) * p.out_stride + h * kD + 2 * t4;
#pragma unroll 1
    for (int c = 0; c < kD; c += 64) {
      uint32_t o[32];
      tmem_ld_16x256b_x8(tmem + lane_base + kColO + c, o);
      if (c + 64 == kD) {  // O is read: the next item's first P V may overwrite it
        tc_fence_before();
        mbar_arrive(oread);
      }
#pragma unroll
      for (int g = 0; g < 8; ++g) {
        if (va) *reinterpret_cast<uint32_t*>(oa + c + 8 * g) =
            pack_half2(__uint_as_float(o[4 * g]) * inv[0], __uint_as_float(o[4 * g + 1]) * inv[0]);
        if (vb) *reinterpret_cast<uint32_t*>(ob + c + 8 * g) =
            pack_half2(__uint_as_float(o[4 * g + 2]) * inv[1], __uint_as_float(o[4 * g + 3]) * inv[1]);
      }
    }
    if (p.lse != nullptr && t4 == 0) {
      float* lrow = p.lse + (static_cast<size_t>(b) * H + h) * p.n_q;
      if (va) lrow[ra] = l_run[0] > 0.f ? (m_run[0] + log2f(l_run[0])) * 0.6931471805599453f : -CUDART_INF_F;
      if (vb) lrow[rbw] = l_run[1] > 0.f ? (m_run[1] + log2f(l_run[1])) * 0.6931471805599453f : -CUDART_INF_F;
    }
    }
    if (SPLIT && !ok) {  // aborted: meet the cluster without pushing
      __syncwarp();
      cluster_barrier();
    }
  }
  if (SPLIT) {
    if (warp >= kSoftmaxWarps) {  // this warp is done with the slots (the softmax warps met this barrier above)
      __syncwarp();
      cluster_barrier();
    }
    cluster_barrier();  // every row pushed
    const int rows_per = (p.n_q + S - 1) / S;
    const float* rows_o = reinterpret_cast<const float*>(smem + SH::kOffK);
    const float* rows_l = rows_o + S * rows_per * kD;
    const int q_lo = rank * rows_per;
    const int b = item(0).b, h = item(0).h;
    const int n_rows = min(p.n_q, q_lo + rows_per) - q_lo;
#pragma unroll 1
    for (int t = tid; t < n_rows * (kD / 4); t += kThreadsTc) {
      const int qq = t / (kD / 4), d = (t % (kD / 4)) * 4;
      float mmax = -CUDART_INF_F;
#pragma unroll 1
      for (int r = 0; r < S; ++r) mmax = fmaxf(mmax, rows_l[r * rows_per + qq]);
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      float wsum = 0.f;
      if (mmax != -CUDART_INF_F)
#pragma unroll 2
        for (int r = 0; r < S; ++r) {  // in split order
          const float w = exp2f(rows_l[r * rows_per + qq] - mmax);
          const float4 v = *reinterpret_cast<const float4*>(rows_o + (r * rows_per + qq) * kD + d);
          wsum += w;
          acc.x += w * v.x;
          acc.y += w * v.y;
          acc.z += w * v.z;
          acc.w += w * v.w;
        }
      const float iw = wsum > 0.f ? 1.f / wsum : 0.f;
      const int q = q_lo + qq;
      float o[4] = {acc.x * iw, acc.y * iw, acc.z * iw, acc.w * iw};
      if (!F32)  // values clipped to +-65536 may leave the fp16 range
#pragma unroll
        for (int e = 0; e < 4; ++e) o[e] = clip_finite(o[e]);
      *reinterpret_cast<uint2*>(p.out + (static_cast<size_t>(b) * p.n_q + q) * p.out_stride + h * kD + d) =
          make_uint2(pack_half2(o[0], o[1]), pack_half2(o[2], o[3]));
      if (p.lse != nullptr && d == 0)
        p.lse[(static_cast<size_t>(b) * H + h) * p.n_q + q] =
            wsum > 0.f ? (mmax + log2f(wsum)) * 0.6931471805599453f : -CUDART_INF_F;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

}  // namespace

bool attention_tc_eligible(const AttnArgs& a, int n_splits) {
  return n_splits >= 1 && n_splits <= kMaxClusterSplits && a.n_q >= 1 && a.n_q <= 48 && a.n_own >= 1 &&
         a.n_own <= kSlotKeys;
}

namespace {
const void* tc_fn(int cache_dtype, bool split) {
  if (cache_dtype == 1)
    return split ? reinterpret_cast<const void*>(&attn_tc_kernel<false, true>)
                 : reinterpret_cast<const void*>(&attn_tc_kernel<false, false>);
  return split ? reinterpret_cast<const void*>(&attn_tc_kernel<true, true>)
               : reinterpret_cast<const void*>(&attn_tc_kernel<true, false>);
}
int tc_smem(int cache_dtype) { return cache_dtype == 1 ? Shape<false>::kSmem : Shape<true>::kSmem; }
}  // namespace

cudaError_t attention_tc_set_attributes(int cache_dtype, bool split) {
  return cudaFuncSetAttribute(tc_fn(cache_dtype, split), cudaFuncAttributeMaxDynamicSharedMemorySize,
                              tc_smem(cache_dtype));
}

// The most splits, at least 2 and at most `wanted`, whose clusters are all resident at once: one
// cluster in a second wave costs as much as the first wave. The occupancy counts clusters at one
// CTA per SM; two share an SM here, so s CTAs take the SMs of (s + 1) / 2 (32 clusters of 8 started
// within 3.3 us of one another, against 15 that it counts for 8 and 36 for 4).
// Split launches check every cache value, so a call that asks for splits keeps two.
static int resident_splits(int wanted, int B, int n_heads, int cache_dtype) {
  int s = wanted;
  while (s > 2 && max_resident_clusters(tc_fn(cache_dtype, true), kThreadsTc, static_cast<size_t>(tc_smem(cache_dtype)),
                                        (s + kCtasPerSm - 1) / kCtasPerSm) < static_cast<long long>(B) * n_heads)
    --s;
  return s;
}

cudaError_t launch_attention_tc(const AttnArgs& a_in, int B, int cache_dtype, cudaStream_t stream, bool pdl) {
  AttnArgs a = a_in;
  if (a.n_splits > 1) a.n_splits = resident_splits(a.n_splits, B, a.n_heads, cache_dtype);
  // a long cache begun last runs alone: 26 B/ns a CTA, so 1000 fp32 rows are 40 us
  int dev = 0, sm_count = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  a.by_length = a.plan == nullptr && a.targs == nullptr && B > 1 && B <= kMaxByLength &&
                static_cast<long long>(B) * a.n_heads * a.n_splits > static_cast<long long>(kCtasPerSm) * sm_count;
  AttnMaps maps{};
  if (!encode_rows_map(&maps.q, a.q, B, a.n_q, a.q_stride, a.n_heads) ||
      !encode_rows_map(&maps.k_own, a.k_own, B, a.n_own, a.own_stride, a.n_heads) ||
      !encode_rows_map(&maps.v_own, a.v_own, B, a.n_own, a.own_stride, a.n_heads))
    return cudaErrorInvalidValue;
  a.param_maps = 0;
  // one layer's caches outside a tick: maps by value (the row count is not known here; a chunk
  // is loaded by TMA only when all of its rows are the vehicle's)
  if (cache_dtype == 1 && a.targs == nullptr && a.k_cache != nullptr && a.v_cache != nullptr &&
      encode_cache_map(&maps.k, a.k_cache, INT32_MAX, static_cast<uint32_t>(a.n_heads)) &&
      encode_cache_map(&maps.v, a.v_cache, INT32_MAX, static_cast<uint32_t>(a.n_heads)))
    a.param_maps = 1;
  const long long items = static_cast<long long>(B) * a.n_heads;
  if (B > 65535 || a.n_heads > 65535 || items > INT32_MAX) return cudaErrorInvalidConfiguration;
  // one wave of CTAs, each with up to kMaxRounds items; more items: as many waves as that takes
  const long long wave = static_cast<long long>(kCtasPerSm) * sm_count;
  const long long waves = (items + wave * kMaxRounds - 1) / (wave * kMaxRounds);
  const dim3 grid = a.n_splits > 1 ? dim3(a.n_splits, a.n_heads, B)
                                   : dim3(static_cast<unsigned>(items < waves * wave ? items : waves * wave));
  void* kargs[] = {&a, &B, &maps};
  return launch_ex(tc_fn(cache_dtype, a.n_splits > 1), grid, dim3(kThreadsTc),
                   static_cast<size_t>(tc_smem(cache_dtype)), stream, pdl, kargs, 1, a.n_splits);
}

}  // namespace fsx
