// Eq. 1 of Sec. 3.1 on the 5th-generation tensor cores: one CTA per (vehicle, head, key split)
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
// its chunk 0 before its cache chunks. Chunk i sits in K / V slot i mod kSlots.
//
// Warp roles: warps 0-2 run the online softmax for query rows
// 16 w .. 16 w + 15, two rows per thread; warp 3 lane 0 issues S and P V as their inputs become
// ready; warps 4-5 stage and convert the K rows, warps 6-7 the V rows, two
// chunks ahead. Two CTAs per SM. bf16 caches: whole chunks by TMA. fp32 caches: 16-key stages by
// 16-byte copies, two in flight per tensor (32 KB a CTA), converted into the slot by the warp that
// copied the rows: another CTA's stream then hides a start-up, which 64-key stages and one CTA per SM
// cannot (24 vehicles with 16-1000 rows, 32 heads: 78 -> 76.8 us).
// Splits: the CTAs of one (vehicle, head) form a thread-block cluster and merge
// (log-sum-exp weights) by pushing each split's normalised fp32 rows to the rank that owns them
// through distributed shared memory. Split and fp32 launches check every cache value they stage
// against the fp16 range.
// Measured against the mma.sync kernel of attention.cu, which split and fp32 launches ran before: a
// tick of 4 vehicles with 0-700 bf16 rows, 8 layers, 2 splits: 740 -> 452 us; one vehicle with 2048
// rows, 8 splits, Eq. 1 alone: 34 -> 27 us a call; 24 vehicles with 16-1000 fp32 rows, Eq. 1
// alone: 104 -> 68 us a call (4.9 TB/s) with the order below.
// Launches of more than one wave without a plan start the longest caches first (each CTA finds its
// vehicle among at most 128 by counting; the 24 fp32 vehicles: 76.8 -> 67.7 us). A tick's plan is sorted already.
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
constexpr int kMaxByLength = 128;  // vehicles a launch without a plan sorts

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
// barriers: kfull[3], kempty[3], vfull[3], vempty[3], sfull[2], pfull[2], pvdone[2], drain, ktma[3], vtma[3]
constexpr int kNumBars = 25;
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
  static constexpr int kSmem = kOffBar + kNumBars * 8 + 8 /*tmem slot + abort*/;
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

// bounded wait that also gives up once another thread of the CTA gave up
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, int* status, volatile int* abort) {
  const uint32_t addr = smem_addr(bar);
  unsigned long long t0 = 0;
  for (uint32_t it = 0;; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
    if ((it & 63u) == 63u) {
      if (*abort) return false;
      const unsigned long long now = global_timer_ns();
      if (t0 == 0) {
        t0 = now;
      } else if (now - t0 > kWaitLimitNs) {
        set_status(status, kStatusTimeout);
        *abort = 1;
        return false;
      }
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

// map_k, map_v: maps of the one layer's caches when p.cache_maps is NULL and p.param_maps is set
template <bool F32, bool SPLIT>
__global__ void __launch_bounds__(kThreadsTc, kCtasPerSm)
    attn_tc_kernel(const AttnArgs p, const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v) {
  using SH = Shape<F32>;
  using CT = typename CacheType<F32>::T;
  constexpr int kSlots = SH::kSlots;
  constexpr bool kCheck = F32 || SPLIT;  // every staged cache value against the fp16 range
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const int lane = tid & 31;
  const int h = blockIdx.y;
  const int H = p.n_heads;
  const int S = SPLIT ? static_cast<int>(gridDim.x) : 1;     // the cluster spans the grid's x extent
  const int rank = SPLIT ? static_cast<int>(blockIdx.x) : 0;
  const int has_own = rank == 0 ? 1 : 0;                     // chunk 0 holds the own keys

  pdl_launch_dependents();
  pdl_wait();
  if ((smem_addr(smem) & 1023u) != 0u) {  // the swizzled operands need a 1024-byte aligned base
    if (tid == 0) set_status(p.status, kStatusDeviceArg);
    return;
  }
  // Start-up is a chain of dependent global loads (vehicle, offsets, queries, own rows),
  // each at the latency of a loaded memory system. The batched tick hands every CTA row
  // its schedule entry (vehicle, first cache row, length: one load); the copies of the
  // vehicle's queries and own keys / values are then in flight while the rest is read.
  const CT* kc;
  const CT* vc;
  if (p.targs != nullptr) {
    kc = static_cast<const CT*>(p.targs->k_cache[p.layer]);
    vc = static_cast<const CT*>(p.targs->v_cache[p.layer]);
  } else {
    kc = static_cast<const CT*>(p.k_cache);
    vc = static_cast<const CT*>(p.v_cache);
  }
  AttnPlan plan_z{0, 0, 0};
  if (p.plan != nullptr) plan_z = p.plan[blockIdx.z];
  int b = p.plan != nullptr ? plan_z.b : static_cast<int>(blockIdx.z);
  if (p.by_length) {  // this CTA's vehicle: the one with blockIdx.z longer caches before it (ties by index)
    long long* len = reinterpret_cast<long long*>(smem + SH::kOffK);
    int* pick = reinterpret_cast<int*>(len + kMaxByLength);
    const int n = static_cast<int>(gridDim.z);
    if (tid < n) len[tid] = p.offsets[tid + 1] - p.offsets[tid];
    __syncthreads();
    if (tid < n) {
      const long long mine = len[tid];
      int before = 0;
#pragma unroll 4
      for (int j = 0; j < n; ++j) before += len[j] > mine || (len[j] == mine && j < tid) ? 1 : 0;
      if (before == static_cast<int>(blockIdx.z)) *pick = tid;
    }
    __syncthreads();
    b = *pick;
    __syncthreads();  // read before the slot is staged into
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
  uint64_t* ktma = bars + 19;    // [3] a whole cache chunk's K rows landed by TMA
  uint64_t* vtma = bars + 22;    // [3] the same for V
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + kNumBars);
  volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);

  // ---- producers' staging of chunk i (own rows fp16, cache rows bf16 converted later)
  const bool is_prod = warp >= kProdWarp0;
  const bool is_v = warp >= kProdWarp0 + kProdWarps;
  const int pw = warp & (kProdWarps - 1);  // warp within the tensor's staging warps
  const int pt = pw * 32 + lane;               // thread within them
  const int pu = pt & 15;                      // 16-byte unit of a 256-byte row
  const int pr0 = pt >> 4;                     // rows pr0, pr0 + kRowStep, ...
  constexpr int kRowStep = kProdThreads / 16;
  const size_t tok = static_cast<size_t>(H) * kD;
  const __half* obase = (is_v ? p.v_own : p.k_own) + static_cast<size_t>(b) * p.n_own * p.own_stride + h * kD + pu * 8;
  const CT* cbase = nullptr;             // this CTA's first cache row of the tensor (its head), set below
  long long L = 0;                       // cache keys of this CTA
  long long row0 = 0;                    // this CTA's first cache row, set below
  unsigned char* pslots = is_v ? vslot : kslot;
  // Whole cache chunks (every cache chunk but a short last one) come by two TMA box loads
  // issued by one thread of the tensor's warps (when the batched tick supplies the cache
  // maps); the own keys and a short last chunk by 16-byte copies of every thread.
  const CUtensorMap* tmap = nullptr;
  if (!F32) {
    if (p.cache_maps != nullptr && p.targs != nullptr)
      tmap = p.cache_maps + 2 * p.layer + (is_v ? 1 : 0);
    else if (p.param_maps)
      tmap = is_v ? &map_v : &map_k;
  }
  uint64_t* tbar = is_v ? vtma : ktma;
  auto is_own = [&](int i) { return i < has_own; };
  auto by_tma = [&](int i) {
    return tmap != nullptr && i >= has_own && static_cast<long long>(i - has_own + 1) * kSlotKeys <= L;
  };
  // the TMA chunks follow the own chunk, so slot s = i mod kSlots sees them in order from its
  // first one (i = kSlots for slot 0 behind an own chunk): the phase of chunk i on its slot's barrier
  auto tma_parity = [&](int i) {
    return static_cast<uint32_t>((i / kSlots - (has_own != 0 && i % kSlots == 0 ? 1 : 0)) & 1);
  };
  auto chunk_rows = [&](int i) {
    return is_own(i) ? p.n_own
                     : static_cast<int>(min(static_cast<long long>(kSlotKeys),
                                            L - (i - has_own) * static_cast<long long>(kSlotKeys)));
  };
  // fp32: raw stage t (keys 16 t .. of this CTA's run), one warp instruction a row; row r of a stage
  // is the warp's that has r mod kProdWarps == pw. Past the run's end an empty group.
  auto issue_raw = [&](int t) {
    const int rows = static_cast<int>(min(static_cast<long long>(kRawKeys), L - static_cast<long long>(t) * kRawKeys));
    const uint32_t raw = smem_addr(smem + SH::kOffRaw + ((is_v ? 2 : 0) + (t & 1)) * kRawBytes) + lane * 16;
    const CT* src = cbase + static_cast<size_t>(t) * kRawKeys * tok + lane * 4;
#pragma unroll
    for (int r = pw; r < kRawKeys; r += kProdWarps)
      if (r < rows) cp_async_16(raw + r * (kD * 4), src + static_cast<size_t>(r) * tok);
    cp_async_commit();
  };
  auto issue = [&](int i) {
    unsigned char* slot = pslots + (i % kSlots) * kSlotBytes;
    const int rows = chunk_rows(i);
    const long long c0 = (i - has_own) * static_cast<long long>(kSlotKeys);
    if (by_tma(i)) {
      if (pt == 0) {
        uint64_t* bar = tbar + i % kSlots;
        const int y = static_cast<int>(row0 + c0);
        mbar_arrive_expect_tx(bar, kSlotBytes);
        tma_load_cache(slot, tmap, 0, h, y, bar);
        tma_load_cache(slot + kSlotBytes / 2, tmap, 64, h, y, bar);
      }
      cp_async_commit();  // an empty group keeps one group per chunk
      return;
    }
#pragma unroll 8
    for (int m = 0; m < kSlotKeys / kRowStep; ++m) {
      const int r = pr0 + kRowStep * m;
      unsigned char* dst = slot + tile128_off(r, pu);
      if (r < rows) {
        const void* src = is_own(i) ? static_cast<const void*>(obase + static_cast<size_t>(r) * p.own_stride)
                                    : static_cast<const void*>(cbase + static_cast<size_t>(c0 + r) * tok + pu * 8);
        cp_async_16(smem_addr(dst), src);
      } else {
        *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);  // keys past the range: finite zeros
      }
    }
    cp_async_commit();
  };
  // queries: 64 rows x 16 units, rows >= n_q zero (one copy group per thread)
  for (int i = tid; i < 64 * 16; i += kThreadsTc) {
    const int r = i >> 4;
    const int u = i & 15;
    unsigned char* dst = qt + tile128_off(r, u);
    if (r < p.n_q)
      cp_async_16(smem_addr(dst), p.q + (static_cast<size_t>(b) * p.n_q + r) * p.q_stride + h * kD + u * 8);
    else
      *reinterpret_cast<uint4*>(dst) = make_uint4(0u, 0u, 0u, 0u);
  }
  cp_async_commit();
  if (is_prod && has_own != 0) issue(0);  // own keys / values

  long long o_lo, o_hi;
  if (p.plan != nullptr) {
    o_lo = plan_z.lo;
    o_hi = o_lo + plan_z.len;  // a length of -1 fails the check below
  } else {
    const int64_t* offs = p.targs != nullptr ? p.targs->offsets : p.offsets;
    const int64_t* starts = p.targs != nullptr ? p.targs->starts : nullptr;
    o_lo = starts != nullptr ? starts[b] : offs[b];
    o_hi = o_lo + (offs[b + 1] - offs[b]);
  }
  if (o_lo < 0 || o_hi < o_lo || o_hi > p.max_total || (o_hi > o_lo && (kc == nullptr || vc == nullptr))) {
    cp_async_wait<0>();  // the query / own-row copies land before the CTA leaves
    set_status(p.status, kStatusDeviceArg);  // never read outside the caller's cache
    return;
  }
  L = o_hi - o_lo;
  row0 = o_lo;
  if (SPLIT) {  // this split's run of whole chunks
    const long long n_cc = (L + kSlotKeys - 1) / kSlotKeys;
    const long long k_lo = n_cc * rank / S * kSlotKeys, k_hi = min(L, n_cc * (rank + 1) / S * kSlotKeys);
    row0 = o_lo + k_lo;
    L = k_hi > k_lo ? k_hi - k_lo : 0;
  }
  const int n_chunks = has_own + static_cast<int>((L + kSlotKeys - 1) / kSlotKeys);  // 0: a split without keys
  cbase = (is_v ? vc : kc) + (static_cast<size_t>(row0) * H + h) * kD;

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
    // a kernel before this one has already abandoned the tick: this CTA stops below
    *abort = *reinterpret_cast<volatile int*>(p.status) != 0 ? 1 : 0;
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const int n_first = min(n_chunks, 2);  // chunks whose loads are issued up front
  if (is_prod) {  // the first cache chunks; then wait for this thread's query copies
    if (pt == 0 && tmap != nullptr) {  // the TMA barriers, before the first TMA chunk; read after the CTA barrier
      for (int i = 0; i < kSlots; ++i) mbar_init(tbar + i, 1);
      fence_proxy_async();
    }
    if (F32) {
      issue_raw(0);
      issue_raw(1);
      if (has_own != 0)
        cp_async_wait<3>();
      else
        cp_async_wait<2>();
    } else {
      for (int i = has_own; i < n_first; ++i) issue(i);
      if (n_first == 2)
        cp_async_wait<2>();
      else if (n_first == 1)
        cp_async_wait<1>();
      else
        cp_async_wait<0>();
    }
  } else {
    cp_async_wait<0>();
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(tmem_slot);
  if (*abort) {  // the tick was abandoned before this kernel: no MMA was issued
    cp_async_wait<0>();
    if (is_prod && pt == 0)
      for (int i = has_own; i < n_first; ++i)  // the first chunks landed
        if (by_tma(i)) mbar_wait(tbar + i % kSlots, tma_parity(i), p.status);
    if (SPLIT) {  // the other splits may not have seen the status yet: they push their rows here
      cluster_barrier();
      cluster_barrier();
    }
    if (warp == kMmaWarp)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    return;
  }

  if (warp == kMmaWarp) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      const uint32_t id_s = idesc_f16_mn(64, kSlotKeys, false);
      const uint32_t id_pv_own = idesc_f16_mn(64, kD, true);       // fp16 P, fp16 own V
      const uint32_t id_pv = idesc_f16_mn(64, kD, true) | (1u << 7) | (1u << 10);  // bf16 P, bf16 cache V
      const uint32_t aq = smem_addr(qt);
      auto issue_s = [&](int i) {  // S of chunk i into buffer i & 1
        const uint32_t d = tmem + kColS + (i & 1) * kSlotKeys;
        const uint32_t kb = smem_addr(kslot + (i % kSlots) * kSlotBytes);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t off = (kk >> 2) * 8192 + (kk & 3) * 32;
          umma_f16(d, sw128_desc(aq + off), sw128_desc(kb + off), id_s, kk > 0 ? 1u : 0u);
        }
        umma_commit(kempty + (i % kSlots));
        umma_commit(sfull + (i & 1));
      };
      auto issue_pv = [&](int i) {  // O (+)= P V of chunk i, P from tensor memory
        const uint32_t pa = tmem + kColS + (i & 1) * kSlotKeys;
        const uint32_t vb = smem_addr(vslot + (i % kSlots) * kSlotBytes);
        const uint32_t idv = F32 || is_own(i) ? id_pv_own : id_pv;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {  // 16 keys = 8 columns of packed fp16 pairs
          const uint64_t bd = sw128_desc_mn(vb + kk * 2048, 8192, 1024);
          umma_f16_ta(tmem + kColO, pa + kk * 8, bd, idv, (i > 0 || kk > 0) ? 1u : 0u);  // P_hi
          umma_f16_ta(tmem + kColO, pa + kSlotKeys / 2 + kk * 8, bd, idv, 1u);          // P_lo
        }
        umma_commit(vempty + (i % kSlots));
        umma_commit(pvdone + (i & 1));
      };
      // S(ns) and P V(npv) are issued as soon as their inputs are ready: S(ns) needs
      // its K rows and P V(ns - 2) done with the buffer it overwrites, P V(npv) needs
      // P(npv) and its V rows. Each test is at most one phase behind its barrier.
      int ns = 0, npv = 0;
      unsigned long long t_idle = 0;
      for (uint32_t it = 0; npv < n_chunks; ++it) {
        bool progressed = false;
        if (ns < n_chunks && (ns < 2 || npv >= ns - 1) && test_bar(kfull + (ns % kSlots), (ns / kSlots) & 1) &&
            (ns < 2 || test_bar(pvdone + (ns & 1), ((ns - 2) >> 1) & 1))) {
          tc_fence_after();
          issue_s(ns);
          ++ns;
          progressed = true;
        }
        if (npv < ns && test_bar(pfull + (npv & 1), (npv >> 1) & 1) &&
            test_bar(vfull + (npv % kSlots), (npv / kSlots) & 1)) {
          tc_fence_after();
          issue_pv(npv);
          ++npv;
          progressed = true;
        }
        if (progressed) {
          t_idle = 0;
        } else if ((it & 63u) == 63u) {
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
    }
    __syncwarp();
  } else if (is_prod) {
    // ---------------------------------------------------------------- producers
    // per chunk i: wait for its rows, convert cache rows bf16 -> fp16 in place (each
    // thread the units it copied), signal, then refill the slot of chunk i - 1 with
    // chunk i + 2 once the MMAs released it
    uint64_t* full = is_v ? vfull : kfull;
    uint64_t* empty = is_v ? vempty : kempty;
    bool ok = true;
    int issued = n_first;  // chunks whose loads were issued
    uint32_t range = 0;    // fp32: largest magnitudes of the staged values; bf16: bits set by out-of-range ones
    int i = 0;
    for (; ok && i < n_chunks; ++i) {
      unsigned char* slot = pslots + (i % kSlots) * kSlotBytes;
      if (F32) {
        if (is_own(i)) {
          cp_async_wait<2>();  // the two raw stages behind it stay in flight
        } else {               // raw rows -> fp16 slot, once its previous chunk is consumed
          ok = wait_bar(empty + i % kSlots, (i / kSlots) & 1, p.status, abort);
          if (!ok) break;
          const int rows = chunk_rows(i);
          const int u = lane & 15;
          const int sw = (lane >> 2) & 1;  // the two 16-byte reads of a unit in an order that spreads the banks
          for (int st = 0; st < kRawPerChunk; ++st) {
            const int t = (i - has_own) * kRawPerChunk + st;
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
              }
              *reinterpret_cast<uint4*>(slot + tile128_off(st * kRawKeys + r, u)) = out;
            }
            __syncwarp();  // the raw rows are read before they are refilled
            issue_raw(t + 2);
          }
        }
        fence_proxy_async();
        mbar_arrive(full + (i % kSlots));
        continue;
      }
      if (i + 1 < n_chunks) cp_async_wait<1>();
      else cp_async_wait<0>();
      if (by_tma(i)) {
        ok = wait_bar(tbar + i % kSlots, tma_parity(i), p.status, abort);
        if (!ok) break;
      }
      // refill first when the slot of chunk i - 1 is already free (the warp agrees on it)
      bool refilled = false;
      if (i + 2 < n_chunks) {
        refilled = __all_sync(0xffffffffu, test_bar(empty + ((i + 2) % kSlots), ((i + 2) / kSlots) & 1));
        if (refilled) {
          issue(i + 2);
          issued = i + 3;
        }
      }
      if (!is_own(i) && (!is_v || kCheck)) {  // cache K rows -> fp16 (V stays bf16): every read before the first write
        uint4 v[kSlotKeys / kRowStep];
#pragma unroll
        for (int m = 0; m < kSlotKeys / kRowStep; ++m)
          v[m] = *reinterpret_cast<const uint4*>(slot + tile128_off(pr0 + kRowStep * m, pu));
        if (kCheck) {
#pragma unroll
          for (int m = 0; m < kSlotKeys / kRowStep; ++m)
            range |= bf16x2_out_of_range(v[m].x) | bf16x2_out_of_range(v[m].y) | bf16x2_out_of_range(v[m].z) |
                     bf16x2_out_of_range(v[m].w);
        }
        if (!is_v) {
#pragma unroll
          for (int m = 0; m < kSlotKeys / kRowStep; ++m)
            *reinterpret_cast<uint4*>(slot + tile128_off(pr0 + kRowStep * m, pu)) =
                make_uint4(bf16x2_to_half2(v[m].x), bf16x2_to_half2(v[m].y), bf16x2_to_half2(v[m].z),
                           bf16x2_to_half2(v[m].w));
        }
      }
      fence_proxy_async();
      mbar_arrive(full + (i % kSlots));
      if (i + 2 < n_chunks && !refilled) {
        ok = wait_bar(empty + ((i + 2) % kSlots), ((i + 2) / kSlots) & 1, p.status, abort);
        if (ok) {
          issue(i + 2);
          issued = i + 3;
        }
      }
    }
    if (F32) flag_range(p.status, range);
    else if (SPLIT && range != 0) set_status(p.status, kStatusRange);
    cp_async_wait<0>();
    // after an abort: the TMA chunks issued but not consumed land before the CTA leaves
    if (pt == 0)
      for (int j = i; j < issued; ++j)
        if (by_tma(j)) mbar_wait(tbar + j % kSlots, tma_parity(j), p.status);
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
    float m_run[2] = {-CUDART_INF_F, -CUDART_INF_F};
    float l_run[2] = {0.f, 0.f};
    bool ok = true;
    for (int i = 0; i < n_chunks; ++i) {
      const int valid = chunk_rows(i);
      ok = wait_bar(sfull + (i & 1), (i >> 1) & 1, p.status, abort);
      if (!ok) break;
      tc_fence_after();
      const uint32_t sbuf = tmem + lane_base + kColS + (i & 1) * kSlotKeys;
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
          const float p0 = ex2_approx(fmaf(s[r][2 * g], scale_log2, nm));
          const float p1 = ex2_approx(fmaf(s[r][2 * g + 1], scale_log2, nm));
          r4[g & 3] += p0 + p1;
          uint32_t hi, lo;
          if (F32 || is_own(i)) {  // fp16 like the V rows
            hi = pack_half2(p0, p1);
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&hi));
            lo = pack_half2(p0 - f.x, p1 - f.y);
          } else {  // bf16 cache chunks: bf16 like the V rows
            hi = pack_bf16x2(p0, p1);
            lo = pack_bf16x2(p0 - __uint_as_float(hi << 16), p1 - __uint_as_float(hi & 0xffff0000u));
          }
          ph[2 * g + r] = hi;
          pl[2 * g + r] = lo;
        }
        float rs = (r4[0] + r4[1]) + (r4[2] + r4[3]);
        rs += __shfl_xor_sync(0xffffffffu, rs, 1);
        rs += __shfl_xor_sync(0xffffffffu, rs, 2);
        l_run[r] = l_run[r] * alpha[r] + rs;
      }
      if (any_grow && i > 0) {
        // rescale this warp's O rows once P V of the previous chunk is done
        ok = wait_bar(pvdone + ((i - 1) & 1), ((i - 1) >> 1) & 1, p.status, abort);
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
      mbar_arrive(pfull + (i & 1));
    }
    ok = ok && wait_bar(drain, 0, p.status, abort);  // every P V done
    tc_fence_after();
    const float inv[2] = {l_run[0] > 0.f ? 1.f / l_run[0] : 0.f, l_run[1] > 0.f ? 1.f / l_run[1] : 0.f};
    const bool va = ra < p.n_q;
    const bool vb = rbw < p.n_q;
    // A cache key beyond the fp16 range became an infinity here; where it raised a
    // score to +inf (or NaN) the row's sum is NaN: report it, the tick is abandoned.
    // (A key whose scores all fell to -inf carries weight 0, as the exact value would.)
    if (ok && ((va && !(l_run[0] == l_run[0])) || (vb && !(l_run[1] == l_run[1])))) set_status(p.status, kStatusRange);
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
      if (ok) {
#pragma unroll 1
        for (int c = 0; c < kD; c += 64) {
          uint32_t o[32];
          __syncwarp();
          tmem_ld_16x256b_x8(tmem + lane_base + kColO + c, o);
          const bool any = n_chunks > 0;  // a split without keys pushes zeros (its accumulator was never written)
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
      }
      __syncwarp();
    } else if (ok) {
      __half* oa = p.out + (static_cast<size_t>(b) * p.n_q + (va ? ra : 0)) * p.out_stride + h * kD + 2 * t4;
      __half* ob = p.out + (static_cast<size_t>(b) * p.n_q + (vb ? rbw : 0)) * p.out_stride + h * kD + 2 * t4;
#pragma unroll 1
      for (int c = 0; c < kD; c += 64) {
        uint32_t o[32];
        tmem_ld_16x256b_x8(tmem + lane_base + kColO + c, o);
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
    const int n_rows = min(p.n_q, q_lo + rows_per) - q_lo;
    for (int t = tid; t < n_rows * (kD / 4); t += kThreadsTc) {
      const int qq = t / (kD / 4), d = (t % (kD / 4)) * 4;
      float mmax = -CUDART_INF_F;
      for (int r = 0; r < S; ++r) mmax = fmaxf(mmax, rows_l[r * rows_per + qq]);
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      float wsum = 0.f;
      if (mmax != -CUDART_INF_F)
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
      *reinterpret_cast<uint2*>(p.out + (static_cast<size_t>(b) * p.n_q + q) * p.out_stride + h * kD + d) =
          make_uint2(pack_half2(acc.x * iw, acc.y * iw), pack_half2(acc.z * iw, acc.w * iw));
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
  // a long cache that starts in the last wave runs alone: 26 B/ns a CTA, so 1000 fp32 rows are 40 us
  int dev = 0, sm_count = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  a.by_length = a.plan == nullptr && a.targs == nullptr && B > 1 && B <= kMaxByLength &&
                static_cast<long long>(B) * a.n_heads * a.n_splits > static_cast<long long>(kCtasPerSm) * sm_count;
  CUtensorMap map_k{}, map_v{};
  a.param_maps = 0;
  // one layer's caches outside a tick: maps by value (the row count is not known here; a chunk
  // is loaded by TMA only when all of its rows are the vehicle's)
  if (cache_dtype == 1 && a.targs == nullptr && a.k_cache != nullptr && a.v_cache != nullptr &&
      encode_cache_map(&map_k, a.k_cache, INT32_MAX, static_cast<uint32_t>(a.n_heads)) &&
      encode_cache_map(&map_v, a.v_cache, INT32_MAX, static_cast<uint32_t>(a.n_heads)))
    a.param_maps = 1;
  void* kargs[] = {&a, &map_k, &map_v};
  return launch_ex(tc_fn(cache_dtype, a.n_splits > 1), dim3(a.n_splits, a.n_heads, B), dim3(kThreadsTc),
                   static_cast<size_t>(tc_smem(cache_dtype)), stream, pdl, kargs, 1, a.n_splits);
}

}  // namespace fsx
