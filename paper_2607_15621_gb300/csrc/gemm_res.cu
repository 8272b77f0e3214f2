// Residual projections of the expert layer (W_o, W_d; Sec. 3.1) for batches whose output tiles
// do not fill the chip: x[m, n] += D, D[128 weight rows, BN tokens] = W_tile[128, K] . A[BN tokens, K]^T
// on tcgen05, K cut over the 2-8 CTAs of a thread-block cluster.
//
// Each CTA runs its K steps into one accumulator in tensor memory, then the cluster
// reduce-scatters the partial tiles through distributed shared memory: every CTA owns a run of
// the tile's 4-token groups, the others send it their fp32 partials of those groups by st.async
// stores that complete on its mbarrier (its own partials too), and it adds them in split order (deterministic), updates
// x, its fp16 copy and the per-token sums of x^2. The partials never pass through L2 and no CTA
// polls global memory. Measured against that path (write the partial tile, fence, counter, poll,
// read back), ticks of 8 layers: 4 vehicles 441 -> 404 us, 16 vehicles 512 -> 484 us, 40 clip blocks
// 848 -> 818 us. In a launch of W_o for 672 tokens (96-token tiles, 4 splits) the K steps took 3.4 us,
// the exchange 3.4 us and the update 1.3 us (device timer, steps of 0.26 us). The last two were long
// for their code: a launch finds its instructions evicted by the layer's other kernels, and 42 KB of
// them, most in this epilogue, came in on its critical path. At 27 KB (destinations from a table made
// before the wait on the previous kernel, one site of the push, one address per token): 4 vehicles
// 405 -> 374 us, 16 vehicles 480 -> 459, the clip 731 -> 724, a two-layer append of 4 tokens 199 -> 194.
//   warp 0: producer (one bulk copy of a packed 16 KB weight image and one 2-D TMA token box per
//           64-wide K step; the first weights before the wait on the previous kernel);
//   warp 1: MMA issue (M = 128, N = BN, K = 16);
//   warps 2-9: epilogue, two groups of four warps (one per tensor-memory lane quadrant) taking
//           16-token chunks in turn; x is requested before the accumulator is ready.
#include <cuda.h>

#include <algorithm>

#include "device_util.cuh"
#include "gemm_tc.h"
#include "tcgen05.cuh"

namespace fsx {

namespace {

constexpr int kRows = kTcTileRows;
constexpr int kWBytes = kTcTileBytes;
constexpr int kMaxCluster = 8;                 // portable cluster size
constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kGroupBytes = kRows * 16;       // partials of 4 tokens: [128 rows][4 tokens] fp32

template <int BN>
__host__ __device__ constexpr int stage_bytes() {
  return kWBytes + BN * kTcTileK * 2;
}
template <int BN>
__host__ __device__ constexpr int recv_bytes() {  // [split][own groups]: rounding adds at most a group per split
  return (BN / 4 + kMaxCluster - 1) * kGroupBytes;
}
template <int BN>
__host__ __device__ constexpr int n_stages() {
  return BN <= 16 ? 10 : BN <= 48 ? 8 : (BN <= 64 ? 7 : (BN <= 96 ? 5 : (BN <= 144 ? 4 : 3)));
}
template <int BN>
__host__ __device__ constexpr int smem_bytes() {
  return 1024 /* alignment */ + 1024 /* barriers */ + recv_bytes<BN>() + n_stages<BN>() * stage_bytes<BN>();
}
static_assert(smem_bytes<16>() <= 232448 && smem_bytes<48>() <= 232448 && smem_bytes<64>() <= 232448 && smem_bytes<96>() <= 232448 &&
                  smem_bytes<128>() <= 232448 && smem_bytes<144>() <= 232448 && smem_bytes<160>() <= 232448,
              "shared memory of a token tile exceeds the per-block limit");
template <int BN>
__host__ __device__ constexpr uint32_t tmem_cols() {
  return BN <= 32 ? 32 : BN <= 64 ? 64 : (BN <= 128 ? 128 : 256);
}

__device__ __forceinline__ void tma_tokens(void* dst, const CUtensorMap* map, int k, int m, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_addr(dst)),
      "l"(map), "r"(k), "r"(m), "r"(smem_addr(bar))
      : "memory");
}
// 16 fp32 columns of the warp's 32 tensor-memory lanes, without waiting
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// the wait for every load of this thread, tied to the registers
__device__ __forceinline__ void tmem_wait16(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}
__device__ __forceinline__ uint32_t peer_addr(uint32_t local, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

template <int BN>
__global__ void __launch_bounds__(kThreads, 1) gemm_res_kernel(const __grid_constant__ CUtensorMap map_a,
                                                              const TcGemmArgs p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  constexpr int kStages = n_stages<BN>();
  constexpr int kStageBytes = stage_bytes<BN>();
  // the same offset in every CTA of the cluster: the dynamic base is the same
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(base);
  uint64_t* empty = full + kStages;
  uint64_t* tmem_full = empty + kStages;  // the accumulator is ready (every MMA of the CTA done)
  uint64_t* rx = tmem_full + 1;           // the other splits' partials of this CTA's groups
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(rx + 1);
  volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  // [n_groups]: where in the cluster this CTA's partials of a 4-token group go, and the barrier they complete on
  uint2* route = reinterpret_cast<uint2*>(base + 256);
  static_assert(256 + BN / 4 * 8 <= 1024 && 2 * kStages * 8 + 24 <= 256, "header");
  unsigned char* recv = base + 1024;
  unsigned char* stages = recv + recv_bytes<BN>();
  static_assert(recv_bytes<BN>() % 1024 == 0, "the stages must stay 1024-byte aligned");

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int KS = gridDim.x, rank = blockIdx.x;  // the cluster spans the grid's x extent
  const int tiles_n = p.N / kRows;
  const int t_n = blockIdx.y % tiles_n, m0 = (blockIdx.y / tiles_n) * BN;
  const int KT = p.K / kTcTileK;
  const int kt0 = rank * KT / KS, kt1 = (rank + 1) * KT / KS;
  // 4-token groups of the tile that hold tokens; this CTA owns groups g_lo .. g_hi - 1
  const int n_groups = min(BN, p.M - m0 + 3) / 4;
  auto group_lo = [&](int r) { return n_groups * r / KS; };
  const int g_lo = group_lo(rank), g_hi = group_lo(rank + 1);
  auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
    if (*abort) return false;
    const bool ok = mbar_wait(bar, parity, p.status);
    if (!ok) *abort = 1;
    return ok;
  };

  pdl_launch_dependents();
  if (tid == 0) {
    *abort = 0;
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    mbar_init(tmem_full, 1);
    mbar_init(rx, 1);
    mbar_arrive_expect_tx(rx, static_cast<uint32_t>(KS * (g_hi - g_lo) * kGroupBytes));
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (tid >= 64 && tid - 64 < n_groups) {
    const int g = tid - 64;
    int o = 0;
    while (g >= group_lo(o + 1)) ++o;
    const int o_lo = group_lo(o), slot = rank * (group_lo(o + 1) - o_lo) + g - o_lo;
    route[g] = make_uint2(peer_addr(smem_addr(recv) + static_cast<uint32_t>(slot * kGroupBytes), o),
                          peer_addr(smem_addr(rx), o));
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                 "r"(tmem_cols<BN>())
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(tmem_slot);
  const unsigned char* w = p.w + (static_cast<size_t>(t_n) * KT + kt0) * kWBytes;
  const int n = kt1 - kt0;
  if (warp == 0 && lane == 0)
    for (int g = 0; g < n && g < kStages; ++g) {
      mbar_arrive_expect_tx(full + g, kStageBytes);
      bulk_g2s(stages + g * kStageBytes, w + static_cast<size_t>(g) * kWBytes, kWBytes, full + g);
    }
  __syncwarp();
  cluster_arrive();  // every CTA's barriers are initialised before any partial is sent
  cluster_wait();
  pdl_wait();

  if (warp == 0) {
    int g = 0;
    for (; g < n; ++g) {
      const int s = g % kStages;
      unsigned char* st = stages + s * kStageBytes;
      // after a timeout no further copy is issued: its stage's last one may still be on its way
      if (g >= kStages && __any_sync(0xffffffffu, !wait(empty + s, static_cast<uint32_t>(((g / kStages) - 1) & 1)))) break;
      if (lane == 0) {
        if (g >= kStages) {
          mbar_arrive_expect_tx(full + s, kStageBytes);
          bulk_g2s(st, w + static_cast<size_t>(g) * kWBytes, kWBytes, full + s);
        }
        tma_tokens(st + kWBytes, &map_a, (kt0 + g) * kTcTileK, m0, full + s);
      }
      __syncwarp();
    }
    // after a timeout the MMA warp may have skipped its waits: the copies still in
    // flight land (bounded) before the shared memory is released
    if (*abort && lane == 0)
      for (int i = g > kStages ? g - kStages : 0; i < g; ++i) {
        const unsigned long long t0 = global_timer_ns();
        uint32_t done = 0;
        while (!done && global_timer_ns() - t0 < 100000000ull)
          asm volatile(
              "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
              : "=r"(done)
              : "r"(smem_addr(full + i % kStages)), "r"(static_cast<uint32_t>((i / kStages) & 1))
              : "memory");
      }
    __syncwarp();
    cluster_arrive();
  } else if (warp == 1) {
    constexpr uint32_t idesc = idesc_f16(kRows, BN);
    for (int g = 0; g < n; ++g) {
      const int s = g % kStages;
      wait(full + s, static_cast<uint32_t>((g / kStages) & 1));
      tc_fence_after();
      if (lane == 0) {
        const uint32_t a_base = smem_addr(stages + s * kStageBytes);
        const uint32_t b_base = a_base + kWBytes;
#pragma unroll
        for (int k = 0; k < kTcTileK / 16; ++k)
          umma_f16(tmem, sw128_desc(a_base + k * 32), sw128_desc(b_base + k * 32), idesc, (g > 0 || k > 0) ? 1u : 0u);
        umma_commit(empty + s);
      }
      __syncwarp();
    }
    if (lane == 0) umma_commit(tmem_full);
    __syncwarp();
    mbar_wait(tmem_full, 0u, p.status);  // every MMA done before the tensor memory is freed
    __syncwarp();
    cluster_arrive();
  } else {
    const int ew = warp - 2, grp = ew >> 2, q = warp & 3, row = q * 32 + lane;
    // epilogue warp ew updates the CTA's groups ew, ew + 8, ...: lane = rows lane + 32 i, 4 tokens
    float x[4][4];  // [i][token]
    auto load_x = [&](int gl) {
      const int m = m0 + 4 * (g_lo + gl);
#pragma unroll
      for (int t = 0; t < 4; ++t) {  // a token's address once, its rows at constant distances
        const float* src = p.xo + static_cast<size_t>(m + t) * p.ldxo + t_n * kRows + lane;
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i][t] = m + t < p.M ? __ldcg(src + 32 * i) : 0.f;
      }
    };
    const int n_own = g_hi - g_lo;
#pragma unroll 1
    for (int it = 0, gl = ew; it == 0 || gl < n_own; ++it, gl += kEpiWarps) {
      if (gl < n_own) load_x(gl);
      if (it == 0) {  // the exchange
        wait(tmem_full, 0u);
        tc_fence_after();
        const uint32_t taddr = tmem + (static_cast<uint32_t>(q * 32) << 16);
        const bool send = *abort == 0;
        // 16-token chunks grp, grp + 2, ... of the tile (BN is a multiple of 16), the next one on its way
        uint32_t ra[16], rb[16];
        int c = grp;
        __syncwarp();
        if (4 * c < n_groups) {
          tmem_ld16_issue(taddr + 16u * c, ra);
          tmem_wait16(ra);
        }
#pragma unroll 1
        for (; 4 * c < n_groups; c += 2) {
          const bool more = 4 * (c + 2) < n_groups;
          if (more) tmem_ld16_issue(taddr + 16u * (c + 2), rb);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (4 * c + e < n_groups && send) {
              const uint2 to = route[4 * c + e];
              st_async_v4(to.x + row * 16, make_uint4(ra[4 * e], ra[4 * e + 1], ra[4 * e + 2], ra[4 * e + 3]), to.y);
            }
          }
          __syncwarp();
          if (more) {
            tmem_wait16(rb);
#pragma unroll
            for (int e = 0; e < 16; ++e) ra[e] = rb[e];
          }
        }
        __syncwarp();
        cluster_arrive();  // this thread sends nothing more
        if (*abort == 0 && !mbar_wait_cluster(rx, 0u, p.status)) *abort = 1;
      }
      if (gl >= n_own) break;
      float acc[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int t = 0; t < 4; ++t) acc[i][t] = 0.f;
#pragma unroll 2
      for (int s = 0; s < KS; ++s) {  // in split order
        const unsigned char* src = recv + (s * n_own + gl) * kGroupBytes + lane * 16;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 v = *reinterpret_cast<const float4*>(src + i * 512);
          acc[i][0] += v.x;
          acc[i][1] += v.y;
          acc[i][2] += v.z;
          acc[i][3] += v.w;
        }
      }
      const int m = m0 + 4 * (g_lo + gl);
      float ss[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const size_t idx = static_cast<size_t>(m + t) * p.ldxo + t_n * kRows + lane;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc[i][t] += x[i][t];
          ss[t] += acc[i][t] * acc[i][t];
        }
        if (m + t < p.M) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            p.xo[idx + 32 * i] = acc[i][t];
            p.xo16[idx + 32 * i] = __float2half_rn(acc[i][t]);
          }
          if (p.x_copy != nullptr) {
#pragma unroll
            for (int i = 0; i < 4; ++i) p.x_copy[idx + 32 * i] = acc[i][t];
          }
        }
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const float s = warp_sum(ss[t]);
        if (lane == 0 && m + t < p.M) p.ss_out[static_cast<size_t>(t_n) * p.ss_stride + m + t] = s;
      }
    }
    __syncwarp();
  }
  // no CTA leaves while a partner may still send to it: in the normal course everything has
  // landed; after a timeout stores already issued are given 1 ms
  cluster_wait();
  if (*abort) {
    const unsigned long long t0 = global_timer_ns();
    while (global_timer_ns() - t0 < 1000000ull) {
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols<BN>()) : "memory");
}

const void* res_fn(int bn, size_t* smem) {
#define FSX_RES(BN_)                                               \
  if (bn == BN_) {                                                 \
    *smem = smem_bytes<BN_>();                                     \
    return reinterpret_cast<const void*>(&gemm_res_kernel<BN_>);   \
  }
  FSX_RES(16)
  FSX_RES(48)
  FSX_RES(64)
  FSX_RES(96)
  FSX_RES(128)
  FSX_RES(144)
  FSX_RES(160)
#undef FSX_RES
  return nullptr;
}

}  // namespace

cudaError_t gemm_res_set_attributes() {
  for (int bn : kResTiles) {
    size_t smem = 0;
    const void* fn = res_fn(bn, &smem);
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// The token tile and the K splits of a residual projection: the pair with the least copy time of a
// CTA, of those whose clusters are resident at once with one to spare (the last one that the
// occupancy allows was placed after the others had finished: 28 clusters of 5, W_o of 16 vehicles,
// 9 us late). A CTA loads its K steps (16 KB of weights and the token rows each) at up to 100 B/ns,
// all CTAs together at about 13 B/ps from L2, and exchanges its partial tile at about 37 B/ns
// (st.async, 18 B a cycle). splits = 1: the tiles fill the chip, or K is too short to cut.
ResPlan gemm_res_plan(int M, int N, int K) {
  ResPlan best{-1, 1};
  double best_ns = 0.;
  const int KT = K / kTcTileK;
  for (int i = 0; i < kResTileCount; ++i) {
    const int bn = kResTiles[i];
    if (bn == 16 && M > 16) continue;  // several tiles of 16 reread the weights as often
    const int tiles = (N / kRows) * ((M + bn - 1) / bn);
    size_t smem = 0;
    const void* fn = res_fn(bn, &smem);
    for (int ks = 2; ks <= kMaxCluster && ks <= KT / 4; ++ks) {  // at least 4 K steps a CTA
      if (tiles >= max_resident_clusters(fn, kThreads, smem, ks)) continue;
      const double rate = std::min(100., 13000. / (tiles * ks));
      const double ns = (KT + ks - 1) / ks * (kWBytes + bn * 128.) / rate + bn * 512. * (ks - 1) / ks / 37.;
      if (best.splits == 1 || ns < best_ns) {
        best = ResPlan{i, ks};
        best_ns = ns;
      }
    }
  }
  return best;
}

cudaError_t launch_gemm_res(const CUtensorMap& map_a, const TcGemmArgs& args, const ResPlan& plan, cudaStream_t stream,
                            bool pdl) {
  size_t smem = 0;
  const int bn = plan.tile >= 0 && plan.tile < kResTileCount ? kResTiles[plan.tile] : 0;
  const void* fn = res_fn(bn, &smem);
  if (fn == nullptr || plan.splits < 2 || plan.splits > kMaxCluster || args.N % kRows != 0 || args.K % kTcTileK != 0 ||
      args.M <= 0 || args.ss_out == nullptr)
    return cudaErrorInvalidValue;
  CUtensorMap map = map_a;
  TcGemmArgs a = args;
  void* kargs[] = {&map, &a};
  const dim3 grid(static_cast<unsigned>(plan.splits), static_cast<unsigned>((a.N / kRows) * ((a.M + bn - 1) / bn)));
  return launch_ex(fn, grid, dim3(kThreads), smem, stream, pdl, kargs, 1, plan.splits);
}

}  // namespace fsx
