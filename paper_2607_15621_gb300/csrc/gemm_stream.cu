// Projection GEMMs for few tokens (the cache append: n_new x B <= 256 token rows against
// a 7B backbone's weights): D[128 weight rows, BN tokens] = W_tile[128, K] . A[BN tokens, K]^T
// on tcgen05, every weight read once and all tokens in one tile, so the call is bound by
// the weight stream.
//
// The weight tiles lie behind one another in HBM (n-tile major, 64-wide K steps of 16 KB),
// so a matrix is one stream of N/128 x K/64 steps. It is cut into equal contiguous
// ranges, one per SM (to one step): no SM waits for a last wave, whatever the number of
// tiles (a whole-tile split left 56 of 152 SMs idle at 96 tiles and a second wave of 20 at
// 172). A tile that a range boundary cuts is written as fp32 partials, one segment per CTA;
// the CTA that arrives last on the tile's counter adds the segments in range order and runs
// the epilogue. No CTA ever waits for another one, so the kernel may share the GPU with
// kernels whose CTAs must all be resident, and the result does not depend on who is last.
// The first steps are requested before the previous kernel has finished (programmatic
// dependent launch): weights depend on no activation.
//   warp 0: producer (one bulk copy of the packed weight image and one 2-D TMA token box a
//           step); warp 1: MMA issue (M = 128, N = BN, two accumulators in tensor memory);
//   warps 2-9: epilogue, two groups of four warps (one per tensor-memory lane quadrant)
//           taking 8-token chunks in turn.
// Measured on the two-layer append (405 MB of weights a layer), against whole-tile CTAs with
// 128-token tiles, waiting K splits and no dependent launch, when W_o and W_d still ran here too:
// 4 tokens 311 -> 237 us a call (QKV 30.1 -> 23.7 us a launch, gate/up 55.8 -> 35.3, W_o and W_d
// together 42.6 -> 36.9), 64 tokens 370 -> 339 us (QKV 30.2 -> 26.7, gate/up 56.4 -> 42.0, W_o and
// W_d 45.5 -> 50.4; they have moved to gemm_res.cu where it has a split for them).
// More tokens, a whole one-layer append with 96-480 cached rows, before this kernel and the fused
// attention -> now: 64 tokens 286 -> 136 us, 96 of 12 vehicles 307 -> 152, 128 of 16 330 -> 174,
// 160 of 20 394 -> 182, 192 of 48 523 -> 234, 256 of 32 495 -> 239.
// Code size: a launch finds its instructions evicted by the layer's other kernels. One copy of the
// epilogue instead of one per chunk in flight and 32-bit step arithmetic (gate/up at 64 tokens
// 73 -> 49 KB, QKV at 16 tokens 33 -> 28): 4 tokens 193.5 -> 187.3 us a call, 64 tokens 266 -> 261.
#include <cuda.h>

#include "device_util.cuh"
#include "gemm_tc.h"
#include "tcgen05.cuh"

namespace fsx {

namespace {

constexpr int kRows = kTcTileRows;            // weight rows per tile
constexpr int kWBytes = kTcTileBytes;         // weight bytes of one K step
constexpr int kGroups = 2;                    // epilogue groups of 4 warps
constexpr int kEpiThreads = kGroups * 128;
constexpr int kThreads = 64 + kEpiThreads;
constexpr int kChunk = 8;                     // tokens per epilogue round of a group
constexpr int kHeader = 4096;                 // barriers, 1/rms [256], x^2 partials

template <int BN>
__host__ __device__ constexpr int stage_bytes() {
  return kWBytes + BN * kTcTileK * 2;
}
// With 16-token tiles a CTA takes half an SM, so that the next GEMM of the stream is resident and
// fills its ring while the last steps and the split sums of this one run (two-layer append of 4
// tokens: 237 -> 218 us a call together with the last GEMM writing the call's result itself).
// From 32 tokens on the sums of the split tiles weigh more than the fill, and one CTA per SM with
// a deeper ring and more registers for the sums is faster (64 tokens: 359 us a call with two CTAs
// of 4 stages, 333 us with one of 9).
template <int BN>
__host__ __device__ constexpr int ctas_per_sm() {
  return BN <= 16 ? 2 : 1;
}
template <int BN>
__host__ __device__ constexpr int n_stages() {  // as many as that share of the shared memory holds
  return BN <= 16 ? 6 : (BN <= 32 ? 10 : (BN <= 64 ? 9 : (BN <= 128 ? 6 : 4)));
}
constexpr int kBatch = 4;  // segments of a split tile in flight at once (QKV and gate/up have at most 3)
template <int BN>
__host__ __device__ constexpr int sum_chunks() {  // token chunks of a group summed at once
  return BN <= 16 ? 1 : (BN <= 32 ? 2 : 4);
}
template <int BN>
__host__ __device__ constexpr int smem_bytes() {
  return 1024 /* alignment of the ring */ + kHeader + n_stages<BN>() * stage_bytes<BN>();
}
template <int BN>
__host__ __device__ constexpr bool smem_fits() {  // 228 KB per SM, 1 KB of it reserved per CTA
  return ctas_per_sm<BN>() * (smem_bytes<BN>() + 1024) <= 228 * 1024;
}
static_assert(smem_fits<16>() && smem_fits<32>() && smem_fits<64>() && smem_fits<128>() && smem_fits<256>(),
              "shared memory of a token tile exceeds its share of an SM");

__device__ __forceinline__ void tma_tokens(void* dst, const CUtensorMap* map, int k, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_addr(dst)),
      "l"(map), "r"(k), "r"(0), "r"(smem_addr(bar))
      : "memory");
}

// 8 consecutive fp32 columns of the warp's 32 tensor-memory lanes
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
               :
               : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, 128;" ::"r"(1 + g) : "memory"); }
__device__ __forceinline__ void epi_sync() {
  asm volatile("bar.sync %0, %1;" ::"n"(1 + kGroups), "n"(kEpiThreads) : "memory");
}

template <int BN, int EPI, bool NORM>
__global__ void __launch_bounds__(kThreads, ctas_per_sm<BN>()) gemm_stream_kernel(const __grid_constant__ CUtensorMap map_a,
                                                                 const TcGemmArgs p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  constexpr int kStages = n_stages<BN>();
  constexpr int kStageBytes = stage_bytes<BN>();
  constexpr int kRound = sum_chunks<BN>();
  constexpr uint32_t kTmemCols = 2 * BN <= 32 ? 32 : 2 * BN;  // two accumulators of BN fp32 columns
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(base);
  uint64_t* empty = full + kStages;
  uint64_t* tmem_full = empty + kStages;  // [2] accumulator ready
  uint64_t* tmem_empty = tmem_full + 2;   // [2] accumulator drained
  uint64_t* drain = tmem_empty + 2;       // every MMA of the CTA done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* last = abort + 1;         // this CTA arrived last on the tile
  float* rstd = reinterpret_cast<float*>(base + 1024);                  // [BN]
  float* ssp = reinterpret_cast<float*>(base + 2048);                   // [groups][4 quadrants][8 tokens]
  unsigned char* stages = base + kHeader;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int KT = p.K / kTcTileK;
  // K steps of the matrix; times the CTAs they fit 32 bits (2^32 / 152 steps are 460 GB of weights)
  const uint32_t total = static_cast<uint32_t>(p.N / kRows) * KT;
  const int G = gridDim.x;
  const uint32_t s0 = total * blockIdx.x / G, s1 = total * (blockIdx.x + 1) / G;  // this CTA's steps
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
    for (int a = 0; a < 2; ++a) {
      mbar_init(tmem_full + a, 1);
      mbar_init(tmem_empty + a, 4 * kGroups);
    }
    mbar_init(drain, 1);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(tmem_slot);

  if (warp == 0) {
    // ---- producer: step s0 + g in stage g mod kStages; the weights of the first
    // kStages steps before the wait on the previous kernel
    const int n = static_cast<int>(s1 - s0);
    const unsigned char* w = p.w + static_cast<size_t>(s0) * kWBytes;
    if (lane == 0)
      for (int g = 0; g < n && g < kStages; ++g) {
        mbar_arrive_expect_tx(full + g, kStageBytes);
        bulk_g2s(stages + g * kStageBytes, w + static_cast<size_t>(g) * kWBytes, kWBytes, full + g);
      }
    __syncwarp();
    pdl_wait();
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
        tma_tokens(st + kWBytes, &map_a, static_cast<int>((s0 + g) % KT) * kTcTileK, full + s);
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
  } else if (warp == 1) {
    // ---- MMA issuer: one accumulator per segment (the CTA's steps of one tile)
    pdl_wait();
    constexpr uint32_t idesc = idesc_f16(kRows, BN);
    int g = 0, i = 0;
    for (uint32_t t = s0; t < s1; ++i) {
      const uint32_t end = min(s1, (t / KT + 1) * KT);
      const int acc = i & 1;
      if (i >= 2) wait(tmem_empty + acc, static_cast<uint32_t>(((i >> 1) - 1) & 1));
      tc_fence_after();
      const uint32_t d = tmem + static_cast<uint32_t>(acc * BN);
      for (bool first = true; t < end; ++t, ++g) {
        const int s = g % kStages;
        wait(full + s, static_cast<uint32_t>((g / kStages) & 1));
        tc_fence_after();
        if (lane == 0) {
          const uint32_t a_base = smem_addr(stages + s * kStageBytes);
          const uint32_t b_base = a_base + kWBytes;
#pragma unroll
          for (int k = 0; k < kTcTileK / 16; ++k)
            umma_f16(d, sw128_desc(a_base + k * 32), sw128_desc(b_base + k * 32), idesc, (!first || k > 0) ? 1u : 0u);
          umma_commit(empty + s);
        }
        first = false;
        __syncwarp();
      }
      if (lane == 0) umma_commit(tmem_full + acc);
      __syncwarp();
    }
    if (lane == 0) umma_commit(drain);  // every MMA done before the tensor memory is freed
    __syncwarp();
    mbar_wait(drain, 0u, p.status);
  } else {
    // ---- epilogue: thread = weight row `row` of the tile, group `grp` takes token chunks
    // grp, grp + 2, ... of 8 tokens
    pdl_wait();
    const int etid = tid - 64, grp = etid >> 7, gtid = etid & 127;
    const int q = warp & 3, row = q * 32 + lane;
    if (NORM) {  // 1/rms of every token from the per-128-column sums of x^2: 8 threads a token
      for (int m0 = 0; m0 < BN; m0 += kEpiThreads / 8) {
        const int m = m0 + (etid >> 3);
        float ss = 0.f;
        if (m < p.M)
          for (int j = etid & 7; j < p.n_ss; j += 8) ss += __ldcg(p.ss_in + static_cast<size_t>(j) * p.ss_stride + m);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        if ((etid & 7) == 0 && m < BN) rstd[m] = rsqrtf(ss / static_cast<float>(p.K) + 1e-6f);
      }
      epi_sync();
    }
    // tokens c0 .. c0 + 7 of tile t_n, this thread's row
    auto finish = [&](int t_n, int c0, float (&v)[kChunk]) {
      const int n0 = t_n * kRows;
      if (EPI == kEpiResidual) {
        float x[kChunk];
        const size_t idx = static_cast<size_t>(c0) * p.ldxo + n0 + row;
#pragma unroll
        for (int j = 0; j < kChunk; ++j)  // every load before the first store
          x[j] = c0 + j < p.M ? __ldcg(p.xo + idx + static_cast<size_t>(j) * p.ldxo) : 0.f;
#pragma unroll
        for (int j = 0; j < kChunk; ++j)
          if (c0 + j < p.M) {
            x[j] += v[j];
            p.xo[idx + static_cast<size_t>(j) * p.ldxo] = x[j];
            p.xo16[idx + static_cast<size_t>(j) * p.ldxo] = __float2half_rn(x[j]);
            if (p.x_copy != nullptr) p.x_copy[idx + static_cast<size_t>(j) * p.ldxo] = x[j];
          }
#pragma unroll
        for (int j = 0; j < kChunk; ++j) {
          const float ss = warp_sum(x[j] * x[j]);
          if (lane == 0) ssp[(grp * 4 + q) * kChunk + j] = ss;
        }
        group_sync(grp);
        if (gtid < kChunk && c0 + gtid < p.M) {  // fixed quadrant order
          const float* s = ssp + grp * 4 * kChunk + gtid;
          p.ss_out[static_cast<size_t>(t_n) * p.ss_stride + c0 + gtid] =
              ((s[0] + s[kChunk]) + s[2 * kChunk]) + s[3 * kChunk];
        }
        group_sync(grp);
      } else {
#pragma unroll
        for (int j = 0; j < kChunk; ++j) {
          const int m = c0 + j;
          const float a = NORM ? v[j] * rstd[m] : v[j];
          if (EPI == kEpiStore) {
            if (m < p.M) p.y[static_cast<size_t>(m) * p.ldy + n0 + row] = __float2half_rn(a);
          } else {  // packed rows 16b .. 16b + 7 are gate rows, 16b + 8 .. 16b + 15 their up rows
            const float up = __shfl_xor_sync(0xffffffffu, a, 8);
            if ((lane & 8) == 0 && m < p.M)
              p.y[static_cast<size_t>(m) * p.ldy + n0 / 2 + (row >> 4) * 8 + (row & 7)] =
                  __float2half_rn(__fdividef(a, 1.f + __expf(-a)) * up);
          }
        }
      }
    };
    const uint32_t lanes = static_cast<uint32_t>(q * 32) << 16;
    // segment of CTA c in a tile it shares: slot 2 c + 1 when the tile starts in its range,
    // else 2 c; [8-token chunk][2][128 rows] groups of 4 tokens
    constexpr size_t kSlot = static_cast<size_t>(BN) * kRows;
    auto cta_of = [&](uint32_t step) { return static_cast<int>(((step + 1) * G - 1) / total); };
    int i = 0;
    for (uint32_t t = s0; t < s1; ++i) {
      const int tile = static_cast<int>(t / KT);
      const uint32_t t_lo = tile * KT, t_hi = t_lo + KT;
      const uint32_t end = min(s1, t_hi);
      const int acc = i & 1;
      const bool whole = t == t_lo && end == t_hi;
      wait(tmem_full + acc, static_cast<uint32_t>((i >> 1) & 1));
      tc_fence_after();
      float* slot = p.part + static_cast<size_t>(2 * blockIdx.x + (t == t_lo ? 1 : 0)) * kSlot;
      for (int c0 = grp * kChunk; c0 < BN && c0 < p.M; c0 += kGroups * kChunk) {
        float v[kChunk];
        __syncwarp();  // tcgen05.ld.sync.aligned needs the whole warp converged
        tmem_ld8(tmem + lanes + static_cast<uint32_t>(acc * BN + c0), v);
        if (whole) {
          finish(tile, c0, v);
        } else {
          float4* d = reinterpret_cast<float4*>(slot) + static_cast<size_t>(c0 / 4) * kRows + row;
          __stcg(d, make_float4(v[0], v[1], v[2], v[3]));
          __stcg(d + kRows, make_float4(v[4], v[5], v[6], v[7]));
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tmem_empty + acc);
      if (!whole) {
        const int first = cta_of(t_lo), n_seg = cta_of(t_hi - 1) - first + 1;
        __threadfence();
        epi_sync();
        if (etid == 0) *last = atomicAdd(p.tile_count + tile, 1) == n_seg - 1;
        epi_sync();
        if (*last) {
          __threadfence();
          if (etid == 0) p.tile_count[tile] = 0;  // zero between launches
          // kRound chunks of the group at a time, kBatch segments of each in flight, added in range order
          for (int c0 = grp * kChunk; c0 < BN && c0 < p.M; c0 += kRound * kGroups * kChunk) {
            float v[kRound][kChunk];
#pragma unroll
            for (int r = 0; r < kRound; ++r)
#pragma unroll
              for (int j = 0; j < kChunk; ++j) v[r][j] = 0.f;
            for (int sg = 0; sg < n_seg; sg += kBatch) {
              float4 w4[kRound][kBatch][2];
#pragma unroll
              for (int r = 0; r < kRound; ++r)
#pragma unroll
                for (int e = 0; e < kBatch; ++e) {
                  const int c = first + sg + e, cr = c0 + r * kGroups * kChunk;
                  const float4* d = reinterpret_cast<const float4*>(p.part + static_cast<size_t>(2 * c + (sg + e == 0 ? 1 : 0)) * kSlot) +
                                    static_cast<size_t>(cr / 4) * kRows + row;
#pragma unroll
                  for (int hh = 0; hh < 2; ++hh)
                    w4[r][e][hh] = sg + e < n_seg && cr < BN && cr < p.M ? __ldcg(d + hh * kRows) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
              for (int r = 0; r < kRound; ++r)
#pragma unroll
                for (int e = 0; e < kBatch; ++e)
#pragma unroll
                  for (int hh = 0; hh < 2; ++hh) {
                    v[r][4 * hh] += w4[r][e][hh].x;
                    v[r][4 * hh + 1] += w4[r][e][hh].y;
                    v[r][4 * hh + 2] += w4[r][e][hh].z;
                    v[r][4 * hh + 3] += w4[r][e][hh].w;
                  }
            }
#pragma unroll 1
            for (int r = 0; r < kRound; ++r) {  // one copy of the code: the chunks move up
              const int cr = c0 + r * kGroups * kChunk;
              if (cr >= BN || cr >= p.M) break;
              finish(tile, cr, v[0]);
#pragma unroll
              for (int e = 1; e < kRound; ++e)
#pragma unroll
                for (int j = 0; j < kChunk; ++j) v[e - 1][j] = v[e][j];
            }
          }
        }
      }
      t = end;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

const void* stream_fn(int bn, int epi, size_t* smem) {
#define FSX_STREAM(BN_)                                                                                           \
  if (bn == BN_) {                                                                                                \
    *smem = smem_bytes<BN_>();                                                                                    \
    if (epi == kEpiStore) return reinterpret_cast<const void*>(&gemm_stream_kernel<BN_, kEpiStore, true>);        \
    if (epi == kEpiSwiglu) return reinterpret_cast<const void*>(&gemm_stream_kernel<BN_, kEpiSwiglu, true>);      \
    if (epi == kEpiResidual) return reinterpret_cast<const void*>(&gemm_stream_kernel<BN_, kEpiResidual, false>); \
  }
  FSX_STREAM(16)
  FSX_STREAM(32)
  FSX_STREAM(64)
  FSX_STREAM(128)
  FSX_STREAM(256)
#undef FSX_STREAM
  return nullptr;
}

int stream_grid(int N, int K, int sm_count) {  // at least 4 steps (16 MMAs) a CTA
  const long long steps = static_cast<long long>(N / kRows) * (K / kTcTileK);
  return static_cast<int>(steps / 4 < 1 ? 1 : (steps / 4 < sm_count ? steps / 4 : sm_count));
}

}  // namespace

cudaError_t gemm_stream_set_attributes() {
  for (int bn : kStreamTiles)
    for (int epi : {kEpiStore, kEpiResidual, kEpiSwiglu}) {
      size_t smem = 0;
      const void* fn = stream_fn(bn, epi, &smem);
      const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

// one 16-token tile up to 16 tokens, then the next power of two
int gemm_stream_tile(int M) {
  for (int i = 0; i < kStreamTileCount; ++i)
    if (M <= kStreamTiles[i]) return i;
  return -1;
}

size_t gemm_stream_part_bytes(int M, int sm_count) {
  const int i = gemm_stream_tile(M);
  return i < 0 ? 0 : static_cast<size_t>(2 * sm_count) * kStreamTiles[i] * kRows * sizeof(float);
}

cudaError_t launch_gemm_stream(const CUtensorMap& map_a, const TcGemmArgs& args, int epi, int sm_count,
                               cudaStream_t stream, bool pdl) {
  const int i = gemm_stream_tile(args.M);
  if (i < 0 || args.M <= 0 || args.N % kRows != 0 || args.K % kTcTileK != 0 || args.part == nullptr ||
      args.tile_count == nullptr)
    return cudaErrorInvalidValue;
  size_t smem = 0;
  const void* fn = stream_fn(kStreamTiles[i], epi, &smem);
  if (fn == nullptr) return cudaErrorInvalidValue;
  CUtensorMap map = map_a;
  TcGemmArgs a = args;
  void* kargs[] = {&map, &a};
  return launch_ex(fn, dim3(static_cast<unsigned>(stream_grid(args.N, args.K, sm_count))), dim3(kThreads), smem, stream,
                   pdl, kargs);
}

}  // namespace fsx
