// Incremental backbone cache append (Sec. 1, Sec. 3.3): the slow system's
// forward of one frame's n_new tokens per vehicle through the frozen causal
// decoder, appending every layer's rotated keys and values to the KV cache
// that the tick reads. Its cost does not depend on the history length.
//
// Per call:  embed -> n_layers x [ RMSNorm+QKV (tcgen05 GEMM) -> rotary
//            embedding, cache-row writes and causal attention over
//            [cached rows ; new rows] -> W_o + residual -> RMSNorm+gate/up+SiLU
//            -> W_d + residual ] -> residual stream out.
// QKV and gate/up run on the few-token tensor-core GEMM (gemm_stream.cu): norm gains
// folded into the packed weights, 1/rms applied in the epilogue from per-128-column
// sums of x^2, the weight stream cut evenly over the SMs. W_o and W_d, whose tiles are
// few, run with K cut over clusters (gemm_res.cu) where gemm_res_plan finds a split (at
// the 7B shape for every token count), else on the streaming GEMM too. The token
// count is n_new * B (4 for one vehicle), so the call streams every backbone
// weight once and is bound by HBM. No kernel of a call waits on other CTAs of its
// grid (those of a cluster are scheduled together).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <thread>
#include <type_traits>
#include <vector>

#include "../../include/fsx.h"
#include "device_util.cuh"
#include "gemm_tc.h"
#include "kernels.h"

namespace fsx {
void set_error_message(const char* msg);
}

namespace {

using fsx::kHeadDim;
constexpr int kMaxNew = 8;         // new tokens per vehicle and call
constexpr int kAttnWarps = 4;
constexpr int kRopePairs = kHeadDim / 2;

fsx_status fail(fsx_status s, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  fsx::set_error_message(buf);
  return s;
}

#define FSX_CUDA(call)                                                                              \
  do {                                                                                              \
    cudaError_t e_ = (call);                                                                        \
    if (e_ != cudaSuccess) return fail(FSX_ERR_CUDA, "%s: %s (%s:%d)", #call, cudaGetErrorString(e_), \
                                       __FILE__, __LINE__);                                         \
  } while (0)

__device__ __forceinline__ int status_set(const int* status) {
  return *reinterpret_cast<const volatile int*>(status);
}

// ---- token rows in: x (fp32 residual stream), its fp16 copy and the per-token
// sums of x^2 over each 128-column group (the RMSNorm input of the QKV GEMM), and the
// cosines and sines of the token's rotary angles, which depend on its position only:
// formed once per call (fp64 angles) and read by every layer. Block 0 also checks the
// offsets and destination rows, its threads sharing the B (B - 1) / 2 pairs of ranges.
struct EmbedArgsA {
  const __nv_bfloat16* x_new;  // [M, d]
  const int64_t* offsets;      // [B + 1]
  const int64_t* dst;          // [B]
  int B, n_new, d;
  long long max_rows;
  const double* inv_freq;      // [64] base^(-2 j / 128)
  float2* rot;                 // [M][64] (cos, sin) of position * inv_freq
  float* x;
  __half* x16;
  float* ss;
  int ss_stride;
  int* status;
};

__global__ void __launch_bounds__(128) append_embed_kernel(const EmbedArgsA a) {
  fsx::pdl_launch_dependents();  // the first GEMM fills its weight ring meanwhile
  const int m = blockIdx.x;
  if (m == 0) {
    const int64_t* off = a.offsets;
    bool ok = off[0] >= 0 && off[a.B] <= a.max_rows;
    for (int b = threadIdx.x; b < a.B; b += blockDim.x) {
      const int64_t lo = a.dst[b], hi = lo + a.n_new;
      ok = ok && off[b + 1] >= off[b] && lo >= 0 && hi <= a.max_rows && (hi <= off[0] || lo >= off[a.B]);
      for (int c = 0; c < b; ++c) {
        const int64_t o = a.dst[c];
        ok = ok && (hi <= o || lo >= o + a.n_new);
      }
    }
    if (!ok) fsx::set_status(a.status, fsx::kStatusDeviceArg);
  }
  if (threadIdx.x < kRopePairs) {
    const int b = m / a.n_new;
    const long long pos = (a.offsets[b + 1] - a.offsets[b]) + (m - b * a.n_new);
    double sd, cd;
    sincos(static_cast<double>(pos) * a.inv_freq[threadIdx.x], &sd, &cd);
    a.rot[static_cast<size_t>(m) * kRopePairs + threadIdx.x] = make_float2(static_cast<float>(cd), static_cast<float>(sd));
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int g = warp; g < a.d / 128; g += 4) {
    const size_t idx = static_cast<size_t>(m) * a.d + g * 128 + lane * 4;
    const uint2 raw = *reinterpret_cast<const uint2*>(a.x_new + idx);
    const float v0 = __uint_as_float(raw.x << 16), v1 = __uint_as_float(raw.x & 0xffff0000u);
    const float v2 = __uint_as_float(raw.y << 16), v3 = __uint_as_float(raw.y & 0xffff0000u);
    *reinterpret_cast<float4*>(a.x + idx) = make_float4(v0, v1, v2, v3);
    *reinterpret_cast<uint2*>(a.x16 + idx) = make_uint2(fsx::pack_half2(v0, v1), fsx::pack_half2(v2, v3));
    const float ss = fsx::warp_sum(v0 * v0 + v1 * v1 + v2 * v2 + v3 * v3);
    if (lane == 0) a.ss[static_cast<size_t>(g) * a.ss_stride + m] = ss;
  }
}

// ---- rotary embedding, cache-row writes and causal attention of the new tokens of
// vehicle b, head h, in one launch. The CTA rotates the new queries and keys itself
// (cos / sin from the embed kernel) and rounds the new keys and values to bf16 in shared
// memory; rank 0 of the cluster writes them to the cache rows dst[b] + i. The keys are the
// vehicle's cached rows (positions 0 .. L_b-1) in 8-key units, then one unit of its new
// rows; new token i sees every cached row and new rows 0 .. i. Everything is fp32.
//
// The keys are few and every row is read once, so the kernel is bound by load latency:
// a warp works on 8-key units, holds one unit's K and V rows (4 KB) in registers and issues
// the next unit's K loads as soon as the scores are formed and its V loads after P V; four
// CTAs share an SM (16 units in flight), and the units go round robin over the 4 warps of
// `cluster` CTAs (as many as keep four CTAs per SM for the batch). No key moves through
// shared memory: 16 lanes share a row in both products (two whole rows an instruction), the
// queries stay in registers, and a transposed reduction over the 16 lanes leaves lane
// 16 h + 4 k + i of the warp with the scores of key 2 k + h for quarter i of the queries. Both
// products use packed fp32 FMAs. The CTAs of a cluster exchange their (max, sum, output) through
// distributed shared memory, each merging its share of the n_new x 128 outputs.
// Measured: from the end of QKV to the last output 7.4 us for one vehicle with 224 rows, about 30 us for
// 16 vehicles with 96-480 rows (issue-bound: 420 instructions per 8 keys); two-layer appends 210 -> 204
// and 322 -> 302 us a call against 16-key units with 4 lanes a row and the queries in shared memory. The
// separate rotary (fp64 pow and sincos per pair and layer) and attention (a lane per key) launches that
// this kernel replaced took 55 and 130 us.
struct AttnArgsA {
  const __half* qkv;   // [M, 3 HD]: q | k | v before the rotation
  int ld;
  int HD;
  const float2* rot;   // [M][64]
  __nv_bfloat16* k_cache;  // this layer's rows
  __nv_bfloat16* v_cache;
  const int64_t* offsets;
  const int64_t* dst;
  int n_new;
  __half* out;  // [M, HD]
  int* status;
};

constexpr int kNewStride = kHeadDim + 8;  // bf16 row stride of the new keys / values in shared memory
constexpr int kMaxSplit = 8;              // CTAs of a cluster
constexpr int kUnit = 8;                  // keys of a warp's unit of work
static_assert(kMaxNew <= kUnit, "the new rows are one unit");

// d += a * b on two packed fp32 values
__device__ __forceinline__ void fma2(uint64_t& d, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}
__device__ __forceinline__ uint64_t bf16x2_to_f32x2(uint32_t v) {
  return pack2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
}
// 2^x on the special-function unit (relative error about 2^-22, as exp2f; -inf -> +0)
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t peer_addr(const void* local, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(fsx::smem_addr(local)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_peer(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

// Two 8-byte accesses in place of one of 16, for a cache that is only 8-byte aligned
template <bool WIDE>
__device__ __forceinline__ uint4 ld_unit(const __nv_bfloat16* p) {
  if (WIDE) return *reinterpret_cast<const uint4*>(p);
  const uint2 a = reinterpret_cast<const uint2*>(p)[0], b = reinterpret_cast<const uint2*>(p)[1];
  return make_uint4(a.x, a.y, b.x, b.y);
}
template <bool WIDE>
__device__ __forceinline__ void st_unit(__nv_bfloat16* p, uint4 v) {
  if (WIDE) {
    *reinterpret_cast<uint4*>(p) = v;
  } else {
    reinterpret_cast<uint2*>(p)[0] = make_uint2(v.x, v.y);
    reinterpret_cast<uint2*>(p)[1] = make_uint2(v.z, v.w);
  }
}

// NQ: query slots (4 or 8) for n_new <= NQ new tokens; VWIDE: the values' cache is 16-byte aligned
// (the keys' always is, the values' needs 8 bytes only)
template <int NQ, bool VWIDE>
__global__ void __launch_bounds__(kAttnWarps * 32, NQ == 4 ? 4 : 2) append_attn_kernel(const AttnArgsA a) {
  __shared__ __align__(16) float qs[NQ][kHeadDim];
  __shared__ __align__(16) __nv_bfloat16 kn[kMaxNew][kNewStride], vn[kMaxNew][kNewStride];
  __shared__ float sm_m[kAttnWarps][NQ], sm_l[kAttnWarps][NQ];
  __shared__ __align__(16) float sm_o[kAttnWarps][NQ][kHeadDim];
  __shared__ float rv_o[NQ * kHeadDim];                       // [split][this rank's share of the outputs]
  __shared__ float rv_m[kMaxSplit][NQ], rv_l[kMaxSplit][NQ];  // every split's running maxima and sums
  constexpr int NH = NQ / 4;  // queries whose scores a lane keeps
  fsx::pdl_launch_dependents();
  fsx::pdl_wait();
  const int S = gridDim.x, rank = blockIdx.x;  // the cluster spans the grid's x extent
  const int h = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nq = a.n_new;
  const long long lo = a.offsets[b], hi = a.offsets[b + 1], d0 = a.dst[b];
  if (status_set(a.status)) return;  // set before this launch or not at all: the same for the whole cluster
  if (S > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");  // this CTA runs
  const int L = static_cast<int>(hi - lo);
  const int n_units = (L + kUnit - 1) / kUnit + 1;  // the last one: the new rows

  // this thread's operands of the rotation, requested ahead of the cache rows
  constexpr int kRot = NQ * kRopePairs / (kAttnWarps * 32);
  float2 cs[kRot];
  __half rq[kRot][2], rk[kRot][2], rv[kRot][2];
#pragma unroll
  for (int t = 0; t < kRot; ++t) {
    const int i = (t * kAttnWarps * 32 + tid) / kRopePairs, jj = tid % kRopePairs;
    if (i < nq) {
      const int m = b * nq + i;
      const __half* q = a.qkv + static_cast<size_t>(m) * a.ld + h * kHeadDim + jj;
      cs[t] = a.rot[static_cast<size_t>(m) * kRopePairs + jj];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        rq[t][e] = q[e * kRopePairs];
        rk[t][e] = q[a.HD + e * kRopePairs];
        rv[t][e] = q[2 * a.HD + e * kRopePairs];
      }
    }
  }

  const int hv = lane >> 4, u = lane & 15;  // key parity, 16-byte unit of a row
  uint4 kraw[4], vraw[4];
  // row loads of unit c: lane's key 2 kk + hv, zeros past the vehicle's rows
  auto unit_keys = [&](int c) { return c == n_units - 1 ? nq : min(kUnit, L - kUnit * c); };
  const size_t lane_off = static_cast<size_t>(hv) * a.HD + u * 8;  // of this lane's first row and dims, in values
  const size_t unit0 = static_cast<size_t>(lo) * a.HD + h * kHeadDim + lane_off;
  const size_t pair = 2 * static_cast<size_t>(a.HD);               // from key 2 kk + hv to key 2 kk + 2 + hv
  auto load_rows = [&](auto wide, int c, const __nv_bfloat16* cache, const __nv_bfloat16* fresh, uint4 (&raw)[4]) {
    constexpr bool kWide = decltype(wide)::value;
    const __nv_bfloat16* row = cache + unit0 + static_cast<size_t>(c) * (kUnit / 2) * pair;
    if (kUnit * c + kUnit <= L) {  // a whole unit of cached rows
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) raw[kk] = ld_unit<kWide>(row + kk * pair);
      return;
    }
    const bool own = c == n_units - 1;
    const int n = unit_keys(c);
    if (own) row = fresh + hv * kNewStride + u * 8;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
      raw[kk] = 2 * kk + hv < n ? ld_unit<kWide>(row + kk * (own ? 2 * static_cast<size_t>(kNewStride) : pair))
                                : make_uint4(0u, 0u, 0u, 0u);
  };
  auto load_k = [&](int c) { load_rows(std::true_type{}, c, a.k_cache, &kn[0][0], kraw); };
  auto load_v = [&](int c) { load_rows(std::integral_constant<bool, VWIDE>{}, c, a.v_cache, &vn[0][0], vraw); };
  const int step = S * kAttnWarps;
  int c = rank * kAttnWarps + warp;
  if (c < n_units - 1) {  // in flight while the new rows are rotated
    load_k(c);
    load_v(c);
  }

  const float scale = 1.4426950408889634f * rsqrtf(static_cast<float>(kHeadDim));  // log2(e) / sqrt(128)
#pragma unroll
  for (int t = 0; t < kRot; ++t) {
    const int i = (t * kAttnWarps * 32 + tid) / kRopePairs, jj = tid % kRopePairs;
    if (i < nq) {
      const float q0 = __half2float(rq[t][0]), q1 = __half2float(rq[t][1]);
      const float k0 = __half2float(rk[t][0]), k1 = __half2float(rk[t][1]);
      qs[i][jj] = (q0 * cs[t].x - q1 * cs[t].y) * scale;
      qs[i][jj + kRopePairs] = (q0 * cs[t].y + q1 * cs[t].x) * scale;
      kn[i][jj] = __float2bfloat16_rn(k0 * cs[t].x - k1 * cs[t].y);
      kn[i][jj + kRopePairs] = __float2bfloat16_rn(k0 * cs[t].y + k1 * cs[t].x);
      vn[i][jj] = __float2bfloat16_rn(__half2float(rv[t][0]));
      vn[i][jj + kRopePairs] = __float2bfloat16_rn(__half2float(rv[t][1]));
    } else {
      qs[i][jj] = qs[i][jj + kRopePairs] = 0.f;
    }
  }
  __syncthreads();
  if (rank == 0)  // the new cache rows, 16 bytes a thread
    for (int t = tid; t < nq * (kHeadDim / 8); t += kAttnWarps * 32) {
      const int i = t / (kHeadDim / 8), uu = t - i * (kHeadDim / 8);
      const size_t o = static_cast<size_t>(d0 + i) * a.HD + h * kHeadDim + uu * 8;
      *reinterpret_cast<uint4*>(a.k_cache + o) = *reinterpret_cast<const uint4*>(&kn[i][uu * 8]);
      st_unit<VWIDE>(a.v_cache + o, *reinterpret_cast<const uint4*>(&vn[i][uu * 8]));
    }

  uint64_t q2[NQ][4];  // dims 8 u .. 8 u + 7 of every query
#pragma unroll
  for (int qi = 0; qi < NQ; ++qi) {
    const ulonglong2 qa = *reinterpret_cast<const ulonglong2*>(&qs[qi][8 * u]);
    const ulonglong2 qb = *reinterpret_cast<const ulonglong2*>(&qs[qi][8 * u + 4]);
    q2[qi][0] = qa.x;
    q2[qi][1] = qa.y;
    q2[qi][2] = qb.x;
    q2[qi][3] = qb.y;
  }
  const int q_lane = (u & 3) * NH;  // this lane's queries q_lane .. q_lane + NH - 1
  float m_run[NH], l_run[NH];       // l_run: this lane's keys only
  uint64_t o[NQ][4];                // this half warp's keys, value dims 8 u .. 8 u + 7
#pragma unroll
  for (int qq = 0; qq < NH; ++qq) {
    m_run[qq] = -INFINITY;
    l_run[qq] = 0.f;
  }
#pragma unroll
  for (int qi = 0; qi < NQ; ++qi)
#pragma unroll
    for (int e = 0; e < 4; ++e) o[qi][e] = 0ull;
  if (c == n_units - 1) {  // a warp whose first unit is the new rows
    load_k(c);
    load_v(c);
  }
#pragma unroll 1
  for (; c < n_units; c += step) {
    const bool own = c == n_units - 1;
    const int n = unit_keys(c);
    const int next = c + step;
    // this lane's 8 dims of every score, then the transposed sum over the row's 16 lanes: key bits
    // (lane bits 3, 2), then query quarter (lane bits 1, 0)
    const bool up8 = (u & 8) != 0, up4 = (u & 4) != 0, up2 = (u & 2) != 0, up1 = (u & 1) != 0;
    float r4[2][NQ];  // [key bit 0], key bit 1 by lane bit 3
#pragma unroll
    for (int k0 = 0; k0 < 2; ++k0) {
      uint64_t kv[2][4];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const uint4 w = kraw[k0 + 2 * e];
        kv[e][0] = bf16x2_to_f32x2(w.x);
        kv[e][1] = bf16x2_to_f32x2(w.y);
        kv[e][2] = bf16x2_to_f32x2(w.z);
        kv[e][3] = bf16x2_to_f32x2(w.w);
      }
#pragma unroll
      for (int qi = 0; qi < NQ; ++qi) {
        float sum[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          uint64_t acc = mul2(kv[e][0], q2[qi][0]);
          fma2(acc, kv[e][1], q2[qi][1]);
          fma2(acc, kv[e][2], q2[qi][2]);
          fma2(acc, kv[e][3], q2[qi][3]);
          const float2 f = unpack2(acc);
          sum[e] = f.x + f.y;
        }
        r4[k0][qi] = (up8 ? sum[1] : sum[0]) + __shfl_xor_sync(0xffffffffu, up8 ? sum[0] : sum[1], 8);
      }
    }
    if (next < n_units) load_k(next);
    float r2[NQ], r1[NQ / 2], p[NH];
#pragma unroll
    for (int qi = 0; qi < NQ; ++qi)
      r2[qi] = (up4 ? r4[1][qi] : r4[0][qi]) + __shfl_xor_sync(0xffffffffu, up4 ? r4[0][qi] : r4[1][qi], 4);
#pragma unroll
    for (int qi = 0; qi < NQ / 2; ++qi)
      r1[qi] = (up2 ? r2[NQ / 2 + qi] : r2[qi]) + __shfl_xor_sync(0xffffffffu, up2 ? r2[qi] : r2[NQ / 2 + qi], 2);
#pragma unroll
    for (int qq = 0; qq < NH; ++qq)
      p[qq] = (up1 ? r1[NH + qq] : r1[qq]) + __shfl_xor_sync(0xffffffffu, up1 ? r1[qq] : r1[NH + qq], 1);
    const int key = 2 * (u >> 2) + hv;
    float alpha[NH];
    bool moved = false;
#pragma unroll
    for (int qq = 0; qq < NH; ++qq) {
      // visible: a real key that is a cached row or a new row <= the query's
      const int qi = q_lane + qq;
      const bool vis = qi < nq && key < n && (!own || key <= qi);
      const float sv = vis ? p[qq] : -INFINITY;
      float mx = sv;  // over the 8 keys: the lanes with this lane's query quarter
#pragma unroll
      for (int sh = 16; sh > 2; sh >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, sh));
      const float m_new = fmaxf(m_run[qq], mx);
      const bool none = m_new == -INFINITY;  // an unused query slot
      alpha[qq] = none ? 1.f : ex2_approx(m_run[qq] - m_new);
      p[qq] = none ? 0.f : ex2_approx(sv - m_new);  // 0 where not visible
      l_run[qq] = l_run[qq] * alpha[qq] + p[qq];
      moved = moved || alpha[qq] != 1.f;
      m_run[qq] = m_new;
    }
    if (__any_sync(0xffffffffu, moved)) {
#pragma unroll
      for (int qi = 0; qi < NQ; ++qi) {
        const float av = __shfl_sync(0xffffffffu, alpha[qi % NH], qi / NH);
        const uint64_t al = pack2(av, av);
#pragma unroll
        for (int e = 0; e < 4; ++e) o[qi][e] = mul2(o[qi][e], al);
      }
    }
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      const uint64_t v0 = bf16x2_to_f32x2(vraw[kk].x), v1 = bf16x2_to_f32x2(vraw[kk].y);
      const uint64_t v2 = bf16x2_to_f32x2(vraw[kk].z), v3 = bf16x2_to_f32x2(vraw[kk].w);
#pragma unroll
      for (int qi = 0; qi < NQ; ++qi) {  // key 2 kk + hv: its probabilities are in this half warp
        const float pk = __shfl_sync(0xffffffffu, p[qi % NH], (lane & 16) | (kk << 2) | (qi / NH));
        const uint64_t pp = pack2(pk, pk);
        fma2(o[qi][0], pp, v0);
        fma2(o[qi][1], pp, v1);
        fma2(o[qi][2], pp, v2);
        fma2(o[qi][3], pp, v3);
      }
    }
    if (next < n_units) load_v(next);
  }
#pragma unroll
  for (int qi = 0; qi < NQ; ++qi) {
    float ov[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 f = unpack2(o[qi][e]);
      ov[2 * e] = f.x + __shfl_xor_sync(0xffffffffu, f.x, 16);
      ov[2 * e + 1] = f.y + __shfl_xor_sync(0xffffffffu, f.y, 16);
    }
    *reinterpret_cast<float4*>(&sm_o[warp][qi][u * 8 + hv * 4]) =
        hv == 0 ? make_float4(ov[0], ov[1], ov[2], ov[3]) : make_float4(ov[4], ov[5], ov[6], ov[7]);
  }
#pragma unroll
  for (int qq = 0; qq < NH; ++qq) {
    float l = l_run[qq];
#pragma unroll
    for (int sh = 16; sh > 2; sh >>= 1) l += __shfl_xor_sync(0xffffffffu, l, sh);
    if (lane < 4) {
      sm_m[warp][q_lane + qq] = m_run[qq];
      sm_l[warp][q_lane + qq] = l;
    }
  }
  __syncthreads();
  // the CTA's four warps, then (S > 1) the cluster's CTAs: output element e = query * 128 + dim
  // belongs to rank e / (n_new * 128 / S)
  if (S > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // every peer runs
  const int share = nq * kHeadDim / S;
  for (int e = tid; e < nq * kHeadDim; e += kAttnWarps * 32) {
    const int qi = e / kHeadDim, dd = e - qi * kHeadDim;
    float mm = -INFINITY;
#pragma unroll
    for (int w = 0; w < kAttnWarps; ++w) mm = fmaxf(mm, sm_m[w][qi]);
    float num = 0.f, den = 0.f;
#pragma unroll
    for (int w = 0; w < kAttnWarps; ++w) {
      const float f = sm_m[w][qi] == -INFINITY ? 0.f : exp2f(sm_m[w][qi] - mm);
      num += f * sm_o[w][qi][dd];
      den += f * sm_l[w][qi];
    }
    if (S == 1) {
      a.out[static_cast<size_t>(b * nq + qi) * a.HD + h * kHeadDim + dd] = __float2half_rn(den > 0.f ? num / den : 0.f);
      continue;
    }
    const int owner = e / share;
    st_peer(peer_addr(&rv_o[rank * share + (e - owner * share)], owner), num);
    if (dd < S) {  // this split's maximum and sum of the query, to every rank
      st_peer(peer_addr(&rv_m[rank][qi], dd), mm);
      st_peer(peer_addr(&rv_l[rank][qi], dd), den);
    }
  }
  if (S == 1) return;
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  for (int t = tid; t < share; t += kAttnWarps * 32) {
    const int e = rank * share + t;
    const int qi = e / kHeadDim, dd = e - qi * kHeadDim;
    float mm = -INFINITY;
    for (int r = 0; r < S; ++r) mm = fmaxf(mm, rv_m[r][qi]);
    float num = 0.f, den = 0.f;
    for (int r = 0; r < S; ++r) {  // a split without keys has the maximum -inf
      const float f = rv_m[r][qi] == -INFINITY ? 0.f : exp2f(rv_m[r][qi] - mm);
      num += f * rv_o[r * share + t];
      den += f * rv_l[r][qi];
    }
    a.out[static_cast<size_t>(b * nq + qi) * a.HD + h * kHeadDim + dd] = __float2half_rn(den > 0.f ? num / den : 0.f);
  }
}

const void* append_attn_fn(int n_new, bool v_wide) {
  if (n_new <= 4)
    return v_wide ? reinterpret_cast<const void*>(&append_attn_kernel<4, true>)
                  : reinterpret_cast<const void*>(&append_attn_kernel<4, false>);
  return v_wide ? reinterpret_cast<const void*>(&append_attn_kernel<kMaxNew, true>)
                : reinterpret_cast<const void*>(&append_attn_kernel<kMaxNew, false>);
}

// CTAs per (vehicle, head): the largest power of two up to 8 that keeps the batch's CTAs
// within two waves of the four that share an SM (16 vehicles: 325 us a call with one CTA each, the
// longest history last to finish, 312 us with two)
int append_attn_splits(int B, int n_heads, int sm_count) {
  int s = kMaxSplit;
  while (s > 1 && static_cast<long long>(B) * n_heads * s > 8ll * sm_count) s >>= 1;
  return s;
}

}  // namespace

struct fsx_append_s {
  fsx_append_config cfg{};
  int device = 0;
  int sm_count = 0;
  int HD = 0;
  void* w_arena = nullptr;
  long long weight_bytes = 0;
  std::vector<const unsigned char*> w_qkv, w_o, w_gu, w_dn;
  CUtensorMap map_x16[fsx::kStreamTileCount], map_o[fsx::kStreamTileCount], map_h[fsx::kStreamTileCount];
  CUtensorMap map_o_res[fsx::kResTileCount], map_h_res[fsx::kResTileCount];
  float* x = nullptr;
  __half* x16 = nullptr;
  float* ss = nullptr;
  int ss_stride = 0;
  __half* qkv = nullptr;
  __half* o = nullptr;
  __half* hbuf = nullptr;
  double* inv_freq = nullptr;  // [64] rotary frequencies
  float2* rot = nullptr;       // [n_new * max_batch][64] (cos, sin) of the current call's positions
  float* gemm_part = nullptr;
  int* tile_count = nullptr;
  int* status = nullptr;
};

namespace {

void free_append(fsx_append_s* h) {
  if (!h) return;
  cudaSetDevice(h->device);
  cudaDeviceSynchronize();
  void* bufs[] = {h->w_arena, h->x, h->x16, h->ss, h->qkv, h->o, h->hbuf,
                  h->inv_freq, h->rot, h->gemm_part, h->tile_count, h->status};
  for (void* p : bufs)
    if (p) cudaFree(p);
  delete h;
}

fsx_status check_append_config(const fsx_append_config* c) {
  if (!c) return fail(FSX_ERR_INVALID_ARG, "config is NULL");
  if (c->n_layers <= 0 || c->d_model <= 0 || c->n_heads <= 0 || c->head_dim <= 0 || c->d_ff <= 0 ||
      c->n_new <= 0 || c->max_batch <= 0 || c->max_cache_rows < 0)
    return fail(FSX_ERR_INVALID_ARG, "config fields must be positive (max_cache_rows >= 0)");
  if (!(c->rope_base > 1.f)) return fail(FSX_ERR_INVALID_ARG, "rope_base must be > 1");
  if (c->head_dim != kHeadDim) return fail(FSX_ERR_UNSUPPORTED, "head_dim must be 128");
  if (c->d_model % 128 != 0) return fail(FSX_ERR_UNSUPPORTED, "d_model must be a multiple of 128");
  if (c->d_ff % 64 != 0) return fail(FSX_ERR_UNSUPPORTED, "d_ff must be a multiple of 64");
  if (c->n_new > kMaxNew) return fail(FSX_ERR_UNSUPPORTED, "n_new must be <= %d", kMaxNew);
  if (static_cast<long long>(c->n_new) * c->max_batch > 256)
    return fail(FSX_ERR_UNSUPPORTED, "n_new * max_batch must be <= 256");
  if (c->n_heads > 4096) return fail(FSX_ERR_UNSUPPORTED, "n_heads too large");
  return FSX_OK;
}

}  // namespace

extern "C" {

fsx_status fsx_append_create(const fsx_append_config* cfg, const fsx_append_weights* w, int device,
                             fsx_append_handle* out) {
  fsx::set_error_message("");
  if (!out) return fail(FSX_ERR_INVALID_ARG, "out handle pointer is NULL");
  *out = nullptr;
  fsx_status st = check_append_config(cfg);
  if (st != FSX_OK) return st;
  if (!w || !w->attn_norm || !w->wq || !w->wk || !w->wv || !w->wo || !w->mlp_norm || !w->w_gate || !w->w_up ||
      !w->w_down)
    return fail(FSX_ERR_INVALID_ARG, "a weight pointer is NULL");
  if (device < 0) return fail(FSX_ERR_INVALID_ARG, "device must be >= 0");
  int n_dev = 0;
  if (cudaGetDeviceCount(&n_dev) != cudaSuccess || n_dev == 0) return fail(FSX_ERR_CUDA, "no CUDA device available");
  if (device >= n_dev) return fail(FSX_ERR_INVALID_ARG, "device %d >= device count %d", device, n_dev);

  fsx_append_s* h = new fsx_append_s();
  h->cfg = *cfg;
  h->device = device;
  h->HD = cfg->n_heads * cfg->head_dim;
  const int L = cfg->n_layers, d = cfg->d_model, HD = h->HD, F = cfg->d_ff;
  auto bail = [&](fsx_status s) {
    free_append(h);
    return s;
  };
#define FSX_CUDA_H(call)                                                                                  \
  do {                                                                                                    \
    cudaError_t e_ = (call);                                                                              \
    if (e_ != cudaSuccess)                                                                                \
      return bail(fail(e_ == cudaErrorMemoryAllocation ? FSX_ERR_OOM : FSX_ERR_CUDA, "%s: %s", #call,    \
                       cudaGetErrorString(e_)));                                                          \
  } while (0)

  FSX_CUDA_H(cudaSetDevice(device));
  FSX_CUDA_H(cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, device));
  FSX_CUDA_H(fsx::gemm_stream_set_attributes());
  FSX_CUDA_H(fsx::gemm_res_set_attributes());

  // ---- weight tiles per layer [QKV | W_o | gate/up | W_d], 128-row x 64-K swizzled
  // images; RMSNorm gains folded into the K columns of QKV and gate/up; gate/up rows
  // interleaved so one 128-row tile holds gate rows 8j..8j+7 next to their up rows
  const size_t tile = fsx::kTcTileBytes;
  const size_t t_qkv = static_cast<size_t>(3 * HD / 128) * (d / 64), t_o = static_cast<size_t>(d / 128) * (HD / 64);
  const size_t t_gu = static_cast<size_t>(2 * F / 128) * (d / 64), t_dn = static_cast<size_t>(d / 128) * (F / 64);
  const size_t per_layer = (t_qkv + t_o + t_gu + t_dn) * tile;
  h->weight_bytes = static_cast<long long>(per_layer) * L;
  FSX_CUDA_H(cudaMalloc(&h->w_arena, per_layer * L));
  {
    std::vector<unsigned char> host(per_layer);
    const size_t hd_d = static_cast<size_t>(HD) * d;
    const int n_threads = std::max(1, std::min<int>(16, static_cast<int>(std::thread::hardware_concurrency())));
    // rows(r) -> source row r of the (row-permuted) matrix, N rows of K columns, optional per-K gain;
    // the n-tiles are spread over the threads
    auto pack_matrix = [&](auto rows, int N, int K, const float* gain, unsigned char* dst) {
      std::vector<std::thread> pool;
      for (int t = 0; t < n_threads; ++t)
        pool.emplace_back([&, t]() {
          const float* rp[128];
          for (int nt = t; nt < N / 128; nt += n_threads)
            for (int kt = 0; kt < K / 64; ++kt) {
              for (int r = 0; r < 128; ++r) rp[r] = rows(nt * 128 + r);
              fsx::pack_tc_tile(rp, gain, kt * 64,
                                reinterpret_cast<__half*>(dst + (static_cast<size_t>(nt) * (K / 64) + kt) * tile));
            }
        });
      for (auto& th : pool) th.join();
    };
    for (int l = 0; l < L; ++l) {
      unsigned char* base = host.data();
      const float* wq = w->wq + hd_d * l;
      const float* wk = w->wk + hd_d * l;
      const float* wv = w->wv + hd_d * l;
      pack_matrix(
          [&](int r) -> const float* {
            if (r < HD) return wq + static_cast<size_t>(r) * d;
            if (r < 2 * HD) return wk + static_cast<size_t>(r - HD) * d;
            return wv + static_cast<size_t>(r - 2 * HD) * d;
          },
          3 * HD, d, w->attn_norm + static_cast<size_t>(l) * d, base);
      const float* wo = w->wo + hd_d * l;
      pack_matrix([&](int r) -> const float* { return wo + static_cast<size_t>(r) * HD; }, d, HD, nullptr,
                  base + t_qkv * tile);
      const float* wg = w->w_gate + static_cast<size_t>(F) * d * l;
      const float* wu = w->w_up + static_cast<size_t>(F) * d * l;
      pack_matrix(
          [&](int q) -> const float* {
            const int blk = q >> 4, r = q & 15;
            return r < 8 ? wg + static_cast<size_t>(blk * 8 + r) * d : wu + static_cast<size_t>(blk * 8 + r - 8) * d;
          },
          2 * F, d, w->mlp_norm + static_cast<size_t>(l) * d, base + (t_qkv + t_o) * tile);
      const float* wd = w->w_down + static_cast<size_t>(d) * F * l;
      pack_matrix([&](int r) -> const float* { return wd + static_cast<size_t>(r) * F; }, d, F, nullptr,
                  base + (t_qkv + t_o + t_gu) * tile);
      FSX_CUDA_H(cudaMemcpy(static_cast<unsigned char*>(h->w_arena) + per_layer * l, host.data(), per_layer,
                            cudaMemcpyHostToDevice));
    }
  }
  for (int l = 0; l < L; ++l) {
    const unsigned char* base = static_cast<const unsigned char*>(h->w_arena) + per_layer * l;
    h->w_qkv.push_back(base);
    h->w_o.push_back(base + t_qkv * tile);
    h->w_gu.push_back(base + (t_qkv + t_o) * tile);
    h->w_dn.push_back(base + (t_qkv + t_o + t_gu) * tile);
  }

  // ---- workspace: token rows padded to whole 256-token tiles
  const size_t m_pad = (static_cast<size_t>(cfg->n_new) * cfg->max_batch + 255) / 256 * 256;
  FSX_CUDA_H(cudaMalloc(&h->x, m_pad * d * sizeof(float)));
  FSX_CUDA_H(cudaMalloc(&h->x16, m_pad * d * sizeof(__half)));
  h->ss_stride = static_cast<int>(m_pad);
  FSX_CUDA_H(cudaMalloc(&h->ss, static_cast<size_t>(d / 128) * m_pad * sizeof(float)));
  FSX_CUDA_H(cudaMalloc(&h->qkv, m_pad * 3 * HD * sizeof(__half)));
  FSX_CUDA_H(cudaMalloc(&h->o, m_pad * HD * sizeof(__half)));
  FSX_CUDA_H(cudaMalloc(&h->hbuf, m_pad * F * sizeof(__half)));
  FSX_CUDA_H(cudaMemset(h->x, 0, m_pad * d * sizeof(float)));
  FSX_CUDA_H(cudaMemset(h->x16, 0, m_pad * d * sizeof(__half)));
  FSX_CUDA_H(cudaMemset(h->ss, 0, static_cast<size_t>(d / 128) * m_pad * sizeof(float)));
  FSX_CUDA_H(cudaMemset(h->qkv, 0, m_pad * 3 * HD * sizeof(__half)));
  FSX_CUDA_H(cudaMemset(h->o, 0, m_pad * HD * sizeof(__half)));
  FSX_CUDA_H(cudaMemset(h->hbuf, 0, m_pad * F * sizeof(__half)));
  {
    for (int i = 0; i < fsx::kStreamTileCount; ++i)
      if (!fsx::encode_act_map(&h->map_x16[i], h->x16, m_pad, d, fsx::kStreamTiles[i]) ||
          !fsx::encode_act_map(&h->map_o[i], h->o, m_pad, HD, fsx::kStreamTiles[i]) ||
          !fsx::encode_act_map(&h->map_h[i], h->hbuf, m_pad, F, fsx::kStreamTiles[i]))
        return bail(fail(FSX_ERR_CUDA, "tensor map encoding of the activation buffers failed"));
    for (int i = 0; i < fsx::kResTileCount; ++i)
      if (!fsx::encode_act_map(&h->map_o_res[i], h->o, m_pad, HD, fsx::kResTiles[i]) ||
          !fsx::encode_act_map(&h->map_h_res[i], h->hbuf, m_pad, F, fsx::kResTiles[i]))
        return bail(fail(FSX_ERR_CUDA, "tensor map encoding of the activation buffers failed"));
  }
  {
    double inv_freq[kRopePairs];
    for (int j = 0; j < kRopePairs; ++j) inv_freq[j] = std::pow(static_cast<double>(cfg->rope_base), -2.0 * j / kHeadDim);
    FSX_CUDA_H(cudaMalloc(&h->inv_freq, sizeof(inv_freq)));
    FSX_CUDA_H(cudaMemcpy(h->inv_freq, inv_freq, sizeof(inv_freq), cudaMemcpyHostToDevice));
  }
  FSX_CUDA_H(cudaMalloc(&h->rot, static_cast<size_t>(cfg->n_new) * cfg->max_batch * kRopePairs * sizeof(float2)));
  FSX_CUDA_H(cudaMalloc(&h->gemm_part, fsx::gemm_stream_part_bytes(cfg->n_new * cfg->max_batch, h->sm_count)));
  const size_t n_tiles = static_cast<size_t>(std::max({3 * HD, 2 * F, d})) / 128;  // of the widest matrix
  FSX_CUDA_H(cudaMalloc(&h->tile_count, sizeof(int) * n_tiles));
  FSX_CUDA_H(cudaMemset(h->tile_count, 0, sizeof(int) * n_tiles));
  FSX_CUDA_H(cudaMalloc(&h->status, sizeof(int)));
  FSX_CUDA_H(cudaMemset(h->status, 0, sizeof(int)));
  FSX_CUDA_H(cudaDeviceSynchronize());
#undef FSX_CUDA_H
  *out = h;
  return FSX_OK;
}

fsx_status fsx_append_set_concurrent(fsx_append_handle h, int enable) {
  if (!h) return fail(FSX_ERR_INVALID_ARG, "handle is NULL");
  (void)enable;  // no append kernel waits on other CTAs under either setting
  return FSX_OK;
}

fsx_status fsx_append(fsx_append_handle h, void* const* k_cache, void* const* v_cache, const int64_t* d_offsets,
                      const int64_t* d_dst_rows, int B, const void* d_x_new, float* d_hidden, void* stream) {
  if (!h) return fail(FSX_ERR_INVALID_ARG, "handle is NULL");
  const fsx_append_config& c = h->cfg;
  if (!k_cache || !v_cache || !d_offsets || !d_dst_rows || !d_x_new || !d_hidden)
    return fail(FSX_ERR_INVALID_ARG, "a pointer argument is NULL");
  if (B < 1 || B > c.max_batch) return fail(FSX_ERR_INVALID_ARG, "B=%d outside 1..max_batch=%d", B, c.max_batch);
  for (int l = 0; l < c.n_layers; ++l) {
    if (!k_cache[l] || !v_cache[l]) return fail(FSX_ERR_INVALID_ARG, "cache layer %d pointer is NULL", l);
    if (reinterpret_cast<uintptr_t>(k_cache[l]) % 16 != 0 || reinterpret_cast<uintptr_t>(v_cache[l]) % 8 != 0)
      return fail(FSX_ERR_INVALID_ARG, "cache layer %d pointer is not aligned (keys 16 bytes, values 8)", l);
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  FSX_CUDA(cudaSetDevice(h->device));
  const int d = c.d_model, HD = h->HD, F = c.d_ff;
  const int M = B * c.n_new;
  const int bn_i = fsx::gemm_stream_tile(M);  // M <= 256: checked at create

  EmbedArgsA ea{};
  ea.x_new = static_cast<const __nv_bfloat16*>(d_x_new);
  ea.offsets = d_offsets;
  ea.dst = d_dst_rows;
  ea.B = B;
  ea.n_new = c.n_new;
  ea.d = d;
  ea.max_rows = c.max_cache_rows;
  ea.inv_freq = h->inv_freq;
  ea.rot = h->rot;
  ea.x = h->x;
  ea.x16 = h->x16;
  ea.ss = h->ss;
  ea.ss_stride = h->ss_stride;
  ea.status = h->status;
  append_embed_kernel<<<M, 128, 0, st>>>(ea);
  FSX_CUDA(cudaGetLastError());

  // The residual projections' tiles are few (d / 128): K is cut over clusters where those fit the
  // chip (gemm_res.cu), else the weight stream is cut evenly like the others'.
  const fsx::ResPlan plan_o = fsx::gemm_res_plan(M, d, HD), plan_d = fsx::gemm_res_plan(M, d, F);
  auto launch_residual = [&](const CUtensorMap* maps, const CUtensorMap* maps_res, const fsx::ResPlan& plan,
                             const fsx::TcGemmArgs& g) {
    if (plan.splits > 1) return fsx::launch_gemm_res(maps_res[plan.tile], g, plan, st, true);
    return fsx::launch_gemm_stream(maps[bn_i], g, fsx::kEpiResidual, h->sm_count, st, true);
  };
  const int attn_splits = append_attn_splits(B, c.n_heads, h->sm_count);
  for (int l = 0; l < c.n_layers; ++l) {
    fsx::TcGemmArgs g{};
    g.M = M;
    g.status = h->status;
    g.w = h->w_qkv[l];
    g.N = 3 * HD;
    g.K = d;
    g.y = h->qkv;
    g.ldy = 3 * HD;
    g.ss_in = h->ss;
    g.n_ss = d / 128;
    g.ss_stride = h->ss_stride;
    g.part = h->gemm_part;
    g.tile_count = h->tile_count;
    FSX_CUDA(fsx::launch_gemm_stream(h->map_x16[bn_i], g, fsx::kEpiStore, h->sm_count, st, true));

    AttnArgsA aa{};
    aa.qkv = h->qkv;
    aa.ld = 3 * HD;
    aa.HD = HD;
    aa.rot = h->rot;
    aa.k_cache = static_cast<__nv_bfloat16*>(k_cache[l]);
    aa.v_cache = static_cast<__nv_bfloat16*>(v_cache[l]);
    aa.offsets = d_offsets;
    aa.dst = d_dst_rows;
    aa.n_new = c.n_new;
    aa.out = h->o;
    aa.status = h->status;
    void* attn_args[] = {&aa};
    FSX_CUDA(fsx::launch_ex(append_attn_fn(c.n_new, reinterpret_cast<uintptr_t>(v_cache[l]) % 16 == 0),
                            dim3(attn_splits, c.n_heads, B), dim3(kAttnWarps * 32), 0, st, true, attn_args, 1,
                            attn_splits));

    fsx::TcGemmArgs go{};
    go.M = M;
    go.status = h->status;
    go.w = h->w_o[l];
    go.N = d;
    go.K = HD;
    go.xo = h->x;
    go.xo16 = h->x16;
    go.ldxo = d;
    go.ss_out = h->ss;
    go.ss_stride = h->ss_stride;
    go.part = h->gemm_part;
    go.tile_count = h->tile_count;
    FSX_CUDA(launch_residual(h->map_o, h->map_o_res, plan_o, go));

    fsx::TcGemmArgs gg{};
    gg.M = M;
    gg.status = h->status;
    gg.w = h->w_gu[l];
    gg.N = 2 * F;
    gg.K = d;
    gg.y = h->hbuf;
    gg.ldy = F;
    gg.ss_in = h->ss;
    gg.n_ss = d / 128;
    gg.ss_stride = h->ss_stride;
    gg.part = h->gemm_part;
    gg.tile_count = h->tile_count;
    FSX_CUDA(fsx::launch_gemm_stream(h->map_x16[bn_i], gg, fsx::kEpiSwiglu, h->sm_count, st, true));

    fsx::TcGemmArgs gd{};
    gd.M = M;
    gd.status = h->status;
    gd.w = h->w_dn[l];
    gd.N = d;
    gd.K = F;
    gd.xo = h->x;
    gd.xo16 = h->x16;
    gd.ldxo = d;
    gd.ss_out = h->ss;
    gd.ss_stride = h->ss_stride;
    gd.part = h->gemm_part;
    gd.tile_count = h->tile_count;
    gd.x_copy = l == c.n_layers - 1 ? d_hidden : nullptr;  // the residual stream after the last layer
    FSX_CUDA(launch_residual(h->map_h, h->map_h_res, plan_d, gd));
  }
  return FSX_OK;
}

fsx_status fsx_append_get_status(fsx_append_handle h, void* stream) {
  if (!h) return fail(FSX_ERR_INVALID_ARG, "handle is NULL");
  FSX_CUDA(cudaSetDevice(h->device));
  FSX_CUDA(cudaStreamSynchronize(static_cast<cudaStream_t>(stream)));
  int v = 0;
  FSX_CUDA(cudaMemcpy(&v, h->status, sizeof(int), cudaMemcpyDeviceToHost));
  FSX_CUDA(cudaMemset(h->status, 0, sizeof(int)));
  return static_cast<fsx_status>(v);
}

long long fsx_append_weight_bytes(fsx_append_handle h) { return h ? h->weight_bytes : 0; }

void fsx_append_destroy(fsx_append_handle h) { free_append(h); }

}  // extern "C"
