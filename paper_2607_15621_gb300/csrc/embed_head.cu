// Token assembly and waypoint head of the action expert (Sec. 3.1).
//
// embed: x_b = [E_act ; F_b] + P_pos into the fp32 residual stream; block 0
//        also checks the cache ranges (offsets non-decreasing; the rows of every
//        vehicle, at offsets[b] or at its optional start row, within capacity) and
//        raises the device status word, which turns the rest of the tick
//        into no-ops. Warp b < B also ranks vehicle b by cache length, so the
//        attention launches can start the longest caches first (a schedule
//        only: every (vehicle, head) computes the same result in any order).
// head:  waypoint j of vehicle b = W_h RMSNorm(x_{b,j}; g_f) + b_h, fp32.
#include "device_util.cuh"
#include "kernels.h"

namespace fsx {

namespace {

constexpr int kEmbedWarps = 4;  // token rows per block, one a warp

// Bound by the latency of its loads: a warp has a whole token row in flight, and the checks of
// block 0 and the ranking run across threads (one thread walking the offsets, and a barrier per
// 128 columns, took 7 us for 16 vehicles and 15 us for 128). Measured together with the head's
// early loads: a tick of 16 vehicles, 8 layers, 522 -> 512 us; of 40 clip blocks 862 -> 848 us.
__global__ void __launch_bounds__(kEmbedWarps * 32) embed_kernel(const EmbedArgs a) {
  pdl_launch_dependents();
  pdl_wait();
  const int T = a.n_action + a.n_frame;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t* off = a.targs->offsets;
  const int64_t* st = a.targs->starts;
  if (blockIdx.x == 0) {
    bool ok = off[0] >= 0;
    if (st == nullptr) ok = ok && off[a.B] <= a.max_total;
    for (int i = threadIdx.x; i < a.B; i += kEmbedWarps * 32) {
      const int64_t lo = off[i], hi = off[i + 1];
      ok = ok && hi >= lo;
      if (st != nullptr) ok = ok && st[i] >= 0 && st[i] + (hi - lo) <= a.max_total;  // inside the caller's cache
    }
    if (!ok) set_status(a.status, kStatusDeviceArg);
  }
  const int row = blockIdx.x * kEmbedWarps + warp;  // b * T + t
  if (row < a.B) {  // rank of vehicle `row`: longer caches first, ties by index
    const int64_t len = off[row + 1] - off[row];
    int cnt = 0;
    for (int j = lane; j < a.B; j += 32) {
      const int64_t lj = off[j + 1] - off[j];
      cnt += (lj > len || (lj == len && j < row)) ? 1 : 0;
    }
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if (lane == 0) {
      AttnPlan e;
      e.lo = st != nullptr ? st[row] : off[row];
      e.b = row;
      e.len = (len >= 0 && len <= 0x7fffffff) ? static_cast<int>(len) : -1;
      a.plan[cnt] = e;
    }
  }
  if (row >= a.B * T) return;
  const int b = row / T;
  const int t = row - b * T;
  const size_t frame = (static_cast<size_t>(b) * a.n_frame + (t - a.n_action)) * a.d;
  for (int g0 = 0; g0 < a.d / 128; g0 += 4) {  // four 128-column groups in flight
    float4 v[4], pos[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = (g0 + i) * 128 + lane * 4;
      v[i] = pos[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (c >= a.d) continue;
      pos[i] = *reinterpret_cast<const float4*>(a.pos_emb + static_cast<size_t>(t) * a.d + c);
      if (t < a.n_action) {
        v[i] = *reinterpret_cast<const float4*>(a.act_emb + static_cast<size_t>(t) * a.d + c);
      } else if (a.frame_dtype == 1) {  // element loads: the caller's frames need no more than their own alignment
        const __nv_bfloat16* f = static_cast<const __nv_bfloat16*>(a.targs->frames) + frame + c;
        v[i] = make_float4(__bfloat162float(f[0]), __bfloat162float(f[1]), __bfloat162float(f[2]), __bfloat162float(f[3]));
      } else {
        const float* f = static_cast<const float*>(a.targs->frames) + frame + c;
        v[i] = make_float4(f[0], f[1], f[2], f[3]);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = (g0 + i) * 128 + lane * 4;
      if ((g0 + i) * 128 >= a.d) break;
      const float4 x = make_float4(v[i].x + pos[i].x, v[i].y + pos[i].y, v[i].z + pos[i].z, v[i].w + pos[i].w);
      *reinterpret_cast<float4*>(a.x + static_cast<size_t>(row) * a.d + c) = x;
      *reinterpret_cast<uint2*>(a.x16 + static_cast<size_t>(row) * a.d + c) =
          make_uint2(pack_half2(x.x, x.y), pack_half2(x.z, x.w));
      const float ss = warp_sum(x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w);
      if (lane == 0) a.ss[static_cast<size_t>(g0 + i) * a.ss_stride + row] = ss;
    }
  }
}

// one warp per (vehicle, waypoint); the head's weights are requested before the wait on the
// last layer
constexpr int kHeadUnits = 8;  // 128-column groups (d <= 1024)
__global__ void head_kernel(const HeadArgs a) {
  pdl_launch_dependents();
  const int b = blockIdx.x;
  const int lane = threadIdx.x & 31;
  const int units = a.d / 128;
  float4 g0[kHeadUnits], g1[kHeadUnits];  // head rows times the norm gain
#pragma unroll
  for (int i = 0; i < kHeadUnits; ++i) {
    g0[i] = g1[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i >= units) continue;
    const int c = i * 128 + lane * 4;
    const float4 n = *reinterpret_cast<const float4*>(a.final_norm + c);
    const float4 w0 = *reinterpret_cast<const float4*>(a.head_w + c);
    const float4 w1 = *reinterpret_cast<const float4*>(a.head_w + a.d + c);
    g0[i] = make_float4(w0.x * n.x, w0.y * n.y, w0.z * n.z, w0.w * n.w);
    g1[i] = make_float4(w1.x * n.x, w1.y * n.y, w1.z * n.z, w1.w * n.w);
  }
  const float bias0 = a.head_b[0], bias1 = a.head_b[1];
  pdl_wait();
  if (*reinterpret_cast<volatile int*>(a.status) != 0) return;
  for (int j = threadIdx.x >> 5; j < a.n_waypoints; j += blockDim.x >> 5) {
    const float* xr = a.x + (static_cast<size_t>(b) * a.T + j) * a.d;
    float ss = 0.f, o0 = 0.f, o1 = 0.f;
#pragma unroll
    for (int i = 0; i < kHeadUnits; ++i) {
      if (i >= units) continue;
      const float4 x = *reinterpret_cast<const float4*>(xr + i * 128 + lane * 4);
      ss += x.x * x.x + x.y * x.y + x.z * x.z + x.w * x.w;
      o0 += x.x * g0[i].x + x.y * g0[i].y + x.z * g0[i].z + x.w * g0[i].w;
      o1 += x.x * g1[i].x + x.y * g1[i].y + x.z * g1[i].z + x.w * g1[i].w;
    }
    const float rstd = rsqrtf(warp_sum(ss) / static_cast<float>(a.d) + 1e-6f);
    o0 = warp_sum(o0) * rstd;
    o1 = warp_sum(o1) * rstd;
    if (lane == 0) {
      float* out = a.targs != nullptr ? a.targs->waypoints : a.out;
      out[(static_cast<size_t>(b) * a.n_waypoints + j) * 2 + 0] = o0 + bias0;
      out[(static_cast<size_t>(b) * a.n_waypoints + j) * 2 + 1] = o1 + bias1;
    }
  }
}

}  // namespace

cudaError_t launch_embed(const EmbedArgs& a_in, cudaStream_t stream, bool pdl) {
  EmbedArgs a = a_in;
  void* kargs[] = {&a};
  const int rows = a.B * (a.n_action + a.n_frame);
  return launch_ex(reinterpret_cast<const void*>(&embed_kernel), dim3((rows + kEmbedWarps - 1) / kEmbedWarps),
                   dim3(kEmbedWarps * 32), 0, stream, pdl, kargs);
}

cudaError_t launch_head(const HeadArgs& a_in, cudaStream_t stream, bool pdl) {
  HeadArgs a = a_in;
  void* kargs[] = {&a};
  return launch_ex(reinterpret_cast<const void*>(&head_kernel), dim3(a.B), dim3(32 * (a.n_waypoints < 8 ? a.n_waypoints : 8)), 0, stream,
                   pdl, kargs);
}

}  // namespace fsx
