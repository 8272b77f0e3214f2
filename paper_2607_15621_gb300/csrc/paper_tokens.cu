// The paper's own ten-token layout of the action expert (Sec. 3.1): per vehicle and
// frame, one state token -- a two-layer MLP of the 16 ego-state values (previous five
// waypoints, control triplet, speed, target point) -- the frame's four visual tokens
// and five learned waypoint queries; after the shared layer stack a two-layer head
// decodes each query token into one (x, y) waypoint.
//
// The layer stack is the tick of fsx.cu unchanged: its own keys are attended
// bidirectionally with learned positions and no rotary phase, so the order in which
// the ten tokens are held does not change the result once the position table follows
// them. The handle therefore holds the queries as its five learned action tokens
// (rows 0-4, read by the head) and the state token plus the four visual tokens as its
// five frame rows (rows 5-9), with the paper's position rows permuted to that order.
// Per tick: state_tokens_kernel writes [state token ; visual tokens] of every
// vehicle into a handle-owned fp32 frame buffer, the tick runs on it, and
// head2_kernel (in place of the single-layer head) decodes the queries.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <vector>

#include "../../include/fsx.h"
#include "device_util.cuh"
#include "kernels.h"

namespace fsx {

void set_error_message(const char* msg);
// hooks into the tick handle (fsx.cu)
fsx_status paper_attach(fsx_handle h, float* d_params, const float* d_head, float* d_frames, const float* d_state_w,
                        int visual_dtype);
float* paper_frames(fsx_handle h);
const float* paper_state_weights(fsx_handle h);
cudaError_t paper_order_after_last_tick(fsx_handle h, cudaStream_t st);
int paper_device(fsx_handle h);
int paper_sm_count(fsx_handle h);
int paper_max_batch(fsx_handle h);
int paper_d(fsx_handle h);
int paper_visual_dtype(fsx_handle h);

namespace {

constexpr int kStateDim = 16;
constexpr int kVisual = 4;
constexpr int kQueries = 5;

__device__ __forceinline__ float silu(float z) { return z / (1.f + expf(-z)); }

// Both kernels are matrix-vector products over 1 MB of fp32 weights (d = 512) that no single SM
// can read in time (one CTA per vehicle took 17-20 us for the state token, one per waypoint 40 us
// for the head), so the rows of a matrix are spread over CTAs, and a warp requests its first
// rows' weights before it needs the vector they multiply: the calls are bound by a few load
// latencies. Measured: a tick of one vehicle, 8 layers and 224 rows, 240 -> 196 us.
constexpr int kMlpThreads = 512;
constexpr int kMlpWarps = kMlpThreads / 32;
constexpr int kMaxUnits = 8;      // 128-wide K units of a row (d <= 1024)
constexpr int kHeadCluster = 8;   // CTAs that share the rows of W_h1 for one vehicle

// two rows of a row-major [*, d] matrix, 4 values a lane and K unit (zeros past row `end`)
struct RowPair {
  float4 w[2][kMaxUnits];
  float bias[2];
  __device__ __forceinline__ void load(const float* __restrict__ W, const float* __restrict__ b, int r0, int end, int d,
                                       int lane) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
      for (int kq = 0; kq < kMaxUnits; ++kq)
        w[i][kq] = r0 + i < end && kq * 128 < d
                       ? __ldg(reinterpret_cast<const float4*>(W + static_cast<size_t>(r0 + i) * d + kq * 128 + lane * 4))
                       : make_float4(0.f, 0.f, 0.f, 0.f);
      bias[i] = r0 + i < end ? __ldg(b + r0 + i) : 0.f;
    }
  }
  // this lane's part of rows . x (x in shared memory)
  __device__ __forceinline__ void dot(const float* x, int d, int lane, float (&acc)[2]) const {
    acc[0] = acc[1] = 0.f;
#pragma unroll
    for (int kq = 0; kq < kMaxUnits; ++kq)
      if (kq * 128 < d) {
        const float4 xv = *reinterpret_cast<const float4*>(x + kq * 128 + lane * 4);
#pragma unroll
        for (int i = 0; i < 2; ++i) acc[i] += w[i][kq].x * xv.x + w[i][kq].y * xv.y + w[i][kq].z * xv.z + w[i][kq].w * xv.w;
      }
  }
};

// Block (s, b): rows d s / n .. d (s + 1) / n - 1 of vehicle b's state token W_s2 silu(W_s1 s_b +
// b_s1) + b_s2 (every block forms the hidden vector, 16 inputs wide, itself) and its share of the
// visual rows. Layout of w: W_s1 [d, 16], b_s1 [d], W_s2 [d, d], b_s2 [d] (fp32, row-major [out, in]).
__global__ void __launch_bounds__(kMlpThreads) state_tokens_kernel(const StateArgs a) {
  __shared__ __align__(16) float s[kStateDim];
  __shared__ __align__(16) float h1[kMaxUnits * 128];
  const int b = blockIdx.y, d = a.d;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* w1 = a.w;
  const float* b1 = w1 + static_cast<size_t>(d) * kStateDim;
  const float* w2 = b1 + d;
  const float* b2 = w2 + static_cast<size_t>(d) * d;
  const int r_lo = d * blockIdx.x / gridDim.x, r_hi = d * (blockIdx.x + 1) / gridDim.x;
  RowPair rows;
  int r0 = r_lo + 2 * warp;
  rows.load(w2, b2, r0, r_hi, d, lane);
  if (threadIdx.x < kStateDim) s[threadIdx.x] = a.state[static_cast<size_t>(b) * kStateDim + threadIdx.x];
  float* out = a.frames + static_cast<size_t>(b) * (1 + kVisual) * d;
  for (int i = blockIdx.x * kMlpThreads + threadIdx.x; i < kVisual * d; i += gridDim.x * kMlpThreads) {
    const size_t src = static_cast<size_t>(b) * kVisual * d + i;
    out[d + i] = a.visual_dtype == 1 ? __bfloat162float(static_cast<const __nv_bfloat16*>(a.visual)[src])
                                     : static_cast<const float*>(a.visual)[src];
  }
  __syncthreads();
  for (int o = threadIdx.x; o < d; o += kMlpThreads) {
    float acc = b1[o];
#pragma unroll
    for (int k = 0; k < kStateDim; k += 4) {
      const float4 wv = __ldg(reinterpret_cast<const float4*>(w1 + static_cast<size_t>(o) * kStateDim + k));
      acc += wv.x * s[k];
      acc += wv.y * s[k + 1];
      acc += wv.z * s[k + 2];
      acc += wv.w * s[k + 3];
    }
    h1[o] = silu(acc);
  }
  __syncthreads();
  for (; r0 < r_hi; r0 += 2 * kMlpWarps) {
    float acc[2];
    rows.dot(h1, d, lane, acc);
    const float bias[2] = {rows.bias[0], rows.bias[1]};
    if (r0 + 2 * kMlpWarps < r_hi) rows.load(w2, b2, r0 + 2 * kMlpWarps, r_hi, d, lane);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float v = warp_sum(acc[i]);
      if (lane == 0 && r0 + i < r_hi) out[r0 + i] = v + bias[i];
    }
  }
}

__device__ __forceinline__ void st_rank0(const float* local, float v) {  // the same offset in cluster CTA 0
  uint32_t addr;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(addr) : "r"(smem_addr(local)));
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

}  // namespace

// One cluster of 8 CTAs per vehicle: w_j = W_h2 silu(W_h1 RMSNorm(x_j; g_f) + b_h1) + b_h2 over the
// final states of the five query tokens, which share every weight row read. Each CTA takes d / 8 rows
// of W_h1 and the matching columns of W_h2; rank 0 adds the CTAs' partial outputs in rank order.
// Layout of a.w: W_h1 [d, d], b_h1 [d], W_h2 [2, d], b_h2 [2].
__global__ void __launch_bounds__(kMlpThreads) head2_kernel(const Head2Args a) {
  __shared__ __align__(16) float n[kQueries][kMaxUnits * 128];
  __shared__ float h1[kQueries][kMaxUnits * 128 / kHeadCluster];
  __shared__ float part[kHeadCluster][2 * kQueries];
  const int d = a.d, rank = blockIdx.x, b = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* w1 = a.w;
  const float* b1 = w1 + static_cast<size_t>(d) * d;
  const float* w2 = b1 + d;
  const float* b2 = w2 + static_cast<size_t>(2) * d;
  const int n_rows = d / kHeadCluster, r_lo = rank * n_rows, r_hi = r_lo + n_rows;
  pdl_launch_dependents();
  RowPair rows;  // weights depend on no other kernel
  int r0 = r_lo + 2 * warp;
  rows.load(w1, b1, r0, r_hi, d, lane);
  float w2v[kMaxUnits * 128 / kHeadCluster / 32];  // warp 2 j + o: output o's columns for waypoint j
#pragma unroll
  for (int i = 0; i < kMaxUnits * 128 / kHeadCluster / 32; ++i)
    w2v[i] = warp < 2 * kQueries && lane + 32 * i < n_rows ? __ldg(w2 + (warp & 1) * d + r_lo + lane + 32 * i) : 0.f;
  pdl_wait();
  if (*reinterpret_cast<volatile int*>(a.status) != 0) return;  // a device-side error: no waypoint (whole cluster)
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");  // this CTA runs
  if (warp < a.n_waypoints) {  // RMSNorm of one token a warp
    const float* xr = a.x + (static_cast<size_t>(b) * a.vehicle_rows + warp) * d;
    float4 x[kMaxUnits];
    float ss = 0.f;
#pragma unroll
    for (int kq = 0; kq < kMaxUnits; ++kq) {
      x[kq] = kq * 128 < d ? __ldcg(reinterpret_cast<const float4*>(xr + kq * 128 + lane * 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
      ss += x[kq].x * x[kq].x + x[kq].y * x[kq].y + x[kq].z * x[kq].z + x[kq].w * x[kq].w;
    }
    const float rstd = rsqrtf(warp_sum(ss) / static_cast<float>(d) + 1e-6f);
#pragma unroll
    for (int kq = 0; kq < kMaxUnits; ++kq)
      if (kq * 128 < d) {
        const float4 g = __ldg(reinterpret_cast<const float4*>(a.final_norm + kq * 128 + lane * 4));
        *reinterpret_cast<float4*>(&n[warp][kq * 128 + lane * 4]) =
            make_float4(x[kq].x * rstd * g.x, x[kq].y * rstd * g.y, x[kq].z * rstd * g.z, x[kq].w * rstd * g.w);
      }
  }
  __syncthreads();
  for (; r0 < r_hi; r0 += 2 * kMlpWarps) {
    float v[kQueries][2];
#pragma unroll
    for (int j = 0; j < kQueries; ++j) rows.dot(n[j], d, lane, v[j]);
    const float bias[2] = {rows.bias[0], rows.bias[1]};
    if (r0 + 2 * kMlpWarps < r_hi) rows.load(w1, b1, r0 + 2 * kMlpWarps, r_hi, d, lane);
#pragma unroll
    for (int j = 0; j < kQueries; ++j)
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float t = warp_sum(v[j][i]);
        if (lane == 0 && r0 + i < r_hi) h1[j][r0 + i - r_lo] = silu(t + bias[i]);
      }
  }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // every CTA of the cluster runs
  __syncthreads();
  if (warp < 2 * a.n_waypoints) {
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < kMaxUnits * 128 / kHeadCluster / 32; ++i)
      if (lane + 32 * i < n_rows) acc += w2v[i] * h1[warp >> 1][lane + 32 * i];
    acc = warp_sum(acc);
    if (lane == 0) st_rank0(&part[rank][warp], acc);
  }
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (rank == 0 && threadIdx.x < 2 * a.n_waypoints) {
    float v = 0.f;
#pragma unroll
    for (int r = 0; r < kHeadCluster; ++r) v += part[r][threadIdx.x];
    a.targs->waypoints[static_cast<size_t>(b) * a.n_waypoints * 2 + threadIdx.x] = v + b2[threadIdx.x & 1];
  }
}

cudaError_t launch_state_tokens(const StateArgs& a_in, int sm_count, cudaStream_t stream) {
  StateArgs a = a_in;
  void* kargs[] = {&a};
  // one pass of 32 rows a block for few vehicles, about two blocks per SM for many
  int slices = 2 * sm_count / a.B;
  slices = slices > a.d / 32 ? a.d / 32 : (slices < 1 ? 1 : slices);
  return launch_ex(reinterpret_cast<const void*>(&state_tokens_kernel), dim3(slices, a.B), dim3(kMlpThreads), 0, stream,
                   false, kargs);
}

cudaError_t launch_head2(const Head2Args& a_in, cudaStream_t stream, bool pdl) {
  Head2Args a = a_in;
  if (a.n_waypoints > kQueries) return cudaErrorInvalidValue;
  void* kargs[] = {&a};
  return launch_ex(reinterpret_cast<const void*>(&head2_kernel), dim3(kHeadCluster, a.B), dim3(kMlpThreads), 0, stream,
                   pdl, kargs, 1, kHeadCluster);
}

}  // namespace fsx

namespace {

fsx_status pfail(fsx_status s, const char* msg) {
  fsx::set_error_message(msg);
  return s;
}

}  // namespace

extern "C" {

fsx_status fsx_paper_create(const fsx_config* cfg, const fsx_paper_weights* w, int device, fsx_handle* out) {
  fsx::set_error_message("");
  if (!out) return pfail(FSX_ERR_INVALID_ARG, "out handle pointer is NULL");
  *out = nullptr;
  if (!cfg || !w) return pfail(FSX_ERR_INVALID_ARG, "config or weights is NULL");
  if (!w->state_w1 || !w->state_b1 || !w->state_w2 || !w->state_b2 || !w->query_emb || !w->pos_emb ||
      !w->head_w1 || !w->head_b1 || !w->head_w2 || !w->head_b2 || !w->final_norm)
    return pfail(FSX_ERR_INVALID_ARG, "a weight pointer is NULL");
  const int d = cfg->d_model;
  if (d <= 0 || d > 1024) return pfail(FSX_ERR_UNSUPPORTED, "d_model must be in 1..1024");
  fsx_config c = *cfg;
  c.n_action = fsx::kQueries;      // the five waypoint queries: the handle's action tokens 0-4
  c.n_frame = 1 + fsx::kVisual;    // the state token and the four visual tokens
  c.n_waypoints = fsx::kQueries;
  c.frame_dtype = FSX_F32;         // the frame rows are assembled in fp32 on the device
  const int paper_visual_dtype = cfg->frame_dtype;
  if (paper_visual_dtype != FSX_F32 && paper_visual_dtype != FSX_BF16)
    return pfail(FSX_ERR_INVALID_ARG, "frame_dtype (of the visual tokens) must be FSX_F32 or FSX_BF16");
  // position rows in the handle's token order: queries 0-4, state, visual 0-3 (paper order:
  // state, visual 0-3, queries 0-4)
  std::vector<float> pos(static_cast<size_t>(10) * d);
  for (int i = 0; i < 10; ++i) {
    const int paper_row = i < 5 ? 5 + i : i - 5;
    std::memcpy(&pos[static_cast<size_t>(i) * d], w->pos_emb + static_cast<size_t>(paper_row) * d, d * sizeof(float));
  }
  std::vector<float> zero_head(static_cast<size_t>(2) * d + 2, 0.f);  // the single-layer head is not used
  fsx_weights tw{};
  tw.act_emb = w->query_emb;
  tw.pos_emb = pos.data();
  tw.attn_norm = w->attn_norm;
  tw.wq = w->wq;
  tw.wk = w->wk;
  tw.wv = w->wv;
  tw.wo = w->wo;
  tw.mlp_norm = w->mlp_norm;
  tw.w_gate = w->w_gate;
  tw.w_up = w->w_up;
  tw.w_down = w->w_down;
  tw.final_norm = w->final_norm;
  tw.head_w = zero_head.data();
  tw.head_b = zero_head.data() + 2 * d;
  fsx_handle h = nullptr;
  fsx_status s = fsx_create(&c, &tw, device, &h);
  if (s != FSX_OK) return s;
  // device copies: head [W_h1; b_h1; W_h2; b_h2], state MLP [W_s1; b_s1; W_s2; b_s2], frame rows
  const size_t n_head = (static_cast<size_t>(d) * d + d + 2 * static_cast<size_t>(d) + 2 + 3) / 4 * 4;  // 16-byte multiple
  const size_t n_state = static_cast<size_t>(d) * fsx::kStateDim + d + static_cast<size_t>(d) * d + d;
  std::vector<float> host(n_head + n_state, 0.f);
  float* p = host.data();
  auto put = [&](const float* src, size_t n) {
    std::memcpy(p, src, n * sizeof(float));
    p += n;
  };
  put(w->head_w1, static_cast<size_t>(d) * d);
  put(w->head_b1, d);
  put(w->head_w2, 2 * static_cast<size_t>(d));
  put(w->head_b2, 2);
  p = host.data() + n_head;
  put(w->state_w1, static_cast<size_t>(d) * fsx::kStateDim);
  put(w->state_b1, d);
  put(w->state_w2, static_cast<size_t>(d) * d);
  put(w->state_b2, d);
  float* dparams = nullptr;
  float* dframes = nullptr;
  cudaError_t e = cudaSetDevice(device);
  if (e == cudaSuccess) e = cudaMalloc(&dparams, host.size() * sizeof(float));
  if (e == cudaSuccess) e = cudaMemcpy(dparams, host.data(), host.size() * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMalloc(&dframes, static_cast<size_t>(cfg->max_batch) * (1 + fsx::kVisual) * d * sizeof(float));
  if (e != cudaSuccess) {
    if (dparams) cudaFree(dparams);
    if (dframes) cudaFree(dframes);
    fsx_destroy(h);
    return pfail(e == cudaErrorMemoryAllocation ? FSX_ERR_OOM : FSX_ERR_CUDA, cudaGetErrorString(e));
  }
  s = fsx::paper_attach(h, dparams, dparams, dframes, dparams + n_head, paper_visual_dtype);
  if (s != FSX_OK) {
    cudaFree(dparams);
    cudaFree(dframes);
    fsx_destroy(h);
    return s;
  }
  *out = h;
  return FSX_OK;
}

fsx_status fsx_paper_tick(fsx_handle h, const void* const* k_cache, const void* const* v_cache,
                          const int64_t* d_offsets, int B, const void* d_visual, const float* d_state,
                          float* d_waypoints, void* stream) {
  fsx::set_error_message("");
  if (!h) return pfail(FSX_ERR_INVALID_ARG, "handle is NULL");
  if (!fsx::paper_frames(h)) return pfail(FSX_ERR_INVALID_ARG, "handle was not created by fsx_paper_create");
  if (!d_visual || !d_state) return pfail(FSX_ERR_INVALID_ARG, "visual tokens or state is NULL");
  if (B < 1 || B > fsx::paper_max_batch(h)) return pfail(FSX_ERR_INVALID_ARG, "B outside 1..max_batch");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaSetDevice(fsx::paper_device(h));
  if (e == cudaSuccess) e = fsx::paper_order_after_last_tick(h, st);
  fsx::StateArgs a{};
  a.state = d_state;
  a.visual = d_visual;
  a.visual_dtype = fsx::paper_visual_dtype(h);
  a.w = fsx::paper_state_weights(h);
  a.frames = fsx::paper_frames(h);
  a.d = fsx::paper_d(h);
  a.B = B;
  if (e == cudaSuccess) e = fsx::launch_state_tokens(a, fsx::paper_sm_count(h), st);
  if (e != cudaSuccess) return pfail(FSX_ERR_CUDA, cudaGetErrorString(e));
  return fsx_tick(h, k_cache, v_cache, d_offsets, B, fsx::paper_frames(h), d_waypoints, stream);
}

}  // extern "C"
