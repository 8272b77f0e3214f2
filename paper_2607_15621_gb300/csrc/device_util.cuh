// Device-side primitives shared by the fsx kernels (sm_103a): tensor-core
// mma.sync, ldmatrix, cp.async, bulk copies with mbarrier completion,
// programmatic dependent launch, bounded waits and the device status word.
#pragma once

#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace fsx {

// Status codes written into the device status word (mirrors fsx_status).
enum : int { kStatusOk = 0, kStatusTimeout = 5, kStatusDeviceArg = 6, kStatusRange = 7 };

// ~1 s bound for every device-side wait (globaltimer counts nanoseconds).
constexpr unsigned long long kWaitLimitNs = 1000000000ull;

__device__ __forceinline__ void set_status(int* status, int code) { atomicCAS(status, 0, code); }

__device__ __forceinline__ unsigned long long global_timer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Programmatic dependent launch: let the next kernel of the stream start its
// prologue now / wait until the previous kernel has completed and flushed.
__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// D[16x8] += A[16x16] * B[16x8], fp16 operands, fp32 accumulators.
__device__ __forceinline__ void mma_f16_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                              uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void ldsm_x4(uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3,
                                        uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}

__device__ __forceinline__ void ldsm_x4_trans(uint32_t& r0, uint32_t& r1, uint32_t& r2,
                                              uint32_t& r3, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}

// 16-byte global->shared asynchronous copy (L2 only).
__device__ __forceinline__ void cp_async_16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ---- mbarrier + bulk (non-tensor) copies -----------------------------------
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}

// Plain arrival (no transaction bytes): completes the phase of a count-1 barrier.
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// `n` arrivals at once.
__device__ __forceinline__ void mbar_arrive_n(uint64_t* bar, uint32_t n) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(n) : "memory");
}

// Bounded wait for phase `parity` of an mbarrier; false (and status set) on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* status) {
  const uint32_t addr = smem_addr(bar);
  unsigned long long t0 = 0;
  for (uint32_t it = 0;; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, "
        "p;\n}"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
    if ((it & 255u) == 0) {
      const unsigned long long now = global_timer_ns();
      if (t0 == 0) {
        t0 = now;
      } else if (now - t0 > kWaitLimitNs) {
        set_status(status, kStatusTimeout);
        return false;
      }
    }
  }
}

// mbarrier_wait with acquire semantics at cluster scope, for phases completed by
// other CTAs' st.async stores; false (and status set) on timeout.
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity, int* status) {
  const uint32_t addr = smem_addr(bar);
  unsigned long long t0 = 0;
  for (uint32_t it = 0;; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, "
        "0, p;\n}"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
    if ((it & 255u) == 0) {
      const unsigned long long now = global_timer_ns();
      if (t0 == 0) {
        t0 = now;
      } else if (now - t0 > kWaitLimitNs) {
        set_status(status, kStatusTimeout);
        return false;
      }
    }
  }
}

// Distributed shared memory stores that complete on the destination CTA's
// mbarrier (transaction bytes): `raddr` and `rbar` are shared::cluster addresses
// of the same CTA. The values come from registers, so the sender's buffers are
// free at once; the receiver's wait on `rbar` orders its reads after the data.
__device__ __forceinline__ void st_async_v4(uint32_t raddr, uint4 v, uint32_t rbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1,%2,%3,%4}, [%5];" ::"r"(raddr),
               "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(rbar)
               : "memory");
}
__device__ __forceinline__ void st_async_v2(uint32_t raddr, uint32_t a, uint32_t b, uint32_t rbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1,%2}, [%3];" ::"r"(raddr), "r"(a),
               "r"(b), "r"(rbar)
               : "memory");
}
__device__ __forceinline__ void st_async_b32(uint32_t raddr, uint32_t a, uint32_t rbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(raddr), "r"(a),
               "r"(rbar)
               : "memory");
}

// Bulk global->shared copy of `bytes` (multiple of 16, both ends 16-byte
// aligned) completing on `bar`; the weights are streamed once per tick.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// Before the first TMA load of a CTA through a tensor map that lies in global memory, by the thread
// that issues its loads: the map may have been rewritten at the same address (by a host copy, hence
// the system scope) since an earlier kernel loaded through it, and TMA reads maps by a proxy of its own.
__device__ __forceinline__ void tensormap_acquire(const void* map) {
  asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(map) : "memory");
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
  __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}

// Cache values the kernels convert to fp16 are expected within +-65504. The converters
// below keep in `peak` the largest magnitudes seen, as two packed fp16 (start at 0): a value
// that rounds beyond 65504 became an infinity and a NaN stays one, so out_of_range(peak) tells
// whether an input lay outside the fp16 range. flag_range() turns that into the FSX_ERR_RANGE
// error status: a tick is abandoned like on any other device-side error, and Eq. 1 alone still
// writes its rows, so once out_of_range(peak) its callers put saturate_half8() between the
// conversion and the operand tile and the rows are those of the cache clipped to +-65504.
// (One max per pair of values and one test per unit, against a saturating conversion and two
// compares per value: the conversions bound the staging warps.)
__device__ __forceinline__ uint32_t peak_of(uint32_t peak, uint32_t h) {
  const __half2 m = __hmax2_nan(*reinterpret_cast<const __half2*>(&peak), __habs2(*reinterpret_cast<const __half2*>(&h)));
  return *reinterpret_cast<const uint32_t*>(&m);
}
__device__ __forceinline__ uint32_t bf16x2_to_half2_peak(uint32_t v, uint32_t& peak) {
  const uint32_t h = pack_half2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
  peak = peak_of(peak, h);
  return h;
}
__device__ __forceinline__ uint32_t f32x2_to_half2_peak(float lo, float hi, uint32_t& peak) {
  const uint32_t h = pack_half2(lo, hi);
  peak = peak_of(peak, h);
  return h;
}
__device__ __forceinline__ bool out_of_range(uint32_t peak) {  // an infinity or a NaN in either half
  return ((peak + 0x04000400u) & 0x80008000u) != 0u;           // magnitudes: no carry between the halves
}
__device__ __forceinline__ uint32_t saturate_half2(uint32_t h) {  // infinities -> +-65504, a NaN stays
  const __half2 lim = __float2half2_rn(65504.f);
  const __half2 v = __hmax2_nan(__hmin2_nan(*reinterpret_cast<const __half2*>(&h), lim), __hneg2(lim));
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ uint4 saturate_half8(uint4 h) {
  return make_uint4(saturate_half2(h.x), saturate_half2(h.y), saturate_half2(h.z), saturate_half2(h.w));
}
__device__ __forceinline__ void flag_range(int* status, uint32_t peak) {
  if (out_of_range(peak)) set_status(status, kStatusRange);
}

// Two bf16 (low half first) -> two fp16, via fp32 (bf16 -> fp32 is exact).
__device__ __forceinline__ uint32_t bf16x2_to_half2(uint32_t v) {
  const float lo = __uint_as_float(v << 16);
  const float hi = __uint_as_float(v & 0xffff0000u);
  return pack_half2(lo, hi);
}

}  // namespace fsx
