// Shared host/device helpers of libqbert: workspace layout, status word, error text.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "qbert.h"

namespace qb {

// ---- workspace layout (device memory owned by the caller) ------------------------------------
// [0]   int32  status   first device-side error, never cleared by a kernel
// [4]   int32  detail   where a bounded wait gave up (role << 16 | stage), diagnostics only
// [16]  uint32 act_absmax_bits   reduction slot of act_absmax_kernel for a single tensor
// [32]  uint64 ticket            launches that cleared slots << 32 | blocks of the running one that have started
// [40]  uint32 cleared           number of the last such launch whose reduction slots are clear
// [44]  uint32 round             counts the launches whose clusters waited for one another
// [64]  uint64 cluster_max[24]   round << 32 | bit pattern of a cluster's max|x|, all of the last such launch
// [256] uint32 range_hi_enc[G], uint32 range_lo_inv[G]   ordered encodings of per-group max / min
//       or, weight_ring_kernel: uint64 [groups][CTAs], encoded max << 32 | inverted encoded min
constexpr size_t kWsStatusOff = 0;
constexpr size_t kWsDetailOff = 4;
constexpr size_t kWsActMaxOff = 16;
constexpr size_t kWsRangeOff = 256;
constexpr size_t kWsMinBytes = 256;
constexpr int kWsClusters = 24;

struct WsHeader {
  int32_t status;
  int32_t detail;
  uint32_t pad[2];
  uint32_t act_absmax_bits;
  uint32_t pad2[3];
  unsigned long long ticket;
  uint32_t cleared;
  uint32_t round;
  uint32_t pad3[4];
  unsigned long long cluster_max[kWsClusters];
};
static_assert(sizeof(WsHeader) == kWsRangeOff, "the tables follow the header");

// What a call on G groups must get, and what qb_workspace_bytes tells callers to give: with a slot per group and CTA
// (for up to kRingMaxGroups groups) the weight quantizer reads W once where groups are too large for a
// cluster's registers.
constexpr int kRingMaxGroups = 128;
constexpr int kRingMaxCtas = 160;
inline size_t ring_table_bytes(size_t groups) { return groups * kRingMaxCtas * 8; }
inline size_t ws_round(size_t b) { return (b + 255) / 256 * 256; }
inline size_t ws_bytes_needed(int groups) { return ws_round(kWsRangeOff + (groups > 0 ? size_t(groups) * 8 : 0)); }
inline size_t ws_bytes_recommended(int groups) {
  if (groups <= 0) return ws_bytes_needed(0);
  const size_t tables = size_t(groups) * 8, ring = ring_table_bytes(groups < kRingMaxGroups ? groups : kRingMaxGroups);
  return ws_round(kWsRangeOff + (tables > ring ? tables : ring));
}

// ---- host-side error plumbing ------------------------------------------------------------------
void set_last_error(const char* fmt, ...);
qb_status cuda_fail(cudaError_t e, const char* what);
// QB_OK if the current device is sm_100; caches the answer and the SM count per device.
qb_status require_sm100(int* sm_count);

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline bool valid_bits(int b) { return b == 2 || b == 3 || b == 4 || b == 8; }

#define QB_CUDA_TRY(expr)                                   \
  do {                                                      \
    cudaError_t e__ = (expr);                               \
    if (e__ != cudaSuccess) return qb::cuda_fail(e__, #expr); \
  } while (0)

// Launch of a kernel that begins with pdl_begin.
// Programmatic stream serialization: the kernel's blocks may be set up while the kernel before it on the stream
// drains, and wait in pdl_begin for its completion.  Back to back launches of 592 blocks: 4.1 us each without it, 2.2 us
// with it.
// `cluster`: CTAs per cluster; `cooperative`: every block must be resident at once (the blocks wait on
// one another).
// `SPLIT`: kMostL1 asks for the SM's data cache as L1, for the kernels that use next to no shared memory and follow a GEMM,
// which takes nearly all of it.  Without the request such a kernel, set up while the GEMM drains, runs under the GEMM's
// split and has little L1 for its loads in flight; with it its blocks come once the SM is free.  A preference of the one
// launch: it can neither fail a call nor outlast it, as one that is set on the function could.
// In us, with new inputs each pass: encoder layer at M = 4096 with the quantizer's first pass launched after the GEMM 78.6,
// set up under it 84.3, that with the request 77.2; two large layers at M = 24576 1,067, 1,136, 1,066.  On both passes rather
// than the first alone: the same on one stream; ten quantizer batches beside five such layers' GEMMs on another stream
// 496, 509 (launched after the GEMM: 509), beside three calls of the ring quantizer 517, 524 (519).
// The other kernels with little shared memory (embeddings, straight-through backward) have not been tried with it.
enum CacheSplit { kAnySplit, kMostL1 };
template <CacheSplit SPLIT = kAnySplit, class... P, class... A>
inline cudaError_t launch_kernel(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream,
                                 unsigned cluster, bool cooperative, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(block, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[4];
  int n = 1;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = 1;
  }
  if (cooperative) {
    attr[n].id = cudaLaunchAttributeCooperative;
    attr[n++].val.cooperative = 1;
  }
  if (SPLIT == kMostL1) {
    attr[n].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[n++].val.sharedMemCarveout = cudaSharedmemCarveoutMaxL1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, std::decay_t<P>(args)...);
}

// Does work on this stream have `sms` SMs?  Asked before a cooperative launch whose grid is made for the whole device: a
// stream of a green context may have fewer.  Outside a capture the driver refuses such a launch (below); under capture
// it does not, and the graph waits for room that never comes.
bool stream_has_sms(cudaStream_t stream, int sms);

// Was a launch refused because its blocks (of a cooperative launch, of a cluster) cannot be resident together?  The
// grids are made for the whole device; a green context or an MPS client may have fewer SMs.  The forms that need
// residency have one beside them that does not, which such a launch falls back to.
inline bool residency_refused(cudaError_t e) {
  if (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorInvalidClusterSize) return false;
  cudaGetLastError();  // not an error of the call
  return true;
}

// ---- device-side helpers -----------------------------------------------------------------------
#ifdef __CUDACC__
// Called by every thread of a kernel started by launch_kernel before it touches global memory: waits until the
// kernel before this one on the stream has completed and its results are visible, and only then lets the
// next kernel's blocks be set up.  In this order every kernel that runs has all kernels but its direct
// predecessor behind it when it is set up.
// The predecessor still writes when this kernel begins, so nothing that it may have written is read-only for this kernel's
// lifetime: such data (inputs included, which another call of the library may have made) is read with ordinary loads.
// A non-coherent one (__ldg, or a const __restrict__ argument that the compiler turns into one) counts as invariant
// and may be moved above the wait.
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ void report_status(void* ws, int32_t code, int32_t detail = 0) {
  WsHeader* h = reinterpret_cast<WsHeader*>(ws);
  if (atomicCAS(&h->status, 0, code) == 0) h->detail = detail;
}

// Monotone map from float bit patterns to unsigned integers (so that integer atomicMax orders floats).
// Written as integer PTX on the register: as C++ the compiler may turn the sign-bit operations into
// floating-point negation, which does not keep the bit pattern of a NaN (and the NaN would then sort
// below the finite values instead of above them).
__device__ __forceinline__ uint32_t float_to_ordered(float f) {
  uint32_t o;
  asm("{\n\t.reg .b32 t, m;\n\tmov.b32 t, %1;\n\tshr.s32 m, t, 31;\n\tor.b32 m, m, 0x80000000;\n\txor.b32 %0, t, m;\n\t}"
      : "=r"(o)
      : "f"(f));
  return o;
}
__device__ __forceinline__ float ordered_to_float(uint32_t e) {
  uint32_t b = (e & 0x80000000u) ? (e & 0x7fffffffu) : ~e;
  return __uint_as_float(b);
}
__device__ __forceinline__ float min3_nan(float a, float b, float c) {
  float d;
  asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float d;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release(unsigned long long* p, unsigned long long v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void st_release(uint32_t* p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Called by one warp of every block: the block that comes first clears the launch's reduction slots and says so
// (whichever block it is, it is running, so nobody waits for a block that has not started).  The others
// look before they publish (h->cleared shows the number returned here); by then they have read their share of the
// input and the wait is over before it begins.  The block that comes last opens the next launch's count, so that nothing
// is left for a later kernel to put back: one that is never launched would leave the next call with slots that
// count as clear.
__device__ __forceinline__ uint32_t clear_slots(uint32_t* slots, int count, WsHeader* h, int lane) {
  unsigned long long t = 0;
  if (lane == 0) {
    t = atomicAdd(&h->ticket, 1ull);
    if ((uint32_t)t == gridDim.x - 1) atomicAdd(&h->ticket, (1ull << 32) - gridDim.x);
  }
  t = __shfl_sync(0xffffffffu, t, 0);
  const uint32_t launch = (uint32_t)(t >> 32) + 1u;
  if ((uint32_t)t == 0u) {
    for (int i = lane; i < count; i += 32) slots[i] = 0u;
    __threadfence();
    __syncwarp();
    if (lane == 0) st_release(&h->cleared, launch);
  }
  return launch;
}
// 16-byte load with an L2 eviction-priority policy (createpolicy).  The two-pass quantizers use it: the
// first pass asks L2 to keep a fraction of what it reads (the second pass reads the same tensor next),
// the second pass marks its reads as the first to go.
__device__ __forceinline__ float4 ldg_policy(const float4* p, uint64_t policy) {
  float4 v;
  asm volatile("ld.global.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p), "l"(policy));
  return v;
}
__device__ __forceinline__ uint64_t policy_evict_last(float fraction) {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, %1;" : "=l"(pol) : "f"(fraction));
  return pol;
}
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

// Share of a first pass's input that L2 is asked to keep: all of it up to 96 MB (what the 126 MB L2 holds
// of a stream besides what the second pass writes), else 96 MB worth.
inline float l2_keep_fraction(double input_bytes) {
  const double keep = 96.0 * 1048576.0;
  return input_bytes <= keep ? 1.0f : (float)(keep / input_bytes);
}

#endif

}  // namespace qb
