// qb_quantize_act(_batch): per-tensor 8-bit activation quantizer (Table 1 caption: 8-bit activations;
// Appendix A's uniform quantizer on the symmetric range [-a, a], a = max|x|), for one tensor or a
// batch of tensors.
//
// The unit of work is a segment: up to eight units of 128 consecutive elements of one row, one float4 per lane
// and unit, so that a warp has 4 KB of loads in flight at once.  A row is cut into ceil(K / 1024) segments.
//
//   act_absmax_kernel    max|x| of every tensor.  The units of all tensors form one sequence that the
//                        blocks cut into equal contiguous shares (a block meets few tensors and publishes
//                        one atomicMax for each).
//   act_quantize_kernel  one warp per segment: x * (127/a), round half to even, four codes per 32-bit
//                        store, row sum by dp4a and a warp reduction (rows of several segments: atomicAdd on
//                        row sums that the first kernel cleared).
//   act_fused_kernel     both for one tensor of up to 2,368 segments, each of which finds a warp on the device: the
//                        segment stays in registers while the blocks agree on a, within a cluster in
//                        distributed shared memory; x is read once and there is one launch instead of two.
//
// Both passes are memory-bound (4 B read per element, then 4 B read, from L2 as far as it holds the
// tensors, and 1 B written).  What bounds them below L2's size is the bytes in flight and the instructions per
// element: 128 KB of loads per SM and about nine instructions per float4 (packed fp32x2, no clamp) instead of
// 64 KB and thirty.  Quantizer and GEMMs of one BERT-base layer at M = 4096 (88 MB of input): 86.9 -> 81.1 us;
// int8 chain at M = 6144 98.0 -> 91.5; query projection at M = 1024 (fused) 20.1 -> 17.4 -> 12.6.
#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "mbar_wait.cuh"
#include "ptx.cuh"

namespace qb {

constexpr int kActThreads = 256;
constexpr int kActWarps = kActThreads / 32;
constexpr int kActBlocksPerSm = 4;
constexpr int kActMaxCluster = 8;     // act_fused_kernel: CTAs of a cluster (the portable size)
constexpr int kActMaxThreads = 1024;  // and threads of such a CTA
constexpr int kSegUnits = 8;      // float4 per lane and segment
constexpr int kMaxActBatch = 64;  // tensors per launch (descriptors travel as kernel parameters, 4.6 KB)

struct ActItem {
  const float* x;
  int8_t* xq;
  float* act_scale;
  int32_t* rowsum;
  int64_t M;
  int64_t unit_begin;   // index of the tensor's first unit in the launch's sequence
  int64_t seg_begin;    // index of the tensor's first segment in the launch's sequence
  int32_t units_per_row;
  int32_t segs_per_row;
  int32_t seg_units;    // units per segment (the last one of a row may be shorter)
};

template <int P>
struct ActBatch {
  ActItem item[P];
  uint32_t* absmax_bits;  // [count] slots in the workspace
  void* ws;
  int64_t units_total, units_per_block;
  int64_t segs_total;
  int32_t count;
  float keep_fraction;  // share of the launch's input that L2 is asked to keep between the two passes
};

// Running extremes of a lane; NaN stays.  Start value 0: only the magnitude matters.
struct Extremes {
  float lo = 0.0f, hi = 0.0f;
  __device__ __forceinline__ void add(const float4& v) {
    lo = min3_nan(min3_nan(lo, v.x, v.y), v.z, v.w);
    hi = max3_nan(max3_nan(hi, v.x, v.y), v.z, v.w);
  }
  // bit pattern of the largest |x| over the warp (NaN and Inf above every finite value)
  __device__ __forceinline__ uint32_t warp_bits() const {
    const uint32_t h = __float_as_uint(hi) & 0x7fffffffu, l = __float_as_uint(lo) & 0x7fffffffu;
    return __reduce_max_sync(0xffffffffu, max(h, l));
  }
};

// scale and reciprocal of a tensor from the bit pattern of its max|x|; false if NaN/Inf was seen
__device__ __forceinline__ bool act_scales(uint32_t mb, float* s, float* inv) {
  *s = 1.0f;
  *inv = 0.0f;
  if (mb >= 0x7f800000u) return false;
  const float a = __uint_as_float(mb);
  const float s1 = __fdiv_rn(a, 127.0f);
  const float inv1 = __fdiv_rn(127.0f, a);
  if (a > 0.0f && inv1 <= 3.402823466e38f) {
    *s = s1;
    *inv = inv1;
  }
  return true;
}

// Four codes of one float4 as bytes.  |x| <= a and inv = 127/a rounded, so |x * inv| < 127.5 and no code needs a
// clamp; adding 1.5 * 2^23 rounds to an integer, half to even, and leaves the code in the low byte as two's
// complement.  The add is written as a fused multiply-add with 1.0: a packed mul and a packed add would be
// contracted into one operation, which rounds the exact product instead of the rounded one.
__device__ __forceinline__ uint32_t quant_word(const float4& v, float inv) {
  uint32_t b0, b1, b2, b3;
  asm("{\n\t.reg .b64 p0, p1, i2, m2, o2;\n\t"
      "mov.b64 p0, {%4, %5};\n\tmov.b64 p1, {%6, %7};\n\t"
      "mov.b64 i2, {%8, %8};\n\tmov.b64 m2, {%9, %9};\n\tmov.b64 o2, {%10, %10};\n\t"
      "mul.rn.f32x2 p0, p0, i2;\n\tmul.rn.f32x2 p1, p1, i2;\n\t"
      "fma.rn.f32x2 p0, p0, o2, m2;\n\tfma.rn.f32x2 p1, p1, o2, m2;\n\t"
      "mov.b64 {%0, %1}, p0;\n\tmov.b64 {%2, %3}, p1;\n\t}"
      : "=r"(b0), "=r"(b1), "=r"(b2), "=r"(b3)
      : "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "f"(inv), "f"(12582912.0f), "f"(1.0f));
  return __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410);
}

// The tensor of the batch that holds unit / segment `x`: the last one that begins at or before it.  (Walking a batch of 48
// from its start cost every block and warp some 50 cycles per tensor.)
template <int P, int64_t ActItem::*BEGIN>
__device__ __forceinline__ int find_item(const ActBatch<P>& b, int64_t x) {
  int lo = 0, hi = b.count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (b.item[mid].*BEGIN <= x) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

template <int P>
__global__ void __launch_bounds__(kActThreads, kActBlocksPerSm)
act_absmax_kernel(const __grid_constant__ ActBatch<P> b) {
  __shared__ uint32_t s_max[P];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  WsHeader* const h = reinterpret_cast<WsHeader*>(b.ws);
  for (int i = threadIdx.x; i < P; i += kActThreads) s_max[i] = 0u;
  pdl_begin();
  __syncthreads();
  const uint64_t pol = policy_evict_last(b.keep_fraction);
  const int64_t u0 = (int64_t)blockIdx.x * b.units_per_block;
  const int64_t u1 = min(u0 + b.units_per_block, b.units_total);
  bool cleared = warp != 0;
  uint32_t launch = 0;
  const int first = find_item<P, &ActItem::unit_begin>(b, u0);
  int it = first;
  for (; it < b.count && b.item[it].unit_begin < u1; ++it) {
    const ActItem& t = b.item[it];
    const int64_t lo = max(u0 - t.unit_begin, (int64_t)0), hi = min(u1 - t.unit_begin, t.M * t.units_per_row);
    if (t.segs_per_row > 1) {  // row sums that several warps will add to: of the rows that begin in this share
      const int64_t m0 = (lo + t.units_per_row - 1) / t.units_per_row, m1 = (hi + t.units_per_row - 1) / t.units_per_row;
      for (int64_t m = m0 + threadIdx.x; m < m1; m += kActThreads) t.rowsum[m] = 0;
    }
    const float4* x = reinterpret_cast<const float4*>(t.x) + lane;
    Extremes ex;
    for (int64_t u = lo + warp * kSegUnits; u < hi; u += kActWarps * kSegUnits) {
      const int n = (int)min(hi - u, (int64_t)kSegUnits);
      float4 v[kSegUnits];
#pragma unroll
      for (int j = 0; j < kSegUnits; ++j)
        if (j < n) v[j] = ldg_policy(x + (u + j) * 32, pol);
      if (!cleared) {  // warp 0, while its first loads are on their way (every block has at least one unit)
        cleared = true;
        launch = clear_slots(b.absmax_bits, b.count, h, lane);
      }
#pragma unroll
      for (int j = 0; j < kSegUnits; ++j)
        if (j < n) ex.add(v[j]);
    }
    const uint32_t m = ex.warp_bits();
    if (lane == 0 && m != 0u) atomicMax(&s_max[it], m);
  }
  __syncthreads();
  if (threadIdx.x == 0 && !poll_word(&h->cleared, launch)) report_status(b.ws, QB_ERR_TIMEOUT);
  __syncthreads();
  for (int i = first + threadIdx.x; i < it; i += kActThreads)
    if (s_max[i] != 0u) atomicMax(b.absmax_bits + i, s_max[i]);
}

// Codes and row sum of one segment held in v[0 .. n).
__device__ __forceinline__ void quantize_segment(const ActItem& t, uint32_t row, int seg, int n, const float4 (&v)[kSegUnits],
                                                 float inv, int lane) {
  uint32_t* dst = reinterpret_cast<uint32_t*>(t.xq) + ((int64_t)row * t.units_per_row + seg * t.seg_units) * 32 + lane;
  int sum = 0;
#pragma unroll
  for (int j = 0; j < kSegUnits; ++j)
    if (j < n) {
      const uint32_t w = quant_word(v[j], inv);
      sum = __dp4a((int)w, 0x01010101, sum);
      dst[j * 32] = w;
    }
  sum = __reduce_add_sync(0xffffffffu, sum);
  if (lane == 0) {
    if (t.segs_per_row == 1) t.rowsum[row] = sum;
    else atomicAdd(t.rowsum + row, sum);
  }
}

template <int P>
__global__ void __launch_bounds__(kActThreads, kActBlocksPerSm)
act_quantize_kernel(const __grid_constant__ ActBatch<P> b) {
  const int lane = threadIdx.x & 31;
  pdl_begin();
  const int64_t warps = (int64_t)gridDim.x * kActWarps;
  const uint64_t pol = policy_evict_first();
  const int64_t s0 = (int64_t)blockIdx.x * kActWarps + (threadIdx.x >> 5);
  int it = find_item<P, &ActItem::seg_begin>(b, s0), cur = -1;
  float inv = 0.0f;
  for (int64_t s = s0; s < b.segs_total; s += warps) {
    while (it + 1 < b.count && s >= b.item[it + 1].seg_begin) ++it;
    const ActItem& t = b.item[it];
    const uint32_t local = (uint32_t)(s - t.seg_begin);  // below 2^24 rows x 64 segments
    const uint32_t row = t.segs_per_row > 1 ? local / (uint32_t)t.segs_per_row : local;
    const int seg = (int)(local - row * t.segs_per_row);
    const int n = min(t.seg_units, t.units_per_row - seg * t.seg_units);
    const float4* src = reinterpret_cast<const float4*>(t.x) + ((int64_t)row * t.units_per_row + seg * t.seg_units) * 32 + lane;
    float4 v[kSegUnits];
#pragma unroll
    for (int j = 0; j < kSegUnits; ++j)
      if (j < n) v[j] = ldg_policy(src + j * 32, pol);
    if (it != cur) {  // warp-uniform: first segment of this warp in tensor `it`
      cur = it;
      float scale;
      const bool finite = act_scales(b.absmax_bits[it], &scale, &inv);
      if (local == 0 && lane == 0) {  // exactly one warp sees the tensor's first segment
        *t.act_scale = scale;
        if (!finite) report_status(b.ws, QB_ERR_NONFINITE);
      }
    }
    quantize_segment(t, row, seg, n, v, inv, lane);
  }
}

// One tensor, one segment per warp; the segment stays in registers while the warps agree on the maximum, which is what
// bounds the kernel.  The blocks of a cluster (of 8 to 32 warps) agree through distributed shared memory: one barrier of
// the cluster.  MANY: the maxima of several clusters, all resident (cooperative launch), meet in the workspace: each
// is stored with the launch's number, and every block polls for all of them, one release and one acquire in all;
// no word has to be cleared first.  All blocks resident that met in one word (clear, maximum, count, go-ahead,
// read: five trips to L2) took, with the GEMM, 12.7 us at M = 32 x 768 (now, one cluster: 9.1), 14.3 at
// 1,024 x 768 (now, 16 clusters: 12.6).
template <bool MANY>
__global__ void __launch_bounds__(kActMaxThreads, 1)
act_fused_kernel(const __grid_constant__ ActBatch<1> b) {
  __shared__ uint32_t s_max, s_peer[kActMaxCluster];
  __shared__ int s_ok;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  WsHeader* const h = reinterpret_cast<WsHeader*>(b.ws);
  const ActItem& t = b.item[0];
  const uint32_t local = blockIdx.x * (blockDim.x >> 5) + warp;
  const bool mine = local < (uint32_t)b.segs_total;
  const uint32_t row = local / (uint32_t)t.segs_per_row;
  const int seg = (int)(local - row * t.segs_per_row);
  const int n = mine ? min(t.seg_units, t.units_per_row - seg * t.seg_units) : 0;
  const float4* src = reinterpret_cast<const float4*>(t.x) + ((int64_t)row * t.units_per_row + seg * t.seg_units) * 32 + lane;
  if (threadIdx.x == 0) s_max = 0u;
  const uint32_t rank = ptx::cluster_ctarank(), ctas = MANY ? kActMaxCluster : gridDim.x;
  ptx::cluster_arrive();  // "this CTA has started": waited for before the first remote store
  pdl_begin();
  float4 v[kSegUnits];
#pragma unroll
  for (int j = 0; j < kSegUnits; ++j)
    if (j < n) v[j] = src[j * 32];
  uint32_t tag = 0u;
  if (MANY && warp == 0) tag = ld_acquire(&h->round) + 1u;  // every CTA reads it before its cluster publishes
  if (mine && t.segs_per_row > 1 && seg == 0 && lane == 0) t.rowsum[row] = 0;  // published by the barrier below
  __syncthreads();
  Extremes ex;
#pragma unroll
  for (int j = 0; j < kSegUnits; ++j)
    if (j < n) ex.add(v[j]);
  const uint32_t m = ex.warp_bits();
  if (lane == 0 && m != 0u) atomicMax(&s_max, m);
  __syncthreads();
  ptx::cluster_wait();
  if (threadIdx.x < ctas)  // this CTA's maximum into its slot of CTA threadIdx.x
    ptx::st_cluster_u32(ptx::map_to_cta(ptx::smem_u32(&s_peer[rank]), threadIdx.x), s_max);
  __syncwarp();
  ptx::cluster_sync_all();  // publishes the row sums set to zero, too
  uint32_t absmax = 0u;
  for (uint32_t i = 0; i < ctas; ++i) absmax = max(absmax, s_peer[i]);
  if constexpr (MANY) {
    if (warp == 0) {
      const uint32_t cluster = blockIdx.x / kActMaxCluster, clusters = gridDim.x / kActMaxCluster;
      if (rank == 0 && lane == 0) st_release(&h->cluster_max[cluster], (unsigned long long)tag << 32 | absmax);
      bool ok = true;
      uint32_t m = 0u;
      if (lane < (int)clusters) {
        unsigned long long w = ld_acquire(&h->cluster_max[lane]);
        if ((uint32_t)(w >> 32) != tag) {
          const long long t0 = clock64();
          do {
            w = ld_acquire(&h->cluster_max[lane]);
            ok = clock64() - t0 <= kWaitLimitCycles;
          } while ((uint32_t)(w >> 32) != tag && ok);
        }
        m = (uint32_t)w;
      } else if (blockIdx.x == 0 && lane < kWsClusters) {  // no slot keeps the number of an older launch
        h->cluster_max[lane] = (unsigned long long)tag << 32;
      }
      ok = __all_sync(0xffffffffu, ok);
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) {
        s_max = m;
        s_ok = ok ? 1 : 0;
        if (!ok) report_status(b.ws, QB_ERR_TIMEOUT);
        if (blockIdx.x == 0) h->round = tag;
      }
    }
    __syncthreads();
    if (!s_ok) return;
    absmax = s_max;
  }
  float scale, inv;
  const bool finite = act_scales(absmax, &scale, &inv);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *t.act_scale = scale;
    if (!finite) report_status(b.ws, QB_ERR_NONFINITE);
  }
  if (mine) quantize_segment(t, row, seg, n, v, inv, lane);
}

// The launches over `count` tensors (<= P).  `absmax_slots` has room for `count` words.
template <int P>
static qb_status launch_act_batch(const qb_act_desc* d, int count, void* ws, uint32_t* absmax_slots, int sm_count,
                                  cudaStream_t stream) {
  ActBatch<P> b;
  b.count = count;
  b.ws = ws;
  b.absmax_bits = absmax_slots;
  const int64_t cap = (int64_t)sm_count * kActBlocksPerSm;  // one full wave
  // Tensors with the longest segments first: kernel 2 hands segments to warps round-robin, and a long one met
  // at the end of a warp's list would be the launch's tail.  Slot i of `absmax_slots` stays with the
  // i-th tensor of this order; nothing outside the two kernels reads the slots.
  int ord[P];
  for (int i = 0; i < count; ++i) ord[i] = i;
  const auto seg_units = [](int64_t K) {
    const int64_t u = K / 128, n = (u + kSegUnits - 1) / kSegUnits;
    return (int)((u + n - 1) / n);
  };
  if (P > 1)
    std::stable_sort(ord, ord + count, [&](int a, int c) { return seg_units(d[a].K) > seg_units(d[c].K); });
  int64_t units = 0, segs = 0;
  for (int i = 0; i < count; ++i) {
    const qb_act_desc& q = d[ord[i]];
    ActItem& t = b.item[i];
    t.x = q.x;
    t.xq = q.xq;
    t.act_scale = q.act_scale;
    t.rowsum = q.rowsum;
    t.M = q.M;
    t.unit_begin = units;
    t.seg_begin = segs;
    t.units_per_row = (int32_t)(q.K / 128);
    t.seg_units = seg_units(q.K);
    t.segs_per_row = (t.units_per_row + t.seg_units - 1) / t.seg_units;
    units += q.M * t.units_per_row;
    segs += q.M * t.segs_per_row;
  }
  b.units_total = units;
  b.segs_total = segs;
  b.keep_fraction = l2_keep_fraction(512.0 * (double)units);
  const int64_t seg_blocks = (segs + kActWarps - 1) / kActWarps;
  if constexpr (P == 1) {
    // A part of the device takes the two launches below, as does a launch that is refused for want of SMs: they need no
    // blocks resident together, neither a grid's nor a cluster's (the CTAs of a cluster need SMs of one GPC).
    const bool together = segs <= (int64_t)sm_count * (kActBlocksPerSm * kActWarps / 2) &&
                          segs <= kWsClusters * kActMaxCluster * 2 * kActWarps && stream_has_sms(stream, sm_count);
    b.units_per_block = 0;
    // With the GEMM behind it, one cluster of up to 8 CTAs (the portable size; 256 segments) against all blocks
    // resident and one word: M = 128 x 768 9.4 us, 14.3; 256 x 768 10.2, 14.3.  CTAs of at least 1, 4 or 16 warps take as
    // long as those of 8, to 0.3 us.
    if (together && segs <= kActMaxCluster * (kActMaxThreads / 32)) {
      const unsigned warps = (unsigned)std::max<int64_t>((segs + kActMaxCluster - 1) / kActMaxCluster, kActWarps);
      const unsigned ctas = (unsigned)((segs + warps - 1) / warps);
      const cudaError_t e = launch_kernel(act_fused_kernel<false>, ctas, warps * 32, 0, stream, ctas, false, b);
      if (!residency_refused(e)) {
        QB_CUDA_TRY(e);
        return QB_OK;
      }
    } else if (together) {
      // Several clusters while they need no more than half of the warps that the device holds, so that clusters of CTAs
      // of 8 or 16 warps find their place.  What they give is a launch less for a call that is waited for; in a row of
      // calls the two launches overlap their neighbours and draw level at about 768 segments of 1,024.  One linear (N = 768),
      // us, one launch / two; in a row: 320 x 1,024 12.4 / 13.0, 768 x 1,024 13.3 / 13.4, 1,024 x 768 13.1 / 12.7, 1,536 x 1,024
      // 14.5 / 14.2, 2,368 x 1,024 15.0 / 14.9; each waited for: 20.8 / 22.3, 20.9 / 22.4, 20.4 / 21.9, 22.2 / 23.3, 22.6 / 24.1.
      // A segment per warp for all the warps there are (one CTA a cluster, cooperative) was slower than two launches even
      // before these overlapped: 4,500 x 768 18.4 / 16.4; 1,000 x 4,096 26.4 / 24.6.
      const int64_t warps = segs <= kWsClusters * kActMaxCluster * kActWarps ? kActWarps : 2 * kActWarps;
      const unsigned clusters = (unsigned)((segs + warps * kActMaxCluster - 1) / (warps * kActMaxCluster));
      const cudaError_t e = launch_kernel(act_fused_kernel<true>, clusters * kActMaxCluster, (unsigned)warps * 32, 0, stream,
                                          kActMaxCluster, true, b);
      if (!residency_refused(e)) {
        QB_CUDA_TRY(e);
        return QB_OK;
      }
    }
  }
  // equal shares of whole batches of kSegUnits units per warp
  int64_t share = (units + cap - 1) / cap;
  share = (share + kSegUnits - 1) / kSegUnits * kSegUnits;
  b.units_per_block = share;
  QB_CUDA_TRY(launch_kernel<kMostL1>(act_absmax_kernel<P>, (unsigned)((units + share - 1) / share), kActThreads, 0, stream, 1, false, b));
  QB_CUDA_TRY(launch_kernel<kMostL1>(act_quantize_kernel<P>, (unsigned)std::min(seg_blocks, cap), kActThreads, 0, stream, 1, false, b));
  return QB_OK;
}

static qb_status validate_act(const char* who, const float* x, int64_t M, int64_t K, const int8_t* xq,
                              const float* act_scale, const int32_t* rowsum) {
  if (!x || !xq || !act_scale || !rowsum || M <= 0 || K <= 0 || M > QB_MAX_MN || K > QB_MAX_K) {
    set_last_error("%s: null pointer or size out of range (M=%lld K=%lld)", who, (long long)M, (long long)K);
    return QB_ERR_INVALID;
  }
  if (K % 128 != 0 || !aligned16(x) || !aligned16(xq)) {
    set_last_error("%s: K must be a multiple of 128 and x, xq 16-byte aligned", who);
    return QB_ERR_ALIGN;
  }
  return QB_OK;
}

}  // namespace qb

extern "C" qb_status qb_quantize_act(const float* x, int64_t M, int64_t K, int8_t* xq, float* act_scale,
                                     int32_t* rowsum, void* ws, size_t ws_bytes, void* cuda_stream) {
  qb_status st = qb::validate_act("qb_quantize_act", x, M, K, xq, act_scale, rowsum);
  if (st != QB_OK) return st;
  if (!ws || ws_bytes < qb::ws_bytes_needed(0)) {
    qb::set_last_error("qb_quantize_act: workspace null or too small");
    return QB_ERR_WORKSPACE;
  }
  int sms = 0;
  st = qb::require_sm100(&sms);
  if (st != QB_OK) return st;
  uint32_t* slot = reinterpret_cast<uint32_t*>(static_cast<char*>(ws) + qb::kWsActMaxOff);
  const qb_act_desc d{x, M, K, xq, act_scale, rowsum};
  return qb::launch_act_batch<1>(&d, 1, ws, slot, sms, (cudaStream_t)cuda_stream);
}

extern "C" qb_status qb_quantize_act_batch(const qb_act_desc* descs, int32_t count, void* ws, size_t ws_bytes,
                                           void* cuda_stream) {
  if (!descs || count <= 0) {
    qb::set_last_error("qb_quantize_act_batch: descs null or count <= 0");
    return QB_ERR_INVALID;
  }
  for (int i = 0; i < count; ++i) {
    qb_status st = qb::validate_act("qb_quantize_act_batch", descs[i].x, descs[i].M, descs[i].K, descs[i].xq,
                                    descs[i].act_scale, descs[i].rowsum);
    if (st != QB_OK) return st;
  }
  // max-abs slots of a launch: the head of the range area of the workspace
  if (!ws || ws_bytes < qb::kWsRangeOff + sizeof(uint32_t) * (size_t)qb::kMaxActBatch) {
    qb::set_last_error("qb_quantize_act_batch: workspace null or smaller than %zu bytes",
                       qb::kWsRangeOff + sizeof(uint32_t) * (size_t)qb::kMaxActBatch);
    return QB_ERR_WORKSPACE;
  }
  int sms = 0;
  qb_status st = qb::require_sm100(&sms);
  if (st != QB_OK) return st;
  uint32_t* slots = reinterpret_cast<uint32_t*>(static_cast<char*>(ws) + qb::kWsRangeOff);
  for (int i = 0; i < count; i += qb::kMaxActBatch) {
    const int n = count - i < qb::kMaxActBatch ? count - i : qb::kMaxActBatch;
    st = qb::launch_act_batch<qb::kMaxActBatch>(descs + i, n, ws, slots, sms, (cudaStream_t)cuda_stream);
    if (st != QB_OK) return st;
  }
  return QB_OK;
}

extern "C" int32_t qb_quantize_act_launch_count(int32_t count) {
  if (count <= 0) return 0;
  return 2 * ((count + qb::kMaxActBatch - 1) / qb::kMaxActBatch);
}
