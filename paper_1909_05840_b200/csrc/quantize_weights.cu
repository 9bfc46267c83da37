// qb_quantize_pack_weights(_batch): group-wise uniform quantizer Q (Section 3.3, Appendix A) and dense
// k-bit packing (Table 1 counts exactly k bits per weight), for one matrix or a batch of matrices.
//
// Three paths, chosen per matrix on the host (a unit is 128 consecutive elements of one row):
//   weight_regs_kernel   one read of W; any bit widths in one launch.  With the group's own [min, max]: groups
//                        of up to 288 units stay in the registers of one CTA between the range and the
//                        rounding, groups of up to 2,304 units in those of a thread-block cluster.  With
//                        caller-supplied ranges: groups of any size (nothing to reduce).
//   weight_ring_kernel   one read of W: own ranges of larger groups (a range per tensor, say) of up to eleven chunks of
//                        16 KB per SM (27 MB on 148), held in the shared memory and registers of the whole device.
//   two passes           own ranges of groups beyond that, or where the workspace has no room for the ring's
//                        slots, or where the stream has too few SMs for the ring's blocks at once.
//
// Two-pass path, first pass: the matrices of a launch are walked as one sequence of units (one float4
// per lane, fully coalesced; K % 128 == 0 so a unit never
// crosses a row).  Each warp owns a contiguous run of units, so it crosses few group (and matrix)
// boundaries: weight_range_kernel keeps a running min/max per lane, reduces over the warp when the group
// changes and publishes with atomicMax on order-preserving integer encodings in the workspace (block-level
// merge of the final partials first).  Second pass: weight_regs_kernel in its supplied-ranges form, reading
// those encodings (the matrix comes from L2 as far as L2 holds it).
#include <algorithm>
#include <atomic>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "mbar_wait.cuh"
#include "ptx.cuh"

namespace qb {

constexpr int kWqThreads = 256;
constexpr int kWqWarps = kWqThreads / 32;
constexpr int kMaxWeightBatch = 96;  // matrices per launch (descriptors travel as kernel parameters)

struct WeightItem {
  const float4* w;
  uint32_t* packed;
  float* delta;
  float* q0;
  const float* range_lo;
  const float* range_hi;
  int64_t unit_begin;      // index of the matrix's first unit in the launch
  int64_t units;           // N * K / 128
  int32_t units_per_row;   // K / 128
  int32_t rows_per_group;  // R
  int32_t group_begin;     // index of the matrix's first group in the launch's range tables
  int32_t pad;
};

struct WeightBatch {
  WeightItem item[kMaxWeightBatch];
  uint32_t* hi_enc;        // [groups of the launch] encoded maxima
  uint32_t* lo_inv;        // [groups of the launch] inverted encoded minima
  void* ws;
  int64_t units_total;
  int64_t units_per_warp;  // contiguous run per warp
  int32_t count;
  float keep_fraction;     // share of the input that L2 is asked to keep between the range pass and the next
};

// Position of a warp in the launch's unit sequence.
struct UnitWalk {
  int it;             // matrix
  int64_t u_local;    // unit inside the matrix
  int col_unit;       // unit inside the row
  int row_in_group;
  int g;              // group, numbered over the whole launch
  __device__ __forceinline__ void seek(const WeightBatch& b, int64_t u) {
    it = 0;
    while (it + 1 < b.count && u >= b.item[it + 1].unit_begin) ++it;
    enter(b, u - b.item[it].unit_begin);
  }
  __device__ __forceinline__ void enter(const WeightBatch& b, int64_t local) {
    const WeightItem& m = b.item[it];
    u_local = local;
    const int64_t row = local / m.units_per_row;
    col_unit = (int)(local - row * m.units_per_row);
    const int gl = (int)(row / m.rows_per_group);
    row_in_group = (int)(row - (int64_t)gl * m.rows_per_group);
    g = m.group_begin + gl;
  }
  // one unit forward; moves to the next matrix at the end of this one
  __device__ __forceinline__ void advance(const WeightBatch& b) {
    const WeightItem& m = b.item[it];
    ++u_local;
    if (++col_unit == m.units_per_row) {
      col_unit = 0;
      if (++row_in_group == m.rows_per_group) {
        row_in_group = 0;
        ++g;
      }
    }
    if (u_local == m.units && it + 1 < b.count) {
      ++it;
      enter(b, 0);
    }
  }
};

__device__ __forceinline__ void flush_range(uint32_t* __restrict__ hi_enc, uint32_t* __restrict__ lo_inv,
                                            int g, float lo, float hi) {
  // all lanes call; lane 0 publishes
  const uint32_t e_hi = __reduce_max_sync(0xffffffffu, float_to_ordered(hi));
  const uint32_t e_lo = __reduce_max_sync(0xffffffffu, ~float_to_ordered(lo));
  if ((threadIdx.x & 31) == 0) {
    atomicMax(hi_enc + g, e_hi);
    atomicMax(lo_inv + g, e_lo);
  }
}

__global__ void __launch_bounds__(kWqThreads)
weight_range_kernel(const __grid_constant__ WeightBatch b) {
  const int lane = threadIdx.x & 31;
  pdl_begin();
  const uint64_t pol = policy_evict_last(b.keep_fraction);
  const int warp_in_block = threadIdx.x >> 5;
  const int64_t gwarp = (int64_t)blockIdx.x * kWqWarps + warp_in_block;
  int64_t u = gwarp * b.units_per_warp;
  int64_t u_end = u + b.units_per_warp;
  if (u_end > b.units_total) u_end = b.units_total;

  __shared__ int s_group[kWqWarps];
  __shared__ uint32_t s_hi[kWqWarps], s_lo[kWqWarps];

  const float kInf = __int_as_float(0x7f800000);
  float lo = kInf, hi = -kInf;
  uint32_t absmax = 0;
  int cur_g = -1;
  if (u < u_end) {
    UnitWalk pos;
    pos.seek(b, u);
    cur_g = pos.g;
    while (u < u_end) {
      // up to four units of the current matrix in flight
      const WeightItem& m = b.item[pos.it];
      const int nload = (int)min(min((int64_t)4, u_end - u), m.units - pos.u_local);
      float4 v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (j < nload) v[j] = ldg_policy(m.w + (pos.u_local + j) * 32 + lane, pol);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (j < nload) {
          if (pos.g != cur_g) {  // warp-uniform
            flush_range(b.hi_enc, b.lo_inv, cur_g, lo, hi);
            cur_g = pos.g;
            lo = kInf;
            hi = -kInf;
          }
          lo = fminf(fminf(lo, v[j].x), fminf(v[j].y, fminf(v[j].z, v[j].w)));
          hi = fmaxf(fmaxf(hi, v[j].x), fmaxf(v[j].y, fmaxf(v[j].z, v[j].w)));
          absmax = max(absmax, max(max(__float_as_uint(v[j].x) << 1, __float_as_uint(v[j].y) << 1),
                                   max(__float_as_uint(v[j].z) << 1, __float_as_uint(v[j].w) << 1)));
          pos.advance(b);
        }
      }
      u += nload;
    }
  }
  // NaN / Inf: exponent all ones survives the shift as >= 0xff000000
  absmax = __reduce_max_sync(0xffffffffu, absmax);
  if (lane == 0 && absmax >= 0xff000000u) report_status(b.ws, QB_ERR_NONFINITE);

  // final partial of each warp: merge equal groups inside the block, then one pair of atomics each
  const uint32_t e_hi = __reduce_max_sync(0xffffffffu, float_to_ordered(hi));
  const uint32_t e_lo = __reduce_max_sync(0xffffffffu, ~float_to_ordered(lo));
  if (lane == 0) {
    s_group[warp_in_block] = cur_g;
    s_hi[warp_in_block] = e_hi;
    s_lo[warp_in_block] = e_lo;
  }
  __syncthreads();
  if (threadIdx.x < kWqWarps) {
    const int my_g = s_group[threadIdx.x];
    bool leader = my_g >= 0;
    for (int j = 0; j < (int)threadIdx.x; ++j) leader = leader && (s_group[j] != my_g);
    if (leader) {
      uint32_t mh = s_hi[threadIdx.x], ml = s_lo[threadIdx.x];
      for (int j = threadIdx.x + 1; j < kWqWarps; ++j)
        if (s_group[j] == my_g) {
          mh = max(mh, s_hi[j]);
          ml = max(ml, s_lo[j]);
        }
      atomicMax(b.hi_enc + my_g, mh);
      atomicMax(b.lo_inv + my_g, ml);
    }
  }
}

struct GroupParams {
  float lo, hi, inv;
};

// Range [lo, hi] of group g -> (q0, qmax, 1/Delta); lane-uniform.  Publishes Delta and q0 if asked.
// A caller-supplied range must be finite and ordered; a constant group gets Delta = 1, all codes 0.
__device__ __forceinline__ GroupParams finish_group(float lo, float hi, bool from_caller, int bits_levels, int g,
                                                    float* __restrict__ delta, float* __restrict__ q0,
                                                    bool publish, void* ws) {
  GroupParams p;
  p.lo = lo;
  p.hi = hi;
  if (from_caller) {
    const bool bad = !(fabsf(p.lo) <= 3.402823466e38f) || !(fabsf(p.hi) <= 3.402823466e38f) || p.hi < p.lo;
    if (bad) {
      if (publish) report_status(ws, QB_ERR_NONFINITE);
      p.lo = 0.0f;
      p.hi = 0.0f;
    }
  }
  float d = __fdiv_rn(__fsub_rn(p.hi, p.lo), (float)bits_levels);
  float inv = __fdiv_rn(1.0f, d);
  if (!(d > 0.0f) || !(inv <= 3.402823466e38f)) {  // constant group
    d = 1.0f;
    inv = 1.0f;
    p.hi = p.lo;
  }
  p.inv = inv;
  if (publish) {
    delta[g] = d;
    q0[g] = p.lo;
  }
  return p;
}

// Delta of a finished group as finish_group publishes it (a constant group comes back with hi == lo: Delta = 1).
__device__ __forceinline__ float group_step(const GroupParams& gp, int bits_levels) {
  const float d = __fdiv_rn(__fsub_rn(gp.hi, gp.lo), (float)bits_levels);
  return d > 0.0f ? d : 1.0f;
}

// ---- straight-through backward (quantization-aware fine-tuning) ----------------------------------------
// Backward (straight-through estimator): the gradient passes where Clamp passes X (lo_g <= x <= hi_g).
// Memory-bound, 12 B per weight; a matrix of a base model is 28 MB, 4.4 us of bandwidth, so what counts is that all
// of it is in flight at once: a warp takes four units (eight 512-byte loads) and works out their group with
// one division.  A fine-tuning step over four BERT-base layers
// (113 MB of weights fake-quantized in one call, then one backward call per matrix): 144.2 -> 119.3 us.
constexpr int kSteUnits = 4;
__global__ void __launch_bounds__(256)
ste_backward_kernel(const float4* grad_q, const float4* w, int64_t units, uint32_t units_per_group,
                    const float* lo, const float* hi, float4* grad_w) {
  pdl_begin();
  const int lane = threadIdx.x & 31;
  const int64_t step = (int64_t)gridDim.x * 8 * kSteUnits;
  for (int64_t u = ((int64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * kSteUnits; u < units; u += step) {
    const int n = (int)min(units - u, (int64_t)kSteUnits);
    float4 x[kSteUnits], g[kSteUnits];
#pragma unroll
    for (int j = 0; j < kSteUnits; ++j)
      if (j < n) {
        x[j] = w[(u + j) * 32 + lane];
        g[j] = grad_q[(u + j) * 32 + lane];  // grad_w may be the same buffer
      }
    uint32_t group = (uint32_t)u / units_per_group, in_group = (uint32_t)u - group * units_per_group;
    float l = lo[group], h = hi[group];
#pragma unroll
    for (int j = 0; j < kSteUnits; ++j)
      if (j < n) {
        if (in_group == units_per_group) {
          in_group = 0;
          ++group;
          l = lo[group];
          h = hi[group];
        }
        ++in_group;
        float4 r = g[j];
        r.x = (x[j].x >= l && x[j].x <= h) ? r.x : 0.0f;
        r.y = (x[j].y >= l && x[j].y <= h) ? r.y : 0.0f;
        r.z = (x[j].z >= l && x[j].z <= h) ? r.z : 0.0f;
        r.w = (x[j].w >= l && x[j].w <= h) ? r.w : 0.0f;
        grad_w[(u + j) * 32 + lane] = r;
      }
  }
}

// ---- register-resident path ---------------------------------------------------------------------------
// Groups of up to 288 units (36,864 weights: all of BERT's matrices at 128 groups, and anything finer) are
// read from HBM once and stay in registers between the range and the rounding: 16 warps per CTA, one CTA
// per SM, every thread holds up to 18 float4 (one warp: 18 consecutive units, 9 KB, all loads in flight at
// once).  A matrix is served in one of two shapes:
//   * teams: a group is cut into contiguous slices over W = 1, 2, 4, 8 or 16 warps (the smallest W whose
//     slices fit), the team agrees on the range through shared memory and a named barrier;
//   * several groups per warp (groups of at most 9 units: one range per output row, say): a warp holds as
//     many whole consecutive groups as fit and reduces them one after the other.
// A CTA item is 16 warps' worth of consecutive groups of one matrix; the items of all matrices of a launch
// (largest items first, any mix of bit widths: the width is a field of the matrix) form one list that the
// CTAs stride over, so a mixed-precision stack is one launch.  Codes go through a 768-byte staging area per
// warp in blocks of six units: the 4k-bit fields laid down in element order are the packed stream for
// k = 2, 4, 8 (copied out with 16-byte stores) and are regrouped (eight 12-bit fields -> three words) for
// k = 3.  The kernel's other forms (template parameters, below): a thread-block cluster per group for
// groups of up to 2,304 units; fp32 Q(w) instead of packed words (fake quantization); supplied ranges
// (the caller's, or the range pass's for groups too large for a cluster), where nothing is reduced and
// the rounding clamps.
constexpr int kRgUnits = 18;                       // float4 per thread
constexpr int kRgBlock = 6;                        // units per staging block
constexpr int kRgWarps = 16;
constexpr int kRgThreads = 32 * kRgWarps;
constexpr int kRgMaxGroupUnits = kRgUnits * kRgWarps;  // 288
constexpr int kRgMaxBatch = 96;                    // matrices per launch

struct RegsItem {
  const float4* w;
  uint32_t* packed;
  float* delta;
  float* q0;
  int32_t ug;               // units per group
  int32_t groups;
  int32_t item_begin;       // first CTA item of this matrix in the launch's list
  int32_t groups_per_item;  // (16 / W) * groups_per_warp
  int16_t team_warps;       // W
  int16_t groups_per_warp;  // > 1 only with W = 1
  int16_t slice_units;      // units per warp of a team: ceil(ug / W)
  int16_t bits;
  const float* range_lo;    // caller-supplied ranges (the kernel that clamps), else null
  const float* range_hi;
  int32_t chunks;           // supplied ranges only: a group of more than 288 units is cut into this many items
  int32_t encoded;          // supplied ranges are the range pass's order-preserving encodings (max, inverted min)
};

struct RegsBatch {
  RegsItem item[kRgMaxBatch];
  void* ws;
  int32_t total_items;
  int32_t count;
};

// What one warp holds of a CTA item.
struct RegsSlice {
  const float4* src;  // first unit of the slice (+ lane)
  int32_t n;          // units held (0: nothing to do)
  int32_t it;         // matrix
  int32_t first_group;
  int32_t ng;         // groups (several-groups shape), 0 or 1 (teams)
  int32_t first_unit; // of the slice inside its group (teams)
};

// Four codes of one float4 as a 4k-bit field in the low bits of the result (k < 8: bits from 22 up are
// left over from the rounding constant and are dropped by the narrow store that follows).
template <int BITS, bool CLAMP>
__device__ __forceinline__ uint32_t quant_field_open(float4 v, const float lo, const float inv, const float hi) {
  constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23: adding it rounds to an integer, half to even
  if (CLAMP) {  // Clamp(X, q0, qmax): a caller's range may leave weights outside
    v.x = fminf(fmaxf(v.x, lo), hi);
    v.y = fminf(fmaxf(v.y, lo), hi);
    v.z = fminf(fmaxf(v.z, lo), hi);
    v.w = fminf(fmaxf(v.w, lo), hi);
  }
  // Two lanes of fp32 per instruction (sub, mul, then the rounding add).  The add is written as a fused
  // multiply-add with 1.0: a packed mul followed by a packed add gets contracted into one fused operation,
  // which rounds the exact product instead of the rounded one and lands on the other side of a tie.
  uint32_t b0, b1, b2, b3;
  asm("{\n\t.reg .b64 p0, p1, l2, i2, m2, o2;\n\t"
      "mov.b64 p0, {%4, %5};\n\tmov.b64 p1, {%6, %7};\n\t"
      "mov.b64 l2, {%8, %8};\n\tmov.b64 i2, {%9, %9};\n\tmov.b64 m2, {%10, %10};\n\tmov.b64 o2, {%11, %11};\n\t"
      "sub.rn.f32x2 p0, p0, l2;\n\tsub.rn.f32x2 p1, p1, l2;\n\t"
      "mul.rn.f32x2 p0, p0, i2;\n\tmul.rn.f32x2 p1, p1, i2;\n\t"
      "fma.rn.f32x2 p0, p0, o2, m2;\n\tfma.rn.f32x2 p1, p1, o2, m2;\n\t"
      "mov.b64 {%0, %1}, p0;\n\tmov.b64 {%2, %3}, p1;\n\t}"
      : "=r"(b0), "=r"(b1), "=r"(b2), "=r"(b3)
      : "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "f"(lo), "f"(inv), "f"(kMagic), "f"(1.0f));
  if constexpr (BITS == 8) {
    return __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410);
  } else {
    return b0 + (b1 << BITS) + (b2 << (2 * BITS)) + (b3 << (3 * BITS));
  }
}

// Parameters of the group a warp is rounding: q0, 1/Delta, and Delta (fake quantization only).
struct RgGroup {
  float lo, inv, d, hi;  // hi: the kernel that clamps only
};
// Several groups per warp: lane gi holds the parameters of the warp's group gi.
__device__ __forceinline__ void rg_next_group(RgGroup& cur, const RgGroup& mine, int& gi, int& next_start, const int ug) {
  cur.lo = __shfl_sync(0xffffffffu, mine.lo, gi);
  cur.inv = __shfl_sync(0xffffffffu, mine.inv, gi);
  cur.d = __shfl_sync(0xffffffffu, mine.d, gi);
  cur.hi = __shfl_sync(0xffffffffu, mine.hi, gi);
  ++gi;
  next_start += ug;
}

// Item `i` of a 3-bit staging area: 32 codes = eight 12-bit fields held in 16-bit cells -> three words.
__device__ __forceinline__ void store_3bit_item(const uint8_t* stg, uint32_t* __restrict__ out, const int i) {
  const uint4 q = reinterpret_cast<const uint4*>(stg)[i];
  const uint32_t f0 = q.x & 0xffffu, f1 = q.x >> 16, f2 = q.y & 0xffffu, f3 = q.y >> 16;
  const uint32_t f4 = q.z & 0xffffu, f5 = q.z >> 16, f6 = q.w & 0xffffu, f7 = q.w >> 16;
  uint32_t* o3 = out + i * 3;
  o3[0] = f0 | (f1 << 12) | (f2 << 24);
  o3[1] = (f2 >> 8) | (f3 << 4) | (f4 << 16) | (f5 << 28);
  o3[2] = (f5 >> 4) | (f6 << 8) | (f7 << 20);
}

// One staging block (units BLK * 6 ... of the slice): fields into the warp's staging area, then out.
template <int BITS, int BLK, bool MULTI, bool CLAMP>
__device__ __forceinline__ void regs_pack_block(float4 (&v)[kRgUnits], const int n, RgGroup& cur, const RgGroup& mine,
                                                int& gi, int& next_start, const int ug, uint8_t* stg,
                                                uint32_t* __restrict__ out, const int lane,
                                                const float4* next_src, const int next_n) {
#pragma unroll
  for (int jj = 0; jj < kRgBlock; ++jj) {
    const int j = BLK * kRgBlock + jj;
    if (j < n) {
      if (MULTI) {
        if (j == next_start) rg_next_group(cur, mine, gi, next_start, ug);  // warp-uniform: the warp's next group begins
      }
      const uint32_t f = quant_field_open<BITS, CLAMP>(v[j], cur.lo, cur.inv, cur.hi);
      const int fi = jj * 32 + lane;  // field index = element index / 4 inside the block
      if (BITS == 8) reinterpret_cast<uint32_t*>(stg)[fi] = f;
      if (BITS == 4 || BITS == 3) reinterpret_cast<uint16_t*>(stg)[fi] = (uint16_t)f;
      if (BITS == 2) stg[fi] = (uint8_t)f;
    }
  }
  // the registers of this block are free: the same units of the warp's next slice start their way here
#pragma unroll
  for (int jj = 0; jj < kRgBlock; ++jj) {
    const int j = BLK * kRgBlock + jj;
    if (j < next_n) v[j] = next_src[j * 32];
  }
  __syncwarp();
  const int nu = min(kRgBlock, n - BLK * kRgBlock);
  uint32_t* const o = out + BLK * kRgBlock * 4 * BITS;
  if (BITS == 3) {
    if (lane < 4 * nu) store_3bit_item(stg, o, lane);  // four items per unit
  } else {
    const int n16 = nu * BITS;  // 16 * BITS bytes per unit
    const uint4* pk = reinterpret_cast<const uint4*>(stg);
    uint4* o4 = reinterpret_cast<uint4*>(o);
#pragma unroll
    for (int r = 0; r < (kRgBlock * BITS + 31) / 32; ++r) {
      const int i = r * 32 + lane;
      if (i < n16) o4[i] = pk[i];
    }
  }
  __syncwarp();  // the staging area is free again
}

// Fake quantization (Appendix A, forward of the fine-tuning step): Q(w) = Delta * code + q0 as fp32, written
// where the packed words would go.  code = (t + 1.5 * 2^23) - 1.5 * 2^23 is the rounded product as a float
// (exact), then one fused multiply-add; packed two lanes wide like the rounding itself.
template <bool CLAMP>
__device__ __forceinline__ float4 fake_quant4(float4 v, const RgGroup& g) {
  constexpr float kMagic = 12582912.0f;
  float4 q;
  if (CLAMP) {
    v.x = fminf(fmaxf(v.x, g.lo), g.hi);
    v.y = fminf(fmaxf(v.y, g.lo), g.hi);
    v.z = fminf(fmaxf(v.z, g.lo), g.hi);
    v.w = fminf(fmaxf(v.w, g.lo), g.hi);
  }
  asm("{\n\t.reg .b64 p0, p1, l2, i2, m2, o2, d2;\n\t"
      "mov.b64 p0, {%4, %5};\n\tmov.b64 p1, {%6, %7};\n\t"
      "mov.b64 l2, {%8, %8};\n\tmov.b64 i2, {%9, %9};\n\tmov.b64 m2, {%10, %10};\n\tmov.b64 o2, {%11, %11};\n\t"
      "mov.b64 d2, {%12, %12};\n\t"
      "sub.rn.f32x2 p0, p0, l2;\n\tsub.rn.f32x2 p1, p1, l2;\n\t"
      "mul.rn.f32x2 p0, p0, i2;\n\tmul.rn.f32x2 p1, p1, i2;\n\t"
      "fma.rn.f32x2 p0, p0, o2, m2;\n\tfma.rn.f32x2 p1, p1, o2, m2;\n\t"
      "sub.rn.f32x2 p0, p0, m2;\n\tsub.rn.f32x2 p1, p1, m2;\n\t"
      "fma.rn.f32x2 p0, d2, p0, l2;\n\tfma.rn.f32x2 p1, d2, p1, l2;\n\t"
      "mov.b64 {%0, %1}, p0;\n\tmov.b64 {%2, %3}, p1;\n\t}"
      : "=f"(q.x), "=f"(q.y), "=f"(q.z), "=f"(q.w)
      : "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "f"(g.lo), "f"(g.inv), "f"(kMagic), "f"(1.0f), "f"(g.d));
  return q;
}

template <int BLK, bool MULTI, bool CLAMP>
__device__ __forceinline__ void regs_fake_block(float4 (&v)[kRgUnits], const int n, RgGroup& cur, const RgGroup& mine,
                                                int& gi, int& next_start, const int ug, float4* __restrict__ out,
                                                const float4* next_src, const int next_n) {
#pragma unroll
  for (int jj = 0; jj < kRgBlock; ++jj) {
    const int j = BLK * kRgBlock + jj;
    if (j < n) {
      if (MULTI) {
        if (j == next_start) rg_next_group(cur, mine, gi, next_start, ug);
      }
      out[j * 32] = fake_quant4<CLAMP>(v[j], cur);
    }
    if (j < next_n) v[j] = next_src[j * 32];
  }
}

template <int BLK, bool MULTI, bool FAKE, bool CLAMP>
__device__ __forceinline__ void regs_pack_block_any(const int bits, float4 (&v)[kRgUnits], const int n, RgGroup& cur,
                                                    const RgGroup& mine, int& gi, int& next_start, const int ug,
                                                    uint8_t* stg, uint32_t* __restrict__ out, const int lane,
                                                    const float4* next_src, const int next_n) {
  if (BLK * kRgBlock >= n) {  // nothing of this slice here: only the next slice's loads
#pragma unroll
    for (int jj = 0; jj < kRgBlock; ++jj) {
      const int j = BLK * kRgBlock + jj;
      if (j < next_n) v[j] = next_src[j * 32];
    }
    return;
  }
  if (FAKE) {
    regs_fake_block<BLK, MULTI, CLAMP>(v, n, cur, mine, gi, next_start, ug, reinterpret_cast<float4*>(out) + lane, next_src, next_n);
    return;
  }
  switch (bits) {  // CTA-uniform
    case 2: regs_pack_block<2, BLK, MULTI, CLAMP>(v, n, cur, mine, gi, next_start, ug, stg, out, lane, next_src, next_n); break;
    case 3: regs_pack_block<3, BLK, MULTI, CLAMP>(v, n, cur, mine, gi, next_start, ug, stg, out, lane, next_src, next_n); break;
    case 4: regs_pack_block<4, BLK, MULTI, CLAMP>(v, n, cur, mine, gi, next_start, ug, stg, out, lane, next_src, next_n); break;
    default: regs_pack_block<8, BLK, MULTI, CLAMP>(v, n, cur, mine, gi, next_start, ug, stg, out, lane, next_src, next_n); break;
  }
}

template <bool CLUSTER>
__device__ __forceinline__ RegsSlice regs_slice(const RegsBatch& b, const int id, int& it, const int warp,
                                                const int lane, const int crank) {
  RegsSlice s;
  s.n = 0;
  s.it = it;
  s.src = nullptr;
  s.first_group = 0;
  s.ng = 0;
  s.first_unit = 0;
  if (id >= b.total_items) return s;
  while (it + 1 < b.count && id >= b.item[it + 1].item_begin) ++it;
  const RegsItem& m = b.item[it];
  s.it = it;
  if (CLUSTER) {
    // one group per cluster item, cut into slices over the 16 warps of each of the cluster's CTAs
    s.first_group = id - m.item_begin;
    s.ng = 1;
    s.first_unit = (crank * kRgWarps + warp) * m.slice_units;
    s.n = min(max(m.ug - s.first_unit, 0), (int)m.slice_units);
  } else {
    const int W = m.team_warps;
    const int team = warp / W, tw = warp - team * W;
    if (m.chunks > 1) {
      // caller-supplied ranges, a group larger than a CTA's registers: no reduction ties the group together,
      // so it is cut into items of 288 units
      const int local = id - m.item_begin;
      s.first_group = local / m.chunks;
      s.ng = 1;
      s.first_unit = (local - s.first_group * m.chunks) * kRgMaxGroupUnits + warp * kRgUnits;
      s.n = min(max(m.ug - s.first_unit, 0), kRgUnits);
      s.src = m.w + ((int64_t)s.first_group * m.ug + s.first_unit) * 32 + lane;
      return s;
    }
    s.first_group = (id - m.item_begin) * m.groups_per_item + team * m.groups_per_warp;
    s.ng = min(max(m.groups - s.first_group, 0), (int)m.groups_per_warp);
    if (s.ng > 0) {
      if (m.groups_per_warp > 1) {
        s.n = s.ng * m.ug;
      } else {
        s.first_unit = tw * m.slice_units;
        s.n = min(max(m.ug - s.first_unit, 0), (int)m.slice_units);
      }
    }
  }
  s.src = m.w + ((int64_t)s.first_group * m.ug + s.first_unit) * 32 + lane;
  return s;
}

__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}

// Supplied range of group g: the caller's floats, or the encodings the range pass of the two-pass path left.
__device__ __forceinline__ GroupParams supplied_group(const RegsItem& m, int g, int L, bool publish, void* ws) {
  if (m.encoded) {
    const float lo = ordered_to_float(~reinterpret_cast<const uint32_t*>(m.range_lo)[g]);
    const float hi = ordered_to_float(reinterpret_cast<const uint32_t*>(m.range_hi)[g]);
    return finish_group(lo, hi, false, L, g, m.delta, m.q0, publish, ws);
  }
  return finish_group(m.range_lo[g], m.range_hi[g], true, L, g, m.delta, m.q0, publish, ws);
}

// CLUSTER = false: the kernel described above.  CLUSTER = true: groups of 289 to 2,304 units; a thread-block
// cluster of 2 to 8 CTAs (the launch's cluster size) holds one group, every CTA reduces its 16 slices,
// writes its range into every CTA's shared memory and the cluster's barrier publishes them.  Every CTA of a
// cluster runs the same number of items, so the barriers pair up; the last one also keeps a CTA's shared
// memory alive until no peer writes to it any more.
// FAKE: the fp32 fake-quantized matrix is written instead of packed words (`packed` of the item points to it).
// CLAMP: the ranges are supplied (`range_lo`, `range_hi` of the item: the caller's, or what the range pass of
// the two-pass path found): no reduction and no exchange, the weights are clamped into the range, and the pass
// over the registers only looks for NaN and Inf.
template <bool CLUSTER, bool FAKE, bool CLAMP>
__global__ void __launch_bounds__(kRgThreads, 1)
weight_regs_kernel(const __grid_constant__ RegsBatch b) {
  __shared__ __align__(16) uint8_t s_stage[kRgWarps][kRgBlock * 128];
  __shared__ uint32_t s_hi[2][kRgWarps], s_lo[2][kRgWarps];
  __shared__ uint32_t x_hi[2][8], x_lo[2][8];  // CLUSTER: the ranges of the cluster's CTAs
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t* const stg = s_stage[warp];
  const float kInf = __int_as_float(0x7f800000);
  const int csize = CLUSTER ? (int)cluster_size() : 1;
  const int crank = CLUSTER ? (int)ptx::cluster_ctarank() : 0;
  const int id0 = (int)blockIdx.x / csize, stride = (int)gridDim.x / csize;  // items go to clusters
  int it = 0, prev_it = 0;
  float4 v[kRgUnits];
  if (CLUSTER) ptx::cluster_sync_all();  // every CTA has started: its shared memory may be written to
  pdl_begin();
  RegsSlice s = regs_slice<CLUSTER>(b, id0, it, warp, lane, crank);
#pragma unroll
  for (int j = 0; j < kRgUnits; ++j)
    if (j < s.n) v[j] = s.src[j * 32];
  for (int id = id0, round = 0; id < b.total_items; id += stride, ++round) {
    const RegsItem& m = b.item[s.it];
    // The exchange buffers below are double-buffered per run of items with the same teams; when the
    // matrix (and with it, possibly, the team size) changes, every warp of the CTA passes here first.
    if (!CLUSTER && s.it != prev_it) __syncthreads();
    prev_it = s.it;
    const int n = s.n;
    // the warp's slice of the CTA's next item: its loads are issued as the registers come free below
    const RegsSlice nx = regs_slice<CLUSTER>(b, id + stride, it, warp, lane, crank);
    const int W = m.team_warps;
    const int bits = m.bits;
    const int L = (1 << bits) - 1;
    // first output word of the slice: 4k packed words per unit, or the unit's 128 floats
    uint32_t* const out = m.packed + ((int64_t)s.first_group * m.ug + s.first_unit) * (FAKE ? 128 : 4 * bits);
    if (!CLUSTER && m.groups_per_warp > 1) {
      // ---- several whole groups in this warp ----
      const int ug = m.ug;
      float lo = kInf, hi = -kInf;
      uint32_t my_hi = 0, my_lo = 0;
      int end = ug, gi = 0;
#pragma unroll
      for (int j = 0; j < kRgUnits; ++j) {
        if (j < n) {
          lo = min3_nan(min3_nan(lo, v[j].x, v[j].y), v[j].z, v[j].w);
          hi = max3_nan(max3_nan(hi, v[j].x, v[j].y), v[j].z, v[j].w);
          if (!CLAMP && j + 1 == end) {  // warp-uniform
            const uint32_t e_hi = __reduce_max_sync(0xffffffffu, float_to_ordered(hi));
            const uint32_t e_lo = __reduce_max_sync(0xffffffffu, ~float_to_ordered(lo));
            if (lane == gi) {
              my_hi = e_hi;
              my_lo = e_lo;
            }
            ++gi;
            end += ug;
            lo = kInf;
            hi = -kInf;
          }
        }
      }
      // lane i finishes group i of the warp
      RgGroup mine{0.0f, 1.0f, 1.0f, 0.0f};
      if (CLAMP) {
        // hi / lo hold this lane's running extremes over all of the warp's groups: NaN or Inf anywhere shows
        if (__any_sync(0xffffffffu, !(fabsf(hi) <= 3.402823466e38f && fabsf(lo) <= 3.402823466e38f)) && lane == 0 && n > 0)
          report_status(b.ws, QB_ERR_NONFINITE);
      }
      if (lane < s.ng) {
        GroupParams gp;
        if (CLAMP) {
          gp = supplied_group(m, s.first_group + lane, L, true, b.ws);
        } else {
          const float g_hi = ordered_to_float(my_hi);
          const float g_lo = ordered_to_float(~my_lo);
          if (!(fabsf(g_hi) <= 3.402823466e38f && fabsf(g_lo) <= 3.402823466e38f)) report_status(b.ws, QB_ERR_NONFINITE);
          gp = finish_group(g_lo, g_hi, false, L, s.first_group + lane, m.delta, m.q0, true, b.ws);
        }
        mine.lo = gp.lo;
        mine.inv = gp.inv;
        mine.d = group_step(gp, L);
        mine.hi = gp.hi;
      }
      RgGroup cur{0.0f, 1.0f, 1.0f, 0.0f};
      int next_start = 0;
      gi = 0;
      regs_pack_block_any<0, true, FAKE, CLAMP>(bits, v, n, cur, mine, gi, next_start, ug, stg, out, lane, nx.src, nx.n);
      regs_pack_block_any<1, true, FAKE, CLAMP>(bits, v, n, cur, mine, gi, next_start, ug, stg, out, lane, nx.src, nx.n);
      regs_pack_block_any<2, true, FAKE, CLAMP>(bits, v, n, cur, mine, gi, next_start, ug, stg, out, lane, nx.src, nx.n);
    } else if (s.ng > 0) {
      // ---- a slice of one group (team-uniform: every warp of the team is here) ----
      float lo = kInf, hi = -kInf;
#pragma unroll
      for (int j = 0; j < kRgUnits; ++j) {
        if (j < n) {
          lo = min3_nan(min3_nan(lo, v[j].x, v[j].y), v[j].z, v[j].w);
          hi = max3_nan(max3_nan(hi, v[j].x, v[j].y), v[j].z, v[j].w);
        }
      }
      // NaN anywhere makes hi NaN (encoded above every number); Inf shows as hi = +Inf or lo = -Inf
      uint32_t e_hi = 0, e_lo = 0;
      if (!CLAMP) {
        e_hi = __reduce_max_sync(0xffffffffu, float_to_ordered(hi));
        e_lo = __reduce_max_sync(0xffffffffu, ~float_to_ordered(lo));
      }
      if (CLAMP) {
        if (__any_sync(0xffffffffu, !(fabsf(hi) <= 3.402823466e38f && fabsf(lo) <= 3.402823466e38f)) && lane == 0 && n > 0)
          report_status(b.ws, QB_ERR_NONFINITE);
      } else if (CLUSTER) {
        const int flip = round & 1;
        if (lane == 0) {
          s_hi[flip][warp] = e_hi;
          s_lo[flip][warp] = e_lo;
        }
        __syncthreads();
        e_hi = __reduce_max_sync(0xffffffffu, lane < kRgWarps ? s_hi[flip][lane] : 0u);
        e_lo = __reduce_max_sync(0xffffffffu, lane < kRgWarps ? s_lo[flip][lane] : 0u);
        if (warp == 0 && lane < csize) {  // this CTA's range into slot `crank` of CTA `lane`
          ptx::st_cluster_u32(ptx::map_to_cta(ptx::smem_u32(&x_hi[flip][crank]), (uint32_t)lane), e_hi);
          ptx::st_cluster_u32(ptx::map_to_cta(ptx::smem_u32(&x_lo[flip][crank]), (uint32_t)lane), e_lo);
        }
        ptx::cluster_sync_all();
        e_hi = __reduce_max_sync(0xffffffffu, lane < csize ? x_hi[flip][lane] : 0u);
        e_lo = __reduce_max_sync(0xffffffffu, lane < csize ? x_lo[flip][lane] : 0u);
      } else if (W > 1) {
        const int flip = round & 1;
        const int team0 = warp - (warp % W);  // first warp of the team
        if (lane == 0) {
          s_hi[flip][warp] = e_hi;
          s_lo[flip][warp] = e_lo;
        }
        asm volatile("bar.sync %0, %1;" ::"r"(1 + team0 / W), "r"(32 * W) : "memory");
        const uint32_t vh = lane < W ? s_hi[flip][team0 + lane] : 0u;
        const uint32_t vl = lane < W ? s_lo[flip][team0 + lane] : 0u;
        e_hi = __reduce_max_sync(0xffffffffu, vh);
        e_lo = __reduce_max_sync(0xffffffffu, vl);
      }
      const bool publish = s.first_unit == 0 && lane == 0;
      GroupParams gp;
      if (CLAMP) {
        gp = supplied_group(m, s.first_group, L, publish, b.ws);
      } else {
        const float g_hi = ordered_to_float(e_hi);
        const float g_lo = ordered_to_float(~e_lo);
        if (publish && !(fabsf(g_hi) <= 3.402823466e38f && fabsf(g_lo) <= 3.402823466e38f))
          report_status(b.ws, QB_ERR_NONFINITE);
        gp = finish_group(g_lo, g_hi, false, L, s.first_group, m.delta, m.q0, publish, b.ws);
      }
      RgGroup cur{gp.lo, gp.inv, group_step(gp, L), gp.hi};
      const RgGroup mine{0.0f, 1.0f, 1.0f, 0.0f};
      int gi = 0, next_start = -1;
      regs_pack_block_any<0, false, FAKE, CLAMP>(bits, v, n, cur, mine, gi, next_start, 0, stg, out, lane, nx.src, nx.n);
      regs_pack_block_any<1, false, FAKE, CLAMP>(bits, v, n, cur, mine, gi, next_start, 0, stg, out, lane, nx.src, nx.n);
      regs_pack_block_any<2, false, FAKE, CLAMP>(bits, v, n, cur, mine, gi, next_start, 0, stg, out, lane, nx.src, nx.n);
    } else {
      // nothing of this item here (a last item with fewer groups than teams): only the next slice's loads
#pragma unroll
      for (int j = 0; j < kRgUnits; ++j)
        if (j < nx.n) v[j] = nx.src[j * 32];
    }
    s = nx;
  }
  if (CLUSTER) ptx::cluster_sync_all();
}

// ---- shared-memory ring path ------------------------------------------------------------------------------
// Groups too large for a cluster's registers (one range per matrix, say), read once: one persistent CTA per SM
// (cooperative launch), every group cut into chunks of 32 units that are dealt round-robin, so that a group of
// 9 MB is spread over all SMs and its range is known a few chunks after its first chunk was loaded.  A chunk
// stays in a CTA's ring of twelve 16 KB stages, then in the registers of a rounding team, until it is:
//   warp 0         brings chunks in with cp.async.bulk, as far ahead as stages are free, and leaves beside each
//                  what the others need to know of it (the one place where the deal is worked out per chunk)
//   warps 1..4     range: every warp reduces a quarter of each chunk, keeps the extremes over the CTA's run of
//                  chunks of one group, and hands them over when the run ends
//   warps 5..12    agents take the CTA's runs in turn: put the run's range into the CTA's slot of the group's
//                  table, wait until the slots of all CTAs that hold a part of the group are in, reduce them,
//                  leave the group's parameters in shared memory.  Eight agents keep eight runs under way.
//   warps 13..28   rounding: four teams of four warps take every fourth chunk into registers, which frees the
//                  stage, wait for the group's parameters, round and pack (or fake-quantize)
// Nobody waits for a later chunk of its own CTA's list, and a group may not span more rounds of the deal than
// a CTA holds chunks (sixteen), so the loads and ranges that a team waits for never depend on that team.
// A chunk is held from its load until its group's range has gone round, and 37 MB are held at once: the exchange's
// latency bounds the rate.  So a slot's two words carry their own tag: no fence, no count, no atomic; one
// store by the writer, one load by the reader.  Memory-bound: 4 + k/8 B per weight.  The BERT-base set at one range
// per matrix, 4 bits (382 MB): 74.3 us; with an atomicMax, a release count and a polling lane per CTA instead of slots
// 97.8, with those per warp and chunk, which met on three words of one L2 slice, 299; two passes 132.5.
constexpr int kRingUnits = 32;                 // per chunk: 16 KB
constexpr int kRingStages = 12;
constexpr int kRingRangeWarps = 4;
constexpr int kRingAgents = 8;
constexpr int kRingPolls = 1;  // runs of a CTA that poll at a time (below)
constexpr int kRingRoundTeams = 4;             // of four warps
constexpr int kRingFirstAgent = 1 + kRingRangeWarps;
constexpr int kRingFirstRound = kRingFirstAgent + kRingAgents;
constexpr int kRingThreads = 32 * (kRingFirstRound + 4 * kRingRoundTeams);
constexpr int kRingWarpUnits = kRingUnits / 4; // of a range or rounding warp
constexpr int kRingSmemBytes = kRingStages * kRingUnits * 512 + 4 * kRingRoundTeams * kRingWarpUnits * 128;
// A CTA's runs (its chunks of one group) use slot run % kRingSlots.  Once a chunk has landed, the one twelve
// chunks before it is in its team's registers, so that all chunks sixteen or more before it have been rounded.
constexpr int kRingSlots = kRingStages + kRingRoundTeams;
// Rounds of the deal that a group may span, so that its last chunk is loaded and reduced while its first one
// is still held, with four stages left for loads in flight.
constexpr int kRingMaxSpan = kRingSlots - 4;
static_assert(kRingStages % kRingRoundTeams == 0, "a stage is always rounded by the same team");

struct RingItem {
  const float4* w;
  uint32_t* packed;
  float* delta;
  float* q0;
  int32_t ug;                // units per group
  int32_t chunks_per_group;
  int32_t chunk_begin;       // of the matrix, in the launch's list
  int32_t group_begin;       // of the matrix, in the launch's tables
  int32_t groups;
  int32_t bits;
};

struct RingBatch {
  RingItem item[kMaxWeightBatch];
  unsigned long long* slots;  // [groups of the launch][CTAs]: encoded max << 32 | inverted encoded min, 0 until written
  void* ws;
  int32_t chunks_total;
  int32_t count;
};

// A chunk of the launch's list.  `it` only moves forward.
struct RingChunk {
  int it, group, first_unit;  // matrix, group inside it, first unit inside the group
  __device__ __forceinline__ void seek(const RingBatch& b, int c) {
    while (it + 1 < b.count && c >= b.item[it + 1].chunk_begin) ++it;
    const RingItem& m = b.item[it];
    const int local = c - m.chunk_begin;
    group = local / m.chunks_per_group;
    first_unit = (local - group * m.chunks_per_group) * kRingUnits;
  }
  // chunks of this group that the CTA meets from here on, one every `step` chunks
  __device__ __forceinline__ int run(const RingBatch& b, int step) const {
    return (b.item[it].chunks_per_group - first_unit / kRingUnits + step - 1) / step;
  }
};

// What the producer leaves beside a stage's chunk.
struct __align__(16) RingStage {
  uint32_t* out;     // where the chunk's codes (or fp32 values) go
  int32_t unit_words;  // output words per unit
  int16_t n;         // units
  int16_t bits;
  int16_t slot;      // of the chunk's run
  int16_t phase;     // of the slot's barriers
  int16_t last;      // the run ends with this chunk
};

__global__ void __launch_bounds__(256) clear_slots_kernel(unsigned long long* p, int n) {
  pdl_begin();
  for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) p[i] = 0ull;
}

// Codes of the warp's units (n <= kRingWarpUnits) to the packed stream.
template <int BITS>
__device__ __forceinline__ void ring_pack(const float4 (&v)[kRingWarpUnits], const int n, const RgGroup& g, uint8_t* stg,
                                          uint32_t* __restrict__ out, const int lane) {
#pragma unroll
  for (int j = 0; j < kRingWarpUnits; ++j) {  // all of them: what lies past the chunk's end is not copied out
    const uint32_t f = quant_field_open<BITS, false>(v[j], g.lo, g.inv, g.hi);
    const int fi = j * 32 + lane;
    if (BITS == 8) reinterpret_cast<uint32_t*>(stg)[fi] = f;
    if (BITS == 4 || BITS == 3) reinterpret_cast<uint16_t*>(stg)[fi] = (uint16_t)f;
    if (BITS == 2) stg[fi] = (uint8_t)f;
  }
  __syncwarp();
  if (BITS == 3) {
    if (lane < 4 * n) store_3bit_item(stg, out, lane);
  } else {
    const int n16 = n * BITS;
#pragma unroll
    for (int r = 0; r < (kRingWarpUnits * BITS + 31) / 32; ++r) {
      const int i = r * 32 + lane;
      if (i < n16) reinterpret_cast<uint4*>(out)[i] = reinterpret_cast<const uint4*>(stg)[i];
    }
  }
  __syncwarp();
}

template <bool FAKE>
__global__ void __launch_bounds__(kRingThreads, 1)
weight_ring_kernel(const __grid_constant__ RingBatch b) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t s_bar[2 * kRingStages + 2 * kRingSlots];
  __shared__ uint32_t s_hi[kRingSlots][kRingRangeWarps], s_lo[kRingSlots][kRingRangeWarps];
  __shared__ RgGroup s_par[kRingSlots];
  __shared__ RingStage s_stage[kRingStages];
  __shared__ volatile int s_abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t ring = ptx::smem_u32(smem), bars = ptx::smem_u32(s_bar);
  auto full = [&](int s) { return bars + 8u * s; };                       // the stage's chunk has landed
  auto empty = [&](int s) { return bars + 8u * (kRingStages + s); };      // range and rounding warps have read it
  auto ranged = [&](int r) { return bars + 8u * (2 * kRingStages + r); }; // the run's range is in s_hi, s_lo
  auto ready = [&](int r) { return bars + 8u * (2 * kRingStages + kRingSlots + r); };  // the group's parameters are in s_par
  if (threadIdx.x == 0) {
    for (int s = 0; s < kRingStages; ++s) {
      ptx::mbar_init(full(s), 1);
      ptx::mbar_init(empty(s), kRingRangeWarps + 4);
    }
    for (int s = 0; s < kRingSlots; ++s) {
      ptx::mbar_init(ranged(s), kRingRangeWarps);
      ptx::mbar_init(ready(s), 1);
    }
    s_abort = 0;
    ptx::fence_mbar_init();
  }
  pdl_begin();
  __syncthreads();
  bool timed_out = false;
  RingChunk c;
  c.it = 0;
  const int step = (int)gridDim.x;
  const int chunks = (b.chunks_total - (int)blockIdx.x + step - 1) / step;  // of this CTA
  if (warp == 0) {
    if (ptx::elect_one()) {
      // One thread serves a chunk every 0.4 us: the walk over the deal is incremental, the matrix's fields stay in
      // registers, and the next chunk is worked out before the wait for its stage.  (With the division of
      // RingChunk::seek and the fields read per chunk it took 800 cycles, and bound the kernel.)
      int stage = 0, slot = -1, left = 0;
      uint32_t phase = 0, slot_phase = 1;
      RingItem m = b.item[0];
      int it = 0, group = 0, pos = (int)blockIdx.x;  // pos: chunk inside the group
      int words = FAKE ? 128 : 4 * m.bits;
      for (int k = 0; k < chunks; ++k) {
        while (pos >= m.chunks_per_group) {
          pos -= m.chunks_per_group;
          left = 0;
          if (++group == m.groups) {
            group = 0;
            m = b.item[++it];
            words = FAKE ? 128 : 4 * m.bits;
          }
        }
        if (left == 0) {  // the CTA's run in this group begins
          left = (m.chunks_per_group - pos + step - 1) / step;
          if (++slot == kRingSlots) slot = 0;
          if (slot == 0) slot_phase ^= 1u;
        }
        --left;
        const int n = min(m.ug - pos * kRingUnits, kRingUnits);
        const int64_t unit = (int64_t)group * m.ug + pos * kRingUnits;
        const RingStage st{m.packed + unit * words, words, (int16_t)n, (int16_t)m.bits, (int16_t)slot, (int16_t)slot_phase,
                           (int16_t)(left == 0)};
        if (!wait_barrier_relaxed(empty(stage), phase ^ 1u, &s_abort)) {
          timed_out = true;
          break;
        }
        s_stage[stage] = st;
        ptx::mbar_arrive_expect_tx(full(stage), (uint32_t)n * 512u);  // publishes s_stage too
        ptx::bulk_load_1d(ring + stage * kRingUnits * 512, m.w + unit * 32, (uint32_t)n * 512u, full(stage));
        pos += step;
        if (++stage == kRingStages) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
  } else if (warp < kRingFirstAgent) {
    const int part = warp - 1;
    const float kInf = __int_as_float(0x7f800000);
    int stage = 0;
    uint32_t phase = 0;
    float lo = kInf, hi = -kInf;
    for (int k = 0; k < chunks; ++k) {
      if (!wait_barrier_relaxed(full(stage), phase, &s_abort)) {
        timed_out = true;
        break;
      }
      const float4* src = reinterpret_cast<const float4*>(smem + stage * kRingUnits * 512) + part * kRingWarpUnits * 32 + lane;
      const int n = s_stage[stage].n - part * kRingWarpUnits, slot = s_stage[stage].slot;
      const bool last = s_stage[stage].last != 0;
      float4 v[kRingWarpUnits];
#pragma unroll
      for (int j = 0; j < kRingWarpUnits; ++j) v[j] = src[j * 32];  // units past the chunk's end: stale, not used
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(empty(stage));
#pragma unroll
      for (int j = 0; j < kRingWarpUnits; ++j)
        if (j < n) {
          lo = min3_nan(min3_nan(lo, v[j].x, v[j].y), v[j].z, v[j].w);
          hi = max3_nan(max3_nan(hi, v[j].x, v[j].y), v[j].z, v[j].w);
        }
      if (last) {
        const uint32_t e_hi = __reduce_max_sync(0xffffffffu, float_to_ordered(hi));
        const uint32_t e_lo = __reduce_max_sync(0xffffffffu, ~float_to_ordered(lo));
        if (lane == 0) {
          s_hi[slot][part] = e_hi;
          s_lo[slot][part] = e_lo;
          ptx::mbar_arrive(ranged(slot));
        }
        lo = kInf;
        hi = -kInf;
      }
      if (++stage == kRingStages) {
        stage = 0;
        phase ^= 1u;
      }
    }
  } else if (warp < kRingFirstRound) {
    const int agent = warp - kRingFirstAgent;
    int slot = 0;
    uint32_t phase = 0;
    int id = blockIdx.x;
    for (int run = 0; id < b.chunks_total; ++run) {
      c.seek(b, id);
      const int len = c.run(b, step);
      if (run % kRingAgents == agent) {
        const RingItem& m = b.item[c.it];
        unsigned long long* const table = b.slots + (size_t)(m.group_begin + c.group) * step;
        if (!wait_barrier_relaxed(ranged(slot), phase, &s_abort)) {
          timed_out = true;
          break;
        }
        const uint32_t my_hi = __reduce_max_sync(0xffffffffu, lane < kRingRangeWarps ? s_hi[slot][lane] : 0u);
        // (a NaN as minimum encodes to 0, which would read as missing; the maximum is then NaN too and reports it)
        const uint32_t my_lo = __reduce_max_sync(0xffffffffu, lane < kRingRangeWarps ? s_lo[slot][lane] : 1u);
        // the CTA that holds the group's chunk j has slot j (chunks j + step, ... are its own too)
        if (lane == 0)
          asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(table + c.first_unit / kRingUnits),
                       "l"((unsigned long long)my_hi << 32 | max(my_lo, 1u)) : "memory");
        const int n = min(m.chunks_per_group, step);  // CTAs that hold a part of the group
        const int prev = slot < kRingPolls ? slot + kRingSlots - kRingPolls : slot - kRingPolls;
        const uint32_t prev_phase = slot < kRingPolls ? phase ^ 1u : phase;
        if (run >= kRingPolls && !wait_barrier_relaxed(ready(prev), prev_phase, &s_abort)) {
          timed_out = true;
          break;
        }
        uint32_t e_hi, e_lo;
        const long long t0 = clock64();
        bool ok = true, all;
        constexpr int kPer = (kRingMaxCtas + 31) / 32;
        unsigned long long v[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) v[i] = lane + 32 * i < n ? 0ull : 1ull;
        for (;;) {  // all of the lane's missing slots in flight at once
#pragma unroll
          for (int i = 0; i < kPer; ++i)
            if (v[i] == 0ull)
              asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v[i]) : "l"(table + lane + 32 * i) : "memory");
          all = true;
#pragma unroll
          for (int i = 0; i < kPer; ++i) all = all && v[i] != 0ull;
          all = __all_sync(0xffffffffu, all);
          ok = !__any_sync(0xffffffffu, !all && (s_abort != 0 || clock64() - t0 > kWaitLimitCycles));
          if (all || !ok) break;
        }
        e_hi = e_lo = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
          e_hi = max(e_hi, (uint32_t)(v[i] >> 32));
          e_lo = max(e_lo, (uint32_t)v[i]);
        }
        e_hi = __reduce_max_sync(0xffffffffu, e_hi);
        e_lo = __reduce_max_sync(0xffffffffu, e_lo);
        if (!ok) {
          timed_out = true;
          break;
        }
        if (lane == 0) {
          const float g_hi = ordered_to_float(e_hi), g_lo = ordered_to_float(~e_lo);
          const int L = (1 << m.bits) - 1;
          const bool publish = c.first_unit == 0;
          if (publish && !(fabsf(g_hi) <= 3.402823466e38f && fabsf(g_lo) <= 3.402823466e38f)) report_status(b.ws, QB_ERR_NONFINITE);
          const GroupParams gp = finish_group(g_lo, g_hi, false, L, c.group, m.delta, m.q0, publish, b.ws);
          s_par[slot] = RgGroup{gp.lo, gp.inv, group_step(gp, L), gp.hi};
          ptx::mbar_arrive(ready(slot));
        }
        __syncwarp();
      }
      id += len * step;
      if (++slot == kRingSlots) {
        slot = 0;
        phase ^= 1u;
      }
    }
  } else {
    const int rw = warp - kRingFirstRound;
    const int team = rw >> 2, part = rw & 3;
    uint8_t* const stg = smem + kRingStages * kRingUnits * 512 + rw * kRingWarpUnits * 128;
    int stage = team;
    uint32_t phase = 0;
    for (int k = team; k < chunks; k += kRingRoundTeams) {
      if (!wait_barrier_relaxed(full(stage), phase, &s_abort)) {
        timed_out = true;
        break;
      }
      const RingStage st = s_stage[stage];
      const int u0 = part * kRingWarpUnits;
      const int n = min((int)st.n - u0, kRingWarpUnits);
      const float4* src = reinterpret_cast<const float4*>(smem + stage * kRingUnits * 512) + u0 * 32 + lane;
      float4 v[kRingWarpUnits];
#pragma unroll
      for (int j = 0; j < kRingWarpUnits; ++j) v[j] = src[j * 32];  // units past the chunk's end: stale, not used
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(empty(stage));
      // After the wait for the chunk, not before: every run that used this slot earlier is then behind us (a
      // barrier's parity is only told apart one phase at a time).
      if (!wait_barrier_relaxed(ready(st.slot), (uint32_t)st.phase, &s_abort)) {
        timed_out = true;
        break;
      }
      const RgGroup cur = s_par[st.slot];
      uint32_t* const out = st.out + u0 * st.unit_words;
      if (FAKE) {
#pragma unroll
        for (int j = 0; j < kRingWarpUnits; ++j)
          if (j < n) reinterpret_cast<float4*>(out)[j * 32 + lane] = fake_quant4<false>(v[j], cur);
      } else {
        switch (st.bits) {  // team-uniform
          case 2: ring_pack<2>(v, n, cur, stg, out, lane); break;
          case 3: ring_pack<3>(v, n, cur, stg, out, lane); break;
          case 4: ring_pack<4>(v, n, cur, stg, out, lane); break;
          default: ring_pack<8>(v, n, cur, stg, out, lane); break;
        }
      }
      stage += kRingRoundTeams;
      if (stage >= kRingStages) {
        stage -= kRingStages;
        phase ^= 1u;
      }
    }
  }
  if (timed_out) {
    s_abort = 1;
    report_status(b.ws, QB_ERR_TIMEOUT);
    // let copies already in flight land before the CTA's shared memory is released
    const long long t0 = clock64();
    while (clock64() - t0 < 400000ll) {
    }
  }
}

struct HostWeight {
  const float* w;
  int64_t N, K;
  int groups;
  const float* range_lo;
  const float* range_hi;
  uint32_t* packed;
  float* delta;
  float* q0;
  int bits;
};

static qb_status launch_regs_single(const HostWeight* m, int count, bool ranged, void* ws, int sm_count,
                                    cudaStream_t stream, bool fake, bool encoded);

// Two-pass path (own ranges over groups too large for a cluster): one pair of launches over `count`
// matrices (<= kMaxWeightBatch).  Their range tables sit back to back in the workspace: maxima at
// ws + kWsRangeOff, inverted minima after them.  The second pass is the register-resident kernel in its
// supplied-ranges form, reading those tables.
static qb_status launch_two_pass(const HostWeight* m, int count, void* ws, int sm_count, cudaStream_t stream,
                                 bool fake = false) {
  WeightBatch b;
  memset(&b, 0, sizeof(b));
  int total_groups = 0;
  int64_t units = 0;
  for (int i = 0; i < count; ++i) {
    WeightItem& it = b.item[i];
    it.w = reinterpret_cast<const float4*>(m[i].w);
    it.packed = m[i].packed;
    it.delta = m[i].delta;
    it.q0 = m[i].q0;
    it.range_lo = m[i].range_lo;
    it.range_hi = m[i].range_hi;
    it.unit_begin = units;
    it.units = m[i].N * m[i].K / 128;
    it.units_per_row = (int32_t)(m[i].K / 128);
    it.rows_per_group = (int32_t)(m[i].N / m[i].groups);
    it.group_begin = total_groups;
    units += it.units;
    total_groups += m[i].groups;
  }
  b.count = count;
  b.ws = ws;
  b.hi_enc = reinterpret_cast<uint32_t*>(static_cast<char*>(ws) + kWsRangeOff);
  b.lo_inv = b.hi_enc + total_groups;
  b.units_total = units;
  b.keep_fraction = l2_keep_fraction(512.0 * (double)units);
  QB_CUDA_TRY(cudaMemsetAsync(b.hi_enc, 0, sizeof(uint32_t) * 2 * (size_t)total_groups, stream));

  const int64_t max_warps = (int64_t)sm_count * 32;  // 4 blocks of 8 warps per SM
  int64_t upw = (units + max_warps - 1) / max_warps;
  if (upw < 4) upw = 4;
  b.units_per_warp = upw;
  const int64_t warps = (units + upw - 1) / upw;
  const unsigned blocks = (unsigned)((warps + kWqWarps - 1) / kWqWarps);

  QB_CUDA_TRY(launch_kernel(weight_range_kernel, blocks, kWqThreads, 0, stream, 1, false, b));
  HostWeight second[kMaxWeightBatch];
  for (int i = 0; i < count; ++i) {
    second[i] = m[i];
    second[i].range_lo = reinterpret_cast<const float*>(b.lo_inv + b.item[i].group_begin);
    second[i].range_hi = reinterpret_cast<const float*>(b.hi_enc + b.item[i].group_begin);
  }
  return launch_regs_single(second, count, true, ws, sm_count, stream, fake, true);
}

static inline int64_t group_units(const HostWeight& h) { return (h.N / h.groups) * (h.K / 128); }

// Does a matrix take the register-resident path?  With its own ranges: groups of at most 288 units in one
// CTA, up to 2,304 in a cluster of up to 8 CTAs.  With the caller's ranges: always (nothing to reduce).
constexpr int kRgMaxCluster = 8;
static inline int regs_cluster_size(const HostWeight& h) {
  if (h.range_lo != nullptr) return 1;
  return (int)((group_units(h) + kRgMaxGroupUnits - 1) / kRgMaxGroupUnits);
}
static inline bool regs_eligible(const HostWeight& h) {
  return h.range_lo != nullptr || group_units(h) <= (int64_t)kRgMaxGroupUnits * kRgMaxCluster;
}

// Clusters of `cl` CTAs that can be resident at once (asked once per device and cluster size).
static qb_status regs_max_clusters(int cl, int* out) {
  static std::atomic<int> cached[64][kRgMaxCluster + 1] = {};
  int dev = 0;
  QB_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) {
    set_last_error("device ordinal %d out of range", dev);
    return QB_ERR_CUDA;
  }
  int n = cached[dev][cl].load(std::memory_order_acquire);
  if (n == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cl * 64u);
    cfg.blockDim = dim3(kRgThreads);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    QB_CUDA_TRY(cudaOccupancyMaxActiveClusters(&n, weight_regs_kernel<true, false, false>, &cfg));
    if (n < 1) {
      set_last_error("no cluster of %d CTAs fits the device", cl);
      return QB_ERR_CUDA;
    }
    cached[dev][cl].store(n, std::memory_order_release);
  }
  *out = n;
  return QB_OK;
}

// Matrices whose groups need a cluster of `cl` CTAs (289 to 2,304 units per group), any bit widths: one
// group per cluster item.
static qb_status launch_regs_cluster(const HostWeight* m, int count, int cl, void* ws, cudaStream_t stream, bool fake) {
  int max_clusters = 0;
  qb_status st = regs_max_clusters(cl, &max_clusters);
  if (st != QB_OK) return st;
  for (int first = 0; first < count; first += kRgMaxBatch) {
    const int n = std::min(kRgMaxBatch, count - first);
    RegsBatch b;
    memset(&b, 0, sizeof(b));
    int items = 0;
    for (int i = 0; i < n; ++i) {
      const HostWeight& h = m[first + i];
      RegsItem& it = b.item[i];
      const int ug = (int)group_units(h);
      it.w = reinterpret_cast<const float4*>(h.w);
      it.packed = h.packed;
      it.delta = h.delta;
      it.q0 = h.q0;
      it.ug = ug;
      it.groups = h.groups;
      it.item_begin = items;
      it.groups_per_item = 1;
      it.team_warps = (int16_t)kRgWarps;
      it.groups_per_warp = 1;
      it.slice_units = (int16_t)((ug + kRgWarps * cl - 1) / (kRgWarps * cl));
      it.bits = (int16_t)h.bits;
      items += h.groups;
    }
    b.ws = ws;
    b.total_items = items;
    b.count = n;
    QB_CUDA_TRY(launch_kernel(fake ? weight_regs_kernel<true, true, false> : weight_regs_kernel<true, false, false>,
                              (unsigned)(std::min(items, max_clusters) * cl), kRgThreads, 0, stream, (unsigned)cl, false, b));
  }
  return QB_OK;
}

// Matrices served by single CTAs (own ranges with groups of at most 288 units, or the caller's ranges with
// groups of any size: `ranged`), any bit widths: launches of up to kRgMaxBatch matrices, inside a launch
// the matrices with the largest CTA items first.
static qb_status launch_regs_single(const HostWeight* m, int count, bool ranged, void* ws, int sm_count,
                                    cudaStream_t stream, bool fake, bool encoded) {
  struct Shape {
    int idx, W, gpw, slice, gpi, chunks;
    int64_t item_units;
  };
  std::vector<Shape> sh(count);
  for (int i = 0; i < count; ++i) {
    const int64_t ug = group_units(m[i]);
    Shape& s = sh[i];
    s.idx = i;
    s.chunks = 1;
    if (ug > kRgMaxGroupUnits) {  // `ranged` only: the group is cut into items of 288 units
      s.W = kRgWarps;
      s.gpw = 1;
      s.slice = kRgUnits;
      s.gpi = 1;
      s.chunks = (int)((ug + kRgMaxGroupUnits - 1) / kRgMaxGroupUnits);
      s.item_units = kRgMaxGroupUnits;
      continue;
    }
    s.W = 1;
    while (s.W * kRgUnits < ug) s.W *= 2;
    s.gpw = s.W == 1 ? std::max(1, kRgUnits / (int)ug) : 1;
    s.slice = ((int)ug + s.W - 1) / s.W;
    s.gpi = (kRgWarps / s.W) * s.gpw;
    s.item_units = (int64_t)std::min(s.gpi, m[i].groups) * ug;
  }
  std::stable_sort(sh.begin(), sh.end(), [](const Shape& a, const Shape& b) { return a.item_units > b.item_units; });
  for (int first = 0; first < count; first += kRgMaxBatch) {
    const int n = std::min(kRgMaxBatch, count - first);
    RegsBatch b;
    memset(&b, 0, sizeof(b));
    int64_t items = 0;
    for (int i = 0; i < n; ++i) {
      const Shape& s = sh[first + i];
      const HostWeight& h = m[s.idx];
      RegsItem& it = b.item[i];
      it.w = reinterpret_cast<const float4*>(h.w);
      it.packed = h.packed;
      it.delta = h.delta;
      it.q0 = h.q0;
      it.ug = (int32_t)group_units(h);
      it.groups = h.groups;
      it.item_begin = (int32_t)items;
      it.groups_per_item = s.gpi;
      it.team_warps = (int16_t)s.W;
      it.groups_per_warp = (int16_t)s.gpw;
      it.slice_units = (int16_t)s.slice;
      it.bits = (int16_t)h.bits;
      it.range_lo = h.range_lo;
      it.range_hi = h.range_hi;
      it.chunks = s.chunks;
      it.encoded = encoded ? 1 : 0;
      items += s.chunks > 1 ? (int64_t)h.groups * s.chunks : (h.groups + s.gpi - 1) / s.gpi;
    }
    if (items > 0x7fffffff) {
      set_last_error("weight batch too large for one launch (%lld items)", (long long)items);
      return QB_ERR_INVALID;
    }
    b.ws = ws;
    b.total_items = (int32_t)items;
    b.count = n;
    const unsigned grid = (unsigned)std::min<int64_t>(items, sm_count);
    auto kernel = ranged ? (fake ? weight_regs_kernel<false, true, true> : weight_regs_kernel<false, false, true>)
                         : (fake ? weight_regs_kernel<false, true, false> : weight_regs_kernel<false, false, false>);
    QB_CUDA_TRY(launch_kernel(kernel, grid, kRgThreads, 0, stream, 1, false, b));
  }
  return QB_OK;
}

// Register-resident path over any number of eligible matrices of any bit widths.  Matrices whose groups
// need a cluster go to launches of their cluster size, matrices with caller-supplied ranges to launches of
// the kernel that clamps.
static qb_status launch_regs(const HostWeight* m_all, int count_all, void* ws, int sm_count, cudaStream_t stream,
                             bool fake = false) {
  std::vector<HostWeight> single, ranged, clustered[kRgMaxCluster + 1];
  for (int i = 0; i < count_all; ++i) {
    if (m_all[i].range_lo != nullptr) {
      ranged.push_back(m_all[i]);
      continue;
    }
    const int cl = regs_cluster_size(m_all[i]);
    (cl <= 1 ? single : clustered[cl]).push_back(m_all[i]);
  }
  for (int cl = 2; cl <= kRgMaxCluster; ++cl) {
    if (clustered[cl].empty()) continue;
    qb_status st = launch_regs_cluster(clustered[cl].data(), (int)clustered[cl].size(), cl, ws, stream, fake);
    if (st != QB_OK) return st;
  }
  if (!ranged.empty()) {
    qb_status st = launch_regs_single(ranged.data(), (int)ranged.size(), true, ws, sm_count, stream, fake, false);
    if (st != QB_OK) return st;
  }
  if (single.empty()) return QB_OK;
  return launch_regs_single(single.data(), (int)single.size(), false, ws, sm_count, stream, fake, false);
}

// One pair of launches (clear, ring kernel) over `count` matrices (<= kMaxWeightBatch) whose groups fit the ring.
template <bool FAKE>
static qb_status launch_ring_form(const RingBatch& b, unsigned grid, cudaStream_t stream, bool* refused) {
  static std::atomic<bool> attr_set[64] = {};
  int dev = 0;
  QB_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64 || !attr_set[dev].load(std::memory_order_acquire)) {
    QB_CUDA_TRY(cudaFuncSetAttribute(weight_ring_kernel<FAKE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingSmemBytes));
    if (dev >= 0 && dev < 64) attr_set[dev].store(true, std::memory_order_release);
  }
  const cudaError_t e = launch_kernel(weight_ring_kernel<FAKE>, grid, kRingThreads, kRingSmemBytes, stream, 1, true, b);
  *refused = residency_refused(e);
  if (!*refused) QB_CUDA_TRY(e);
  return QB_OK;
}
// `refused`: nothing was rounded, the blocks cannot all be resident.
static qb_status launch_ring(const HostWeight* m, int count, void* ws, int sm_count, cudaStream_t stream, bool fake,
                             bool* refused) {
  RingBatch b;
  int groups = 0, chunks = 0;
  for (int i = 0; i < count; ++i) {
    const HostWeight& h = m[i];
    RingItem& it = b.item[i];
    it.w = reinterpret_cast<const float4*>(h.w);
    it.packed = h.packed;
    it.delta = h.delta;
    it.q0 = h.q0;
    it.ug = (int32_t)group_units(h);
    it.chunks_per_group = (it.ug + kRingUnits - 1) / kRingUnits;
    it.chunk_begin = chunks;
    it.group_begin = groups;
    it.groups = h.groups;
    it.bits = h.bits;
    chunks += it.chunks_per_group * h.groups;
    groups += h.groups;
  }
  b.ws = ws;
  b.slots = reinterpret_cast<unsigned long long*>(static_cast<char*>(ws) + kWsRangeOff);
  b.chunks_total = chunks;
  b.count = count;
  const unsigned grid = (unsigned)std::min(chunks, std::min(sm_count, kRingMaxCtas));
  const int slots = groups * (int)grid;
  QB_CUDA_TRY(launch_kernel(clear_slots_kernel, (unsigned)std::min((slots + 255) / 256, sm_count), 256, 0, stream, 1, false,
                            b.slots, slots));
  return fake ? launch_ring_form<true>(b, grid, stream, refused) : launch_ring_form<false>(b, grid, stream, refused);
}

// Matrices whose groups do not fit a cluster's registers: the ring as long as a group spans few enough rounds of
// its deal (up to 148 * 11 chunks of 16 KB, 27 MB), else, and where the workspace has no room for the
// slots, the two passes.  Both are a pair of launches per job.
static inline bool ring_eligible(const HostWeight& h, int sm_count) {
  return (group_units(h) + kRingUnits - 1) / kRingUnits <= (int64_t)(kRingMaxSpan - 1) * std::min(sm_count, kRingMaxCtas) &&
         h.groups <= kRingMaxGroups;
}
struct LargeJob {
  std::vector<HostWeight> m;  // at most kMaxWeightBatch matrices
  int64_t groups = 0;         // of all of them; a ring job has at most kRingMaxGroups
  bool ring = false;
};
static std::vector<LargeJob> plan_large_groups(const std::vector<HostWeight>& m, int sm_count) {
  std::vector<LargeJob> jobs;
  for (const bool ring : {true, false}) {
    bool open = false;
    for (const HostWeight& h : m) {
      if (ring_eligible(h, sm_count) != ring) continue;
      if (!open || (int)jobs.back().m.size() == kMaxWeightBatch || (ring && jobs.back().groups + h.groups > kRingMaxGroups)) {
        jobs.emplace_back();
        jobs.back().ring = ring;
        open = true;
      }
      jobs.back().m.push_back(h);
      jobs.back().groups += h.groups;
    }
  }
  return jobs;
}
static qb_status launch_large_groups(const std::vector<HostWeight>& m, void* ws, size_t ws_bytes, int sm_count,
                                     cudaStream_t stream, bool fake) {
  for (const LargeJob& j : plan_large_groups(m, sm_count)) {
    bool two_pass = !j.ring || kWsRangeOff + ring_table_bytes((size_t)j.groups) > ws_bytes || !stream_has_sms(stream, sm_count);
    qb_status st = QB_OK;
    if (!two_pass) st = launch_ring(j.m.data(), (int)j.m.size(), ws, sm_count, stream, fake, &two_pass);
    if (st == QB_OK && two_pass) st = launch_two_pass(j.m.data(), (int)j.m.size(), ws, sm_count, stream, fake);
    if (st != QB_OK) return st;
  }
  return QB_OK;
}

// All matrices of a call, any bit widths.
static qb_status launch_weights(const std::vector<HostWeight>& m, void* ws, size_t ws_bytes, int sm_count,
                                cudaStream_t stream, bool fake) {
  std::vector<HostWeight> regs, rest;
  for (const HostWeight& h : m) (regs_eligible(h) ? regs : rest).push_back(h);
  if (!regs.empty()) {
    qb_status st = launch_regs(regs.data(), (int)regs.size(), ws, sm_count, stream, fake);
    if (st != QB_OK) return st;
  }
  return launch_large_groups(rest, ws, ws_bytes, sm_count, stream, fake);
}

qb_status launch_quantize_pack_weights(const float* w, int64_t N, int64_t K, int bits, int groups,
                                       const float* range_lo, const float* range_hi, uint32_t* packed,
                                       float* delta, float* q0, void* ws, size_t ws_bytes, int sm_count,
                                       cudaStream_t stream) {
  return launch_weights({HostWeight{w, N, K, groups, range_lo, range_hi, packed, delta, q0, bits}}, ws, ws_bytes, sm_count,
                        stream, false);
}

static qb_status validate_weight(const char* who, const float* w, int64_t N, int64_t K, int bits, int groups,
                                 const float* range_lo, const float* range_hi, const uint32_t* packed,
                                 const float* delta, const float* q0) {
  if (!w || !packed || !delta || !q0 || N <= 0 || K <= 0 || N > QB_MAX_MN || K > QB_MAX_K || !valid_bits(bits) ||
      groups < 1 || N % groups != 0 || ((range_lo == nullptr) != (range_hi == nullptr))) {
    set_last_error("%s: invalid argument (N=%lld K=%lld bits=%d groups=%d)", who, (long long)N, (long long)K, bits,
                   groups);
    return QB_ERR_INVALID;
  }
  if (K % 128 != 0 || !aligned16(w) || !aligned16(packed)) {
    set_last_error("%s: K must be a multiple of 128 and w, packed 16-byte aligned", who);
    return QB_ERR_ALIGN;
  }
  return QB_OK;
}

}  // namespace qb

extern "C" qb_status qb_quantize_pack_weights(const float* w, int64_t N, int64_t K, int bits, int groups,
                                              const float* range_lo, const float* range_hi, uint32_t* packed,
                                              float* delta, float* q0, void* ws, size_t ws_bytes,
                                              void* cuda_stream) {
  qb_status st = qb::validate_weight("qb_quantize_pack_weights", w, N, K, bits, groups, range_lo, range_hi, packed,
                                     delta, q0);
  if (st != QB_OK) return st;
  if (!ws || ws_bytes < qb::ws_bytes_needed(groups)) {
    qb::set_last_error("qb_quantize_pack_weights: workspace null or smaller than %zu bytes",
                       qb::ws_bytes_needed(groups));
    return QB_ERR_WORKSPACE;
  }
  int sms = 0;
  st = qb::require_sm100(&sms);
  if (st != QB_OK) return st;
  return qb::launch_quantize_pack_weights(w, N, K, bits, groups, range_lo, range_hi, packed, delta, q0, ws, ws_bytes,
                                          sms, (cudaStream_t)cuda_stream);
}

static std::vector<qb::HostWeight> host_weights(const qb_weight_desc* descs, int32_t count) {
  std::vector<qb::HostWeight> m(count);
  for (int i = 0; i < count; ++i) {
    const qb_weight_desc& d = descs[i];
    m[i] = qb::HostWeight{d.w, d.N, d.K, d.groups, d.range_lo, d.range_hi, d.packed, d.delta, d.q0, d.bits};
  }
  return m;
}

extern "C" qb_status qb_quantize_pack_weights_batch(const qb_weight_desc* descs, int32_t count, void* ws,
                                                    size_t ws_bytes, void* cuda_stream) {
  if (!descs || count <= 0) {
    qb::set_last_error("qb_quantize_pack_weights_batch: descs null or count <= 0");
    return QB_ERR_INVALID;
  }
  int64_t total_groups = 0;
  for (int i = 0; i < count; ++i) {
    const qb_weight_desc& d = descs[i];
    qb_status st = qb::validate_weight("qb_quantize_pack_weights_batch", d.w, d.N, d.K, d.bits, d.groups, d.range_lo,
                                       d.range_hi, d.packed, d.delta, d.q0);
    if (st != QB_OK) return st;
    total_groups += d.groups;
  }
  if (total_groups > (1 << 24) || !ws || ws_bytes < qb::ws_bytes_needed((int)total_groups)) {
    qb::set_last_error("qb_quantize_pack_weights_batch: workspace null or smaller than %zu bytes (sum of groups %lld)",
                       qb::ws_bytes_needed((int)total_groups), (long long)total_groups);
    return QB_ERR_WORKSPACE;
  }
  int sms = 0;
  qb_status st = qb::require_sm100(&sms);
  if (st != QB_OK) return st;
  return qb::launch_weights(host_weights(descs, count), ws, ws_bytes, sms, (cudaStream_t)cuda_stream, false);
}

extern "C" int32_t qb_quantize_pack_weights_launch_count(const qb_weight_desc* descs, int32_t count) {
  if (!descs || count <= 0) return 0;
  for (int i = 0; i < count; ++i) {
    const qb_weight_desc& d = descs[i];
    if (d.N <= 0 || d.K <= 0 || d.groups < 1 || d.N % d.groups != 0 || d.K % 128 != 0) return 0;
  }
  int sms = 148;
  qb::require_sm100(&sms);  // without a device: the plan for a 148-SM part
  int per_cluster[qb::kRgMaxCluster + 1] = {};
  int ranged = 0;
  std::vector<qb::HostWeight> large;
  for (const qb::HostWeight& h : host_weights(descs, count)) {
    if (!qb::regs_eligible(h))
      large.push_back(h);
    else if (h.range_lo != nullptr)
      ++ranged;
    else
      ++per_cluster[std::max(1, qb::regs_cluster_size(h))];
  }
  const auto launches = [](int matrices, int per_launch) { return (matrices + per_launch - 1) / per_launch; };
  int32_t n = launches(ranged, qb::kRgMaxBatch);
  for (int cl = 1; cl <= qb::kRgMaxCluster; ++cl) n += launches(per_cluster[cl], qb::kRgMaxBatch);
  n += 2 * (int32_t)qb::plan_large_groups(large, sms).size();
  return n;
}

extern "C" qb_status qb_fake_quantize_weights(const float* w, int64_t N, int64_t K, int bits, int groups,
                                              const float* range_lo, const float* range_hi, float* wq, float* delta,
                                              float* q0, void* ws, size_t ws_bytes, void* cuda_stream) {
  qb_status st = qb::validate_weight("qb_fake_quantize_weights", w, N, K, bits, groups, range_lo, range_hi,
                                     reinterpret_cast<const uint32_t*>(wq), delta, q0);
  if (st != QB_OK) return st;
  if (!ws || ws_bytes < qb::ws_bytes_needed(groups)) {
    qb::set_last_error("qb_fake_quantize_weights: workspace null or smaller than %zu bytes",
                       qb::ws_bytes_needed(groups));
    return QB_ERR_WORKSPACE;
  }
  int sms = 0;
  st = qb::require_sm100(&sms);
  if (st != QB_OK) return st;
  // `packed` of the descriptor points to the fp32 output
  return qb::launch_weights({qb::HostWeight{w, N, K, groups, range_lo, range_hi, reinterpret_cast<uint32_t*>(wq), delta, q0, bits}},
                            ws, ws_bytes, sms, (cudaStream_t)cuda_stream, true);
}

extern "C" qb_status qb_fake_quantize_weights_batch(const qb_weight_desc* descs, int32_t count, void* ws,
                                                    size_t ws_bytes, void* cuda_stream) {
  if (!descs || count <= 0) {
    qb::set_last_error("qb_fake_quantize_weights_batch: descs null or count <= 0");
    return QB_ERR_INVALID;
  }
  int64_t total_groups = 0;
  for (int i = 0; i < count; ++i) {
    const qb_weight_desc& d = descs[i];
    qb_status st = qb::validate_weight("qb_fake_quantize_weights_batch", d.w, d.N, d.K, d.bits, d.groups, d.range_lo,
                                       d.range_hi, d.packed, d.delta, d.q0);
    if (st != QB_OK) return st;
    total_groups += d.groups;
  }
  if (total_groups > (1 << 24) || !ws || ws_bytes < qb::ws_bytes_needed((int)total_groups)) {
    qb::set_last_error("qb_fake_quantize_weights_batch: workspace null or smaller than %zu bytes (sum of groups %lld)",
                       qb::ws_bytes_needed((int)total_groups), (long long)total_groups);
    return QB_ERR_WORKSPACE;
  }
  int sms = 0;
  qb_status st = qb::require_sm100(&sms);
  if (st != QB_OK) return st;
  return qb::launch_weights(host_weights(descs, count), ws, ws_bytes, sms, (cudaStream_t)cuda_stream, true);
}

extern "C" qb_status qb_ste_backward(const float* grad_wq, const float* w, int64_t N, int64_t K, int groups,
                                     const float* range_lo, const float* range_hi, float* grad_w,
                                     void* cuda_stream) {
  if (!grad_wq || !w || !grad_w || N <= 0 || K <= 0 || N > QB_MAX_MN || K > QB_MAX_K || groups < 1 ||
      N % groups != 0 || ((range_lo == nullptr) != (range_hi == nullptr))) {
    qb::set_last_error("qb_ste_backward: invalid argument (N=%lld K=%lld groups=%d)", (long long)N, (long long)K,
                       groups);
    return QB_ERR_INVALID;
  }
  if (K % 128 != 0 || !qb::aligned16(grad_wq) || !qb::aligned16(w) || !qb::aligned16(grad_w)) {
    qb::set_last_error("qb_ste_backward: K must be a multiple of 128 and grad_wq, w, grad_w 16-byte aligned");
    return QB_ERR_ALIGN;
  }
  int sms = 0;
  qb_status st = qb::require_sm100(&sms);
  if (st != QB_OK) return st;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  if (range_lo == nullptr) {  // the group's own [min, max]: every element is inside, the gradient passes unchanged
    if (grad_w != grad_wq)
      QB_CUDA_TRY(cudaMemcpyAsync(grad_w, grad_wq, sizeof(float) * (size_t)N * (size_t)K, cudaMemcpyDeviceToDevice,
                                  stream));
    return QB_OK;
  }
  const int64_t units = N * (K / 128);  // below 2^33; a tensor that large does not exist, but the division is 32-bit
  if (units > 0xffffffffll) {
    qb::set_last_error("qb_ste_backward: matrix too large (N=%lld K=%lld)", (long long)N, (long long)K);
    return QB_ERR_INVALID;
  }
  const int64_t blocks = std::min((units + 8 * qb::kSteUnits - 1) / (8 * qb::kSteUnits), (int64_t)sms * 64);
  QB_CUDA_TRY(qb::launch_kernel(qb::ste_backward_kernel, (unsigned)blocks, 256, 0, stream, 1, false,
                                reinterpret_cast<const float4*>(grad_wq), reinterpret_cast<const float4*>(w), units,
                                (uint32_t)(N / groups * (K / 128)), range_lo, range_hi, reinterpret_cast<float4*>(grad_w)));
  return QB_OK;
}
