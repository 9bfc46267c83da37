// qb_quantize_embedding, qb_embedding_lookup: group-wise quantized embedding tables (Section 5.1 and the
// appendix on mixed-precision embedding: the embedding dimensions are bucketed into groups, 4-bit word
// and 8-bit position embedding) and the lookup that dequantizes the rows it gathers.
//
// The table stays in lookup order, E[v][d], so that a token's row of codes is one contiguous run of
// D*k/8 bytes; a group is therefore a block of D/G consecutive COLUMNS over all V rows.
//
// One thread owns four consecutive columns (a warp = 128 columns = one packing unit); a block reads several
// rows side by side, so that it has about 512 threads whatever D is.
//   emb_range_kernel   two blocks per SM stride over the rows, eight rows in flight per thread; per-thread running
//                      min / max of its four columns, merged per group in shared memory, one atomicMax per
//                      group and block on order-preserving encodings in the workspace
//   emb_pack_kernel    blocks stride over the rows, last rows first (what the range pass read last is still in
//                      L2), four rows in flight per thread: packed fp32x2 arithmetic, no clamp (the range is
//                      the group's own), narrow stores that lay the fields down in stream order (k = 3:
//                      assembled with warp shuffles)
//   emb_lookup_kernel  blocks stride over the tokens: the thread's 4k-bit field of the row, four fused
//                      multiply-adds with its columns' (Delta, q0), one float4 store (or add-and-store, then
//                      last tokens first: what was written last is still in L2).  One token per thread at a
//                      time and 32 registers: the stores need warps, not loads in flight (two and four tokens
//                      per thread: 40.0 and 48.8 us against 35.0 for the lookups below)
// All three are streams: 4 B, 4 B + k/8 B per table element, and k/8 B + 4 B (8 B) per looked-up element.
// 30,522 x 768 at 4 bits, 128 groups (94 MB): 52.6 us with 36 scalar operations per float4, an
// atomic per column and a memset, 35.5 now.  24,576 tokens, word table at 4 bits then position table at 8 bits
// accumulated: 41.4 -> 34.3 us.
#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "mbar_wait.cuh"

namespace qb {

constexpr int kEmbMaxD = 4096;  // D/4 <= 1024 threads
constexpr int kEmbThreads = 512;
constexpr int kEmbRangeRows = 8, kEmbRows = 4;  // in flight per thread, range pass and packing

__device__ __forceinline__ bool finite_f(float x) { return fabsf(x) <= 3.402823466e38f; }

__global__ void __launch_bounds__(1024)
emb_range_kernel(const float4* e, int64_t V, int d4, int slots, int cols_per_group, int groups, float keep_fraction,
                 uint32_t* g_hi, uint32_t* g_lo_inv, void* ws) {
  extern __shared__ uint32_t emb_smem[];  // [slots][2][4 * d4] encoded maxima / inverted minima
  pdl_begin();
  const uint64_t pol = policy_evict_last(keep_fraction);
  WsHeader* const h = reinterpret_cast<WsHeader*>(ws);
  const int q = threadIdx.x % d4, slot = threadIdx.x / d4;
  const float kInf = __int_as_float(0x7f800000);
  float lo[4] = {kInf, kInf, kInf, kInf}, hi[4] = {-kInf, -kInf, -kInf, -kInf};
  const int64_t step = (int64_t)gridDim.x * slots;
  bool cleared = threadIdx.x >= 32;
  uint32_t launch = 0;
  for (int64_t r = (int64_t)blockIdx.x * slots + slot; r < V; r += kEmbRangeRows * step) {
    float4 v[kEmbRangeRows];
#pragma unroll
    for (int j = 0; j < kEmbRangeRows; ++j)  // past the end: the row of this round that is there, once more
      v[j] = ldg_policy(e + (r + j * step < V ? r + j * step : r) * d4 + q, pol);
    if (!cleared) {  // the block's first warp (its first row exists), while its first loads are on their way
      cleared = true;
      launch = clear_slots(g_hi, 2 * groups, h, threadIdx.x);
    }
#pragma unroll
    for (int j = 0; j < kEmbRangeRows; j += 2) {
      lo[0] = min3_nan(lo[0], v[j].x, v[j + 1].x);
      lo[1] = min3_nan(lo[1], v[j].y, v[j + 1].y);
      lo[2] = min3_nan(lo[2], v[j].z, v[j + 1].z);
      lo[3] = min3_nan(lo[3], v[j].w, v[j + 1].w);
      hi[0] = max3_nan(hi[0], v[j].x, v[j + 1].x);
      hi[1] = max3_nan(hi[1], v[j].y, v[j + 1].y);
      hi[2] = max3_nan(hi[2], v[j].z, v[j + 1].z);
      hi[3] = max3_nan(hi[3], v[j].w, v[j + 1].w);
    }
  }
  const int D = 4 * d4;
  uint32_t* mine = emb_smem + (size_t)slot * 2 * D;
#pragma unroll
  for (int i = 0; i < 4; ++i) {  // a thread that saw no row contributes the neutral encodings of -inf / +inf
    mine[4 * q + i] = float_to_ordered(hi[i]);
    mine[D + 4 * q + i] = ~float_to_ordered(lo[i]);
  }
  if (threadIdx.x == 0 && !poll_word(&h->cleared, launch)) report_status(ws, QB_ERR_TIMEOUT);
  __syncthreads();
  // groups of few columns: a thread each; of many: a warp each
  const bool by_warp = cols_per_group >= 16;
  const int lane = threadIdx.x & 31;
  const int first = by_warp ? (int)threadIdx.x >> 5 : (int)threadIdx.x, stride = by_warp ? (int)blockDim.x >> 5 : (int)blockDim.x;
  for (int g = first; g < groups; g += stride) {
    uint32_t eh = 0, el = 0;
    for (int s2 = 0; s2 < slots; ++s2) {
      const uint32_t* col = emb_smem + (size_t)s2 * 2 * D + g * cols_per_group;
      for (int c = by_warp ? lane : 0; c < cols_per_group; c += by_warp ? 32 : 1) {
        eh = max(eh, col[c]);
        el = max(el, col[D + c]);
      }
    }
    if (by_warp) {
      eh = __reduce_max_sync(0xffffffffu, eh);
      el = __reduce_max_sync(0xffffffffu, el);
      if (lane != 0) continue;
    }
    // the slots in the workspace only ever grow: skip the atomic when it cannot change anything
    const uint32_t have_h = __ldcg(g_hi + g), have_l = __ldcg(g_lo_inv + g);
    if (eh > have_h) atomicMax(g_hi + g, eh);
    if (el > have_l) atomicMax(g_lo_inv + g, el);
  }
}

// Encoded range of a group -> q0, 1/Delta, Delta; `report`: the one thread that says that the table is not finite.
__device__ __forceinline__ void embed_group(uint32_t hi_enc, uint32_t lo_inv, int levels, float* lo, float* inv, float* d,
                                            bool report, void* ws) {
  float l = ordered_to_float(~lo_inv), h = ordered_to_float(hi_enc);
  if (!(finite_f(l) && finite_f(h))) {
    if (report) report_status(ws, QB_ERR_NONFINITE);
    l = 0.0f;
    h = 0.0f;
  }
  float dl = __fdiv_rn(__fsub_rn(h, l), (float)levels);
  float iv = __fdiv_rn(1.0f, dl);
  if (!(dl > 0.0f) || !(iv <= 3.402823466e38f)) {  // constant group: Delta = 1, all codes 0
    dl = 1.0f;
    iv = 0.0f;
  }
  *lo = l;
  *inv = iv;
  *d = dl;
}

// Four codes of one float4 (columns of possibly different groups) as a 4k-bit field in the low bits.
// (x - q0) * (1/Delta), rounded half to even by adding 1.5 * 2^23; the add is written as a fused multiply-add with
// 1.0, since a packed mul and a packed add would be contracted and round the exact product.  x lies in the
// group's range, so the code needs no clamp; `& 2^k - 1` keeps a non-finite table's garbage in its field.
template <int BITS>
__device__ __forceinline__ uint32_t quant_columns(const float4& v, const float (&lo)[4], const float (&inv)[4]) {
  uint32_t b0, b1, b2, b3;
  asm("{\n\t.reg .b64 p0, p1, l0, l1, i0, i1, m2, o2;\n\t"
      "mov.b64 p0, {%4, %5};\n\tmov.b64 p1, {%6, %7};\n\t"
      "mov.b64 l0, {%8, %9};\n\tmov.b64 l1, {%10, %11};\n\t"
      "mov.b64 i0, {%12, %13};\n\tmov.b64 i1, {%14, %15};\n\t"
      "mov.b64 m2, {%16, %16};\n\tmov.b64 o2, {%17, %17};\n\t"
      "sub.rn.f32x2 p0, p0, l0;\n\tsub.rn.f32x2 p1, p1, l1;\n\t"
      "mul.rn.f32x2 p0, p0, i0;\n\tmul.rn.f32x2 p1, p1, i1;\n\t"
      "fma.rn.f32x2 p0, p0, o2, m2;\n\tfma.rn.f32x2 p1, p1, o2, m2;\n\t"
      "mov.b64 {%0, %1}, p0;\n\tmov.b64 {%2, %3}, p1;\n\t}"
      : "=r"(b0), "=r"(b1), "=r"(b2), "=r"(b3)
      : "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "f"(lo[0]), "f"(lo[1]), "f"(lo[2]), "f"(lo[3]), "f"(inv[0]), "f"(inv[1]),
        "f"(inv[2]), "f"(inv[3]), "f"(12582912.0f), "f"(1.0f));
  if constexpr (BITS == 8) {
    return __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410);
  } else {
    constexpr uint32_t cm = (1u << BITS) - 1u;
    return (b0 & cm) | ((b1 & cm) << BITS) | ((b2 & cm) << (2 * BITS)) | ((b3 & cm) << (3 * BITS));
  }
}

template <int BITS>
__global__ void __launch_bounds__(1024)
emb_pack_kernel(const float4* e, int64_t V, int d4, int slots, int cols_per_group,
                const uint32_t* g_hi, const uint32_t* g_lo_inv, uint32_t* packed, float* delta, float* q0, void* ws) {
  constexpr int L = (1 << BITS) - 1;
  pdl_begin();
  const int q = threadIdx.x % d4, slot = threadIdx.x / d4, lane = threadIdx.x & 31;
  const uint64_t pol = policy_evict_first();
  const int64_t step = (int64_t)gridDim.x * slots;
  float lo[4], inv[4];
  bool first = true;
  for (int64_t i = (int64_t)blockIdx.x * slots + slot; i < V; i += kEmbRows * step) {  // warp-uniform
    float4 v[kEmbRows];
#pragma unroll
    for (int j = 0; j < kEmbRows; ++j)
      if (i + j * step < V) v[j] = ldg_policy(e + (V - 1 - (i + j * step)) * d4 + q, pol);
    if (first) {  // the parameters, while the first rows are on their way
      first = false;
      uint32_t eh[4], el[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {  // all of them before the first store below, which may not be passed by a load
        eh[k] = g_hi[(4 * q + k) / cols_per_group];
        el[k] = g_lo_inv[(4 * q + k) / cols_per_group];
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int c = 4 * q + k, g = c / cols_per_group;
        const bool publish = blockIdx.x == 0 && slot == 0 && c == g * cols_per_group;  // first column of a group
        float d;
        embed_group(eh[k], el[k], L, &lo[k], &inv[k], &d, publish, ws);
        if (publish) {
          delta[g] = d;
          q0[g] = lo[k];
        }
      }
    }
#pragma unroll
    for (int j = 0; j < kEmbRows; ++j)
      if (i + j * step < V) {
        const int64_t r = V - 1 - (i + j * step);
        const uint32_t f = quant_columns<BITS>(v[j], lo, inv);
        uint8_t* row = reinterpret_cast<uint8_t*>(packed) + r * ((int64_t)d4 * BITS / 2);
        if (BITS == 8) reinterpret_cast<uint32_t*>(row)[q] = f;
        if (BITS == 4) reinterpret_cast<uint16_t*>(row)[q] = (uint16_t)f;
        if (BITS == 2) row[q] = (uint8_t)f;
        if (BITS == 3) {
          // output word `lane` (of the unit's twelve) = bits 32 lane .. of the lanes' 12-bit fields
          const int src = 32 * lane / 12, off = 32 * lane - 12 * src;
          const uint32_t f0 = __shfl_sync(0xffffffffu, f, src & 31), f1 = __shfl_sync(0xffffffffu, f, (src + 1) & 31);
          const uint32_t f2 = __shfl_sync(0xffffffffu, f, (src + 2) & 31), f3 = __shfl_sync(0xffffffffu, f, (src + 3) & 31);
          const uint64_t bits = (uint64_t)f0 | ((uint64_t)f1 << 12) | ((uint64_t)f2 << 24) | ((uint64_t)f3 << 36);
          if (lane < 12) reinterpret_cast<uint32_t*>(row)[(q >> 5) * 12 + lane] = (uint32_t)(bits >> off);
        }
      }
  }
}

template <int BITS, bool ADD>
__global__ void __launch_bounds__(1024)
emb_lookup_kernel(const int32_t* ids, int64_t T, const uint32_t* packed, int64_t V, int d4, int slots,
                  int cols_per_group, const float* delta, const float* q0, float4* out,
                  void* ws) {
  constexpr uint32_t cm = (1u << BITS) - 1u;
  pdl_begin();
  const int q = threadIdx.x % d4, slot = threadIdx.x / d4;
  const int64_t step = (int64_t)gridDim.x * slots;
  const int64_t words_per_row = (int64_t)d4 * BITS / 8;
  const int bit = 4 * q * BITS;  // position of this thread's field in the row's bit stream
  const int wi = bit >> 5, sh = bit & 31;
  float d[4], z[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int g = (4 * q + k) / cols_per_group;
    d[k] = delta[g];
    z[k] = q0[g];
  }
  for (int64_t i = (int64_t)blockIdx.x * slots + slot; i < T; i += step) {
    const int64_t t = ADD ? T - 1 - i : i;
    const int id = ids[t];
    float4* const o = out + t * d4 + q;
    float4 a;
    if (ADD) a = *o;
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
    if (id >= 0 && id < V) {
      const uint32_t* row = packed + (int64_t)id * words_per_row + wi;
      uint32_t f = row[0];
      if (BITS == 3 && sh + 12 > 32) f = __funnelshift_r(f, row[1], sh);
      else f >>= sh;
      r.x = __fmaf_rn(d[0], (float)(f & cm), z[0]);
      r.y = __fmaf_rn(d[1], (float)((f >> BITS) & cm), z[1]);
      r.z = __fmaf_rn(d[2], (float)((f >> (2 * BITS)) & cm), z[2]);
      r.w = __fmaf_rn(d[3], (float)((f >> (3 * BITS)) & cm), z[3]);
    } else if (q == 0) {
      report_status(ws, QB_ERR_INVALID, (int)t);
    }
    if (ADD) {
      r.x = __fadd_rn(a.x, r.x);
      r.y = __fadd_rn(a.y, r.y);
      r.z = __fadd_rn(a.z, r.z);
      r.w = __fadd_rn(a.w, r.w);
    }
    *o = r;
  }
}

// Rows that a block of about `threads` threads reads side by side, and the blocks that fill the device.
static int emb_slots(int d4) { return std::max(1, kEmbThreads / d4); }
// (resident blocks depend on the kernel and the block size alone: asked once for each)
enum { kEmbPack = 0, kEmbLookup = 1, kEmbLookupAdd = 2 };
template <class K>
static qb_status emb_grid(K kernel, int kind, int bits, int d4, int64_t rows, int sms, unsigned* grid) {
  static std::atomic<int> resident[3][9][kEmbMaxD / 128 + 1] = {};
  std::atomic<int>& known = resident[kind][bits][d4 / 32];
  const int slots = emb_slots(d4);
  int per_sm = known.load(std::memory_order_relaxed);
  if (per_sm == 0) {
    QB_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, d4 * slots, 0));
    per_sm = std::max(1, per_sm);
    known.store(per_sm, std::memory_order_relaxed);
  }
  *grid = (unsigned)std::min((rows + slots - 1) / slots, (int64_t)sms * per_sm);
  return QB_OK;
}

static qb_status validate_embedding(const char* who, int64_t V, int64_t D, int bits, int groups) {
  if (V <= 0 || D <= 0 || V > QB_MAX_MN || D > kEmbMaxD || !valid_bits(bits) || groups < 1 || D % groups != 0) {
    set_last_error("%s: invalid argument (V=%lld D=%lld bits=%d groups=%d; D <= %d)", who, (long long)V, (long long)D,
                   bits, groups, kEmbMaxD);
    return QB_ERR_INVALID;
  }
  if (D % 128 != 0) {
    set_last_error("%s: D must be a multiple of 128", who);
    return QB_ERR_ALIGN;
  }
  return QB_OK;
}

}  // namespace qb

extern "C" qb_status qb_quantize_embedding(const float* table, int64_t V, int64_t D, int bits, int groups,
                                           uint32_t* packed, float* delta, float* q0, void* ws, size_t ws_bytes,
                                           void* cuda_stream) {
  if (!table || !packed || !delta || !q0) {
    qb::set_last_error("qb_quantize_embedding: null pointer");
    return QB_ERR_INVALID;
  }
  qb_status st = qb::validate_embedding("qb_quantize_embedding", V, D, bits, groups);
  if (st != QB_OK) return st;
  if (!qb::aligned16(table) || !qb::aligned16(packed)) {
    qb::set_last_error("qb_quantize_embedding: table and packed must be 16-byte aligned");
    return QB_ERR_ALIGN;
  }
  if (!ws || ws_bytes < qb::ws_bytes_needed((int)D)) {
    qb::set_last_error("qb_quantize_embedding: workspace null or smaller than %zu bytes (8 bytes per column)",
                       qb::ws_bytes_needed((int)D));
    return QB_ERR_WORKSPACE;
  }
  int sms = 0;
  st = qb::require_sm100(&sms);
  if (st != QB_OK) return st;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  uint32_t* g_hi = reinterpret_cast<uint32_t*>(static_cast<char*>(ws) + qb::kWsRangeOff);
  uint32_t* g_lo = g_hi + groups;
  const int d4 = (int)(D / 4), slots = qb::emb_slots(d4), block = d4 * slots;
  const float4* e4 = reinterpret_cast<const float4*>(table);
  const int cpg = (int)(D / groups);
  // two blocks per SM; slots * D <= 4096 columns: at most 32 KB of shared memory
  const unsigned rblocks = (unsigned)std::min((V + slots - 1) / slots, (int64_t)sms * 2);
  QB_CUDA_TRY(qb::launch_kernel(qb::emb_range_kernel, rblocks, (unsigned)block, (size_t)slots * 2 * (size_t)D * sizeof(uint32_t), stream,
                                1, false, e4, V, d4, slots, cpg, groups, qb::l2_keep_fraction(4.0 * (double)V * (double)D), g_hi,
                                g_lo, ws));
  auto pack = bits == 2 ? qb::emb_pack_kernel<2> : (bits == 3 ? qb::emb_pack_kernel<3> : (bits == 4 ? qb::emb_pack_kernel<4> : qb::emb_pack_kernel<8>));
  unsigned grid = 0;
  st = qb::emb_grid(pack, qb::kEmbPack, bits, d4, V, sms, &grid);
  if (st != QB_OK) return st;
  QB_CUDA_TRY(qb::launch_kernel(pack, grid, (unsigned)block, 0, stream, 1, false, e4, V, d4, slots, cpg, g_hi, g_lo, packed, delta, q0,
                                ws));
  return QB_OK;
}

extern "C" qb_status qb_embedding_lookup(const int32_t* ids, int64_t T, const uint32_t* packed, const float* delta,
                                         const float* q0, int64_t V, int64_t D, int bits, int groups,
                                         int accumulate, float* out, void* ws, size_t ws_bytes, void* cuda_stream) {
  if (!ids || !packed || !delta || !q0 || !out || T <= 0 || T > QB_MAX_MN) {
    qb::set_last_error("qb_embedding_lookup: null pointer or T out of range (T=%lld)", (long long)T);
    return QB_ERR_INVALID;
  }
  qb_status st = qb::validate_embedding("qb_embedding_lookup", V, D, bits, groups);
  if (st != QB_OK) return st;
  if (!qb::aligned16(packed) || !qb::aligned16(out)) {
    qb::set_last_error("qb_embedding_lookup: packed and out must be 16-byte aligned");
    return QB_ERR_ALIGN;
  }
  if (!ws || ws_bytes < qb::kWsMinBytes) {
    qb::set_last_error("qb_embedding_lookup: workspace null or too small");
    return QB_ERR_WORKSPACE;
  }
  int sms = 0;
  st = qb::require_sm100(&sms);
  if (st != QB_OK) return st;
  cudaStream_t stream = (cudaStream_t)cuda_stream;
  const int d4 = (int)(D / 4), slots = qb::emb_slots(d4), block = d4 * slots;
  auto lookup = accumulate ? (bits == 2 ? qb::emb_lookup_kernel<2, true> : (bits == 3 ? qb::emb_lookup_kernel<3, true> : (bits == 4 ? qb::emb_lookup_kernel<4, true> : qb::emb_lookup_kernel<8, true>)))
                           : (bits == 2 ? qb::emb_lookup_kernel<2, false> : (bits == 3 ? qb::emb_lookup_kernel<3, false> : (bits == 4 ? qb::emb_lookup_kernel<4, false> : qb::emb_lookup_kernel<8, false>)));
  unsigned grid = 0;
  st = qb::emb_grid(lookup, accumulate ? qb::kEmbLookupAdd : qb::kEmbLookup, bits, d4, T, sms, &grid);
  if (st != QB_OK) return st;
  QB_CUDA_TRY(qb::launch_kernel(lookup, grid, (unsigned)block, 0, stream, 1, false, ids, T, packed, V, d4, slots, (int)(D / groups),
                                delta, q0, reinterpret_cast<float4*>(out), ws));
  return QB_OK;
}
