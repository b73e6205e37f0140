// Search over the compressed layouts (Section 3.5: compressed representations
// are duplicated for every assignment, the high-bitrate rows are stored once
// and rescore the best candidates): per query the R best approximate scores
// of its probed union, each point once, rescored exactly, the best k kept.
// Two layouts: per-row scaled E4M3 codes of every copy (approximate score
// s_q * s_x * sum q8 x8), and 4-bit PQ codes of every copy's residual x - C_p
// (approximate score <q, C_p> + sum_s <q_s, B[s][code_s]>).  A point counts by
// its copy in the partition the query probed earliest.
//
//   score_items    (partition, up to 32 of its queries): the partition's
//                  rows times the queries on the tensor cores, one 4-byte key
//                  per (query, row) written at the pair's place in the
//                  query's slice; 0 for a copy that does not count
//   finish_slices  a block per query: the R best rows of its slice, rescored
//                  exactly from the stored rows, and the best k of those
//
// Exactness.  The shortlist is defined on approximate scores summed in fp32 in
// a fixed order (`Rows::exact`).  The tensor cores add in another order, so a
// key holds such a score within delta only (`Rows::delta`).  With T the R-th
// largest key of a slice, a row above T + 2 delta is in the shortlist and one
// below T - 2 delta is not; those between are scored again in the defined
// order and ranked by it (score descending, lower id first), so the shortlist
// is the defined one.
//
// Why partition-major: a warp per (query, probe) pair read a partition's codes
// once per query and spent one table look-up or one fp8 conversion a term
// (10 000 queries, 10^7 x 96 fp8, t = 6, R = 1 000: scoring 6 230, selecting
// 2 990, rescoring 2 810 us; 1.18 M x 100 PQ4, t = 14, R = 100: 4 076, 1 884
// and 398 us).  Here the codes are read and decoded once for up to 32 queries:
// 768 and 954 us, 769 and 549 us.  The product is a few
// percent of the work, so warp-level MMAs fed from registers are used: a key
// leaves the registers it was computed in, with no TMEM round trip.
#include <algorithm>

#include "internal.cuh"
#include "scan_common.cuh"

namespace soar {

namespace {

constexpr int kWarps = 8;
constexpr int kThreads = 32 * kWarps;

// the values of two e4m3 codes, the low byte's first
__device__ __forceinline__ float2 fp8_pair_values(uint32_t two) {
  const __half2_raw h = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)two, __NV_E4M3);
  return __half22float2(__half2(h));
}

// D (16 x 8, fp32) += A (16 x 32 e4m3) B (32 x 8 e4m3)
__device__ __forceinline__ void mma_e4m3(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k32.row.col.f32.e4m3.e4m3.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// D (16 x 8, fp32) += A (16 x 16 bf16) B (16 x 8 bf16)
__device__ __forceinline__ void mma_bf16x16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                            uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// (x, y) as a bf16 pair (x in the low half), and what it leaves over
__device__ __forceinline__ uint32_t bf16_pair(float x, float y, float& rx, float& ry) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  const float2 f = __bfloat1622float2(h);
  rx = x - f.x;
  ry = y - f.y;
  return *reinterpret_cast<const uint32_t*>(&h);
}

// A layout gives: the queries of an item in shared memory, a fragment of 16
// rows' codes, its product with 8 * nt queries (accumulator element i of tile n:
// row lane / 4 + 8 * (i / 2), query 8 n + 2 * (lane % 4) + i % 2), and the score
// in the defined order.
struct Frag {
  uint4 a[2], b[2];
};

// Per-row scaled E4M3 codes.
struct Fp8Rows {
  static constexpr int kTiles = 4;      // most 8-query tiles per item
  static constexpr bool kScaled = true;
  const uint8_t* codes;
  int code_stride;
  const float* row_scales;
  const float* Qf;        // [nq][code_stride] code values
  const float* qscale;
  int k64;                // 64-byte steps of a row
  int tiles;              // 8-query tiles staged per item, at most kTiles

  __host__ __device__ int query_stride() const { return 64 * k64 + 16; }   // bytes; + 16: conflict-free reads
  __host__ __device__ size_t item_smem() const { return (size_t)8 * tiles * query_stride(); }
  __device__ void stage_shared(unsigned char*) const {}
  __device__ void stage_query(unsigned char* sm, int slot, int64_t q, int lane) const {
    uint8_t* dst = sm + slot * query_stride();
    for (int i = lane; i < 64 * k64; i += 32)
      dst[i] = (q >= 0 && i < code_stride)
                   ? (uint8_t)__nv_cvt_float_to_fp8(Qf[q * code_stride + i], __NV_SATFINITE, __NV_E4M3)
                   : (uint8_t)0;
  }
  // The K order is free as long as both operands agree: lane % 4 takes a 16-byte
  // chunk of each 64 bytes of a row, whose four words serve two MMAs.  A fragment
  // is two such steps of rows lane / 4 and lane / 4 + 8.
  __host__ __device__ int fragments() const { return (k64 + 1) / 2; }
  __device__ void load(Frag& f, const uint8_t* xa, const uint8_t* xb, int part, int lane) const {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int o = 64 * (2 * part + u) + 16 * (lane & 3);
      f.a[u] = f.b[u] = make_uint4(0u, 0u, 0u, 0u);
      if (o < code_stride) {
        f.a[u] = __ldg(reinterpret_cast<const uint4*>(xa + o));
        f.b[u] = __ldg(reinterpret_cast<const uint4*>(xb + o));
      }
    }
  }
  __device__ void multiply(const unsigned char* sm, const Frag& f, int part, int nt, int lane, float (&acc)[kTiles][4]) const {
    const unsigned char* qw = sm + (lane >> 2) * query_stride() + 16 * (lane & 3) + 128 * part;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (2 * part + u >= k64) break;
#pragma unroll
      for (int n = 0; n < kTiles; ++n)
        if (n < nt) {
          const uint4 w = *reinterpret_cast<const uint4*>(qw + 8 * n * query_stride() + 64 * u);
          mma_e4m3(acc[n], f.a[u].x, f.b[u].x, f.a[u].y, f.b[u].y, w.x, w.y);
          mma_e4m3(acc[n], f.a[u].z, f.b[u].z, f.a[u].w, f.b[u].w, w.z, w.w);
        }
    }
  }
  __device__ float row_factor(int64_t r) const { return row_scales[r]; }
  __device__ float query_factor(int64_t q, int64_t) const { return qscale[q]; }
  __device__ static float combine(float acc, float rf, float qf) { return acc * qf * rf; }
  // finishing: the query's code values in shared memory
  __host__ __device__ int query_floats() const { return code_stride; }
  __device__ float3 stage_finish(float* qs, int64_t q, const float*, int) const {
    float n2 = 0.f;
    for (int i = threadIdx.x; i < code_stride; i += kThreads) {
      const float v = Qf[q * (int64_t)code_stride + i];
      qs[i] = v;
      n2 = fmaf(v, v, n2);
    }
    return make_float3(n2, 0.f, 0.f);
  }
  // |key's score - defined score|: both sums of exact products have at most
  // code_stride fp32 additions, off by 2^-24 (defined order) and at most 2^-23
  // (tensor cores: their width is not documented; whole shortlists of rows that one
  // large product and many small ones make up are compared with the defined ones in
  // tests/test_gpu_shortlist_defined.py) of a partial sum that stays below ||q8||
  // ||x8||, and ||x8|| <= 448 sqrt(d); the rest covers the scaling.
  // The scale of a row that the query meets is at most smax.
  __device__ float delta(float3 v, int64_t q, float smax) const {
    return ldexpf((float)code_stride, -22) * sqrtf(v.x) * 448.f * sqrtf((float)code_stride) * qscale[q] * smax;
  }
  __device__ bool tabulate(const float*, float*, int) const { return false; }
  __device__ float exact_tabulated(const float*, int64_t, float) const { return 0.f; }
  __device__ float exact(const float* qs, int64_t q, int64_t r, float) const {
    const uint4* x = reinterpret_cast<const uint4*>(codes + r * (int64_t)code_stride);
    float acc = 0.f;
    for (int c = 0; c < code_stride / 16; ++c) {
      const uint4 v = __ldg(x + c);
      const uint32_t wv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int b = 0; b < 4; b += 2) {
          const float2 w = fp8_pair_values((wv[i] >> (8 * b)) & 0xffffu);
          acc = fmaf(qs[16 * c + 4 * i + b], w.x, acc);
          acc = fmaf(qs[16 * c + 4 * i + b + 1], w.y, acc);
        }
    }
    return acc * qscale[q] * row_scales[r];
  }
};

// PQ4 codes: approx = <q, C_p> + sum_s LUT[s][code_s], LUT[s][j] = <q_s, B[s][j]>.
// A subspace's two dimensions are one bf16 pair of an MMA operand, so decoding
// a code is one shared-memory read of its centre (hi and lo parts); centres and
// queries enter as hi + lo and the lo lo product is dropped.
struct Pq4Rows {
  static constexpr bool kScaled = false;
  static constexpr int kTiles = 4;      // (eight took 122 registers: two blocks an SM, 1 346 us)
  const uint8_t* codes;
  int code_stride, m, d;
  const float* B;         // [m][16][2]
  const float* Qf;        // [nq][qstride] fp32
  int qstride;
  const float* base;      // [pairs] <q, C_p>
  int steps;              // K steps of 8 subspaces
  int tiles;

  // a query's K step holds, for each lane % 4, its four operand words (hi, hi + 4 pairs on, lo, lo + 4 pairs on)
  __host__ __device__ int query_stride() const { return 64 * steps + 16; }   // bytes; + 16: conflict-free reads
  __host__ __device__ size_t item_smem() const {
    return (size_t)8 * steps * 16 * 8 + (size_t)8 * tiles * query_stride();
  }
  __device__ void stage_shared(unsigned char* sm) const {
    uint2* lut = reinterpret_cast<uint2*>(sm);
    for (int e = threadIdx.x; e < 8 * steps * 16; e += kThreads) {
      float x = 0.f, y = 0.f, rx, ry, u, v;
      if (e < m * 16) {
        const float2 c = reinterpret_cast<const float2*>(B)[e];
        x = c.x;
        y = c.y;
      }
      const uint32_t hi = bf16_pair(x, y, rx, ry);
      lut[e] = make_uint2(hi, bf16_pair(rx, ry, u, v));
    }
  }
  __device__ void stage_query(unsigned char* sm, int slot, int64_t q, int lane) const {
    uint32_t* dst = reinterpret_cast<uint32_t*>(sm + (size_t)8 * steps * 16 * 8 + slot * query_stride());
    for (int i = lane; i < 8 * steps; i += 32) {
      float x = 0.f, y = 0.f, rx, ry, u, v;
      if (q >= 0 && i < m) {
        const float2 w = *reinterpret_cast<const float2*>(Qf + q * (int64_t)qstride + 2 * i);
        x = w.x;
        y = w.y;
      }
      uint32_t* at = dst + 16 * (i / 8) + 4 * (i % 4) + (i / 4) % 2;
      at[0] = bf16_pair(x, y, rx, ry);
      at[2] = bf16_pair(rx, ry, u, v);
    }
  }
  // A fragment is 32 code bytes (eight K steps) of rows lane / 4 and lane / 4 + 8.
  __host__ __device__ int fragments() const { return (steps + 7) / 8; }
  __device__ void load(Frag& f, const uint8_t* xa, const uint8_t* xb, int part, int) const {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int o = 32 * part + 16 * u;
      f.a[u] = f.b[u] = make_uint4(0u, 0u, 0u, 0u);
      if (o < code_stride) {
        f.a[u] = __ldg(reinterpret_cast<const uint4*>(xa + o));
        f.b[u] = __ldg(reinterpret_cast<const uint4*>(xb + o));
      }
    }
  }
  __device__ void multiply(const unsigned char* sm, const Frag& f, int part, int nt, int lane, float (&acc)[kTiles][4]) const {
    const uint2* lut = reinterpret_cast<const uint2*>(sm) + (lane & 3) * 16 + 1024 * part;
    const unsigned char* qw = sm + (size_t)8 * steps * 16 * 8 + (lane >> 2) * query_stride() + 16 * (lane & 3) + 512 * part;
    const int sh = 4 * (lane & 3);
#pragma unroll
    for (int ks = 0; ks < 8; ++ks) {
      if (8 * part + ks >= steps) break;
      const uint4 ca = f.a[ks / 4], cb = f.b[ks / 4];
      const uint32_t wa = (ks % 4 == 0 ? ca.x : ks % 4 == 1 ? ca.y : ks % 4 == 2 ? ca.z : ca.w) >> sh;
      const uint32_t wb = (ks % 4 == 0 ? cb.x : ks % 4 == 1 ? cb.y : ks % 4 == 2 ? cb.z : cb.w) >> sh;
      const uint2* l0 = lut + 128 * ks;
      const uint2 a0 = l0[wa & 15u], a1 = l0[wb & 15u], a2 = l0[64 + ((wa >> 16) & 15u)], a3 = l0[64 + ((wb >> 16) & 15u)];
#pragma unroll
      for (int n = 0; n < kTiles; ++n)
        if (n < nt) {
          const uint4 v = *reinterpret_cast<const uint4*>(qw + 8 * n * query_stride() + 64 * ks);
          mma_bf16x16(acc[n], a0.x, a1.x, a2.x, a3.x, v.x, v.y);
          mma_bf16x16(acc[n], a0.y, a1.y, a2.y, a3.y, v.x, v.y);
          mma_bf16x16(acc[n], a0.x, a1.x, a2.x, a3.x, v.z, v.w);
        }
    }
  }
  __device__ float row_factor(int64_t) const { return 0.f; }
  __device__ float query_factor(int64_t, int64_t pair) const { return base[pair]; }
  __device__ static float combine(float acc, float, float qf) { return qf + acc; }
  __host__ __device__ int query_floats() const { return qstride; }
  // this thread's shares of ||q||^2 and of sum_s max_j ||B[s][j]||^2, and its largest |<q, C_p>|
  __device__ float3 stage_finish(float* qs, int64_t q, const float* bases, int tq) const {
    float3 v = make_float3(0.f, 0.f, 0.f);
    for (int i = threadIdx.x; i < qstride; i += kThreads) {
      const float x = Qf[q * (int64_t)qstride + i];
      qs[i] = x;
      v.x = fmaf(x, x, v.x);
    }
    for (int s = threadIdx.x; s < m; s += kThreads) {
      float most = 0.f;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float2 c = reinterpret_cast<const float2*>(B)[16 * s + j];
        most = fmaxf(most, fmaf(c.y, c.y, c.x * c.x));
      }
      v.y += most;
    }
    for (int j = threadIdx.x; j < tq; j += kThreads) v.z = fmaxf(v.z, fabsf(bases[j]));
    return v;
  }
  // 3 * 2^-18 ||q|| ||r|| for the dropped parts, 2^-23 of it for each of the
  // 3 d + d / 2 additions, and the rounding of base + sum; a factor to spare.
  __device__ float delta(float3 v, int64_t, float) const {
    const float qb = sqrtf(v.x) * sqrtf(v.y);
    return qb * (ldexpf(1.f, -14) + ldexpf((float)d, -20)) + ldexpf(v.z + qb, -21);
  }
  // the query's products with every centre, for many rows (all threads), where they fit `room` floats
  __device__ bool tabulate(const float* qs, float* table, int room) const {
    if (16 * m > room) return false;
    for (int e = threadIdx.x; e < 16 * m; e += kThreads) {
      const float2 c = reinterpret_cast<const float2*>(B)[e];
      table[e] = fmaf(qs[2 * (e / 16) + 1], c.y, qs[2 * (e / 16)] * c.x);
    }
    return true;
  }
  __device__ float exact_tabulated(const float* table, int64_t r, float pair_base) const {
    const uint32_t* x = reinterpret_cast<const uint32_t*>(codes + r * (int64_t)code_stride);
    float acc = 0.f;
#pragma unroll 4
    for (int w = 0; w < m / 8; ++w) {
      const uint32_t v = __ldg(x + w);
#pragma unroll
      for (int b = 0; b < 8; ++b) acc += table[16 * (8 * w + b) + ((v >> (4 * b)) & 15u)];
    }
    for (int s = m / 8 * 8; s < m; ++s) acc += table[16 * s + ((__ldg(x + s / 8) >> (4 * (s % 8))) & 15u)];
    return pair_base + acc;
  }
  __device__ float exact(const float* qs, int64_t, int64_t r, float pair_base) const {
    const uint32_t* x = reinterpret_cast<const uint32_t*>(codes + r * (int64_t)code_stride);
    float acc = 0.f;
    for (int s = 0; s < m; ++s) {
      const float2 c = reinterpret_cast<const float2*>(B)[16 * s + ((__ldg(x + s / 8) >> (4 * (s % 8))) & 15u)];
      acc += fmaf(qs[2 * s + 1], c.y, qs[2 * s] * c.x);
    }
    return pair_base + acc;
  }
};

// base[e] = <q, C_p> of every probed pair in fp32 (a warp per pair: lanes over
// the dimensions, a fixed shuffle tree).
__global__ void pair_bases(const float* __restrict__ Qf, int qstride, const float* __restrict__ C, int d,
                           const int32_t* __restrict__ top, const int32_t* __restrict__ tpq, int64_t q0, int64_t nq,
                           int t, float* __restrict__ base) {
  const int64_t e = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (e >= nq * t) return;
  const int64_t q = q0 + e / t;
  if (tpq && (int)(e % t) >= min(max(tpq[q], 0), t)) return;
  const float* qrow = Qf + q * (int64_t)qstride;
  const float* cp = C + (int64_t)top[q0 * t + e] * d;
  float v = 0.f;
  for (int k = lane; k < d; k += 32) v = fmaf(qrow[k], cp[k], v);
  v = warp_sum(v);
  if (lane == 0) base[e] = v;
}

// Where the queries' keys lie.  Slices of the longest possible length where those
// fit (start null); else one behind the other, each on 16 bytes, a pass taking
// those that start in [from, to).
struct Slices {
  uint32_t* keys;
  const int64_t* start;     // [queries + 1]
  int64_t stride, from, to;
  __device__ int64_t at(int64_t ql) const { return (start ? start[ql] : ql * stride) - from; }
  __device__ bool in_pass(int64_t ql) const { return !start || (start[ql] >= from && start[ql] < to); }
};

// Each probed pair's first position in its query's slice (the sizes of the
// query's earlier probed partitions added up) and the slice's length, in packed
// (unless null, [nq + 1]) rounded up to four; smax cleared; a warp per query.
__global__ void pair_offsets(const int64_t* __restrict__ off, const int32_t* __restrict__ top,
                             const int32_t* __restrict__ tpq, int64_t q0, int64_t nq, int t,
                             int64_t* __restrict__ pos, int64_t* __restrict__ counts, int64_t* __restrict__ packed,
                             int* __restrict__ smax) {
  const int64_t ql = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (ql >= nq) return;
  const int64_t q = q0 + ql;
  const int tq = tpq ? min(max(tpq[q], 0), t) : t;
  int64_t acc = 0;
  for (int j0 = 0; j0 < tq; j0 += 32) {
    const int j = j0 + lane;
    int64_t v = 0;
    if (j < tq) {
      const int p = top[q * (int64_t)t + j];
      v = off[p + 1] - off[p];
    }
    int64_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (j < tq) pos[ql * t + j] = acc + x - v;
    acc += __shfl_sync(0xffffffffu, x, 31);
  }
  if (lane == 0) {
    counts[ql] = acc;
    if (smax) smax[ql] = 0;
    if (packed) packed[ql] = (acc + 3) / 4 * 4;
    if (packed && ql == 0) packed[nq] = 0;
  }
}

// The probe counts of the queries in a pass, 0 for the others.
__global__ void pass_counts(Slices sl, const int32_t* __restrict__ tpq, int64_t q0, int64_t nq, int t,
                            int32_t* __restrict__ counts) {
  const int64_t ql = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (ql < nq) counts[ql] = !sl.in_pass(ql) ? 0 : tpq ? min(max(tpq[q0 + ql], 0), t) : t;
}

// Which of an item's queries probed a partition before this one: a hash table
// in shared memory from partition to a mask of the item's query slots, so that a
// row looks its point's other partitions up once for all queries (comparing each
// query's earlier probes row by row was two thirds of the scoring's
// instructions).  The table is as large as the item's earlier probes or the
// partitions need, whichever are fewer; an item with more of both compares
// (50 queries of 200 probes over 400 partitions, two spills: 1 111 us compared, 152
// hashed).
constexpr int kHashSize = 2048, kHashMost = 1536;
struct ProbeMasks {
  int32_t key[kHashSize];
  uint32_t mask[kHashSize];
  __device__ static int at(int32_t p, int bits) { return (int)(((uint32_t)p * 2654435769u) >> (32 - bits)); }
  __device__ void clear(int bits) {
    for (int i = threadIdx.x; i < 1 << bits; i += blockDim.x) {
      key[i] = -1;
      mask[i] = 0u;
    }
  }
  __device__ void add(int32_t p, uint32_t bit, int bits) {
    for (int h = at(p, bits);; h = (h + 1) & ((1 << bits) - 1)) {
      const int32_t old = atomicCAS(&key[h], -1, p);
      if (old == -1 || old == p) {
        atomicOr(&mask[h], bit);
        return;
      }
    }
  }
  __device__ uint32_t find(int32_t p, int bits) const {
    for (int h = at(p, bits);; h = (h + 1) & ((1 << bits) - 1)) {
      const int32_t k = key[h];
      if (k == p) return mask[h];
      if (k == -1) return 0u;
    }
  }
};

// Work items (partition, up to 32 of its queries; blockIdx.y takes every
// gridDim.y-th step of 128 rows): keys of every (query, row).  A key is the
// order-preserving image of the score, 0 for a copy that does not count.  smax
// (FP8, [queries of the pass], zero before the launch): the largest scale of the
// rows each query met, which are positive and so ordered like their bits.
template <typename Rows>
__global__ void __launch_bounds__(kThreads, 3) score_items(Rows rows, IvfWork work, const int32_t* __restrict__ ids,
                                                        const int32_t* __restrict__ assign, int a,
                                                        const int32_t* __restrict__ top, int64_t q0, Slices sl,
                                                        const int64_t* __restrict__ pos, int* __restrict__ smax) {
  constexpr unsigned kFull = 0xffffffffu;
  constexpr int QB = 8 * Rows::kTiles;
  static_assert(QB <= 32, "a mask word holds the item's queries");
  extern __shared__ __align__(16) unsigned char sl_smem[];
  __shared__ uint32_t* out_s[QB];               // where the pair's keys start
  __shared__ const int32_t* list_s[QB];         // the query's probes
  __shared__ int32_t j_s[QB];                   // how many of them come before this partition
  __shared__ float qf_s[QB];
  __shared__ int64_t q_s[QB];
  __shared__ ProbeMasks masks;
  __shared__ int earlier_s, most_s;
  const int item = blockIdx.x;
  if (item >= work.count()) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // the item's partition: the last entry of item_base at or below it, 32 probes at a time
  int oi = 0;
  for (int len = work.c; len > 1;) {
    const int step = (len + 31) / 32, at = oi + lane * step;
    const unsigned below = __ballot_sync(kFull, lane * step < len && work.item_base[min(at, work.c)] <= item);
    const int take = __popc(below) - 1;
    oi += take * step;
    len = min(step, len - take * step);
  }
  const int p = work.order[oi];
  const int64_t e0 = work.pair_off[p] + (int64_t)(item - work.item_base[oi]) * work.qb;
  const int nqi = (int)min((int64_t)work.qb, work.pair_off[p + 1] - e0);
  const int64_t r0 = work.part_off[p], r1 = work.part_off[p + 1];
  const int nrows = (int)(r1 - r0);
  rows.stage_shared(sl_smem);
  static_assert(QB <= 32, "a warp fills the slots");
  if (threadIdx.x < 32) {                       // a thread per query slot
    const int i = threadIdx.x;
    int64_t q = -1;
    int j = 0;
    if (i < nqi) {
      const int pr = work.pair_vals[e0 + i];    // ql * t + j
      const int64_t ql = pr / work.tmax;
      j = (int)(pr - ql * work.tmax);
      q = q0 + ql;
      out_s[i] = sl.keys + sl.at(ql) + pos[pr];
      list_s[i] = top + q * (int64_t)work.tmax;
      j_s[i] = j;
      qf_s[i] = rows.query_factor(q, pr);
    }
    if (i < QB) q_s[i] = q;
    j = warp_sum(j);
    if (i == 0) {
      earlier_s = j;
      most_s = 0;
    }
  }
  __syncthreads();
#pragma unroll 4
  for (int i = w; i < 8 * rows.tiles; i += kWarps) rows.stage_query(sl_smem, i, q_s[i], lane);
  const int probed = min(earlier_s, work.c);    // distinct partitions among the earlier probes, at most
  const bool hashed = probed <= kHashMost;
  int bits = 6;
  while (hashed && (1 << bits) < kHashSize && (1 << bits) < 8 * probed) ++bits;
  if (a > 1 && hashed) masks.clear(bits);
  __syncthreads();
  if (a > 1 && hashed) {
    for (int i = w; i < nqi; i += kWarps)
      for (int jj = lane; jj < j_s[i]; jj += 32) masks.add(list_s[i][jj], 1u << i, bits);
    __syncthreads();
  }
  const int nt = (nqi + 7) / 8, g = lane >> 2, tig = lane & 3;
  // the item's queries whose earlier probes hold the row's point
  const auto dropped = [&](int32_t o) -> uint32_t {
    if (hashed) return masks.find(o, bits);
    uint32_t m = 0u;
    for (int i = 0; i < nqi; ++i)
      for (int jj = 0; jj < j_s[i]; ++jj)
        if (list_s[i][jj] == o) {
          m |= 1u << i;
          break;
        }
    return m;
  };
  float most = 0.f;
  const int step = 16 * kWarps * (int)gridDim.y;
  int t0 = 16 * (w + kWarps * (int)blockIdx.y);
  const int32_t* pids = ids + r0;
  const auto fetch_id = [&](int tile) { return tile + (lane & 15) < nrows ? pids[tile + (lane & 15)] : -1; };
  int32_t id = fetch_id(t0), next_id = fetch_id(t0 + step);
  int2 next_assign = make_int2(-1, -1);
  float next_rf = 0.f;
  const auto fetch_row = [&](int tile) {        // of the rows whose ids are in `id`
    next_rf = 0.f;
    if (id < 0) return;
    next_rf = rows.row_factor(r0 + tile + (lane & 15));
    if (a == 2) next_assign = __ldg(reinterpret_cast<const int2*>(assign) + id);
  };
  fetch_row(t0);
  // rows past the end read the partition's first row instead
  const auto row_codes = [&](int r) { return rows.codes + (r0 + (r < nrows ? r : 0)) * rows.code_stride; };
  const int parts = rows.fragments();
  for (; t0 < nrows; t0 += step) {
    float acc[Rows::kTiles][4];
#pragma unroll
    for (int n = 0; n < Rows::kTiles; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[n][i] = 0.f;
    const float rf = next_rf;
    const int2 as = next_assign;
    const int32_t id_now = id;
    // the next step's assignments and the ids of the step after it are on their way during this one
    id = next_id;
    fetch_row(t0 + step);
    next_id = fetch_id(t0 + 2 * step);
    Frag f;
    rows.load(f, row_codes(t0 + g), row_codes(t0 + g + 8), 0, lane);
    most = fmaxf(most, rf);
    // lane l: the queries for which row l % 16 does not count
    uint32_t drop = 0u;
    if (a == 2) {
      if (id_now >= 0) drop = dropped(as.x == p ? as.y : as.x);
    } else if (a > 2 && id_now >= 0) {
      for (int i = 0; i < a; ++i) {
        const int v = assign[(int64_t)id_now * a + i];
        if (v != p) drop |= dropped(v);
      }
    }
    rows.multiply(sl_smem, f, 0, nt, lane, acc);
    for (int part = 1; part < parts; ++part) {                  // wide rows
      rows.load(f, row_codes(t0 + g), row_codes(t0 + g + 8), part, lane);
      rows.multiply(sl_smem, f, part, nt, lane, acc);
    }
    const float rfa = __shfl_sync(kFull, rf, g), rfb = __shfl_sync(kFull, rf, g + 8);
    const uint32_t da = __shfl_sync(kFull, drop, g) >> (2 * tig), db = __shfl_sync(kFull, drop, g + 8) >> (2 * tig);
    const bool ina = t0 + g < nrows, inb = t0 + g + 8 < nrows;
#pragma unroll
    for (int n = 0; n < Rows::kTiles; ++n) {
      if (n >= nt) break;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int slot = 8 * n + 2 * tig + i;
        if (slot >= nqi) continue;
        uint32_t* out = out_s[slot] + (t0 + g);
        const float qf = qf_s[slot];
        if (ina) out[0] = (da >> (8 * n + i)) & 1u ? 0u : float_key(Rows::combine(acc[n][i], rfa, qf));
        if (inb) out[8] = (db >> (8 * n + i)) & 1u ? 0u : float_key(Rows::combine(acc[n][2 + i], rfb, qf));
      }
    }
  }
  if (smax) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) most = fmaxf(most, __shfl_xor_sync(kFull, most, o));
    if (lane == 0) atomicMax(&most_s, __float_as_int(most));
    __syncthreads();
    if ((int)threadIdx.x < nqi) atomicMax(smax + (q_s[threadIdx.x] - q0), most_s);
  }
}

// One 16-byte chunk of a stored row, elements in ascending order.
__device__ __forceinline__ float chunk_dot(const float* q, uint4 v, float s, float) {
  const float4 a = *reinterpret_cast<const float4*>(q);
  s = fmaf(a.x, __uint_as_float(v.x), s);
  s = fmaf(a.y, __uint_as_float(v.y), s);
  s = fmaf(a.z, __uint_as_float(v.z), s);
  return fmaf(a.w, __uint_as_float(v.w), s);
}
__device__ __forceinline__ float chunk_dot(const float* q, uint4 v, float s, __nv_bfloat16) {
  const float4 a = *reinterpret_cast<const float4*>(q), b = *reinterpret_cast<const float4*>(q + 4);
  s = fmaf(a.x, __uint_as_float(v.x << 16), s);
  s = fmaf(a.y, __uint_as_float(v.x & 0xffff0000u), s);
  s = fmaf(a.z, __uint_as_float(v.y << 16), s);
  s = fmaf(a.w, __uint_as_float(v.y & 0xffff0000u), s);
  s = fmaf(b.x, __uint_as_float(v.z << 16), s);
  s = fmaf(b.y, __uint_as_float(v.z & 0xffff0000u), s);
  s = fmaf(b.z, __uint_as_float(v.w << 16), s);
  return fmaf(b.w, __uint_as_float(v.w & 0xffff0000u), s);
}

// Exact fp32 <q, x> of 32 stored rows, lane l's row l (id < 0: none), each sum
// in ascending order by its lane.  The rows pass through shared memory nine
// 16-byte chunks at a time, copied by the whole warp so that a row's bytes are
// read together: a lane reading its own row touches 32 lines an instruction
// (10^7 rows of 192 bytes: 1 150 of 1 654 us, about 480 staged).  Nine chunks a row also
// keep the lanes' 16-byte reads on distinct banks.
constexpr int kRowChunks = 9;
template <typename OT>
__device__ float warp_rows_dot(const float* q, const OT* __restrict__ rows, int stride, int32_t id, uint4* buf, int lane) {
  constexpr unsigned kFull = 0xffffffffu;
  constexpr int E = 16 / (int)sizeof(OT);
  const int chunks = stride / E, blocks = (chunks + kRowChunks - 1) / kRowChunks, per = (chunks + blocks - 1) / blocks;
  const int many = 32 - __clz(__ballot_sync(kFull, id >= 0));      // rows up to the last one there is
  float s = 0.f;
  for (int c0 = 0; c0 < chunks; c0 += per) {
    const int m = min(per, chunks - c0);
    __syncwarp();
    for (int i0 = 0; i0 < many * m; i0 += 32) {
      const int i = i0 + lane, r = i / m, c = i - r * m;
      const int32_t rid = __shfl_sync(kFull, id, r & 31);
      if (r < many && rid >= 0)
        cp_async16(buf + r * kRowChunks + c, reinterpret_cast<const uint4*>(rows + (int64_t)rid * stride) + c0 + c);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    if (id >= 0)
      for (int c = 0; c < m; ++c) s = chunk_dot(q + (c0 + c) * E, buf[lane * kRowChunks + c], s, OT());
  }
  return s;
}

constexpr int kBins = 2048;
constexpr int kBand = 1024;         // rows near the R-th score ranked in the defined order
constexpr int kSample = 8;          // keys a thread samples
constexpr int kProbeTable = 64;     // probes looked up in shared memory up to this t

// Rows of a slice kept in shared memory: those at or above a bound that a
// sample puts somewhat below the R-th best.
__host__ __device__ inline int kept_rows(int R) { return 2 * R + 1024; }

// Ascending bitonic sort of buf[0, N), N a power of two (all threads).
__device__ void block_sort(uint64_t* buf, int N) {
  for (int size = 2; size <= N; size <<= 1)
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int i = threadIdx.x; i < N / 2; i += kThreads) {
        const int a = 2 * i - (i & (stride - 1)), b = a + stride;
        const uint64_t x = buf[a], y = buf[b];
        if ((x > y) == ((a & size) == 0)) {
          buf[a] = y;
          buf[b] = x;
        }
      }
      __syncthreads();
    }
}

// A block per query: the R best rows of its slice (see the file comment), their
// exact scores, the best k.
//   keep     2 048 sampled keys put a bound somewhat below the R-th best; the
//            rows at or above it go to shared memory in one pass over the slice
//            (where the sample misleads, the passes below run over the slice)
//   bins     the kept rows are counted in 2 048 linear bins (keys outside their
//            range fall into the end bins, which keeps the bins ordered); the
//            R-th best lies in one bin, and the bins within 2 delta of that
//            one are the band
//   list     every row above the band, then the band's best in the defined
//            order.  Where linear bins cannot tell (rows of very uneven length, a
//            misleading sample, infinities), the R-th largest key of the slice is
//            found byte by byte and the band is taken around it; a band that does
//            not fit (thousands of near-equal scores, or a delta as wide as the
//            scores' spread) has its defined scores computed once, in place of its
//            keys.  (A radix select that computed every row's defined score nine
//            times took its place before: 10 000 queries, 10^6 x 96 in 1 000
//            partitions, t = 6, one row in a thousand 1 000 times longer, FP8 with
//            R = 1 000 42.0 ms, now 7.8; PQ4 with R = 100 34.6, now 6.1; 1.6 and
//            1.3 with rows of equal length)
//   rescore  a thread per row; the best k by per-warp sorted lists (k <= 32) or
//            a sort
// Bound: the latency of one pass over the slice and of the scattered rows.
template <typename Rows, typename OT>
__global__ void __launch_bounds__(kThreads) finish_slices(
    Rows rows, Slices sl, const int64_t* __restrict__ counts, const int64_t* __restrict__ pos, const int32_t* __restrict__ top, const int32_t* __restrict__ tpq, int64_t q0,
    int t, const int64_t* __restrict__ off, const int32_t* __restrict__ ids, const float* __restrict__ base,
    const float* __restrict__ smax, const void* __restrict__ Q, int qdt, int d, const OT* __restrict__ orig,
    int ostride, int R, int k, int stage_at, int64_t* __restrict__ ids_out, float* __restrict__ scores_out) {
  constexpr unsigned kFull = 0xffffffffu;
  extern __shared__ __align__(16) unsigned char fs_smem[];
  __shared__ int32_t warp_s[32];
  __shared__ float red_s[5][kWarps];
  __shared__ int n_list, n_band, n_kept, bin_s, above_s;
  __shared__ float lo_s, hi_s, delta_s;
  __shared__ int at_s[kProbeTable];             // where the probes' rows start in the slice
  __shared__ int64_t row_s[kProbeTable];        // and the index row of the slice's position 0 in that probe
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int64_t ql = blockIdx.x, q = q0 + ql;
  if (!sl.in_pass(ql)) return;
  uint32_t* K = sl.keys + sl.at(ql);            // (rewritten in place by the rarest branch)
  const int n = (int)counts[ql];
  const int tq = tpq ? min(max(tpq[q], 0), t) : t;
  const int64_t* qpos = pos + ql * t;
  const int32_t* probes = top + q * (int64_t)t;
  // shared memory: query row, query for the defined order, histogram / band
  // keys, band, list, kept rows / exact keys
  const int cap = kept_rows(R);
  float* qrow = reinterpret_cast<float*>(fs_smem);
  float* qs = qrow + (ostride + 3) / 4 * 4;
  int* hist = reinterpret_cast<int*>(qs + (rows.query_floats() + 3) / 4 * 4);
  uint64_t* band_key = reinterpret_cast<uint64_t*>(hist);                 // over the histogram once the bin is known
  int32_t* band = reinterpret_cast<int32_t*>(hist + kBins);               // [kBand]
  int32_t* list = band + kBand;                                           // [R] positions in the slice, then ids
  uint32_t* kept = reinterpret_cast<uint32_t*>(
      fs_smem + (reinterpret_cast<unsigned char*>(list + (R + 1) / 2 * 2) - fs_smem + 15) / 16 * 16);   // [cap] keys
  int32_t* kept_at = reinterpret_cast<int32_t*>(kept + cap);              // [cap] positions
  // once the list is known: the exact keys and a warp's staged rows (over each
  // other for k <= 32, where the keys are the warps' few best)
  uint64_t* ex = reinterpret_cast<uint64_t*>(kept);                       // [sorted]
  uint4* stage = reinterpret_cast<uint4*>(fs_smem + stage_at) + 32 * kRowChunks * w;

  for (int i = tid; i < ostride; i += kThreads)
    qrow[i] = i >= d ? 0.f
              : qdt == SOAR_F32 ? static_cast<const float*>(Q)[q * d + i]
                                : __bfloat162float(static_cast<const __nv_bfloat16*>(Q)[q * d + i]);
  if (tid == 0) n_list = n_band = n_kept = 0;
  if (tid < tq && tid < kProbeTable) {
    at_s[tid] = (int)qpos[tid];
    row_s[tid] = off[probes[tid]] - qpos[tid];
  }
  const bool short_slice = n <= R;              // every row that counts is listed
  uint32_t sample[kSample];
  float lo = INFINITY, hi = -INFINITY, delta = 0.f;
  if (!short_slice) {
    float3 norms = rows.stage_finish(qs, q, base ? base + ql * t : nullptr, tq);
    norms.x = warp_sum(norms.x);
    norms.y = warp_sum(norms.y);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) norms.z = fmaxf(norms.z, __shfl_xor_sync(kFull, norms.z, o));
    // a sample and its range
#pragma unroll
    for (int u = 0; u < kSample; ++u) {
      const int64_t i = (int64_t)(u * kThreads + tid) * n / (kSample * kThreads);
      sample[u] = i < n ? K[i] : 0u;
    }
#pragma unroll
    for (int u = 0; u < kSample; ++u)
      if (sample[u]) {
        lo = fminf(lo, key_float(sample[u]));
        hi = fmaxf(hi, key_float(sample[u]));
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo = fminf(lo, __shfl_xor_sync(kFull, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(kFull, hi, o));
    }
    if (lane == 0) {
      red_s[0][w] = lo;
      red_s[1][w] = hi;
      red_s[2][w] = norms.x;
      red_s[3][w] = norms.y;
      red_s[4][w] = norms.z;
    }
    __syncthreads();
    if (tid == 0) {
      for (int u = 1; u < kWarps; ++u) {
        lo = fminf(lo, red_s[0][u]);
        hi = fmaxf(hi, red_s[1][u]);
        norms.x += red_s[2][u];
        norms.y += red_s[3][u];
        norms.z = fmaxf(norms.z, red_s[4][u]);
      }
      lo_s = lo;
      hi_s = hi;
      delta_s = rows.delta(norms, q, smax ? smax[ql] : 0.f);
    }
    __syncthreads();
    lo = lo_s;
    hi = hi_s;
    delta = delta_s;
  }
  // position i of the slice: its probe, its row
  const bool in_table = tq <= kProbeTable;
  const auto probe_of = [&](int i) {
    int a = 0, b = tq - 1;
    while (a < b) {
      const int mid = (a + b + 1) >> 1;
      if ((in_table ? at_s[mid] : (int)qpos[mid]) <= i) a = mid;
      else b = mid - 1;
    }
    return a;
  };
  const auto row_of = [&](int i, int j) { return in_table ? row_s[j] + i : off[probes[j]] - qpos[j] + i; };
  const auto defined_key = [&](int i) {
    const int j = probe_of(i);
    const int64_t r = row_of(i, j);
    return rank_key(rows.exact(qs, q, r, base ? base[ql * t + j] : 0.f), (uint32_t)ids[r]);
  };
  const auto append = [&](bool in, int* count, int32_t* to, int cap, int32_t v) {
    const unsigned b = __ballot_sync(kFull, in);
    int at = 0;
    if (lane == 0 && b) at = atomicAdd(count, __popc(b));
    at = __shfl_sync(kFull, at, 0) + __popc(b & ((1u << lane) - 1u));
    if (in && at < cap) to[at] = v;
  };

  // kBins linear bins of [lo, hi]; false where the range is not a finite interval
  float scale = 0.f;
  const auto set_bins = [&]() {
    scale = (float)(kBins - 1) / (hi - lo);
    for (int i = tid; i < kBins; i += kThreads) hist[i] = 0;
    __syncthreads();
    return scale > 0.f && scale < INFINITY && delta < INFINITY;
  };
  const auto bin_of = [&](uint32_t key) {
    return (int)fminf(fmaxf((key_float(key) - lo) * scale, 0.f), (float)(kBins - 1));
  };
  // counted rows, and bin_s = the bin that holds the want-th best of them
  const auto find_bin = [&](int want) {
    constexpr int kOwn = kBins / kThreads;
    __syncthreads();
    int mine = 0, all;
#pragma unroll
    for (int u = 0; u < kOwn; ++u) mine += hist[kBins - 1 - (tid * kOwn + u)];
    int c = block_exclusive_scan<int>(mine, warp_s, all);
    if (c < want && c + mine >= want)
      for (int u = 0; u < kOwn; ++u) {
        const int b = kBins - 1 - (tid * kOwn + u);
        c += hist[b];
        if (c >= want) {
          bin_s = b;
          break;
        }
      }
    __syncthreads();
    return all;
  };
  // n_list rows of the list so far, as positions, and m <= kBand rows of the band:
  // the rows as ids, then the band's best in the defined order
  const auto finish_band = [&](int m) {
    int N = 2;
    while (N < m) N <<= 1;
    for (int i = tid; i < N; i += kThreads) band_key[i] = i < m ? defined_key(band[i]) : ~0ull;   // (bins: no longer read)
    __syncthreads();
    block_sort(band_key, N);
    const int have = n_list;
    for (int i = tid; i < have; i += kThreads) list[i] = ids[row_of(list[i], probe_of(list[i]))];
    for (int i = tid; i < R - have; i += kThreads) list[have + i] = (int32_t)(band_key[i] & 0xffffffffu);
    __syncthreads();
    if (tid == 0) n_list = R;
  };
  // The list from `count` rows (key_at, pos_at), all rows of the slice that count
  // or (open) all at or above lo; false where linear bins cannot tell.
  const auto choose = [&](int count, auto key_at, auto pos_at, bool open) {
    if (!set_bins()) return false;
    for (int i = tid; i < count; i += kThreads) {
      const uint32_t key = key_at(i);
      if (key) atomicAdd(&hist[bin_of(key)], 1);
    }
    if (find_bin(R) <= R) return false;
    const float wide = ceilf(2.f * delta * scale) + 1.f;
    const int mb = wide < (float)kBins ? (int)wide : kBins;
    if (open && bin_s < mb) return false;                                // rows below lo might be in the band
    const int b_lo = max(0, bin_s - mb), b_hi = min(kBins - 1, bin_s + mb);
    int in_band = 0, m;
    for (int b = b_lo + tid; b <= b_hi; b += kThreads) in_band += hist[b];
    block_exclusive_scan<int>(in_band, warp_s, m);
    if (m > kBand) return false;
    for (int i0 = 0; i0 < count; i0 += kThreads) {
      const int i = i0 + tid;
      const uint32_t key = i < count ? key_at(i) : 0u;
      const int b = key ? bin_of(key) : -1;
      if (!__any_sync(kFull, b >= b_lo)) continue;
      append(b > b_hi, &n_list, list, R, b > b_hi ? pos_at(i) : 0);
      append(b >= b_lo && b <= b_hi, &n_band, band, kBand, b >= b_lo ? pos_at(i) : 0);
    }
    __syncthreads();
    finish_band(m);
    return true;
  };
  // The need-th largest of the values value(i) > 0, i in [0, n), and (in need) how
  // many of its equals count; at least `need` values are positive.
  const auto nth_largest = [&](int& need, auto value) {
    uint32_t prefix = 0u, mask = 0u;
    for (int shift = 24; shift >= 0; shift -= 8) {
      __syncthreads();
      hist[tid] = 0;
      __syncthreads();
      int last = 0, run = 0;                            // (a thread's keys mostly share their leading bytes)
      for (int i = tid; i < n; i += kThreads) {
        const uint32_t v = value(i);
        if (!v || (v & mask) != prefix) continue;
        const int b = (v >> shift) & 0xffu;
        if (b != last) {
          if (run) atomicAdd(&hist[last], run);
          last = b;
          run = 0;
        }
        ++run;
      }
      if (run) atomicAdd(&hist[last], run);
      __syncthreads();
      int all;
      const int mine = hist[255 - tid], c = block_exclusive_scan<int>(mine, warp_s, all);
      if (c < need && c + mine >= need) {
        bin_s = 255 - tid;
        above_s = c;
      }
      __syncthreads();
      need -= above_s;
      prefix |= (uint32_t)bin_s << shift;
      mask |= 0xffu << shift;
    }
    return prefix;
  };

  uint32_t floor_key = 1u;                              // every row that counts
  const bool finite = !short_slice && (n <= cap || set_bins());
  if (n > cap && finite) {
#pragma unroll
    for (int u = 0; u < kSample; ++u)
      if (sample[u]) atomicAdd(&hist[bin_of(sample[u])], 1);
    const float expect = (float)R * (kSample * kThreads) / (float)n;
    const int want = (int)(1.25f * expect + 4.f * sqrtf(expect) + 8.f);
    if (find_bin(want) > want) floor_key = max(1u, float_key(lo + (float)(bin_s - 1) / scale));
  }
  // one pass: four keys a load (slices start on 16 bytes), two loads in flight, one counter step a warp and load
  if (finite) {
    constexpr int kPass = 2;
    const int n4 = n / 4;
    for (int i0 = 32 * w; i0 <= n4; i0 += kPass * kThreads) {
      uint4 v[kPass];
#pragma unroll
      for (int u = 0; u < kPass; ++u) {
        const int i = i0 + u * kThreads + lane;
        v[u] = make_uint4(0u, 0u, 0u, 0u);
        if (i < n4) {
          v[u] = reinterpret_cast<const uint4*>(K)[i];
        } else if (i == n4) {                           // the last one to three keys
          if (n % 4 > 0) v[u].x = K[4 * i];
          if (n % 4 > 1) v[u].y = K[4 * i + 1];
          if (n % 4 > 2) v[u].z = K[4 * i + 2];
        }
      }
#pragma unroll
      for (int u = 0; u < kPass; ++u) {
        const uint32_t key[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
        int mine = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) mine += key[e] >= floor_key ? 1 : 0;
        if (!__any_sync(kFull, mine)) continue;
        int incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(kFull, incl, o);
          if (lane >= o) incl += y;
        }
        int at = 0;
        if (lane == 31) at = atomicAdd(&n_kept, incl);
        at = __shfl_sync(kFull, at, 31) + incl - mine;
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (key[e] >= floor_key) {
            if (at < cap) {
              kept[at] = key[e];
              kept_at[at] = 4 * (i0 + u * kThreads + lane) + e;
            }
            ++at;
          }
      }
    }
  }
  __syncthreads();
  const int m_kept = n_kept;
  bool done = false, few = short_slice;                 // few: at most R rows count
  if (finite && m_kept <= cap) {
    if (floor_key == 1u && m_kept <= R) {
      few = true;
    } else if (m_kept > R) {
      if (floor_key > 1u) lo = key_float(floor_key);
      done = choose(m_kept, [&](int i) { return kept[i]; }, [&](int i) { return kept_at[i]; }, floor_key > 1u);
    }
  }
  if (!done && !few) {                                  // (a long slice has more rows above the floor than are kept)
    lo = lo_s;
    done = choose(n, [&](int i) { return K[i]; }, [&](int i) { return i; }, false);
  }
  __syncthreads();
  if (!done) {
    if (tid == 0) n_list = n_band = 0;
    int cnt = 0, total;
    for (int i = tid; i < n; i += kThreads) cnt += K[i] != 0u;
    block_exclusive_scan<int>(cnt, warp_s, total);
    if (few || total <= R) {
      for (int i0 = 0; i0 < n; i0 += kThreads) {
        const int i = i0 + tid;
        const bool in = i < n && K[i] != 0u;
        append(in, &n_list, list, R, in ? ids[row_of(i, probe_of(i))] : -1);
      }
    } else {
      // the band around the R-th largest key itself; all rows where that or delta is not finite
      int need = R;
      const float f = key_float(nth_largest(need, [&](int i) { return K[i]; }));
      uint32_t lo_key = 1u, hi_key = ~0u;
      if (fabsf(f) < INFINITY && delta < INFINITY) {
        lo_key = max(1u, float_key(__fsub_rd(f, 2.f * delta)));
        hi_key = float_key(__fadd_ru(f, 2.f * delta));
      }
      int in_band = 0, m;
      for (int i = tid; i < n; i += kThreads) in_band += K[i] >= lo_key && K[i] <= hi_key ? 1 : 0;
      block_exclusive_scan<int>(in_band, warp_s, m);
      const bool fits = m <= kBand;
      float* table = reinterpret_cast<float*>(kept);      // (the kept rows: no longer read)
      const bool tabulated = !fits && rows.tabulate(qs, table, 2 * cap);
      __syncthreads();
      const auto defined = [&](int i) {
        const int j = probe_of(i);
        const int64_t r = row_of(i, j);
        const float b = base ? base[ql * t + j] : 0.f;
        return max(1u, float_key(tabulated ? rows.exact_tabulated(table, r, b) : rows.exact(qs, q, r, b)));
      };
      // a band too large for shared memory: its keys become those of the defined
      // scores, in place, and the other rows' zero
      for (int i0 = 0; i0 < n; i0 += kThreads) {
        const int i = i0 + tid;
        const uint32_t key = i < n ? K[i] : 0u;
        const bool in = key >= lo_key && key <= hi_key;
        append(key > hi_key, &n_list, list, R, i);
        if (fits) append(in, &n_band, band, kBand, i);
        else if (i < n) K[i] = in ? defined(i) : 0u;
      }
      __syncthreads();
      if (fits) {
        finish_band(m);
      } else {
        need = R - n_list;
        const uint32_t least = nth_largest(need, [&](int i) { return K[i]; });
        // of the rows that score as the last one does, those of the lowest ids
        const auto tie = [&](int i) { return K[i] == least ? ~(uint32_t)ids[row_of(i, probe_of(i))] : 0u; };
        const uint32_t last = nth_largest(need, tie);
        for (int i0 = 0; i0 < n; i0 += kThreads) {
          const int i = i0 + tid;
          append(i < n && (K[i] > least || tie(i) >= last), &n_list, list, R, i);
        }
        __syncthreads();
        for (int i = tid; i < R; i += kThreads) list[i] = ids[row_of(list[i], probe_of(list[i]))];
      }
    }
    __syncthreads();
  }
  // ---- exact scores of the listed rows, the best k
  const int have = min(n_list, R);
  if (k <= 32) {
    uint64_t best = ~0ull, thr = ~0ull;         // lane j < k: the warp's j-th best key
    const auto insert = [&](uint64_t key) {
      unsigned bal = __ballot_sync(kFull, key < thr);
      while (bal) {
        const int src = __ffs(bal) - 1;
        bal &= bal - 1;
        const uint64_t kk = __shfl_sync(kFull, key, src);
        if (kk >= thr) continue;
        const int at = __popc(__ballot_sync(kFull, lane < k && best < kk));
        const uint64_t up = __shfl_up_sync(kFull, best, 1);
        if (lane > at && lane < k) best = up;
        if (lane == at) best = kk;
        thr = __shfl_sync(kFull, best, k - 1);
      }
    };
    for (int i0 = 32 * w; i0 < have; i0 += kThreads) {
      const int i = i0 + lane;
      const int32_t id = i < have ? list[i] : -1;
      const float s = warp_rows_dot(qrow, orig, ostride, id, stage, lane);
      insert(id >= 0 && s == s ? rank_key(s, (uint32_t)id) : ~0ull);
    }
    __syncthreads();                              // (the staged rows lie over ex)
    ex[32 * w + lane] = lane < k ? best : ~0ull;
    __syncthreads();
    if (w == 0) {
      for (int u = 1; u < kWarps; ++u) insert(ex[32 * u + lane]);
      if (lane < k) {
        ids_out[q * k + lane] = best != ~0ull ? (int64_t)(uint32_t)(best & 0xffffffffu) : -1;
        scores_out[q * k + lane] = best != ~0ull ? key_float(~(uint32_t)(best >> 32)) : -INFINITY;
      }
    }
  } else {
    int N = 2;
    while (N < max(have, k)) N <<= 1;           // (k <= R: within ex)
    for (int i0 = 32 * w; i0 < N; i0 += kThreads) {
      const int i = i0 + lane;
      const int32_t id = i < have ? list[i] : -1;
      const float s = warp_rows_dot(qrow, orig, ostride, id, stage, lane);
      if (i < N) ex[i] = id >= 0 && s == s ? rank_key(s, (uint32_t)id) : ~0ull;
    }
    __syncthreads();
    block_sort(ex, N);
    for (int i = tid; i < k; i += kThreads) {
      const uint64_t key = ex[i];
      ids_out[q * k + i] = key != ~0ull ? (int64_t)(uint32_t)(key & 0xffffffffu) : -1;
      scores_out[q * k + i] = key != ~0ull ? key_float(~(uint32_t)(key >> 32)) : -INFINITY;
    }
  }
}

// Keys a query may need, a multiple of four (slices are read 16 bytes at a time).
int64_t slice_rows(const IndexData& ix, int t) {
  return (std::max<int64_t>(1, std::min<int64_t>((int64_t)t * ix.max_partition, ix.rows)) + 3) / 4 * 4;
}
// The key buffer holds 2 GB at most (or eight slices).  A slice of the longest
// possible length is mostly a third full, so a batch whose slices do not fit
// that way has them packed, and only what does not fit then takes another pass
// over the partitions: passes cover windows of the packed keys, as many as the
// longest slices could fill; the ones that stay empty end at once.  Chunks of a
// batch are small enough that there are few of those.  (10 000 queries over 10^7
// x 96 FP8, at most 2.4 GB of keys and 0.6 in fact: 2 768 us in two passes of
// 8 945 and 1 055 queries, 2 458 packed, 2 391 in a 4 GB buffer.)
constexpr int64_t kKeysMost = (int64_t)1 << 29;
struct KeyPlan {
  int64_t slice, room, queries, window;     // keys: a slice at most, the buffer; queries a chunk; keys a pass (0: one pass)
};
KeyPlan key_plan(const IndexData& ix, int64_t nq, int t) {
  KeyPlan p;
  p.slice = slice_rows(ix, t);
  p.room = std::max(kKeysMost, 8 * p.slice);
  // (the buffers of a chunk's pairs: 2^24 pairs at most)
  p.queries = std::min({nq, std::max<int64_t>(8, ((int64_t)1 << 24) / t), std::max<int64_t>(8, 4 * p.room / p.slice)});
  p.window = p.queries * p.slice > p.room ? (p.room - p.slice) / 4 * 4 : 0;
  if (!p.window) p.room = p.queries * p.slice;
  return p;
}

template <typename Rows>
void run(const IndexData& ix, Rows rws, float* base, const float* Qf, int qstride, const void* Q,
         soar_dtype dt, const int32_t* top, const int32_t* tpq, int64_t nq, int t, int R, int k, int64_t* ids_out,
         float* scores_out, cudaStream_t s, Scratch& scr) {
  rws.tiles = Rows::kTiles;
  while (rws.tiles > 1 && rws.item_smem() > 180 * 1024) --rws.tiles;     // wide rows: fewer queries an item
  const int QB = 8 * rws.tiles;
  const KeyPlan plan = key_plan(ix, nq, t);
  const int64_t cq = plan.queries;
  uint32_t* keys = scr.get<uint32_t>((size_t)plan.room);
  int64_t* counts = scr.get<int64_t>(cq);
  int64_t* start = plan.window ? scr.get<int64_t>((size_t)cq + 1) : nullptr;
  int32_t* taken = plan.window ? scr.get<int32_t>(cq) : nullptr;
  int* smax = Rows::kScaled ? scr.get<int>(cq) : nullptr;
  int64_t* pos = scr.get<int64_t>((size_t)cq * t);
  int32_t* inv = scr.get<int32_t>((size_t)cq * t);
  const int a = 1 + ix.spills;
  const int ostride = ix.dtype == SOAR_F32 ? (ix.d + 3) / 4 * 4 : (ix.d + 7) / 8 * 8;
  int sorted = kThreads;                                  // exact keys: the warps' lists, or R of them to sort
  if (k > 32)
    while (sorted < R) sorted <<= 1;
  const auto up = [](size_t b) { return (b + 15) / 16 * 16; };
  const size_t kept_at = up(sizeof(float) * ((size_t)(ostride + 3) / 4 * 4 + (rws.query_floats() + 3) / 4 * 4) +
                            sizeof(int) * (size_t)(kBins + kBand) + sizeof(int32_t) * (size_t)((R + 1) / 2 * 2));
  const size_t stage_at = kept_at + (k > 32 ? up(sizeof(uint64_t) * (size_t)sorted) : 0);
  const size_t fin_smem = std::max(kept_at + sizeof(uint64_t) * (size_t)std::max(kept_rows(R), sorted),
                                   stage_at + sizeof(uint4) * 32 * kRowChunks * kWarps);
  const size_t item_smem = rws.item_smem();
  allow_smem(score_items<Rows>, item_smem);
  const auto finish = [&](auto elem, const Slices& sl, int64_t q0, int64_t m) {
    using OT = decltype(elem);
    auto kern = finish_slices<Rows, OT>;
    allow_smem(kern, fin_smem);
    kern<<<(unsigned)m, kThreads, fin_smem, s>>>(rws, sl, counts, pos, top, tpq, q0, t, ix.offsets, ix.ids, base,
                                                 reinterpret_cast<const float*>(smax), Q, (int)dt, ix.d,
                                                 static_cast<const OT*>(ix.originals), ostride, R, k, (int)stage_at,
                                                 ids_out, scores_out);
    SOAR_LAUNCHED();
  };
  for (int64_t q0 = 0; q0 < nq; q0 += cq) {
    const int64_t m = std::min(cq, nq - q0);
    Scratch cs(s);
    stage_mark(s, "scan", true);
    pair_offsets<<<ceil_div(m * 32, 256), 256, 0, s>>>(ix.offsets, top, tpq, q0, m, t, pos, counts, start, smax);
    SOAR_LAUNCHED();
    if (start) exclusive_scan_i64(start, start, m + 1, s, cs);
    if (base) {
      pair_bases<<<ceil_div(m * t * 32, 256), 256, 0, s>>>(Qf, qstride, ix.centroids, ix.d, top, tpq, q0, m, t, base);
      SOAR_LAUNCHED();
    }
    stage_mark(s, "scan", false);
    const int64_t passes = start ? (m * plan.slice + plan.window - 1) / plan.window : 1;
    for (int64_t pass = 0; pass < passes; ++pass) {
      Scratch ps(s);
      const Slices sl{keys, start, plan.slice, pass * plan.window, (pass + 1) * plan.window};
      const int32_t* tp = tpq ? tpq + q0 : nullptr;
      if (start) {
        pass_counts<<<ceil_div(m, 256), 256, 0, s>>>(sl, tpq, q0, m, t, taken);
        SOAR_LAUNCHED();
        tp = taken;
      }
      const Grouped g = group_pairs(ix, m, t, tp, QB, top + q0 * t, inv, s, ps, false, false);
      stage_mark(s, "scan", true);
      // a batch of few pairs splits each partition's rows over several blocks
      const int64_t items = std::min<int64_t>(m * t, g.max_items);
      const unsigned split = (unsigned)std::max<int64_t>(1, std::min<int64_t>(16, 8 * num_sms() / std::max<int64_t>(1, items)));
      const IvfWork work{ix.offsets, g.pair_off, g.vals, g.order, g.item_base, ix.c, t, QB};
      score_items<Rows><<<dim3((unsigned)items, split), kThreads, item_smem, s>>>(rws, work, ix.ids, ix.assign, a, top,
                                                                                 q0, sl, pos, smax);
      SOAR_LAUNCHED();
      stage_mark(s, "scan", false);
      stage_mark(s, "rescore", true);
      if (ix.dtype == SOAR_F32) finish(float{}, sl, q0, m);
      else finish(__nv_bfloat16{}, sl, q0, m);
      stage_mark(s, "rescore", false);
    }
  }
}

}  // namespace

void fp8_search(const IndexData& ix, const float* Qf, const float* qscale, const void* Q, soar_dtype dt,
                const int32_t* top, const int32_t* tpq, int64_t nq, int t, int R, int k, int64_t* ids_out,
                float* scores_out, cudaStream_t s, Scratch& scr) {
  const Fp8Rows rws{static_cast<const uint8_t*>(ix.vectors), ix.code_stride, ix.row_scales, Qf, qscale,
                    (ix.code_stride + 63) / 64, 0};
  run(ix, rws, nullptr, Qf, ix.code_stride, Q, dt, top, tpq, nq, t, R, k, ids_out, scores_out, s, scr);
}

void pq_search(const IndexData& ix, const float* Qf, int qstride, const void* Q, soar_dtype dt, const int32_t* top,
               const int32_t* tpq, int64_t nq, int t, int R, int k, int64_t* ids_out, float* scores_out,
               cudaStream_t s, Scratch& scr) {
  float* base = scr.get<float>((size_t)key_plan(ix, nq, t).queries * t);
  const Pq4Rows rws{static_cast<const uint8_t*>(ix.vectors), ix.code_stride, ix.pq_m, ix.d, ix.pq_cb, Qf, qstride,
                    base, (ix.pq_m + 7) / 8, 0};
  run(ix, rws, base, Qf, qstride, Q, dt, top, tpq, nq, t, R, k, ids_out, scores_out, s, scr);
}

}  // namespace soar
