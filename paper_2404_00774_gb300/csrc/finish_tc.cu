// Exact finishing of the tensor-core partition scan (scan_tc.cu): the
// screened candidate lists of every (query, partition) pair are rescored
// exactly in fp32 (fp32 rows, or bf16 rows widened exactly) from the
// row-major copy of the index, the partitions
// whose lists overflowed are rescanned exactly, spilled copies of a point
// are dropped (Section 3.5: a spilled point's copies carry bit-identical
// exact scores) and each query keeps its top k (Section 2.2).
//   finish_queries  a warp per query (k <= 32, batches that fill the chip)
//   finish_block    a block per query (k <= 128)
#include "scan_common.cuh"

namespace soar {

namespace {

// Largest batch finished by a block per query when k <= 32.  Finishing, us, a warp /
// a block per query (Glove-shaped, t = 14): k = 10 2 048 queries 33 / 34, 3 000 36 /
// 36, 4 096 44 / 49, 6 000 56 / 63, 10 000 70 / 102; k = 32, where lists overflow and
// partitions are rescanned, 1 216 1 721 / 1 115, 2 048 1 856 / 1 618, 4 096 2 707 /
// 2 849, 10 000 4 986 / 6 314; in tight clusters (bf16) k = 10 2 048 28 / 27, 4 096 35
// / 39, 10 000 67 / 79, k = 32 2 048 3 166 / 1 752, 4 096 4 019 / 3 081, 10 000 7 458 /
// 6 751.  The line gives up 5 us without overflow below it for what it saves with.
constexpr int64_t kBlockFinishMax = 4096;
// Queries per SM up to which their blocks are of 512 threads, above that of 128
// (finishing, us, 128 against 512 threads; 152 SMs: k = 100 of about 270 lists,
// 70 queries 64 / 32, 300 queries 67 / 42, 600 queries 94 / 69, 1 024 queries
// 103 / 103; k = 10 of 14 lists, 300 queries 20 / 19, 608 21 / 32, 1 216 22 / 57;
// k = 32 with overflows, 300 761 / 325, 608 821 / 470, 1 216 1 115 / 810).
constexpr int64_t kWideBlockMax = 4;

// Exact fp32 <q, x> of row-major row `pos` (row stride rs; k ascending, the
// same order for every copy of a point).  fp32 rows: rs a multiple of 4.
__device__ __forceinline__ float exact_dot_rm(const float* __restrict__ q, const float* __restrict__ vec, int rs,
                                              int64_t pos) {
  const float* x = vec + pos * (int64_t)rs;
  float acc = 0.f;
#pragma unroll 8
  for (int k4 = 0; k4 < rs / 4; ++k4) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(q + 4 * k4));
    const float4 v = __ldg(reinterpret_cast<const float4*>(x + 4 * k4));
    acc = fmaf(a.x, v.x, acc);
    acc = fmaf(a.y, v.y, acc);
    acc = fmaf(a.z, v.z, acc);
    acc = fmaf(a.w, v.w, acc);
  }
  return acc;
}

// bf16 rows (rs a multiple of 8): each element widened to fp32 exactly.
__device__ __forceinline__ float exact_dot_rm(const float* __restrict__ q, const __nv_bfloat16* __restrict__ vec,
                                              int rs, int64_t pos) {
  const __nv_bfloat16* x = vec + pos * (int64_t)rs;
  float acc = 0.f;
#pragma unroll 4
  for (int k8 = 0; k8 < rs / 8; ++k8) {
    const uint4 w = __ldg(reinterpret_cast<const uint4*>(x + 8 * k8));
    const float4 a0 = __ldg(reinterpret_cast<const float4*>(q + 8 * k8));
    const float4 a1 = __ldg(reinterpret_cast<const float4*>(q + 8 * k8 + 4));
    acc = fmaf(a0.x, __uint_as_float(w.x << 16), acc);
    acc = fmaf(a0.y, __uint_as_float(w.x & 0xffff0000u), acc);
    acc = fmaf(a0.z, __uint_as_float(w.y << 16), acc);
    acc = fmaf(a0.w, __uint_as_float(w.y & 0xffff0000u), acc);
    acc = fmaf(a1.x, __uint_as_float(w.z << 16), acc);
    acc = fmaf(a1.y, __uint_as_float(w.z & 0xffff0000u), acc);
    acc = fmaf(a1.z, __uint_as_float(w.w << 16), acc);
    acc = fmaf(a1.w, __uint_as_float(w.w & 0xffff0000u), acc);
  }
  return acc;
}


// Finishing pass of a block per query (k <= 128).  The query's bound L* (the
// largest L_k its finished partitions published) bounds its final k-th best
// exact score from below; the candidates of all its lists whose upper bound
// reaches L* are gathered in shared memory, rescored exactly a thread each,
// sorted with the best k so far, and equal neighbours (a spilled point's
// copies have bit-identical keys) dropped.  A partition whose list overflowed
// is rescanned exactly by the whole block.
// Bound: latency (a few hundred scattered 16-byte loads a query).  It replaces
// a warp per (query, partition) list plus a k-way merge of t sorted lists by
// a warp (k = 100, 1 024 queries of 272 lists: 870 us with its helper kernels,
// 99 now), and takes k <= 32 too for batches that do not fill the chip
// with a warp per query, where one warp rescanning overflowed partitions set
// the time of a small batch (100 queries: 147 us before, 18 now; most of that
// since small batches get lists long enough not to overflow).
constexpr int fb_keys(int threads) { return threads == 128 ? 1024 : 2048; }   // the best k so far and the pending
constexpr int fb_pend(int threads) { return fb_keys(threads) - kTcWideK; }
constexpr int fb_unroll(int threads) { return threads == 128 ? 4 : 2; }       // list entries a thread loads per round

template <typename RowT, int T>
__global__ void __launch_bounds__(T) finish_block(
    const Cand* __restrict__ cand, const int2* __restrict__ hdr, const unsigned* __restrict__ gbound,
    const int32_t* __restrict__ inv, int t, const int32_t* __restrict__ tpq, const float* __restrict__ Qf, int kp,
    const RowT* __restrict__ rows, int rs, const int32_t* __restrict__ ids, const int32_t* __restrict__ top,
    const int64_t* __restrict__ part_off, int k, int kc, int64_t* __restrict__ ids_out,
    float* __restrict__ scores_out) {
  constexpr unsigned kFull = 0xffffffffu;
  constexpr int kPend = fb_pend(T), kUnroll = fb_unroll(T);
  static_assert(T * kUnroll <= kPend, "a round's entries fit behind an empty list");
  __shared__ uint64_t buf[fb_keys(T)];         // [0, best) ascending distinct keys
  __shared__ int32_t pend[kPend];              // row positions
  __shared__ int32_t pre_s[T], e_s[T], warp_s[32];
  __shared__ unsigned ovf_s[T / 32];
  __shared__ int fill_s;
  const int64_t q = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int tq = tpq ? min(max(tpq[q], 0), t) : t;
  const float lstar = key_float(gbound[q]);
  const float* qv = Qf + q * (int64_t)kp;
  int best = 0;                                // uniform
  if (tid == 0) fill_s = 0;
  __syncthreads();
  // the pending rows rescored and merged into the best k (all threads; fill_s visible)
  const auto flush = [&]() {
    const int n = fill_s;
    if (n == 0) return;
    for (int i = tid; i < n; i += T) {
      const int32_t pos = pend[i];
      buf[best + i] = rank_key_of_number(exact_dot_rm(qv, rows, rs, pos), (uint32_t)ids[pos]);
    }
    int N = 2;
    while (N < best + n) N <<= 1;
    for (int i = best + n + tid; i < N; i += T) buf[i] = ~0ull;
    __syncthreads();
    if (tid == 0) fill_s = 0;
    for (int size = 2; size <= N; size <<= 1)
      for (int stride = size >> 1; stride > 0; stride >>= 1) {
        for (int i = tid; i < N / 2; i += T) {
          const int a = 2 * i - (i & (stride - 1)), b = a + stride;
          const uint64_t x = buf[a], y = buf[b];
          if ((x > y) == ((a & size) == 0)) {
            buf[a] = y;
            buf[b] = x;
          }
        }
        __syncthreads();
      }
    // distinct keys move down, chunk by chunk (a key never moves up, and the
    // entry before a chunk is read before anything is written there)
    int m = 0;
    for (int base = 0; base < N && m < k; base += T) {
      const int i = base + tid;
      const uint64_t x = i < N ? buf[i] : ~0ull, y = (i > 0 && i < N) ? buf[i - 1] : ~0ull;
      const int take = (x != ~0ull && (i == 0 || x != y)) ? 1 : 0;
      int total;
      const int r = m + block_exclusive_scan<int>(take, warp_s, total);   // (synchronises: every read is done)
      if (take && r < k) buf[r] = x;
      m += total;
      __syncthreads();
    }
    best = min(m, k);
  };
  for (int j0 = 0; j0 < tq; j0 += T) {
    const int j = j0 + tid;
    int e_l = 0, cnt_l = 0;
    bool ovf_l = false;
    if (j < tq) {
      e_l = inv[q * t + j];
      const int hy = hdr[e_l].y;
      ovf_l = hy < 0;
      cnt_l = ovf_l ? 0 : min(hy & 0x7fffffff, kc);
    }
    int total;
    const int ex = block_exclusive_scan<int>(cnt_l, warp_s, total);
    pre_s[tid] = ex;
    e_s[tid] = e_l;
    const unsigned ob = __ballot_sync(kFull, ovf_l);
    if (lane == 0) ovf_s[w] = ob;
    __syncthreads();
    for (int base = 0; base < total; base += T * kUnroll) {
      if (fill_s + T * kUnroll > kPend) flush();     // (fill_s last written before a barrier: uniform)
      bool keep[kUnroll];
      int32_t pos[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const int f = base + u * T + tid;
        keep[u] = false;
        pos[u] = 0;
        if (f < total) {
          int lo = 0;                           // the last list that starts at or before f: the one holding entry f
#pragma unroll
          for (int step = T / 2; step > 0; step >>= 1)
            if (pre_s[lo + step] <= f) lo += step;
          const Cand c = cand[(int64_t)e_s[lo] * kc + (f - pre_s[lo])];
          keep[u] = c.s >= lstar;
          pos[u] = c.id;
        }
      }
      __syncthreads();                          // every thread has read fill_s
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const unsigned kb = __ballot_sync(kFull, keep[u]);
        int at = 0;
        if (lane == 0 && kb) at = atomicAdd(&fill_s, __popc(kb));
        at = __shfl_sync(kFull, at, 0);
        if (keep[u]) pend[at + __popc(kb & ((1u << lane) - 1u))] = pos[u];
      }
      __syncthreads();
    }
    // partitions whose lists overflowed: rescanned exactly
    for (int word = 0; word < T / 32; ++word)
      for (unsigned bits = ovf_s[word]; bits; bits &= bits - 1) {
        const int p = top[q * t + j0 + 32 * word + __ffs(bits) - 1];
        const int64_t r1 = part_off[p + 1];
        for (int64_t r0 = part_off[p]; r0 < r1; r0 += T) {
          if (best < k || fill_s + T > kPend) flush();   // early rows fill the best k, then only better ones wait
          const uint64_t thr = best == k ? buf[k - 1] : ~0ull;
          __syncthreads();
          const int64_t r = r0 + tid;
          const bool in = r < r1 && rank_key_of_number(exact_dot_rm(qv, rows, rs, r), (uint32_t)ids[r]) < thr;
          const unsigned kb = __ballot_sync(kFull, in);
          int at = 0;
          if (lane == 0 && kb) at = atomicAdd(&fill_s, __popc(kb));
          at = __shfl_sync(kFull, at, 0);
          if (in) pend[at + __popc(kb & ((1u << lane) - 1u))] = (int32_t)r;
          __syncthreads();
        }
      }
    __syncthreads();                            // pre_s, e_s and ovf_s are rewritten next
  }
  flush();
  for (int i = tid; i < k; i += T) {
    const bool have = i < best;
    ids_out[q * k + i] = have ? (int64_t)(uint32_t)(buf[i] & 0xffffffffu) : -1;
    scores_out[q * k + i] = have ? key_float(~(uint32_t)(buf[i] >> 32)) : -INFINITY;
  }
}

// Finishing pass for k <= 32, a warp per query: the query's bound L* (the
// largest L_k its finished partitions published) bounds its final k-th best exact score from
// below; every candidate whose upper bound reaches L* (and beats the current
// k-th best) is rescored exactly, and every partition whose list overflowed
// is rescanned exactly.  The exact results go into a lane-distributed sorted
// top-k (lane j: j-th best rank key), dropping the second copy of a spilled
// point (its exact score is bit-identical, so its key is too).  Writes the
// query's ids / scores, padded with -1 / -inf.
template <typename RowT>
__global__ void __launch_bounds__(256) finish_queries(
    const Cand* __restrict__ cand, const int2* __restrict__ hdr, const unsigned* __restrict__ gbound,
    const int32_t* __restrict__ inv, int64_t nq, int t, const int32_t* __restrict__ tpq, const float* __restrict__ Qf,
    int kp, const RowT* __restrict__ rows, int rs, const int32_t* __restrict__ ids, const int32_t* __restrict__ top,
    const int64_t* __restrict__ part_off, int k, int kc, int64_t* __restrict__ ids_out,
    float* __restrict__ scores_out) {
  constexpr unsigned kFull = 0xffffffffu;
  constexpr int kPend = 256;                    // pending candidates per warp
  __shared__ int32_t pend_s[8][kPend];
  const int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (q >= nq) return;
  const int tq = tpq ? min(max(tpq[q], 0), t) : t;
  const float lstar = key_float(gbound[q]);
  const float* qv = Qf + q * (int64_t)kp;
  uint64_t mine = ~0ull;          // lane j < k: the j-th best key so far (empty: after every real key)
  uint64_t thr = ~0ull;           // the k-th best key
  // inserts the keys of this round (one per lane, ~0 for none)
  auto insert_round = [&](uint64_t key) {
    unsigned bal = __ballot_sync(kFull, key < thr);
    while (bal) {
      const int src = __ffs(bal) - 1;
      bal &= bal - 1;
      const uint64_t kk = __shfl_sync(kFull, key, src);
      if (kk >= thr) continue;                                   // the same in every lane
      if (__ballot_sync(kFull, lane < k && mine == kk)) continue;  // spilled copy already in
      const int pos = __popc(__ballot_sync(kFull, lane < k && mine < kk));
      const uint64_t up = __shfl_up_sync(kFull, mine, 1);
      if (lane > pos && lane < k) mine = up;
      if (lane == pos) mine = kk;
      thr = __shfl_sync(kFull, mine, k - 1);
    }
  };
  // candidates whose upper bound reaches L*, gathered over all of the
  // query's partitions (padded row positions), then rescored 32 at a time so
  // that the exact dot products of a round overlap
  int32_t* pend = pend_s[threadIdx.x >> 5];
  int npend = 0;
  auto flush = [&]() {
    for (int b = 0; b < npend; b += 32) {
      const float kth = thr == ~0ull ? -INFINITY : key_float(~(uint32_t)(thr >> 32));
      uint64_t key = ~0ull;
      if (b + lane < npend) {
        const int32_t pos = pend[b + lane];
        const float v = exact_dot_rm(qv, rows, rs, pos);
        if (v >= kth) key = rank_key(v, (uint32_t)ids[pos]);
      }
      insert_round(key);
    }
    npend = 0;
    __syncwarp();
  };
  // the query's probes 32 at a time: lane l holds probe j0 + l's slot and
  // list length; a warp prefix sum over the lengths lets every lane load one
  // candidate of any of the 32 lists in the same round
  for (int j0 = 0; j0 < tq; j0 += 32) {
    const int j = j0 + lane;
    int64_t e_l = 0;
    int cnt_l = 0;
    bool ovf_l = false;
    if (j < tq) {
      e_l = inv[q * t + j];
      const int hy = hdr[e_l].y;
      ovf_l = hy < 0;
      cnt_l = ovf_l ? 0 : min(hy & 0x7fffffff, kc);
    }
    int incl = cnt_l;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += v;
    }
    const int total = __shfl_sync(kFull, incl, 31);
    for (int base = 0; base < total; base += 32) {
      const int f = base + lane;
      // the list holding entry f: the first lane whose inclusive sum exceeds f
      int lo = 0;
#pragma unroll
      for (int step = 16; step > 0; step >>= 1) {
        const int probe = __shfl_sync(kFull, incl, lo + step - 1);
        if (probe <= f) lo += step;
      }
      const int64_t e = __shfl_sync(kFull, e_l, lo);
      const int first = __shfl_sync(kFull, incl, lo) - __shfl_sync(kFull, cnt_l, lo);
      bool keep = false;
      int32_t pos = 0;
      if (f < total) {
        const Cand c = cand[e * kc + (f - first)];
        keep = c.s >= lstar;
        pos = c.id;
      }
      const unsigned kb = __ballot_sync(kFull, keep);
      if (npend + __popc(kb) > kPend) flush();
      if (keep) pend[npend + __popc(kb & ((1u << lane) - 1u))] = pos;
      npend += __popc(kb);
      __syncwarp();
    }
    // lists that overflowed: rescan their partitions exactly
    for (unsigned ob = __ballot_sync(kFull, ovf_l); ob; ob &= ob - 1) {
      const int l = __ffs(ob) - 1;
      flush();
      const int p = top[q * t + j0 + l];
      const int64_t r0 = part_off[p];
      const int64_t nrows = part_off[p + 1] - part_off[p];
      for (int64_t rb = 0; rb < nrows; rb += 32) {
        const int64_t r = rb + lane;
        const uint64_t key =
            r < nrows ? rank_key_of_number(exact_dot_rm(qv, rows, rs, r0 + r), (uint32_t)ids[r0 + r]) : ~0ull;
        insert_round(key);
      }
    }
  }
  flush();
  if (lane < k) {
    const bool have = mine != ~0ull;
    ids_out[q * k + lane] = have ? (int64_t)(uint32_t)(mine & 0xffffffffu) : -1;
    scores_out[q * k + lane] = have ? key_float(~(uint32_t)(mine >> 32)) : -INFINITY;
  }
}

}  // namespace

void finish_tc_queries(const IndexData& ix, const Cand* lists, const int2* hdr, const unsigned* gbound,
                       const int32_t* inv, int64_t nq, int t, const int32_t* tpq, const float* Qf,
                       const int32_t* top, int k, int kc, int64_t* ids_out, float* scores_out, cudaStream_t s) {
  const auto launch = [&](auto row) {
    using RowT = decltype(row);
    const RowT* rows = static_cast<const RowT*>(ix.vectors);
    // a warp per query once that fills the chip; a block per query below that and for k > 32
    if (k <= 32 && nq > kBlockFinishMax)
      finish_queries<RowT><<<ceil_div(nq * 32, 256), 256, 0, s>>>(lists, hdr, gbound, inv, nq, t, tpq, Qf, ix.tc_kp,
                                                                  rows, ix.row_stride, ix.ids, top, ix.offsets, k, kc,
                                                                  ids_out, scores_out);
    else if (nq > kWideBlockMax * num_sms())
      finish_block<RowT, 128><<<(unsigned)nq, 128, 0, s>>>(lists, hdr, gbound, inv, t, tpq, Qf, ix.tc_kp, rows,
                                                           ix.row_stride, ix.ids, top, ix.offsets, k, kc, ids_out,
                                                           scores_out);
    else
      finish_block<RowT, 512><<<(unsigned)nq, 512, 0, s>>>(lists, hdr, gbound, inv, t, tpq, Qf, ix.tc_kp, rows,
                                                           ix.row_stride, ix.ids, top, ix.offsets, k, kc, ids_out,
                                                           scores_out);
  };
  if (ix.dtype == SOAR_F32) launch(float{});
  else launch(__nv_bfloat16{});
  SOAR_LAUNCHED();
}

}  // namespace soar
