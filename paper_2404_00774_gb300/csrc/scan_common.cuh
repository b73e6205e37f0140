// Types shared by the partition-scan kernels (SIMT and tensor-core).
#pragma once

#include "internal.cuh"

namespace soar {

// One candidate of a per-query top-k list.
struct Cand {
  float s;
  int32_t id;
};

// Order of the top-k lists: higher score first, lower id first on ties
// (id -1, the empty slot, loses every tie).
__device__ __forceinline__ bool better(float a, int ia, float b, int ib) {
  return a > b || (a == b && (unsigned)ia < (unsigned)ib);
}

// Work items of the batched IVF scan: (partition, chunk of <= qb of the
// (query, probe) pairs that probe it), partitions visited in `order`
// (largest first).  Pairs are sorted by partition; pair e belongs to query
// pair_vals[e] / tmax and writes its list to slot e.
struct IvfWork {
  const int64_t* part_off;
  const int64_t* pair_off;
  const int32_t* pair_vals;
  const int32_t* order;
  const int32_t* item_base;   // [c + 1], item_base[c] = total
  int c, tmax, qb;
  __device__ int count() const { return item_base[c]; }
  __device__ int partition_of(int item) const {
    int lo = 0, hi = c - 1;
    while (lo < hi) {
      int mid = (lo + hi + 1) >> 1;
      if (item_base[mid] <= item) lo = mid; else hi = mid - 1;
    }
    return lo;   // index into `order`
  }
  __device__ void describe(int item, int64_t& r0, int64_t& r1, int64_t& e0, int& nqi) const {
    const int lo = partition_of(item);
    const int p = order[lo];
    e0 = pair_off[p] + (int64_t)(item - item_base[lo]) * qb;
    nqi = (int)min((int64_t)qb, pair_off[p + 1] - e0);
    r0 = part_off[p];
    r1 = part_off[p + 1];
  }
  __device__ int64_t query(int64_t e) const { return pair_vals[e] / tmax; }
  __device__ int64_t slot(int64_t e) const { return e; }
};

// Largest k of the tensor-core scan (its heap mode) and the largest
// candidate list per pair slot in that mode.
constexpr int kTcWideK = 128;
constexpr int kTcWideList = 256;

// Finishing of the tensor-core scan (finish_tc.cu), on the scan's candidate
// lists [nq * t][kc], headers [nq * t] (L_k, count | overflow << 31) and the
// queries' bounds [nq] (ordered key of the largest L_k): the exact top k
// (k <= 128) of every query into ids_out / scores_out.
void finish_tc_queries(const IndexData& ix, const Cand* lists, const int2* hdr, const unsigned* gbound,
                       const int32_t* inv, int64_t nq, int t, const int32_t* tpq, const float* Qf,
                       const int32_t* top, int k, int kc, int64_t* ids_out, float* scores_out, cudaStream_t s);

// Tensor-core scan (scan_tc.cu) of a full-vector index (rows in the
// core-matrix layout of tc.cuh, queries as fp32 rows of tc_kp columns):
// screening on the tensor cores, then exact rescoring; the final top k of
// every query goes to ids_out / scores_out.  counter: zero; hdr [nq * t]:
// cleared headers of the grouped pairs; gbound [nq]: the ordered key of -inf;
// lists: room for kc = scan_tc_list_len(k, nq * t) candidates a pair.
// k <= scan_tc_max_k(ix) (at most 128).
void scan_tc_search(const IndexData& ix, const IvfWork& work, int max_items, const float* Qf, const float* qnorm,
                    const int32_t* top, const int32_t* inv, const int32_t* tpq, int64_t nq, int t, int k,
                    Cand* lists, int kc, int* counter, int2* hdr, unsigned* gbound, int* err, int64_t* ids_out,
                    float* scores_out, cudaStream_t s, Scratch& scr);
int scan_tc_max_k(const IndexData& ix);
// Group-maxima scan (scan_gm.cu), which takes k <= 16 when its shared memory fits
// the row width; lists [pairs][kc].  Headers cleared, bounds -inf and the work
// counter zero before the launch.
bool scan_gm_usable(const IndexData& ix, int k);
void scan_gm_launch(const IndexData& ix, const IvfWork& work, int grid, const float* Qf, const float* qnorm,
                    int64_t nq, int k, int kc, float dscale, long long wait_limit, int* counter, int* err,
                    unsigned* gbound, Cand* lists, int2* hdr, cudaStream_t s, Scratch& scr);
// SM cycles a pipeline wait of the scan may take before its CTA gives up
// (0: the default of about a second); the teardown's waits keep the default.
void set_scan_wait_limit(long long cycles);
// Candidate-list length per pair slot for a batch of `pairs` (query, probe) pairs.
int scan_tc_list_len(int k, int64_t pairs);

// Query-major exact scan (scan_query.cu): one or more warps per (query, probe)
// pair (top [nq][t], tpq per-query counts or null) over the core-matrix rows;
// the exact top k (k <= 32) of every query into ids_out / scores_out.  Usable when
// the batch probes few pairs per partition (nq * t <= 2c), k <= 32 and the
// rows have at most 1 024 columns.
bool scan_by_query_usable(const IndexData& ix, int64_t nq, int t, int k);
void scan_by_query(const IndexData& ix, const float* Qf, int qstride, const int32_t* top, const int32_t* tpq,
                   int64_t nq, int t, int k, int64_t* ids_out, float* scores_out, cudaStream_t s, Scratch& scr);

// Search over the compressed layouts (shortlist.cu): for every query the R best
// approximate scores over its probed union, each point once (its copy in the
// earliest-probed partition), rescored exactly against Q (dt), the best k
// (k <= R <= 4 096) into ids_out / scores_out.
//   FP8  approximate score s_q * s_x * sum q8 x8; Qf the queries' code values
//        (code_stride columns), qscale their scales
//   PQ4  approximate score <q, C_p> + sum_s <q_s, B[s][code_s]>; Qf fp32 rows of
//        qstride columns
void fp8_search(const IndexData& ix, const float* Qf, const float* qscale, const void* Q, soar_dtype dt,
                const int32_t* top, const int32_t* tpq, int64_t nq, int t, int R, int k, int64_t* ids_out,
                float* scores_out, cudaStream_t s, Scratch& scr);
void pq_search(const IndexData& ix, const float* Qf, int qstride, const void* Q, soar_dtype dt, const int32_t* top,
               const int32_t* tpq, int64_t nq, int t, int R, int k, int64_t* ids_out, float* scores_out,
               cudaStream_t s, Scratch& scr);

// (query, probe) pairs of a batch grouped by partition (search.cu).
struct Grouped {
  const int32_t* order;    // [c] partitions in the order their items are handed out
  int64_t* pair_off;       // [c + 1]
  const int32_t* vals;     // pairs sorted by partition (value q * t + j)
  int32_t* item_base;      // [c + 1]
  int* counter;            // work items handed out so far, zero
  int max_items;
  int2* hdr;               // tensor-core scan: cleared headers of the pair slots, bounds of the queries
  unsigned* gbound;
};
Grouped group_pairs(const IndexData& ix, int64_t nq, int t, const int32_t* tpq, int qb, const int32_t* top,
                    int32_t* inv, cudaStream_t s, Scratch& scr, bool tc, bool first_probes_first);

}  // namespace soar
