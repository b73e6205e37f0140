// Primary and first spilled assignment on the 5th-generation tensor cores.
//
// One persistent CTA per SM takes items of points whose rows form two A operands
// of 128 rows in shared memory (fp32 in the K-major core-matrix layout of
// tc.cuh, staged by cp.async): for the primary assignment two blocks of 128
// points, for the spill 128 points and their unit residuals r_hat = (x -
// C[pi(x)]) / ||x - C[pi(x)]|| (one A operand where rows are too wide for two).
// The codebook, packed once per pass in that layout as B tiles of 128
// centroids split into 8-column K steps, streams through a shared-memory ring
// of those K steps, copied by cp.async.bulk (it stays in L2: every CTA reads
// all of it, each starting at its own tile); every B tile serves both A
// operands, which halves that traffic.  Per K step one thread issues the
// kind::tf32 MMAs into a double-buffered TMEM accumulator.  Eight epilogue
// warps read the scores back, one point per TMEM lane (the spill: two warps a
// lane, half of the tile's columns each), and evaluate the expanded loss of
// Theorem 3.1
//     L(c') = ||c'||^2 - 2<x, c'> + lambda (<x, r_hat> - <c', r_hat>)^2
// (||x||^2 dropped: constant per point; lambda term absent for the primary).
//
// Rigorous screening.  Both operands are rounded to the nearest tf32 value
// before the MMA (an error of 2^-11 each; the hardware would truncate, 2^-10), so
// |<a, b>~ - <a, b>| < 2^-10 (1 + 2^-12) ||a|| ||b||, and the fp32 accumulation
// adds at most 2^-16 ||a|| ||b||.  The screened loss of a pair is within
//     delta = 2^-9 (1 + 2^-4) ||x|| ||c'|| + lambda e (2 |t~| + e),
//     e = 2^-10 (1 + 2^-4) ||c'||,
// (t~ = <x, r_hat> - <c', r_hat>~) plus an allowance for the fp32 rounding of the
// loss and of the exact decision.  Per point the epilogue keeps the smallest
// upper bound U = min(L~ + delta) so far and the pairs with L~ - delta <= U; the
// true minimiser is among them unless more than the list holds are (the point
// is then flagged and its refine pass scores every centroid).  Centroids the
// point is already assigned to are excluded.  A point with one candidate left
// is decided; the others are queued, and the refine kernel decides among the
// candidates with the direct form ||x - c'||^2 + lambda <x - c', r_hat>^2, lower
// index on ties.
//
// Bound of the primary: the epilogue's issue slots and the codebook stream from
// L2 (tf32 floor 0.51 ms for 1.18 M x 100 against 2 000 centroids).  Keeping the
// sixteen smallest lower bounds sorted cost 37 of 47 instructions a pair (5.9 ms
// a pass, the spill 6.8); most pairs are now dismissed eight at a time by a
// maximum that the TMEM load computes: 1.36 ms, the spill 3.50 (of which copies and
// MMAs 0.88 and 1.73, staging the operands 0.27 and 0.63, the survivors 0.2 and
// 0.57).
//
// Warp roles: 0 = bulk-copy producer, 1 = TMEM owner and MMA issuer,
// 2 = gate, 3..10 = epilogue and A-operand loaders.  Every mbarrier wait is bounded;
// on expiry the CTA raises *err, stops, waits (bounded) for its copies and
// MMAs in flight, frees its TMEM and returns.
#include <type_traits>

#include "internal.cuh"
#include "tc.cuh"

namespace soar {

namespace {

constexpr int kTM = 128;       // rows of an A operand (MMA M)
constexpr int kN = 128;        // centroids of a B tile (MMA N): two operands x two buffers fill the 512 TMEM columns
constexpr int kEpi = 256;      // epilogue threads (8 warps: 4 lane quarters x 2)
constexpr int kThr = 96 + kEpi;   // producer, MMA issuer, gate, epilogue
constexpr int kStagesMax = 8;
constexpr int kStepBytes = kN * 32;   // a K step (8 columns) of a codebook tile
constexpr int kList = 16;      // candidates handed to the refine per point

// v rounded to the nearest value with 10 explicit mantissa bits (ties away from
// zero); infinities and NaNs pass through.
__device__ __forceinline__ float round_tf32(float v) {
  uint32_t u = __float_as_uint(v);
  if ((u & 0x7f800000u) == 0x7f800000u) return v;
  u = (u + 0x1000u) & 0xffffe000u;
  return __uint_as_float(u);
}

template <typename XT>
struct AsgParams {
  const XT* X;
  int64_t n;
  int d, kp;
  const float* Cc;        // [ctiles][kp / 8][kN][8] packed codebook (padding rows: zeros, +inf norm)
  const float* tmax;      // [ctiles] largest ||c|| of each B tile
  const float* C;         // [c][d] row-major
  int c, ctiles;
  int32_t* assign;        // [n][astride]: column 0 = primary (read by the spill pass); decided points written
  int astride;
  const float* inv_rn;    // [n][4] 1 / ||x - C[pi(x)]|| (0 for a zero residual)
  float lambda;
  int stages, steps;      // codebook stages, K steps in each
  int cap;                // candidates an epilogue thread holds
  int* err;
  int32_t* cand;          // [n][kList] candidate centroids, -1 padded
  int32_t* queue;         // [n] points left to the refine: with candidates from the front, flagged ones from the back
  uint64_t* best;         // [n] the flagged points' best keys so far (set to none here)
  int* qcount;            // [2] how many of each
  int vec;                // rows of whole 16-byte pieces, X and C 16-byte aligned: 16-byte copies (fp32) or loads
};

__device__ __forceinline__ float ld(const float* p) { return __ldg(p); }
__device__ __forceinline__ float ld(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// OPS = A operands: 2 (primary: two blocks of points; spill: points and
// residuals) or, for the primary only, 1.
template <int NDIR, int OPS, typename XT>
__global__ void __launch_bounds__(kThr, 1) assign_tc_kernel(AsgParams<XT> P) {
  constexpr bool kSplit = NDIR > 0 || OPS == 1;    // two epilogue threads a point, half of the columns each
  constexpr int kPts = kSplit ? kTM : 2 * kTM;  // points per item
  constexpr int kCols = kSplit ? kN / 2 : kN;   // columns per epilogue thread and tile
  constexpr uint32_t kW = OPS * kN;             // TMEM columns per accumulator buffer
  // the no-swizzle operand layout needs 16-byte alignment only
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  const int kp = P.kp, S = P.stages, ksteps = kp / 8, per = P.steps;
  const int nch = (ksteps + per - 1) / per;     // stages per B tile
  const uint32_t stage_bytes = (uint32_t)per * kStepBytes;
  const uint32_t sbo = (uint32_t)kp * 32u;
  const uint32_t a_bytes = (uint32_t)kTM * kp * 4u;
  unsigned char* sA = base;                                                  // OPS operands
  unsigned char* sB = base + (size_t)OPS * a_bytes;
  float* list_lb = reinterpret_cast<float*>(sB + (size_t)S * stage_bytes);   // [cap][kEpi]
  int* list_id = reinterpret_cast<int*>(list_lb + P.cap * kEpi);             // [cap][kEpi]
  float* nx_s = reinterpret_cast<float*>(list_id + P.cap * kEpi);            // [kEpi] ||x||^2 (one operand: of either half of the columns)
  float* mu_s = nx_s + kEpi;                                                // [kTM] U of the second half
  float* mev_s = mu_s + kTM;                                                // [kTM]
  int* mcnt_s = reinterpret_cast<int*>(mev_s + kTM);                        // [kTM]
  float* xr_s = reinterpret_cast<float*>(mcnt_s + kTM);                     // [kTM] <x, r_hat>
  float* rn_s = xr_s + kTM;                                                 // [kTM] 1 or 0 (zero residual)
  int* prior_s = reinterpret_cast<int*>(rn_s + kTM);                        // [kTM]
  uint64_t* bars = reinterpret_cast<uint64_t*>(prior_s + kTM);
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s, issued_s, consumed_s, committed_s;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto full = [&](int s) { return tc::smem_u32(&bars[s]); };
  auto empty = [&](int s) { return tc::smem_u32(&bars[S + s]); };
  auto tfull = [&](int b) { return tc::smem_u32(&bars[2 * S + b]); };
  auto tempty = [&](int b) { return tc::smem_u32(&bars[2 * S + 2 + b]); };
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      tc::bar_init(full(s), 1);
      tc::bar_init(empty(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::bar_init(tfull(b), 1);
      tc::bar_init(tempty(b), kEpi / 32);
    }
    tc::bar_init_fence();
    abort_s = 0;
    issued_s = consumed_s = committed_s = 0;
  }
  if (warp == 1) tc::tmem_alloc(tc::smem_u32(&tmem_base_s), 2 * kW);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_base_s;
  const uint32_t idesc = tc::idesc_tf32(kTM, kN);
  volatile int* abort_v = &abort_s;
  auto give_up = [&]() {
    if (atomicExch(&abort_s, 1) == 0) atomicExch(P.err, 1);
  };
  // epilogue thread: TMEM lane 32 (warp % 4) + lane = row m of an operand; hh: its
  // operand (two blocks of points) or its half of the columns
  const int m = 32 * (warp & 3) + lane;
  const int hh = (warp - 3) >> 2;
  const int mp = kSplit ? m : m + kTM * hh;     // point within the item
  const int et = threadIdx.x - 96;              // epilogue thread index (list column)

  // static schedule: items blockIdx.x, blockIdx.x + gridDim.x, ... so that the
  // producer can stream the codebook across item boundaries
  const int ntiles_pts = (int)((P.n + kPts - 1) / kPts);
  const int nitems = ntiles_pts > (int)blockIdx.x ? (ntiles_pts - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  // each CTA sweeps the codebook from its own starting tile, so that the SMs
  // do not all read the same L2 lines at the same moment
  const int rot = (int)(((int64_t)blockIdx.x * P.ctiles) / gridDim.x);

  if (warp == 0) {
    // ---- producer: the codebook stages of every item, back to back
    if (lane == 0) {
      uint32_t C = 0;
      bool stop = false;
      for (int it = 0; it < nitems && !stop; ++it)
        for (int i = 0; i < P.ctiles && !stop; ++i) {
          const int ti = (i + rot) % P.ctiles;
          for (int g = 0; g < nch; ++g, ++C) {
            const uint32_t s = C % S, ph = (C / S) & 1;
            if (!tc::bar_wait(empty(s), ph ^ 1, abort_v)) { give_up(); stop = true; break; }
            const int k0 = g * per, kn = min(per, ksteps - k0);
            const uint32_t bytes = (uint32_t)kn * kN * 32;
            tc::bar_arrive_expect_tx(full(s), bytes);
            tc::bulk_copy_g2s(tc::smem_u32(sB) + s * stage_bytes, P.Cc + ((int64_t)ti * ksteps + k0) * kN * 8,
                              bytes, full(s));
            issued_s = (int)(C + 1);
          }
        }
    }
  } else {
    uint32_t tile_ctr = 0, chunk_ctr = 0;
    uint32_t committed = 0;                     // MMA issuer: tiles whose tfull commit was issued
    for (int it = 0; it < nitems; ++it) {
      if (tc::named_bar_or(3, kThr - 32, *abort_v != 0)) break;   // (also ends the previous item)
      const int item = (int)blockIdx.x + it * (int)gridDim.x;
      const int64_t p = (int64_t)item * kPts + mp;
      const bool active = warp >= 3 && p < P.n;

      // ---- A operands: a thread stages one row, rounded to tf32 and closed by
      // (-1/2, -1/2) in columns d, d + 1 against the codebook's (hi, lo) split of
      // ||c||^2; with residuals, the second half of the threads stages those, with a
      // single operand the second half of its columns
      if (warp >= 3) {
        const bool resid = NDIR > 0 && hh == 1;
        float* row = reinterpret_cast<float*>(sA + (size_t)(OPS == 2 ? hh : 0) * a_bytes) + (m >> 3) * (kp * 8) + (m & 7) * 4;
        float inv = 0.f;
        int prior = -1;
        const float* cr = nullptr;
        if (resid && active) {
          prior = P.assign[p * P.astride];
          inv = P.inv_rn[p * 4];
          cr = assigned_row(P.C, prior, P.d);
        }
        float ss = 0.f, xd = 0.f;
        const int d4 = P.vec ? P.d / 4 : 0;             // 4-column chunks in 16-byte copies or loads
        const int mid = OPS == 1 ? kp / 16 * 2 : 0;
        const int c0 = OPS == 1 && hh == 1 ? mid : 0, c1 = OPS == 1 && hh == 0 ? mid : kp / 4;   // this thread's chunks
        const int cv1 = min(c1, d4);
        const auto put = [&](int k4, const float (&xv)[4], const float (&cv)[4]) {
          float av[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int k = 4 * k4 + u;
            if (resid) {
              const float rv = (xv[u] - cv[u]) * inv;
              xd = fmaf(xv[u], rv, xd);
              av[u] = round_tf32(rv);
            } else {
              ss = fmaf(xv[u], xv[u], ss);
              av[u] = (k == P.d || k == P.d + 1) ? -0.5f : round_tf32(xv[u]);
            }
          }
          *reinterpret_cast<float4*>(row + k4 * 32) = make_float4(av[0], av[1], av[2], av[3]);
        };
        const auto centroid4 = [&](int k4) {
          return resid && active ? __ldg(reinterpret_cast<const float4*>(cr + 4 * k4)) : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        if constexpr (std::is_same<XT, float>::value) {
          const float* xsrc = P.X + p * P.d;
          if (active)
            for (int k4 = c0; k4 < cv1; ++k4) tc::cp_async16(tc::smem_u32(row + k4 * 32), xsrc + 4 * k4);
          tc::cp_async_wait_all();
#pragma unroll 4
          for (int k4 = c0; k4 < cv1; ++k4) {
            const float4 x = active ? *reinterpret_cast<const float4*>(row + k4 * 32) : make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 cc = centroid4(k4);
            put(k4, {x.x, x.y, x.z, x.w}, {cc.x, cc.y, cc.z, cc.w});
          }
        } else {
#pragma unroll 4
          for (int k4 = c0; k4 < cv1; k4 += 2) {        // 8 columns a load (c0 and cv1 are even)
            const uint4 x = active ? __ldg(reinterpret_cast<const uint4*>(P.X + p * P.d + 4 * k4)) : make_uint4(0u, 0u, 0u, 0u);
            const float4 ca = centroid4(k4), cb = centroid4(k4 + 1);
            put(k4, {__uint_as_float(x.x << 16), __uint_as_float(x.x & 0xffff0000u), __uint_as_float(x.y << 16),
                     __uint_as_float(x.y & 0xffff0000u)}, {ca.x, ca.y, ca.z, ca.w});
            put(k4 + 1, {__uint_as_float(x.z << 16), __uint_as_float(x.z & 0xffff0000u), __uint_as_float(x.w << 16),
                         __uint_as_float(x.w & 0xffff0000u)}, {cb.x, cb.y, cb.z, cb.w});
          }
        }
#pragma unroll 4
        for (int k4 = max(c0, cv1); k4 < c1; ++k4) {    // rows of other widths, and the padding
          float xv[4], cv[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int k = 4 * k4 + u;
            xv[u] = (active && k < P.d) ? ld(P.X + p * P.d + k) : 0.f;
            cv[u] = (resid && active && k < P.d) ? __ldg(cr + k) : 0.f;
          }
          put(k4, xv, cv);
        }
        if (resid) {
          xr_s[m] = xd;                                  // <x, r_hat> of the fp32 r_hat
          rn_s[m] = inv > 0.f ? 1.f : 0.f;
          prior_s[m] = prior;
        } else {
          nx_s[OPS == 1 ? m + kTM * hh : mp] = ss;
        }
        tc::fence_async_smem();
      }
      asm volatile("bar.sync 3, %0;" ::"n"(kThr - 32) : "memory");

      if (warp == 1) {
        // ---- MMA issuer.  It never touches an mbarrier (an mbarrier access
        // right after tcgen05.mma stalls the thread until the MMA pipe
        // drains): the gate warp waits for it and hands each codebook stage
        // over through a named barrier that also carries the stop flag.
        bool stop = false;
        for (int i = 0; i < P.ctiles && !stop; ++i) {
          const uint32_t T = tile_ctr + i, b = T & 1;
          for (int g = 0; g < nch; ++g) {
            stop = tc::named_bar_or(2, 64, false);
            if (stop) break;
            if (lane == 0) {
              const uint32_t C = chunk_ctr + i * nch + g, s = C % S;
              tc::fence_after_sync();
              const int k0 = g * per, kn = min(per, ksteps - k0);
              for (int jj = 0; jj < kn; ++jj) {
                const int j = k0 + jj;
                const uint64_t bd = tc::smem_desc(tc::smem_u32(sB) + s * stage_bytes + jj * kN * 32, 128, 256);
#pragma unroll
                for (int o = 0; o < OPS; ++o)
                  tc::mma_tf32(tmem + b * kW + o * kN,
                               tc::smem_desc(tc::smem_u32(sA) + o * a_bytes + j * 256, 128, sbo), bd, idesc, j > 0);
              }
              tc::mma_commit(empty(s));              // the stage is free once these MMAs completed
            }
            __syncwarp();
          }
          if (lane == 0) tc::mma_commit(tfull(b));   // (also after a stop: MMAs in flight land first)
          committed = T + 1;
        }
        if (lane == 0) committed_s = (int)committed;
      } else if (warp == 2) {
        // ---- gate: waits for the TMEM buffer and each codebook stage, then
        // releases the MMA issuer
        bool stop = false;
        for (int i = 0; i < P.ctiles && !stop; ++i) {
          const uint32_t T = tile_ctr + i, b = T & 1, tph = (T >> 1) & 1;
          for (int g = 0; g < nch; ++g) {
            const uint32_t C = chunk_ctr + i * nch + g, s = C % S, ph = (C / S) & 1;
            int ok = 1;
            if (lane == 0) {
              ok = (g > 0 || tc::bar_wait(tempty(b), tph ^ 1, abort_v)) && tc::bar_wait(full(s), ph, abort_v);
              if (!ok) give_up();
              else consumed_s = (int)(C + 1);
              tc::fence_before_sync();
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            stop = tc::named_bar_or(2, 64, !ok);
            if (stop) break;
          }
        }
      } else {
        // ---- epilogue: kCols of each B tile's columns per thread
        float* lbs = list_lb + et;                     // [cap] lower bounds and ids of the candidates so far
        int* ids = list_id + et;
        int cnt = 0;
        float U = INFINITY, packed = INFINITY;         // packed: U when the list was last cleared of stale entries
        float ev = INFINITY;                           // the smallest lower bound the list had no room for
        const float nx = sqrtf(OPS == 1 ? nx_s[m] + nx_s[m + kTM] : nx_s[mp]), nx2 = nx * nx;
        const float xr = NDIR > 0 ? xr_s[m] : 0.f, er0 = NDIR > 0 ? ldexpf(rn_s[m], -10) * 1.0625f : 0.f;
        const int prior = NDIR > 0 ? prior_s[m] : -1;
        const float lam = P.lambda;
        for (int i = 0; i < P.ctiles; ++i) {
          const uint32_t T = tile_ctr + i, b = T & 1, tph = (T >> 1) & 1;
          const bool ok = tc::bar_wait(tfull(b), tph, abort_v);
          if (!ok) give_up();
          tc::fence_after_sync();
          // per-tile bound: |L~ - L| <= dlc + 2 lambda e |t~| for every column
          const int ti = (i + rot) % P.ctiles;
          const float cmax = __ldg(P.tmax + ti), c2max = cmax * cmax;
          const float e = er0 * cmax;
          float dlc = fmaf(ldexpf(nx, -9) * 1.0625f, cmax, ldexpf(fmaf(nx, cmax, c2max), -14) + ldexpf(nx2, -16));
          if (NDIR > 0) dlc = fmaf(lam * e, e, fmaf(ldexpf(lam, -14), (nx + cmax) * (nx + cmax), dlc));
          const float two_le = 2.f * lam * e;
          const uint32_t tbase = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + b * kW +
                                 (kSplit ? hh * kCols : hh * kN);
#pragma unroll 1
          for (int rd = 0; rd < kCols / 32 && ok; ++rd) {
            const uint32_t taddr = tbase + 32 * rd;
            const int cbase = ti * kN + (kSplit ? hh * kCols : 0) + 32 * rd;
            float v[32];                               // primary: <x, c> - ||c||^2 / 2; spill: lower bounds
            uint32_t gm = 0u;                          // groups of eight columns that hold a candidate
            if constexpr (NDIR == 0) {
              uint32_t rx[32];
              float g[4];
#pragma unroll
              for (int q8 = 0; q8 < 4; ++q8) tc::tmem_ld8_max(taddr + 8 * q8, rx + 8 * q8, g[q8]);
              tc::tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(rx[j]);
              // (padded centroids carry ||c||^2 = +inf: their product is -inf)
              U = fminf(U, fmaf(-2.f, fmaxf(fmaxf(g[0], g[1]), fmaxf(g[2], g[3])), dlc));
              const float cut = -0.5f * (U + dlc);     // L~ - delta <= U
#pragma unroll
              for (int q8 = 0; q8 < 4; ++q8) gm |= (g[q8] >= cut ? 1u : 0u) << q8;
            } else {
              uint32_t rx[32], rr[32];
              tc::tmem_ld32(taddr, rx);
              tc::tmem_ld32(taddr + kN, rr);
              tc::tmem_ld_wait();
              float um[4] = {INFINITY, INFINITY, INFINITY, INFINITY}, lm[4] = {INFINITY, INFINITY, INFINITY, INFINITY};
              const int jskip = prior - cbase;         // the point's own centroid
              if (__any_sync(0xffffffffu, (unsigned)jskip < 32u)) {
#pragma unroll
                for (int j = 0; j < 32; ++j)
                  if (j == jskip) rx[j] = 0xff800000u;   // -inf: an infinite loss
              }
#pragma unroll
              for (int j = 0; j < 32; ++j) {
                const float t = xr - __uint_as_float(rr[j]);
                const float L = fmaf(lam * t, t, -2.f * __uint_as_float(rx[j]));
                const float dl = fmaf(two_le, fabsf(t), dlc);
                v[j] = L - dl;
                um[j & 3] = fminf(um[j & 3], L + dl);
                lm[j >> 3] = fminf(lm[j >> 3], v[j]);
              }
              U = fminf(U, fminf(fminf(um[0], um[1]), fminf(um[2], um[3])));
#pragma unroll
              for (int q8 = 0; q8 < 4; ++q8) gm |= (lm[q8] <= U ? 1u : 0u) << q8;
            }
            // an idle row (past the last point) is zero: it would be near all
            // centroids of equal norm at once, and its warp's time the whole pass's
            if (!active) gm = 0u;
            // one trip per surviving group of the lane with the most of them, in it
            // one per candidate (kept small: this code unrolled over the rounds ran
            // at half the speed, short of instructions)
            while (__any_sync(0xffffffffu, gm != 0u)) {
              const int q8 = __ffs(gm) - 1;            // -1: this lane has none left
              gm &= gm - 1u;
              float w[8];
              uint32_t em = 0u;
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                const float lo = q8 & 1 ? v[8 + u] : v[u], hi = q8 & 1 ? v[24 + u] : v[16 + u];
                w[u] = q8 & 2 ? hi : lo;
                if (NDIR == 0) w[u] = fmaf(-2.f, w[u], -dlc);
                em |= (w[u] <= U ? 1u : 0u) << u;
              }
              if (q8 < 0) em = 0u;
              while (__any_sync(0xffffffffu, em != 0u)) {
                const int u = __ffs(em) - 1;
                em &= em - 1u;
                const float a0 = u & 1 ? w[1] : w[0], a1 = u & 1 ? w[3] : w[2], a2 = u & 1 ? w[5] : w[4],
                            a3 = u & 1 ? w[7] : w[6];
                const float b0 = u & 2 ? a1 : a0, b1 = u & 2 ? a3 : a2;
                const float lb = u & 4 ? b1 : b0;
                const bool take = u >= 0 && lb < INFINITY;
                if (__any_sync(0xffffffffu, take && cnt == P.cap && U < packed)) {
                  if (cnt == P.cap && U < packed) {    // candidates that fell behind make room, once per fall of U
                    packed = U;
                    int k = 0;
#pragma unroll 1
                    for (int j = 0; j < cnt; ++j) {
                      const float o = lbs[j * kEpi];
                      if (o <= U) {
                        lbs[k * kEpi] = o;
                        ids[k * kEpi] = ids[j * kEpi];
                        ++k;
                      }
                    }
                    cnt = k;
                  }
                }
                const bool room = cnt < P.cap;
                if (take && room) {
                  lbs[cnt * kEpi] = lb;
                  ids[cnt * kEpi] = cbase + 8 * q8 + u;
                }
                if (take && !room) ev = fminf(ev, lb);
                cnt += take && room ? 1 : 0;
              }
            }
          }
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::bar_arrive(tempty(b));
          if (!ok) break;
        }
        if constexpr (kSplit) {                        // the second half's bounds and count for the first
          if (hh == 1) {
            mu_s[m] = U;
            mev_s[m] = ev;
            mcnt_s[m] = cnt;
          }
          asm volatile("bar.sync 1, %0;" ::"n"(kEpi) : "memory");
        }
        if ((!kSplit || hh == 0) && active && !abort_s) {
          int other = 0;
          if constexpr (kSplit) {
            U = fminf(U, mu_s[m]);
            ev = fminf(ev, mev_s[m]);
            other = mcnt_s[m];
          }
          int ncand = 0, only = -1;
          int32_t* cand = P.cand + p * kList;
          for (int j = 0; j < cnt + other; ++j) {
            const int at = j < cnt ? j * kEpi : (j - cnt) * kEpi + kTM;    // (et + kTM: the second half's list)
            if (lbs[at] <= U) {
              only = ids[at];
              if (ncand < kList) cand[ncand] = only;
              ++ncand;
            }
          }
          // (no candidate at all: no finite loss)
          const bool over = ev <= U || ncand > kList || ncand == 0;
          if (ncand == 1 && !over) {
            P.assign[p * P.astride + NDIR] = only;     // the bounds leave one centroid: decided
          } else if (!over) {
            for (int q = ncand; q < kList; ++q) cand[q] = -1;
          }
          // queue the undecided points for the direct-form refine (an atomic per warp and queue)
          const unsigned am = __activemask();
          const unsigned listed = __ballot_sync(am, ncand != 1 && !over), flagged = __ballot_sync(am, over);
          const int leader = __ffs(am) - 1;
          int lbase = 0, fbase = 0;
          if (lane == leader && listed) lbase = atomicAdd(P.qcount, __popc(listed));
          if (lane == leader && flagged) fbase = atomicAdd(P.qcount + 1, __popc(flagged));
          lbase = __shfl_sync(am, lbase, leader);
          fbase = __shfl_sync(am, fbase, leader);
          const unsigned before = (1u << lane) - 1;
          if (listed & (1u << lane)) P.queue[lbase + __popc(listed & before)] = (int32_t)p;
          if (flagged & (1u << lane)) {
            const int f = fbase + __popc(flagged & before);
            P.queue[P.n - 1 - f] = (int32_t)p;
            P.best[f] = ~0ull;
          }
        }
      }
      tile_ctr += P.ctiles;
      chunk_ctr += (uint32_t)P.ctiles * nch;
    }
  }

  __syncthreads();
  if (abort_s && threadIdx.x == 0) {
    volatile int never = 0;
    for (int C = consumed_s; C < issued_s; ++C) tc::bar_wait(full(C % S), (C / S) & 1, &never);
  }
  if (abort_s && threadIdx.x == 64 && committed_s > 0) {
    volatile int never = 0;
    const int T = committed_s - 1;
    tc::bar_wait(tfull(T & 1), (T >> 1) & 1, &never);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 1) tc::tmem_dealloc(tmem, 2 * kW);
}

// ||c||^2 and ||c|| of every centroid (a warp each); clears the pass's queue counters.
__global__ void codebook_norms(const float* __restrict__ C, int c, int d, float* __restrict__ n2,
                               float* __restrict__ n1, int* __restrict__ qcount) {
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (w >= c) return;
  if (w == 0 && lane < 2) qcount[lane] = 0;
  float s = 0.f;
  for (int k = lane; k < d; k += 32) {
    const float v = C[(int64_t)w * d + k];
    s = fmaf(v, v, s);
  }
  s = warp_sum(s);
  if (lane == 0) {
    n2[w] = s;
    n1[w] = sqrtf(s);
  }
}

// Codebook as B tiles of kN rows, each split into K steps of 8 columns stored
// contiguously in the core-matrix layout of tc.cuh (8-row groups 256 bytes
// apart), rounded to tf32: rows padded to ctiles * kN and columns to kp with
// zeros, except columns d and d + 1 holding ||c||^2 split into its tf32 part and
// the remainder (the MMA then adds -||c||^2 / 2 to <x, c> at full fp32 accuracy);
// padding rows hold +inf there.
__global__ void pack_codebook(const float* __restrict__ C, const float* __restrict__ n2, int c, int d, int kp,
                              int rows_pad, float* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)rows_pad * kp) return;
  const int r = (int)(i / kp), k = (int)(i % kp);
  float v = 0.f;
  if (r < c) {
    if (k < d) {
      v = round_tf32(C[(int64_t)r * d + k]);
    } else if (k <= d + 1) {
      const float hi = __uint_as_float(__float_as_uint(n2[r]) & 0xffffe000u);   // tf32 truncation
      v = k == d ? hi : round_tf32(n2[r] - hi);
    }
  } else if (k == d) {
    v = INFINITY;           // padding rows: infinite loss for every point
  }
  const int ti = r / kN, rr = r % kN, j = k >> 3, kk = k & 7;
  out[((int64_t)ti * (kp / 8) + j) * kN * 8 + (rr >> 3) * 64 + (kk >> 2) * 32 + (rr & 7) * 4 + (kk & 3)] = v;
}

// Largest ||c|| of each tile (warp per tile).
__global__ void tile_max_norms(const float* __restrict__ n1, int c, int ctiles, float* __restrict__ tmax) {
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (w >= ctiles) return;
  float v = 0.f;
  for (int j = lane; j < kN; j += 32) {
    const int r = w * kN + j;
    if (r < c) v = fmaxf(v, n1[r]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if (lane == 0) tmax[w] = v;
}

// ||r||^2, r = x - c_prior, by a warp.
template <typename XT>
__device__ __forceinline__ float residual_norm2(const XT* x, const float* cr, int d, int lane) {
  float s = 0.f;
  for (int k = lane; k < d; k += 32) {
    const float v = load_elem(x, k) - cr[k];
    s = fmaf(v, v, s);
  }
  return warp_sum(s);
}

// Direct-form losses of the flagged points (the last qcount[1] of the queue)
// against every centroid not yet assigned to them, as keys (loss, centroid)
// that order like losses, lower index first, the least kept in best[f].  A
// block takes 64 points and a share of the codebook in tiles of 64 centroids, 4 x
// 4 pairs a thread, staged 16 columns at a time; every sum runs over k in
// ascending order in one fp32 accumulator, the order of the listed decision's
// two halves apart.  Few flagged points split the codebook over more blocks.
// Bound: the FMA pipe, two (primary) or three operations a pair and column.  In
// clusters tighter than the screening band every point is flagged, and a warp
// per point with a centroid per lane, whose loads touch 32 rows at once, took
// 72 ms for 200 000 x 150 against 2 000 (the pass now 5.8; the spill 77, now 9.3)
// and 454 at 320 columns (13.4); the general kernels of assign.cu take 13.5 for
// that spill and 14.9 at 320 columns.
constexpr int kFt = 64, kFk = 16, kFlagThreads = 256;
template <int NDIR, typename XT>
__global__ void __launch_bounds__(kFlagThreads) refine_flagged(const XT* __restrict__ X, int64_t n, int d,
                                                               const float* __restrict__ C, int c,
                                                               const int32_t* __restrict__ assign, int astride,
                                                               float lambda, const int32_t* __restrict__ queue,
                                                               const int* __restrict__ qcount,
                                                               uint64_t* __restrict__ best) {
  __shared__ __align__(16) float xs[kFk][kFt + 4], cs[kFk][kFt + 4], rs[NDIR > 0 ? kFk : 1][kFt + 4];
  __shared__ int32_t pt_s[kFt], prior_s[kFt];
  __shared__ float rn2_s[kFt];
  const int total = qcount[1], tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int pblocks = (total + kFt - 1) / kFt, ctiles = (c + kFt - 1) / kFt;
  if (pblocks == 0) return;
  const int slices = max(1, min(ctiles, (int)gridDim.x / pblocks)), per = (ctiles + slices - 1) / slices;
  const int tx = tid % 16, ty = tid / 16;        // centroids 4 tx .., points 4 ty ..
  for (int64_t item = blockIdx.x; item < (int64_t)pblocks * slices; item += gridDim.x) {
    const int f0 = (int)(item % pblocks) * kFt, t0 = (int)(item / pblocks) * per, t1 = min(ctiles, t0 + per);
    __syncthreads();
    if (tid < kFt) {
      const int32_t p = f0 + tid < total ? queue[n - 1 - f0 - tid] : -1;
      pt_s[tid] = p;
      prior_s[tid] = NDIR > 0 && p >= 0 ? assign[(int64_t)p * astride] : -1;
    }
    __syncthreads();
    if constexpr (NDIR > 0)
      for (int i = w; i < kFt; i += kFlagThreads / 32) {
        const int64_t p = pt_s[i];
        const float r = p >= 0 ? residual_norm2(X + p * d, assigned_row(C, prior_s[i], d), d, lane) : 0.f;
        if (lane == 0) rn2_s[i] = r;
      }
    uint64_t key[4] = {~0ull, ~0ull, ~0ull, ~0ull};
    for (int t = t0; t < t1; ++t) {
      float dist[4][4], pr[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) dist[i][j] = pr[i][j] = 0.f;
      for (int k0 = 0; k0 < d; k0 += kFk) {
        __syncthreads();
#pragma unroll
        for (int i = tid; i < kFt * kFk; i += kFlagThreads) {
          const int r = i / kFk, kk = i % kFk, k = k0 + kk;
          const int64_t p = pt_s[r];
          const int cq = t * kFt + r;
          const float xv = p >= 0 && k < d ? load_elem(X, p * d + k) : 0.f;
          xs[kk][r] = xv;
          cs[kk][r] = cq < c && k < d ? C[(int64_t)cq * d + k] : 0.f;
          if constexpr (NDIR > 0) rs[kk][r] = p >= 0 && k < d ? xv - assigned_row(C, prior_s[r], d)[k] : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < kFk; ++kk) {
          if (kk >= d - k0) break;                   // uniform
          const float4 xq = *reinterpret_cast<const float4*>(&xs[kk][4 * ty]);
          const float4 cq = *reinterpret_cast<const float4*>(&cs[kk][4 * tx]);
          const float xv[4] = {xq.x, xq.y, xq.z, xq.w}, cv[4] = {cq.x, cq.y, cq.z, cq.w};
          float rv[4] = {0.f, 0.f, 0.f, 0.f};
          if constexpr (NDIR > 0) {
            const float4 rq = *reinterpret_cast<const float4*>(&rs[kk][4 * ty]);
            rv[0] = rq.x; rv[1] = rq.y; rv[2] = rq.z; rv[3] = rq.w;
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float v = xv[i] - cv[j];
              dist[i][j] = fmaf(v, v, dist[i][j]);
              if constexpr (NDIR > 0) pr[i][j] = fmaf(v, rv[i], pr[i][j]);
            }
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int prior = prior_s[4 * ty + i];
        const float rn2 = NDIR > 0 ? rn2_s[4 * ty + i] : 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int cq = t * kFt + 4 * tx + j;
          const float l = NDIR > 0 && rn2 > 0.f ? fmaf(lambda, pr[i][j] * pr[i][j] / rn2, dist[i][j]) : dist[i][j];
          if (cq < c && cq != prior && l == l)       // losses are not negative: ordered like their bits
            key[i] = min(key[i], ((uint64_t)__float_as_uint(l) << 32) | (uint32_t)cq);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) key[i] = min(key[i], (uint64_t)__shfl_xor_sync(0xffffffffu, key[i], o));
      const int f = f0 + 4 * ty + i;
      if (tx == 0 && f < total)
        atomicMin(reinterpret_cast<unsigned long long*>(best + f), (unsigned long long)key[i]);
    }
  }
}

// Direct-form decision among the candidates of each listed point (warp per
// point, persistent over the queue, two lanes per candidate), lower index on
// equal losses; the flagged points' best centroids (-1 where no loss is a
// number) are written out.
template <typename XT>
__global__ void refine_list(const XT* __restrict__ X, int64_t n, int d, const float* __restrict__ C,
                            int32_t* __restrict__ assign, int astride, int col, float lambda,
                            const int32_t* __restrict__ cand, const int32_t* __restrict__ queue,
                            const uint64_t* __restrict__ best_flagged, const int* __restrict__ qcount) {
  constexpr unsigned kFull = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int64_t nthreads = (int64_t)gridDim.x * blockDim.x, thread = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int total = qcount[0], flagged = qcount[1];
  for (int64_t f = thread; f < flagged; f += nthreads)
    assign[(int64_t)queue[n - 1 - f] * astride + col] = (int32_t)(uint32_t)best_flagged[f];
  for (int64_t qi = thread >> 5; qi < total; qi += nthreads >> 5) {
    const int64_t p = queue[qi];
    const XT* x = X + p * d;
    const float* cr = assigned_row(C, col > 0 ? assign[p * astride] : 0, d);
    const float rn2 = col > 0 ? residual_norm2(x, cr, d, lane) : 0.f;
    static_assert(kList * 2 == 32, "two lanes per candidate");
    const int g = lane >> 1, part = lane & 1;
    const int cq = cand[p * kList + g];
    float dist = 0.f, pr = 0.f;
    if (cq >= 0) {
      const float* cv = C + (int64_t)cq * d;
      for (int k = part; k < d; k += 2) {
        const float xv = load_elem(x, k);
        const float v = xv - cv[k];
        dist = fmaf(v, v, dist);
        if (col > 0) pr = fmaf(v, xv - cr[k], pr);
      }
    }
    dist += __shfl_xor_sync(kFull, dist, 1);
    pr += __shfl_xor_sync(kFull, pr, 1);
    float best = INFINITY;
    int bi = -1;
    if (cq >= 0) {
      best = (col > 0 && rn2 > 0.f) ? fmaf(lambda, pr * pr / rn2, dist) : dist;
      bi = cq;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ob = __shfl_xor_sync(kFull, best, o);
      const int oi = __shfl_xor_sync(kFull, bi, o);
      if (oi >= 0 && (bi < 0 || ob < best || (ob == best && oi < bi))) { best = ob; bi = oi; }
    }
    if (lane == 0) assign[p * astride + col] = bi;
  }
}

size_t smem_for(int kp, int ops, int s, int steps, int cap) {
  return 128 + (size_t)ops * kTM * kp * 4 + (size_t)s * steps * kStepBytes + (size_t)cap * kEpi * 8 + (size_t)kEpi * 4 +
         (size_t)6 * kTM * 4 + (size_t)(2 * s + 4) * 8;
}

// K of the MMAs: d columns plus the two norm columns, a multiple of 8
int kp_for(int d) { return (d + 2 + 7) / 8 * 8; }

// A operands, codebook stages and list length that fit: two operands before one
// (half the codebook traffic), stages of 32 KB before 16 KB (fewer, larger copies),
// lists of 16 before 8, those before deep rings.  A point in the band of more
// centroids than its list holds is scored against all of them, which costs less
// than shorter stages or a second codebook stream (lists of 8 in 32 KB stages
// against lists of 16 in 16 KB ones, 4 M x 128 bf16 points: 40 000 centroids 90.5
// / 97.0 ms, with the spill 298 / 327; 4 000 centroids 10.0 / 11.2; two operands and
// lists of 8 against one and lists of 16, 200 000 x 152 points: 2 000 centroids
// 0.49 / 0.55 ms, 20 000, forty to a cluster, 3.30 / 3.49; 2 000, twenty tight ones to
// a cluster, every list full either way, 7.8 / 5.7).
struct Shape {
  int ops = 0, stages = 0, steps = 0, cap = 0;
};
Shape shape_for(int kp, int ndir, int most_ops = 2) {
  for (int ops = most_ops; ops >= (ndir ? 2 : 1); --ops)
    for (int steps : {8, 4})
      for (int cap : {16, 8})
        for (int s = kStagesMax; s >= 2; --s)
          if (smem_for(kp, ops, s, steps, cap) <= 227 * 1024 - 256)   // room for the static shared variables
            return Shape{ops, s, steps, cap};
  return Shape{};
}

}  // namespace

// Wide rows (a primary past 278 columns, a spill past 134) of few points against a
// small codebook go to the general kernels, which take fewer launches (us, here /
// there: primary of 300 columns, 2 000 x 64 81 / 57, 10 000 x 64 82 / 76, 10 000 x
// 128 74 / 116, 100 000 x 2 225 / 342; spill of 150, 2 000 x 64 66 / 38, 10 000 x 64
// 70 / 64, 10 000 x 128 71 / 101, 100 000 x 2 227 / 312).
bool assign_tc_usable(int64_t n, int d, int c, int ndir) {
  if (ndir > 1 || shape_for(kp_for(d), ndir).ops == 0) return false;
  return d <= (ndir ? 134 : 278) || n > 16384 || c > 64;
}

template <typename XT>
void assign_tc_pass(const XT* X, int64_t n, int d, const float* C, int c, int ndir, int32_t* assign, int astride,
                    const float* inv_rn, float lambda, cudaStream_t s, Scratch& scr) {
  const int kp = kp_for(d);
  // few points: 128 of them a block, so that twice as many SMs work (1 000 to 19 000
  // x 100 against 500 centroids: 72 -> 65 us)
  const Shape sh = shape_for(kp, ndir, ndir == 0 && n <= (int64_t)kTM * num_sms() ? 1 : 2);
  if (ndir > 1 || sh.ops == 0) fail(SOAR_EUNSUPPORTED, "tensor-core assignment: unsupported shape");
  const int ctiles = (c + kN - 1) / kN;
  float* Cc = scr.get<float>((size_t)ctiles * kN * kp);
  float* n2 = scr.get<float>(c);
  float* n1 = scr.get<float>(c);
  float* tmax = scr.get<float>(ctiles);
  int* qcount = scr.get<int>(2);             // queued points
  codebook_norms<<<ceil_div((int64_t)c * 32, 256), 256, 0, s>>>(C, c, d, n2, n1, qcount);
  SOAR_LAUNCHED();
  pack_codebook<<<ceil_div((int64_t)ctiles * kN * kp, 256), 256, 0, s>>>(C, n2, c, d, kp, ctiles * kN, Cc);
  SOAR_LAUNCHED();
  tile_max_norms<<<ceil_div((int64_t)ctiles * 32, 256), 256, 0, s>>>(n1, c, ctiles, tmax);
  SOAR_LAUNCHED();
  int32_t* cand = scr.get<int32_t>((size_t)n * kList);
  int32_t* queue = scr.get<int32_t>(n);
  uint64_t* best = scr.get<uint64_t>(n);
  const int vec = d * sizeof(XT) % 16 == 0 && reinterpret_cast<uintptr_t>(X) % 16 == 0 &&
                  reinterpret_cast<uintptr_t>(C) % 16 == 0;
  AsgParams<XT> prm{X, n, d, kp, Cc, tmax, C, c, ctiles, assign, astride, inv_rn, lambda, sh.stages,
                    sh.steps, sh.cap, device_error_word(), cand, queue, best, qcount, vec};
  const size_t smem = smem_for(kp, sh.ops, sh.stages, sh.steps, sh.cap);
  auto kern = ndir == 0 ? (sh.ops == 2 ? assign_tc_kernel<0, 2, XT> : assign_tc_kernel<0, 1, XT>)
                        : assign_tc_kernel<1, 2, XT>;
  allow_smem(kern, smem);
  const int pts = ndir == 0 && sh.ops == 2 ? 2 * kTM : kTM;
  const int grid = (int)std::min<int64_t>((n + pts - 1) / pts, num_sms());
  kern<<<grid, kThr, smem, s>>>(prm);
  SOAR_LAUNCHED();
  auto flagged = ndir == 0 ? refine_flagged<0, XT> : refine_flagged<1, XT>;
  flagged<<<num_sms() * 4, kFlagThreads, 0, s>>>(X, n, d, C, c, assign, astride, lambda, queue, qcount, best);
  SOAR_LAUNCHED();
  refine_list<XT><<<num_sms() * 8, 256, 0, s>>>(X, n, d, C, assign, astride, ndir, lambda, cand, queue, best, qcount);
  SOAR_LAUNCHED();
}

template void assign_tc_pass<float>(const float*, int64_t, int, const float*, int, int, int32_t*, int, const float*,
                                    float, cudaStream_t, Scratch&);
template void assign_tc_pass<__nv_bfloat16>(const __nv_bfloat16*, int64_t, int, const float*, int, int, int32_t*,
                                            int, const float*, float, cudaStream_t, Scratch&);

}  // namespace soar
