// Selector over every candidate (candidate_factor = 0 with Lc above the pooled
// selector's 512-slot pool): step 3 of the eviction step with C = Lc, one CTA per
// unit. Section 3.2 restricts the greedy to the top 4B tokens for speed; this path
// is the unrestricted ablation and admits exactly what the full greedy of Eq. 5
// admits over all Lc candidates.
//
//  1. max-pool mu and sigma over 0 .. Lc-1 (odd kernel, window clipped to the
//     range) and form s_i = mu_i + lambda1 sigma_i; s~ = s / max(max s, eps);
//  2. greedy admissions by s~_i + lambda2 corr_i, ties to the lower position, with
//     corr_i = max over admitted j of cos(k_i, k_j) (clamped at 0 by starting at 0).
//     With lambda2 <= 0 a value can only fall as the admitted set grows, so a value
//     computed against fewer admitted keys is an upper bound: each step takes the
//     best value; if it is stale, the threads whose own best candidate is stale and
//     could still be the admission bring it up to date (in parallel) and the search
//     repeats; a candidate whose value is current when it is the best is the full
//     greedy's choice (any candidate with an equal bound has a higher position).
//     With lambda2 > 0 every candidate is brought up to date after each admission, by
//     warps that take 32 candidates at a time through the tensor cores.
//     When margins are requested the runner-up is brought up to date the same way.
//  3. write the admitted positions ascending (and in admission order, with margins).
// Values live in shared memory (C <= 32768); s~, corr and the inverse key norms in
// the workspace; the first 96 admitted keys are staged in shared memory, later ones
// are read from K in global memory (L2). For lambda2 <= 0 a warp refreshes its lanes'
// stale bests together on the tensor cores; for lambda2 > 0 a warp forms the dots of 32
// candidates with the key just admitted.
#include "kve_internal.h"

namespace kve {
namespace {

// 128 registers a thread: with 1024 threads of 64 the selector spilled, and shared memory leaves the
// spills hardly any L1 (lambda2 > 0 over 4064 candidates: 1.28 ms against 0.82).
constexpr int kAllThreads = 512;
constexpr int kAllWarps = kAllThreads / 32;
constexpr int kAdmStage = 96;          // admitted keys staged in shared memory
constexpr int kAdmStride = 17;         // uint4 per staged row (16 + 1 against bank conflicts)
// Bits of the value of an admitted candidate: a NaN that no arithmetic returns. (-inf cannot stand for
// it: a caller may mask tokens by a base score of -inf, and those are admitted, lowest position
// first, once no other is left. A mark in `applied` made the searches 1.5 % slower.)
constexpr uint32_t kAdmitted = 0xFFFFFFFFu;

__device__ __forceinline__ uint32_t ord_key_all(float f) {
  const uint32_t u = __float_as_uint(f + 0.0f);   // -0 -> +0
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float unord_key_all(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The 32 candidate rows base .. base + 31 of a warp (rows past the last stand for it), 16 bytes
// per load: lane (g, t) holds of row base + 8 r + g the 16-byte chunks 4 s + t (r, s = 0 .. 3), so
// that a load instruction reads 64 contiguous bytes of each of 8 rows.
__device__ __forceinline__ void load_rows(const uint16_t* kb, int64_t kst, int base, int C, uint4 (&x)[4][4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, tq = lane & 3;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const uint4* row = reinterpret_cast<const uint4*>(kb + static_cast<int64_t>(min(base + 8 * r + g, C - 1)) * kst);
#pragma unroll
    for (int s = 0; s < 4; ++s) x[r][s] = __ldg(row + 4 * s + tq);
  }
}

// Of four values, one per row set r, the one of r = lane % 4: that lane's candidate is row
// base + 8 (lane % 4) + lane / 4.
__device__ __forceinline__ float own_row(const float (&y)[4]) {
  const int tq = threadIdx.x & 3;
  return tq < 2 ? (tq == 0 ? y[0] : y[1]) : (tq == 2 ? y[2] : y[3]);
}

struct AllSmall {
  uint32_t wkey[kAllWarps];    // per warp: its owners' best, and the best that is current
  uint32_t widx[kAllWarps];
  uint32_t wcur[kAllWarps];
  float wmax[kAllWarps];
  uint32_t best_key, best_idx, cur_key;
  bool stale;                  // the block's best is a bound, not its current value
};

// Block argmax of the owners' bests: the largest key, ties to the lowest index; and the largest
// of the owners' best current keys, `cur` (0: none has one).
__device__ __forceinline__ void block_best(uint32_t key, uint32_t idx, uint32_t cur, const uint16_t* applied, int t,
                                           AllSmall& sh) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t wk = __reduce_max_sync(0xffffffffu, key);
  const uint32_t wi = __reduce_min_sync(0xffffffffu, key == wk ? idx : 0xFFFFFFFFu);
  const uint32_t wc = __reduce_max_sync(0xffffffffu, cur);
  if (lane == 0) {
    sh.wkey[warp] = wk;
    sh.widx[warp] = wi;
    sh.wcur[warp] = wc;
  }
  __syncthreads();
  if (warp == 0) {
    const bool hold = lane < kAllWarps;
    const uint32_t k = hold ? sh.wkey[lane] : 0u, i = hold ? sh.widx[lane] : 0xFFFFFFFFu;
    const uint32_t bk = __reduce_max_sync(0xffffffffu, k);
    const uint32_t bi = __reduce_min_sync(0xffffffffu, k == bk ? i : 0xFFFFFFFFu);
    const uint32_t bc = __reduce_max_sync(0xffffffffu, hold ? sh.wcur[lane] : 0u);
    if (lane == 0) {
      sh.best_key = bk;
      sh.best_idx = bi;
      sh.cur_key = bc;
      // read here, between the barriers: the owner may bring it up to date after the second
      sh.stale = bi != 0xFFFFFFFFu && applied[bi] < t;
    }
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kAllThreads, 1) select_all_kernel(const __grid_constant__ SelectParams P) {
  wait_previous_kernel();   // mu and sigma come from the score kernel launched before
  __shared__ AllSmall sh;
  extern __shared__ __align__(16) uint8_t dyn[];
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;

  const UnitInfo u = unit_info(P.g, blockIdx.x);
  const int W = P.g.window;
  const int C = u.L - W;                      // every candidate
  const int B = P.budget;
  const int Bl = P.layer_budget[u.layer];
  const int nsel = min(Bl, C);
  const float lambda1 = P.lambda1[u.layer];
  const float lambda2 = P.lambda2[u.layer];
  const bool lazy = !(lambda2 > 0.f);
  const float* mu = P.mu + u.mu_off;
  const float* sg = P.sigma + u.mu_off;
  float* st = reinterpret_cast<float*>(P.keys + u.mu_off);   // s~ per candidate
  float2* cinv = reinterpret_cast<float2*>(P.corr) + u.mu_off;   // (corr_i, 1 / |k_i|)
  const uint16_t* kb = P.k + u.k_off;   // key i at kb + i * k_st
  const int64_t kst = P.g.k_st;
  const int h = P.pool_kernel / 2;

  float* v = reinterpret_cast<float*>(dyn);                         // [kMaxAllCand]
  uint16_t* applied = reinterpret_cast<uint16_t*>(v + kMaxAllCand);  // [kMaxAllCand]
  int32_t* adm = reinterpret_cast<int32_t*>(applied + kMaxAllCand);  // [kMaxAllBudget]
  float* adm_inv = reinterpret_cast<float*>(adm + kMaxAllBudget);    // [kMaxAllBudget]
  uint4* admk = reinterpret_cast<uint4*>(adm_inv + kMaxAllBudget);    // [kAdmStage][kAdmStride]

  // 1. pooled base score and its maximum
  float lmax = -INFINITY;
  for (int i = tid; i < C; i += kAllThreads) {
    const int a = max(i - h, 0), b = min(i + h, C - 1);
    float mh = -INFINITY, shh = -INFINITY;
    for (int j = a; j <= b; ++j) {
      mh = fmaxf(mh, __ldg(mu + j));
      shh = fmaxf(shh, __ldg(sg + j));
    }
    const float s = fmaf(lambda1, shh, mh);
    st[i] = s;
    lmax = fmaxf(lmax, s);
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
  if (lane == 0) sh.wmax[warp] = lmax;
  __syncthreads();
  float smax = sh.wmax[0];
  for (int w = 1; w < kAllWarps; ++w) smax = fmaxf(smax, sh.wmax[w]);
  smax = fmaxf(smax, P.norm_eps);
  // the owner of candidate i is the thread with own = i % kAllThreads: the lane whose row it is
  // in load_rows; it keeps the best of its own candidates
  const int own = warp * 32 + 8 * (lane & 3) + (lane >> 2);
  for (int base = warp * 32; base < C; base += kAllThreads) {
    uint4 x[4][4];
    load_rows(kb, kst, base, C, x);
    float ss[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float e0 = 0.f, e1 = 0.f;
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const uint32_t w4[4] = {x[r][s].x, x[r][s].y, x[r][s].z, x[r][s].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          e0 = fmaf(bf16_lo(w4[e]), bf16_lo(w4[e]), e0);
          e1 = fmaf(bf16_hi(w4[e]), bf16_hi(w4[e]), e1);
        }
      }
      ss[r] = e0 + e1;
      ss[r] += __shfl_xor_sync(0xffffffffu, ss[r], 1);
      ss[r] += __shfl_xor_sync(0xffffffffu, ss[r], 2);
    }
    const float n2 = own_row(ss);
    const int i = base + 8 * (lane & 3) + (lane >> 2);
    if (i < C) {
      const float s = __fdiv_rn(st[i], smax);
      st[i] = s;
      v[i] = s;                     // corr = 0: s~ + lambda2 * 0
      applied[i] = 0;
      cinv[i] = make_float2(0.f, n2 > 0.f ? __fdiv_rn(1.0f, sqrtf(n2)) : 0.f);
    }
  }
  __syncthreads();

  uint32_t my_key = 0, my_idx = 0xFFFFFFFFu;
  uint32_t my_cur = 0;   // and the best key of those that hold t applied admissions
  auto rescan = [&](int t) {
    my_cur = 0;
    my_key = 0;
    my_idx = 0xFFFFFFFFu;
    for (int i = own; i < C; i += kAllThreads) {
      const float x = v[i];
      if (__float_as_uint(x) == kAdmitted) continue;
      const uint32_t k = ord_key_all(x);
      if (applied[i] >= t) my_cur = max(my_cur, k);
      if (k > my_key || my_idx == 0xFFFFFFFFu) {
        my_key = k;
        my_idx = static_cast<uint32_t>(i);
      }
    }
  };
  rescan(0);

  // lambda2 > 0: every candidate brought up to date with the admission of key a, and the owners'
  // new bests. The dots of 32 candidates with that key are 16 mma.m16n8k16 per warp: candidate
  // rows as A fragments straight from the 16-byte loads (a dot does not depend on the order of
  // its elements, so chunk 4 s + t of a row and of the admitted key stand for the k-steps' lane t),
  // the key in every column of B. Bound by the keys' read from L2 (1 MB per admission at 4064
  // candidates): 64 admissions over 4064 candidates take 0.82 ms, against 2.88 with a thread per
  // candidate on the FMA pipe.
  auto refresh_all = [&](int a) {
    const uint4* src = a < kAdmStage ? admk + a * kAdmStride
                                     : reinterpret_cast<const uint4*>(kb + static_cast<int64_t>(adm[a]) * kst);
    uint4 y[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) y[s] = src[4 * s + (lane & 3)];
    const float inv_a = adm_inv[a];
    my_key = 0;
    my_idx = 0xFFFFFFFFu;
    for (int base = warp * 32; base < C; base += kAllThreads) {
      uint4 x[4][4];
      load_rows(kb, kst, base, C, x);
      const int i = base + 8 * (lane & 3) + (lane >> 2);
      const float2 ci = i < C ? cinv[i] : make_float2(0.f, 0.f);
      const float si = i < C ? st[i] : 0.f;
      float d[2][2][4];   // [m-tile][chain]
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int e = 0; e < 4; ++e) d[m][c][e] = 0.f;
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const uint4 r0 = x[2 * m][s], r1 = x[2 * m + 1][s];
          mma_bf16(d[m][0], r0.x, r1.x, r0.y, r1.y, y[s].x, y[s].y);
          mma_bf16(d[m][1], r0.z, r1.z, r0.w, r1.w, y[s].z, y[s].w);
        }
      // element 0 is row g of the m-tile, element 2 row g + 8; every column holds the same dot
      const float dots[4] = {d[0][0][0] + d[0][1][0], d[0][0][2] + d[0][1][2],
                             d[1][0][0] + d[1][1][0], d[1][0][2] + d[1][1][2]};
      const float dot = own_row(dots);
      if (i < C && __float_as_uint(v[i]) != kAdmitted) {
        const float cm = fmaxf(ci.x, dot * ci.y * inv_a);
        const float val = fmaf(lambda2, cm, si);
        cinv[i].x = cm;
        v[i] = val;
        applied[i] = static_cast<uint16_t>(a + 1);
        const uint32_t k = ord_key_all(val);
        if (k > my_key || my_idx == 0xFFFFFFFFu) {
          my_key = k;
          my_idx = static_cast<uint32_t>(i);
        }
      }
    }
  };
  // lambda2 <= 0: after a search whose best is stale, the owners whose stale best could still be
  // the admission bring it up to date and take their new best: those at or above the best current
  // value, or, while there is no current value, the best of each warp. A round is a chain of
  // latencies, so that few rows a round pay although they make more rounds. 64 admissions at
  // lambda2 = -0.9: over 4064 candidates 0.61 ms, over 19968 2.01 ms; with every owner's stale best
  // brought up to date in each round (512 to 1024 rows, 34 to 50 % fewer rounds) 1.73 and 3.27 ms.
  // A warp does this for its lanes together on the tensor cores: lane r's candidate row is row r
  // of the A operand of mma.m16n8k16 (two m-tiles, each skipped when no lane of it takes part),
  // the admitted keys a_lo .. t-1 form the B operand, 8 per pass, where a_lo is the smallest count
  // applied among these bests; a dot with an admission already applied leaves the running maximum
  // unchanged. The rows are loaded 16 bytes at a time, as in load_rows.
  auto refresh_bests = [&](int t) {
    const uint32_t cur = sh.cur_key;
    const bool want = my_idx != 0xFFFFFFFFu && applied[my_idx] < t &&
                      (cur != 0u ? my_key >= cur : my_idx == sh.widx[warp]);
    const uint32_t wants = __ballot_sync(0xffffffffu, want);
    if (wants) {
      const int a_lo = static_cast<int>(__reduce_min_sync(
          0xffffffffu, want ? static_cast<uint32_t>(applied[my_idx]) : static_cast<uint32_t>(t)));
      const float2 ci = want ? cinv[my_idx] : make_float2(0.f, 0.f);
      const int any = __shfl_sync(0xffffffffu, static_cast<int>(my_idx), __ffs(wants) - 1);
      const int row = want ? static_cast<int>(my_idx) : any;   // a valid stand-in
      float cm = ci.x;
      const int g = lane >> 2, tq = lane & 3;
#pragma unroll 1
      for (int m = 0; m < 2; ++m) {
        if (((wants >> (16 * m)) & 0xFFFFu) == 0u) continue;
        // rows g and g + 8 of the m-tile belong to lanes 16m + g and 16m + 8 + g
        const uint4* r0 = reinterpret_cast<const uint4*>(
            kb + static_cast<int64_t>(__shfl_sync(0xffffffffu, row, 16 * m + g)) * kst);
        const uint4* r1 = reinterpret_cast<const uint4*>(
            kb + static_cast<int64_t>(__shfl_sync(0xffffffffu, row, 16 * m + 8 + g)) * kst);
        const float i0 = __shfl_sync(0xffffffffu, ci.y, 16 * m + g);
        const float i1 = __shfl_sync(0xffffffffu, ci.y, 16 * m + 8 + g);
        uint4 x0[4], x1[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          x0[s] = __ldg(r0 + 4 * s + tq);
          x1[s] = __ldg(r1 + 4 * s + tq);
        }
        float c0 = -INFINITY, c1 = -INFINITY;
#pragma unroll 1
        for (int a0 = a_lo; a0 < t; a0 += 8) {
          // column g is admission a0 + g (past t: one that stands, its dots unused)
          const int an = a0 + g < t ? a0 + g : a0;
          const uint4* src = an < kAdmStage ? admk + an * kAdmStride
                                            : reinterpret_cast<const uint4*>(kb + static_cast<int64_t>(adm[an]) * kst);
          float d[2][4];
#pragma unroll
          for (int e = 0; e < 4; ++e) d[0][e] = d[1][e] = 0.f;
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            const uint4 y = src[4 * s + tq];
            mma_bf16(d[0], x0[s].x, x1[s].x, x0[s].y, x1[s].y, y.x, y.y);
            mma_bf16(d[1], x0[s].z, x1[s].z, x0[s].w, x1[s].w, y.z, y.w);
          }
          // elements e and 2 + e: rows g and g + 8, admission a0 + 2tq + e
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int a = a0 + 2 * tq + e;
            if (a < t) {
              const float ia = adm_inv[a];
              c0 = fmaxf(c0, (d[0][e] + d[1][e]) * i0 * ia);
              c1 = fmaxf(c1, (d[0][2 + e] + d[1][2 + e]) * i1 * ia);
            }
          }
        }
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) {
          c0 = fmaxf(c0, __shfl_xor_sync(0xffffffffu, c0, o));
          c1 = fmaxf(c1, __shfl_xor_sync(0xffffffffu, c1, o));
        }
        // lane 16m + 8hh + gg takes its row's from lane 4gg
        const float y0 = __shfl_sync(0xffffffffu, c0, 4 * (lane & 7));
        const float y1 = __shfl_sync(0xffffffffu, c1, 4 * (lane & 7));
        if ((lane >> 4) == m) cm = fmaxf(cm, (lane >> 3) & 1 ? y1 : y0);
      }
      if (want) {
        cinv[my_idx].x = cm;
        v[my_idx] = fmaf(lambda2, cm, st[my_idx]);
        applied[my_idx] = static_cast<uint16_t>(t);
        rescan(t);
      }
    }
  };

  int32_t* order = P.order ? P.order + u.unit * B : nullptr;
  float* margins = P.margins ? P.margins + u.unit * B : nullptr;
  int t = 0;
  bool again = false, all = false, second = false;   // second: the search is for the runner-up
  uint32_t best = 0;
#pragma unroll 1
  while (t < nsel) {
    if (again) {
      if (all)
        refresh_all(t - 1);
      else
        refresh_bests(t);
    }
    block_best(my_key, my_idx, my_cur, applied, t, sh);
    again = sh.stale;                 // a bound: bring what could beat it up to date, search again
    all = false;
    if (again) continue;
    if (!second) {
      // the full greedy's admission at step t
      const int bi = static_cast<int>(sh.best_idx);
      best = sh.best_key;
      if (own == (bi % kAllThreads)) {
        v[bi] = __uint_as_float(kAdmitted);
        rescan(t);
        adm[t] = bi;
        adm_inv[t] = cinv[bi].y;      // the admitted key's inverse norm
        if (order) order[t] = bi;
      }
      if (t < kAdmStage && tid < kHeadDim / 8)
        admk[t * kAdmStride + tid] =
            __ldg(reinterpret_cast<const uint4*>(kb + static_cast<int64_t>(bi) * kst) + tid);
      second = margins != nullptr;
      if (second) continue;           // against admissions 0 .. t-1 too
    } else {
      if (tid == 0)
        margins[t] = sh.best_idx == 0xFFFFFFFFu ? INFINITY : unord_key_all(best) - unord_key_all(sh.best_key);
      second = false;
    }
    ++t;
    my_cur = 0;
    // lambda2 > 0: values grow with corr, so every candidate is brought up to date
    if (!lazy && t < nsel) {
      again = all = true;
      __syncthreads();                // the admitted key and its norm are in place
    }
  }

  // 3. admitted positions ascending, then -1: entry a of the admission order goes to
  //    its rank among the admitted positions (all distinct); nsel <= kMaxAllBudget
  __syncthreads();
  int32_t* out = P.indices + u.unit * B;
  for (int a = tid; a < nsel; a += kAllThreads) {
    const int pos = adm[a];
    int rank = 0;
    for (int c = 0; c < nsel; ++c) rank += (adm[c] < pos);
    out[rank] = pos;
  }
  for (int r = nsel + tid; r < B; r += kAllThreads) out[r] = -1;
  if (order)
    for (int r = nsel + tid; r < B; r += kAllThreads) order[r] = -1;
  if (margins)
    for (int r = nsel + tid; r < B; r += kAllThreads) margins[r] = 0.f;
}

}  // namespace

cudaError_t launch_select_all(const kve_plan& plan, const SelectParams& p, cudaStream_t stream) {
  constexpr size_t smem = kMaxAllCand * (sizeof(float) + sizeof(uint16_t)) +
                          kMaxAllBudget * (sizeof(int32_t) + sizeof(float)) +
                          kAdmStage * kAdmStride * sizeof(uint4);
  cudaError_t e = cudaFuncSetAttribute(select_all_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  return launch_after_previous(select_all_kernel, dim3(static_cast<unsigned>(plan.geo.n_units)),
                               dim3(kAllThreads), smem, stream, p);
}

}  // namespace kve
