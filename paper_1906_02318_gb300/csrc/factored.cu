// Factorised read-out rollout: an ablation of Alg. 2's prediction step.
//
// The candidate's input is held over the horizon and the lifting is affine in
// the input monomials, z_0 = a(x_t) + sum_k p_k(xi) b_k(x_t) (Sec. IV-A), so
// every predicted state coordinate j is
//     z_t[j] = e_j K^t a + sum_k p_k(xi) e_j K^t b_k,
// exact in real arithmetic.  Only the coordinates the safety test reads (those
// with a finite bound, and the position when a track is set) are needed.  Once
// per session `powers_kernel` forms the rows C K^t (C = the n_x state rows) for
// t = 1..H; per tick every block folds them with the split of the lifting at
// x_t into the table V[t][r] = (e_r K^t a, e_r K^t b_1, ...), after which a
// candidate-step costs (1 + P) FMAs per read-out coordinate instead of the n^2
// of z <- K z, and the steps of a candidate no longer depend on each other: the
// warp tests 32 of them at once.  Rounding differs from the full rollout.  The per-step noise of
// Alg. 2 enters after K and does not factor, so noisy sessions cannot use this.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "internal.h"
#include "tick_kernel.cuh"

namespace mpmi {

// Most threads of a block.  One block per SM stages the track grid and builds V once
// for all of its warps (64 registers each); five blocks of 128 threads did both five
// times per SM.
constexpr int kFactBlock = 1024;

// Rows P_t = C K^t, t = 1..H: P_1 is the first NX rows of K and P_t = P_{t-1} K
// (each entry one FMA chain over i = 0..n-1).  One block of NX * N threads;
// out[((t - 1) NX + r) N + j].
template <int N, int NX>
__global__ void __launch_bounds__(256) powers_kernel(const float* K, int H, float* out) {
  __shared__ float sK[N][N];
  __shared__ float buf[2][NX][N];
  const int tid = threadIdx.x;
  for (int i = tid; i < N * N; i += blockDim.x) sK[i / N][i % N] = K[i];
  const int r = tid / N, j = tid % N;
  const bool act = tid < NX * N;
  if (act) {
    buf[0][r][j] = K[r * N + j];
    out[r * N + j] = K[r * N + j];
  }
  __syncthreads();
  for (int t = 2; t <= H; ++t) {
    const int src = t & 1, dst = src ^ 1;
    if (act) {
      float acc = 0.f;
      for (int i = 0; i < N; ++i) acc = __fmaf_rn(buf[src][r][i], sK[i][j], acc);
      buf[dst][r][j] = acc;
      out[((size_t)(t - 1) * NX + r) * N + j] = acc;
    }
    __syncthreads();
  }
}

// Steps t0 + 1 .. t0 + 32 of a candidate with input monomials p, one per lane: the lane
// of the first that violates the safety set, or 32.  RO read-outs (0: ro_n of them).
// Only the first violation counts, so open positions (settle_open) are settled in the
// order of their steps, and none after a step that is known to violate.
template <int KIND, int RO>
__device__ __forceinline__ int first_violation(const DevTrack& tr, const TrackView& tv, bool track,
                                               const float4* V, int ro_n, int H, int t0,
                                               const float* lo, const float* hi, float4 p) {
  constexpr int NX = BasisTraits<KIND>::NX, NP = BasisTraits<KIND>::NP;
  const int lane = threadIdx.x & 31, t = t0 + lane + 1;
  const int n = RO ? RO : ro_n;
  bool ok = true;
  float px = 0.f, py = 0.f;
  if (t <= H) {
    const float4* Vt = V + (t - 1) * n;
#pragma unroll
    for (int r = 0; r < (RO ? RO : NX); ++r) {
      if (RO || r < n) {
        const float4 w = Vt[r];
        float v = __fmaf_rn(p.x, w.y, w.x);
        if constexpr (NP > 1) v = __fmaf_rn(p.y, w.z, v);
        if constexpr (NP > 2) v = __fmaf_rn(p.z, w.w, v);
        ok = ok & (v > lo[r]) & (v < hi[r]);
        if (r == 0) px = v;
        if (r == 1) py = v;
      }
    }
  }
  unsigned int bad;
  if (BasisTraits<KIND>::TRACK && track) {
    const TrackCell cell = track_cell(tr, tv, px, py, ok && t <= H);
    ok = ok && (cell.ok || cell.open || t > H);
    bad = __ballot_sync(kFull, !ok);
    unsigned int todo = __ballot_sync(kFull, cell.open), taken;
    if (bad != 0u) todo &= (bad & (0u - bad)) - 1u;  // before the first violation
    while (todo != 0u) {
      const unsigned int got = settle_open<1>(tr, tv, px, py, cell, todo, &taken);
      if ((taken & ~got) != 0u) {  // an earlier violation than any left open
        bad |= taken & ~got;
        break;
      }
    }
  } else {
    bad = __ballot_sync(kFull, !ok);
  }
  return bad != 0u ? __ffs(bad) - 1 : 32;
}

// The lifting's feature codes of a basis.
struct FeatureCodes {
  uint32_t c[32];
};
constexpr FeatureCodes feature_codes(int kind, int n) {
  FeatureCodes f{};
  for (int j = 0; j < n; ++j) f.c[j] = feature_code(kind, j);
  return f;
}
template <int KIND>
__device__ const FeatureCodes g_codes = feature_codes(KIND, BasisTraits<KIND>::N);

// One tick in the factorised form.  Dynamic shared memory: [track grid (race
// car)] [V: H x ro_n float4, (a, b_1, b_2, b_3) coefficients per read-out].
// One block per SM.  A block draws up to a thread's candidate each, then its warps take
// the drawn candidates from a counter and test 32 steps of one at a time (the read-outs
// of different steps do not depend on each other; lane l: step t0 + l + 1), until the
// first violation.  Bound: issue, about 190 instructions per 32 steps, the track test
// most of them.  GB300, race car, N = 30001, H = 100: 19.6 us; 56.7 with 760 blocks of
// 128 threads that each staged the grid and built V, gave some warps two tiles and
// others one, and tested every listed segment of every step; 28.0 with equal tiles per
// warp; 25.6 with the lifting's features in code (a 32-way switch, or one after the
// other by a whole warp: 11k cycles) instead of one per lane from their codes (300).
template <int KIND>
__global__ void __launch_bounds__(kFactBlock) factored_kernel(const __grid_constant__ TickArgs a) {
  using B = BasisTraits<KIND>;
  constexpr int N = B::N, NX = B::NX, NU = B::NU, NP = B::NP;
  constexpr int ANG = (KIND == kBot) ? 0 : ((KIND == kCar) ? 2 : -1);
  extern __shared__ uint4 s_dyn[];
  __shared__ float4 s_f[N];  // split of the lifting at x_t: a_j, b_1j, b_2j, b_3j
  __shared__ float4 s_cand[kFactBlock];  // drawn candidates: monomials (up to 3), cost
  __shared__ int s_ttv[kFactBlock];
  __shared__ int s_next;
  __shared__ uint64_t s_bar;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // a launch over every slot that is sure to run stages the session's constants while
  // the kernel before it ends; the others look at that kernel's results first
  const bool sure = a.skip_if_safe == nullptr && a.n_list == nullptr;
  if (!sure) grid_dep_wait();
  if (fallback_not_needed(a)) return;
  const int n_eval = a.n_list ? *a.n_list : a.n_slots;
  const int H = a.horizon, ro_n = a.ro_n;
  // the blocks that a short device-side list leaves without a share return at once
  const int wpb = blockDim.x >> 5;
  const FactShare in(n_eval, (int)gridDim.x, wpb, (int)blockIdx.x);
  const int n_active = in.stride;
  if ((int)blockIdx.x >= n_active) {
    if (sure) grid_dep_wait();
    return;
  }

  // the track grid arrives by bulk copy while the table V is built
  const bool track_on = B::TRACK && a.safety.has_track;
  if (track_on) {
    if (tid == 0) bar_init(&s_bar);
    __syncthreads();
    if (tid == 0)
      stage_issue(&s_bar, s_dyn, nullptr, 0, 0, 0, a.safety.track.blob, a.safety.track.blob_bytes,
                  a.withhold_staging != 0);
  }
  TrackView tv{nullptr, nullptr, nullptr, nullptr};
  int track_words = 0;
  if constexpr (B::TRACK) {
    if (a.safety.has_track) {
      track_words = a.safety.track.blob_bytes >> 4;
      const char* base = reinterpret_cast<const char*>(s_dyn);
      tv.cells = reinterpret_cast<const uint32_t*>(base);
      tv.list = reinterpret_cast<const uint16_t*>(base + a.safety.track.off_list);
      tv.seg = reinterpret_cast<const float4*>(base + a.safety.track.off_seg);
      tv.inv = reinterpret_cast<const float*>(base + a.safety.track.off_inv);
    }
  }
  float4* V = reinterpret_cast<float4*>(s_dyn + track_words);
  // this thread's first row C K^t, in flight during the wait and the lifting
  constexpr int N4 = N % 4 == 0 ? N / 4 : 0;
  const auto row_of = [&](int e) {
    const int t = e / ro_n, r = e - t * ro_n;
    return a.ck + ((size_t)t * NX + a.ro_idx[r]) * N;
  };
  float4 p4[N4 ? N4 : 1];
  if (N4 && tid < H * ro_n) {
    const float4* row = reinterpret_cast<const float4*>(row_of(tid));
#pragma unroll
    for (int j = 0; j < N4; ++j) p4[j] = __ldg(row + j);
  }
  const uint32_t code = warp == 0 && lane < N ? g_codes<KIND>.c[lane] : 0u;
  if (sure) grid_dep_wait();

  float uh[NU];
#pragma unroll
  for (int j = 0; j < NU; ++j) uh[j] = __double2float_rn(a.u_h[j]);
  if (warp == 0) {
    // one feature per lane; lane i holds v[i] of the feature codes
    float v = 0.f;
    if (lane >= (int)kVX && lane < (int)kVX + NX) v = __double2float_rn(a.x_t[lane - kVX]);
    if (lane == (int)kVOne) v = 1.f;
    if constexpr (ANG >= 0) {
      float sn, cs;
      sincosf(__shfl_sync(kFull, v, kVX + ANG), &sn, &cs);
      if (lane == (int)kVSin) v = sn;
      if (lane == (int)kVCos) v = cs;
    }
    const float f0 = __shfl_sync(kFull, v, code & 15), f1 = __shfl_sync(kFull, v, code >> 4 & 15);
    const float f2 = __shfl_sync(kFull, v, code >> 8 & 15);
    const float b = __shfl_sync(kFull, v, code >> 12 & 15);
    const uint32_t m = code >> 16;
    if (lane < N)
      s_f[lane] = make_float4(__fmul_rn(__fmul_rn(f0, f1), f2), m == 0 ? b : 0.f,
                              m == 1 ? b : 0.f, m == 2 ? b : 0.f);
  }
  __syncthreads();
  // V[t][r] = (P_t row ro_idx[r]) . (a, b_1, b_2, b_3)
  for (int e = tid; e < H * ro_n; e += blockDim.x) {
    float v0 = 0.f, v1 = 0.f, v2 = 0.f, v3 = 0.f;
    const auto add = [&](int j, float pj) {
      const float4 f = s_f[j];
      v0 = __fmaf_rn(pj, f.x, v0);
      v1 = __fmaf_rn(pj, f.y, v1);
      v2 = __fmaf_rn(pj, f.z, v2);
      v3 = __fmaf_rn(pj, f.w, v3);
    };
    if constexpr (N4 > 0) {  // rows of whole float4s: all of a row's loads in flight
      if (e != tid) {
        const float4* row = reinterpret_cast<const float4*>(row_of(e));
#pragma unroll
        for (int j = 0; j < N4; ++j) p4[j] = __ldg(row + j);
      }
#pragma unroll
      for (int j = 0; j < N4; ++j) {
        add(4 * j, p4[j].x);
        add(4 * j + 1, p4[j].y);
        add(4 * j + 2, p4[j].z);
        add(4 * j + 3, p4[j].w);
      }
    } else {
      const float* row = row_of(e);
#pragma unroll
      for (int j = 0; j < N; ++j) add(j, __ldg(row + j));
    }
    V[e] = make_float4(v0, v1, v2, v3);
  }
  bool failed = false;
  if (track_on) {
    bool ok = bar_wait(&s_bar, 0);
    if (!ok) ok = bar_wait(&s_bar, 0);
    failed = __syncthreads_or(!ok) != 0;
  }

  // bounds of the read-out coordinates, in registers
  float lo[NX], hi[NX];
#pragma unroll
  for (int r = 0; r < NX; ++r) {
    lo[r] = r < ro_n ? a.safety.lo[a.ro_idx[r]] : -INFINITY;
    hi[r] = r < ro_n ? a.safety.hi[a.ro_idx[r]] : INFINITY;
  }

  unsigned long long best = ~0ull;
  unsigned int n_safe = 0, n_exec = 0;
  const int mine = failed ? 0 : in.count(n_eval);
  for (int base = 0; base < mine; base += (int)blockDim.x) {
    const int cnt = min((int)blockDim.x, mine - base);
    int slot = 0;
    float cost = 0.f;
    if (tid < cnt) {
      slot = in.slot(base + tid);
      if (a.slot_list) slot = a.slot_list[slot];
      float xi[NU], p[NP];
      candidate_value<NU>(a, slot, uh, xi);
#pragma unroll
      for (int j = 0; j < NU; ++j) {
        const float d = __fsub_rn(xi[j], uh[j]);
        cost = __fmaf_rn(d, d, cost);
      }
      monomials32<KIND>(xi, p);
      s_cand[tid] = make_float4(p[0], NP > 1 ? p[NP > 1 ? 1 : 0] : 0.f,
                                NP > 2 ? p[NP > 2 ? 2 : 0] : 0.f, cost);
    }
    if (tid == 0) s_next = wpb;  // the warps' first candidates are 0 .. wpb - 1
    __syncthreads();             // also: V is written
    int c = warp;
    while (c < cnt) {
      int next = 0;
      if (lane == 0) next = atomicAdd(&s_next, 1);
      const float4 p = s_cand[c];
      int ttv = H;
      for (int t0 = 0; t0 < H; t0 += 32) {
        // the usual numbers of read-outs in straight-line code: position and speed bound
        // (race car), two bounded coordinates (balance bot)
        constexpr int RO = KIND == kCar ? 3 : (NX >= 2 ? 2 : 0);
        int at;
        if (RO > 0 && ro_n == RO)
          at = first_violation<KIND, RO>(a.safety.track, tv, track_on, V, RO, H, t0, lo, hi, p);
        else
          at = first_violation<KIND, 0>(a.safety.track, tv, track_on, V, ro_n, H, t0, lo, hi, p);
        if (at < 32) {
          ttv = t0 + at;
          break;
        }
      }
      if (lane == 0) s_ttv[c] = ttv;
      c = __shfl_sync(kFull, next, 0);
    }
    __syncthreads();
    if (tid < cnt) {
      const int ttv = s_ttv[tid];
      const unsigned long long key = ((unsigned long long)(H - ttv) << 55) |
                                     ((unsigned long long)__float_as_uint(cost) << 23) |
                                     (unsigned long long)slot;
      best = key < best ? key : best;
      n_exec += (unsigned int)min(ttv + 1, H);
      n_safe += ttv == H;
      if (a.ttv_out) a.ttv_out[slot] = ttv;
      if (a.cost_out) a.cost_out[slot] = cost;
    }
  }
  grid_dep_release();
  session_epilogue<NU, TickArgs, kFactBlock / 32>(a, best, n_safe, n_exec, uh, failed,
                                                  (unsigned int)n_active);
}

template <int KIND>
static void (*factored_fn())(TickArgs) {
  return &factored_kernel<KIND>;
}

static void (*pick_factored(int kind))(TickArgs) {
  switch (kind) {
    case kBot: return factored_fn<kBot>();
    case kCar: return factored_fn<kCar>();
    case kLin11: return factored_fn<kLin11>();
    case kLin22: return factored_fn<kLin22>();
    case kLin41: return factored_fn<kLin41>();
  }
  return nullptr;
}

int compute_powers(int kind, const float* K, int H, float* out, cudaStream_t st) {
  switch (kind) {
    case kBot: powers_kernel<12, 4><<<1, 4 * 12, 0, st>>>(K, H, out); break;
    case kCar: powers_kernel<32, 6><<<1, 6 * 32, 0, st>>>(K, H, out); break;
    case kLin11: powers_kernel<2, 1><<<1, 32, 0, st>>>(K, H, out); break;
    case kLin22: powers_kernel<4, 2><<<1, 32, 0, st>>>(K, H, out); break;
    case kLin41: powers_kernel<5, 4><<<1, 32, 0, st>>>(K, H, out); break;
    default: return fail(MPMI_E_UNSUPPORTED, "powers: unknown basis");
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(MPMI_E_CUDA, std::string("powers kernel: ") + cudaGetErrorString(e));
  return MPMI_OK;
}

int launch_factored(mpmi_session* s, TickArgs& a, cudaStream_t st, int n_hint) {
  void (*const fn)(TickArgs) = pick_factored(s->model->kind);
  if (!fn) return fail(MPMI_E_UNSUPPORTED, "factored kernel not compiled for this basis");
  const size_t track = a.safety.has_track ? (size_t)a.safety.track.blob_bytes : 0;
  const size_t smem = track + (size_t)a.horizon * a.ro_n * sizeof(float4);
  const int n_work = (n_hint > 0 && n_hint < s->n_slots) ? n_hint : s->n_slots;
  const int sms = s->ctx->sm_count;
  int wpb, grid;
  fact_launch(n_work, sms, kFactBlock / 32, &wpb, &grid);
  if (s->fact_grid == 0 || s->fact_smem != smem) {
    if (smem > 0) {
      const size_t cap = kMaxTrackBytes + (size_t)MPMI_MAX_HORIZON * MPMI_MAX_NX * sizeof(float4);
      cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)cap);
      if (e != cudaSuccess) return fail(MPMI_E_CUDA, "cudaFuncSetAttribute (factored)");
    }
    int nb = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, 32 * wpb, smem);
    if (e != cudaSuccess || nb < 1)
      return fail(MPMI_E_UNSUPPORTED, "factored kernel cannot be resident");
    s->fact_grid = sms;  // the check is done
    s->fact_smem = smem;
  }
  const cudaError_t e = launch_dependent(fn, grid, 32 * wpb, smem, st, a);
  if (e != cudaSuccess)
    return fail(MPMI_E_CUDA, std::string("factored kernel launch: ") + cudaGetErrorString(e));
  return MPMI_OK;
}

}  // namespace mpmi
