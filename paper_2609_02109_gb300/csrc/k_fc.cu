// Fixed-context mode (arXiv 2609.02109, Sec. III-B): the observed GPU state s_t is
// held fixed during the search, so predictor g_i(lambda_i, s_t) depends on model i's
// option only.  The sum K_i local predictions are evaluated once (k_fc_local) into a
// per-option table of the utility term of Eq. 3,
//   u = omega_i f Q - alpha eta c_i - beta max(0, tau_i + delta - f)^2,
//   f = (fhat - f_min) / (f_max - f_min)   (per-variant normalisation),
// and a joint configuration's J is the sum of its options' terms (Eq. 3), -inf when a
// floor f_i >= tau_i or the VRAM bound of Eq. 4 fails.  The exhaustive search is then
// a table-lookup scan (k_fc_scan, ALU-bound); k_vram_count / k_vram_write build the
// VRAM-feasible space (Lambda without its VRAM-infeasible configurations) as an
// ascending index list.
#include <cfloat>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "mf_internal.cuh"

namespace mf {

// Device layout of mf_ctx::d_fc.
struct FcLayout {
  float2* tab;       // [sumK] (u, or -inf below the floor; VRAM of the option)
  float* fhat;       // [sumK]
  float* f;          // [sumK]
  float* u;          // [sumK]
  uint8_t* ok;       // [sumK]
};

// The inputs of mf_fc_set, in pinned host memory: every CTA of k_fc_local reads the few
// values of its option itself, early and used last, so no copy comes before the kernel.
struct FcInputs {
  float* obs;        // [4]
  int32_t* variant;  // [sumK]
  float* quality;    // [sumK]
  float* f_min;      // [sumK]
  float* f_max;      // [sumK]
  float* omega;      // [N]
  float* tau;        // [N]
  float* cost;       // [N]
  int32_t* prev;     // [N]
};

static size_t fc_bytes(int sumK, FcLayout* L, char* base) {
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = (o + bytes + 255) / 256 * 256;
    return base ? base + at : nullptr;
  };
  char* p;
  p = take(sizeof(float2) * sumK); if (L) L->tab = (float2*)p;
  p = take(sizeof(float) * sumK); if (L) L->fhat = (float*)p;
  p = take(sizeof(float) * sumK); if (L) L->f = (float*)p;
  p = take(sizeof(float) * sumK); if (L) L->u = (float*)p;
  p = take(sumK); if (L) L->ok = (uint8_t*)p;
  return o;
}

static size_t fc_input_bytes(int sumK, int N, FcInputs* L, char* base) {
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = (o + bytes + 15) / 16 * 16;
    return base ? base + at : nullptr;
  };
  char* p;
  p = take(sizeof(float) * 4); if (L) L->obs = (float*)p;
  p = take(sizeof(int32_t) * sumK); if (L) L->variant = (int32_t*)p;
  p = take(sizeof(float) * sumK); if (L) L->quality = (float*)p;
  p = take(sizeof(float) * sumK); if (L) L->f_min = (float*)p;
  p = take(sizeof(float) * sumK); if (L) L->f_max = (float*)p;
  p = take(sizeof(float) * N); if (L) L->omega = (float*)p;
  p = take(sizeof(float) * N); if (L) L->tau = (float*)p;
  p = take(sizeof(float) * N); if (L) L->cost = (float*)p;
  p = take(sizeof(int32_t) * N); if (L) L->prev = (int32_t*)p;
  return o;
}

struct FcConst {
  float alpha, beta, delta;
};

// ---------------------------------------------------------------------------
// Local predictions: one CTA per option row.  z = [x_i(o) | obs * s_A]; the hidden
// layers spread their units over the threads; the throughput head reduces over
// warp 0.  Thread 0 forms f, the floor flag and u.
//
// Bound by latency: the model's weights (the transposed copy) come into shared memory with
// one round of wide loads where they fit kFcStage, since a row read as it was needed cost
// an L2 round trip per few inputs (12->64->64->2, 144 rows: 7.1 us, staged 5).
// ---------------------------------------------------------------------------
constexpr size_t kFcStage = 96 * 1024;

template <bool ST>
__global__ void __launch_bounds__(256)
k_fc_local(const Params P, const FcLayout L, const FcInputs I, const FcConst C) {
  extern __shared__ __align__(16) float sw[];
  __shared__ float z[MF_MAX_D_LOCAL + 4];
  __shared__ float h1[MF_MAX_HIDDEN], h2[MF_MAX_HIDDEN];
  const int r = blockIdx.x, tid = threadIdx.x;
  const int N = P.n_models;
  int m = 0;
#pragma unroll
  for (int i = 1; i < MF_MAX_MODELS; ++i) m += i < N && r >= P.off[i] ? 1 : 0;
  const int dl = P.d_local, din = P.d_in, H1 = P.h1, H2 = P.h2;
  const float* w = P.wT + (size_t)m * P.per_model;
  if (ST) {
    const float4* src = reinterpret_cast<const float4*>(w);
    float4* dst = reinterpret_cast<float4*>(sw);
#pragma unroll 8
    for (int e = tid; e < (int)(P.per_model >> 2); e += 256) dst[e] = __ldg(src + e);
    w = sw;
  }
  float f_min = 0.f, f_max = 0.f, tau = 0.f, omega = 0.f, cost = 0.f, quality = 0.f, vram = 0.f;
  int variant = 0, prev = 0;
  if (tid == 0) {
    f_min = I.f_min[r]; f_max = I.f_max[r]; quality = I.quality[r]; variant = I.variant[r];
    tau = I.tau[m]; omega = I.omega[m]; cost = I.cost[m]; prev = I.prev[m];
    vram = P.dem[r].y;
  }
  if (tid < dl) z[tid] = P.x[(size_t)r * dl + tid];
  if (tid >= 32 && tid < 36) z[dl + tid - 32] = I.obs[tid - 32] * P.agg_scale[tid - 32];
  __syncthreads();
  const float* b1 = w + (size_t)H1 * din;
  for (int j = tid; j < H1; j += 256) {
    float s = b1[j];
#pragma unroll 4
    for (int k = 0; k < din; ++k) s = fmaf(w[(size_t)k * H1 + j], z[k], s);
    h1[j] = relu(s);
  }
  __syncthreads();
  const float* next = b1 + H1;
  const float* h = h1;
  int hl = H1;
  if (H2 > 0) {
    const float* b2 = next + (size_t)H2 * H1;
    for (int j = tid; j < H2; j += 256) {
      float s = b2[j];
#pragma unroll 16
      for (int k = 0; k < H1; ++k) s = fmaf(next[(size_t)k * H2 + j], h1[k], s);
      h2[j] = relu(s);
    }
    __syncthreads();
    next = b2 + H2;
    h = h2;
    hl = H2;
  }
  if (tid < 32) {
    const float* W3 = next;  // row 0: the throughput head
    float s = 0.f;
    for (int k = tid; k < hl; k += 32) s = fmaf(W3[k], h[k], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (tid == 0) {
      const float fhat = out_act(P, s + W3[2 * hl]);
      const float f = (fhat - f_min) / (f_max - f_min);
      const bool ok = f >= tau;
      const float eta = (prev >= 0 && variant != prev) ? 1.f : 0.f;
      const float margin = tau + C.delta - f;
      const float u = omega * f * quality - C.alpha * eta * cost - C.beta * (margin > 0.f ? margin * margin : 0.f);
      L.fhat[r] = fhat;
      L.f[r] = f;
      L.u[r] = u;
      L.ok[r] = ok ? 1 : 0;
      L.tab[r] = make_float2(ok ? u : -INFINITY, vram);
    }
  }
}

// ---------------------------------------------------------------------------
// Table-lookup scan.  J and the VRAM demand V of a configuration are summed in model order,
// but configurations are not looked at one by one: fp32 addition is monotone (a <= b gives
// fl(p + a) <= fl(p + b)), so
//   - for one setting of the leading N - 1 models, the last model's options within the cap
//     are a prefix of its options in VRAM order: a binary search counts them;
//   - for one setting of the leading N - 2 models, the sums of the extreme demands tell
//     whether all or none of the K_{N-2} K_{N-1} configurations fit, and where some do, the
//     boundary moves one way as model N - 2's demand grows: two pointers count them in
//     K_{N-2} + K_{N-1} steps;
//   - the sums with the largest terms bound every J below from above, and where that bound
//     does not reach the list's k-th entry no candidate is looked at; where it only equals it,
//     none of a setting that comes after that entry (so equal scores, which enter by index,
//     are not looked at over and over).
// The counts and the top-k are exactly those of the sums taken one by one.  This needs sums
// that do not turn to NaN (REG): no demand of -inf, and +inf only under a finite cap, where such
// options fit nowhere.  Other tables are scanned one candidate at a time.
//
// The bar starts high: J is a sum of per-model terms, so the best configurations sit where
// every model has one of its best options.  Every CTA first scores a corner of the space, the
// few best options of each model (m_i, 2^kFcCornerBits configurations), by J - lambda V
// for four weights lambda of the VRAM demand; the k-th best feasible score of the corner
// with the smallest lambda that has k of them bounds the k-th best of the range from below.
//
// The unit of work is one setting of the leading N - 2 models (short ranges: N - 1).  Units
// go round the threads of the grid, so that neighbours, which hold good scores together,
// land on different SMs.  A lane settles its unit by the bounds and counts; the units in
// which a score might beat the bar are then looked at by the whole warp, one after another.
//
// Running top-k: a warp queues the configurations that beat the bar and merges before the
// queue might overflow.  WL (k <= kFcWarpK): each warp keeps its own list and queue and
// merges with warp barriers only, the CTA's list taking the warps' lists at the end;
// otherwise one list and queue per CTA, whose warps meet for a merge when it fills up.
//
// Bound by latency (shared-memory chains of the counts; the prologue's ranking and corner).
// 24^6, VRAM binding: one launch of 23 us at k = 1, 27 at k = 32, 35 at k = 100; everything fits:
// 15.  The scan of every candidate took 12 launches of 75-125 us, each of which also filled its
// lists from nothing.
// ---------------------------------------------------------------------------
constexpr int kFcThreads = 512;
constexpr int kFcWarpK = 64, kFcWarps = kFcThreads / 32;
// A CTA's and a warp's queue.  (128 for a warp: with 256, warps that queue equal scores sorted
// twice as many before the list's bar stopped them: 3^14 of one score 194 us, 171 with 128.)
constexpr int kFcCtaQ = 4096, kFcWarpQ = 128;
constexpr int kFcEndQ = kFcWarps * kFcWarpK;          // the warps' lists, merged at the end (a power of two)
constexpr int kFcLambdas = 4, kFcCornerOpts = 64;     // corner sets, options of a model in one
constexpr int kFcCornerBits = 10;                     // configurations of a corner: 2^10
constexpr int kFcCornerRows = 1024;                   // option rows up to which the corners are ranked
constexpr size_t kFcScanSmem = 226 * 1024;            // dynamic shared memory a launch may take

struct FcScan {
  const float2* tab;
  int32_t corner;                     // score the corners first
  int32_t bits[MF_MAX_MODELS];        // m_i = 2^bits (where the model has as many usable options)
  // units: one setting of models 0 .. lead - 1 (lead = N - 2 or N - 1); the radix digits of
  // the grid's thread count in those models
  int32_t lead;
  uint32_t step[MF_MAX_MODELS];
};

// Shared-memory bytes of k_fc_scan<.., WL> after the table and the two VRAM orders.
__host__ __device__ inline size_t fc_scan_list_bytes(int k, bool wl) {
  const size_t e = sizeof(uint64_t) + sizeof(float);
  if (!wl) return e * (2 * (size_t)k + kFcCtaQ) + 16;
  return e * (2 * (size_t)k + kFcEndQ) + 16 + kFcWarps * (e * (2 * (size_t)k + kFcWarpQ) + 16);
}
__host__ __device__ inline size_t fc_scan_table_bytes(int sumK) {
  return (((size_t)sumK * sizeof(float2) + 15) & ~(size_t)15) + 2 * 256 * sizeof(float);
}

// The extremes of a model's usable options (their VRAM in the CTA's table is not NaN).
struct FcSpan {
  float jmax, jmin, vmin, vmax;
  int n;
};

template <int NMAX, bool WL, bool REG>
__global__ void __launch_bounds__(kFcThreads, 1)
k_fc_scan(const Params P, const FcScan S, const RangeArgs R) {
  // NMAX: a bound on N for the unrolled per-model loops
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ FcSpan s_span[MF_MAX_MODELS];
  stamp_start(R);
  const int N = P.n_models;
  const int sumK = pick(P.off, N - 1) + pick(P.K, N - 1);
  constexpr int QCAP = WL ? kFcEndQ : kFcCtaQ;
  float2* tab = reinterpret_cast<float2*>(sm);
  float* sv = reinterpret_cast<float*>(sm + (((size_t)sumK * sizeof(float2) + 15) & ~(size_t)15));  // last model, VRAM order
  float* sa = sv + 256;                                                                             // model N - 2
  unsigned char* q = reinterpret_cast<unsigned char*>(sa + 256);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // one list + queue block: li, ni [k], qi [qcap], ls, ns [k], qs [qcap], qn
  auto carve = [&](CtaTopK& t, int qcap) {
    t.li = reinterpret_cast<uint64_t*>(q); q += sizeof(uint64_t) * R.k;
    t.ni = reinterpret_cast<uint64_t*>(q); q += sizeof(uint64_t) * R.k;
    t.qi = reinterpret_cast<uint64_t*>(q); q += sizeof(uint64_t) * qcap;
    t.ls = reinterpret_cast<float*>(q); q += sizeof(float) * R.k;
    t.ns = reinterpret_cast<float*>(q); q += sizeof(float) * R.k;
    t.qs = reinterpret_cast<float*>(q); q += sizeof(float) * qcap;
    t.qn = reinterpret_cast<int*>(q); q += 16;
    t.k = R.k;
  };
  CtaTopK tk, wt;  // the CTA's list; this warp's (WL), else the CTA's again
  carve(tk, QCAP);
  if (WL) {  // the warps' blocks follow the CTA's, in warp order
    q += (size_t)warp * ((sizeof(uint64_t) + sizeof(float)) * (2 * (size_t)R.k + kFcWarpQ) + 16);
    carve(wt, kFcWarpQ);
    for (int e = lane; e < R.k; e += 32) { wt.ls[e] = -INFINITY; wt.li[e] = kEmptyIdx; }
    if (lane == 0) *wt.qn = 0;
  } else {
    wt = tk;
  }
  // an option below its floor (utility -inf, or NaN) carries VRAM NaN here, so one compare
  // against the cap decides feasibility, whatever the cap; REG: so does an option whose demand
  // no cap allows
  for (int e = tid; e < sumK; e += blockDim.x) {
    float2 v = S.tab[e];
    if (!(v.x > -INFINITY) || (REG && !(v.y < INFINITY))) v.y = NAN;
    tab[e] = v;
  }
  const size_t gl = (size_t)blockIdx.x * R.k;
  for (int e = tid; e < R.k; e += blockDim.x) {
    tk.ls[e] = R.first ? -INFINITY : R.lists_s[gl + e];
    tk.li[e] = R.first ? kEmptyIdx : R.lists_i[gl + e];
  }
  if (tid == 0) *tk.qn = 0;
  const int last = N - 1;
  const int off_last = pick(P.off, last), klast = pick(P.K, last);
  const int off_prev = last >= 1 ? pick(P.off, last - 1) : 0, kprev = last >= 1 ? pick(P.K, last - 1) : 1;
  const float cap = P.vram_cap;
  __syncthreads();
  // the bar: the CTA's k-th entry, or the corner's k-th best score (entries equal to it enter)
  float thr0_s = tk.ls[R.k - 1];
  uint64_t thr0_i = tk.li[R.k - 1];
  if (REG) {
    // per model: the extremes of its usable options; models N - 2 and N - 1: their demands in order
    for (int i = warp; i < N; i += kFcWarps) {
      const int off = pick(P.off, i), K = pick(P.K, i);
      FcSpan sp{-INFINITY, INFINITY, INFINITY, -INFINITY, 0};
      for (int o = lane; o < K; o += 32) {
        const float2 e = tab[off + o];
        if (e.y < INFINITY) {
          sp.jmax = fmaxf(sp.jmax, e.x);
          sp.jmin = fminf(sp.jmin, e.x);
          sp.vmin = fminf(sp.vmin, e.y);
          sp.vmax = fmaxf(sp.vmax, e.y);
          ++sp.n;
        }
      }
#pragma unroll
      for (int w = 16; w > 0; w >>= 1) {
        sp.jmax = fmaxf(sp.jmax, __shfl_xor_sync(0xffffffffu, sp.jmax, w));
        sp.jmin = fminf(sp.jmin, __shfl_xor_sync(0xffffffffu, sp.jmin, w));
        sp.vmin = fminf(sp.vmin, __shfl_xor_sync(0xffffffffu, sp.vmin, w));
        sp.vmax = fmaxf(sp.vmax, __shfl_xor_sync(0xffffffffu, sp.vmax, w));
        sp.n += __shfl_xor_sync(0xffffffffu, sp.n, w);
      }
      if (lane == 0) s_span[i] = sp;
    }
    __syncthreads();
    // Rankings, one warp per task, an option per lane (all-to-all by shuffles): tasks 0 and 1
    // order the demands of models N - 1 and N - 2, the others a model's usable options by
    // J - lambda V for one lambda, best first (in the queue's memory).
    uint16_t* order = reinterpret_cast<uint16_t*>(tk.qi);  // [lambda][model][kFcCornerOpts]
    float lam1 = 0.f;
    if (S.corner) {
      float sj = 0.f, sy = 0.f;
#pragma unroll
      for (int i = 0; i < NMAX; ++i)
        if (i < N) { sj += s_span[i].jmax - s_span[i].jmin; sy += s_span[i].vmax - s_span[i].vmin; }
      lam1 = sj / sy;
      if (!(lam1 > 0.f && lam1 < 1e30f)) lam1 = 0.f;
    }
    for (int task = warp; task < 2 + (S.corner ? kFcLambdas * N : 0); task += kFcWarps) {
      const int g = task < 2 ? 0 : (task - 2) / N;
      const int i = task == 0 ? last : task == 1 ? max(last - 1, 0) : task - 2 - g * N;
      const float lam = g == 0 ? 0.f : g == 1 ? 0.3f * lam1 : g == 2 ? lam1 : 3.f * lam1;
      const int off = pick(P.off, i), K = pick(P.K, i);
      // the value a task ranks by, highest first: -V, or J - lambda V (unusable options last,
      // also where lambda V overflows: a model's usable options take its first ranks, so every
      // slot of `order` that the corner reads is written)
      auto value = [&](int o) {
        const float2 e = o < K ? tab[off + o] : make_float2(-INFINITY, INFINITY);
        if (task < 2) return e.y < INFINITY ? -e.y : -INFINITY;
        return e.y < INFINITY ? fmaxf(__fsub_rn(e.x, __fmul_rn(lam, e.y)), -FLT_MAX) : -INFINITY;
      };
      for (int c0 = 0; c0 < K; c0 += 32) {
        const int o = c0 + lane;
        const float mine = value(o);
        int rank = 0;
        for (int d0 = 0; d0 < K; d0 += 32) {
          const float other = value(d0 + lane);
#pragma unroll
          for (int u = 0; u < 32; ++u) {
            const float v = __shfl_sync(0xffffffffu, other, u);
            rank += v > mine || (v == mine && d0 + u < o) ? 1 : 0;
          }
        }
        if (o < K) {
          const float y = tab[off + o].y;
          if (task == 0) sv[rank] = y;
          else if (task == 1) sa[rank] = y;
          else if (rank < kFcCornerOpts && y < INFINITY)
            order[(g * MF_MAX_MODELS + i) * kFcCornerOpts + rank] = (uint16_t)(off + o);
        }
      }
    }
    __syncthreads();
    if (S.corner) {
      const bool whole = R.base == 0 && R.len == P.total;
      constexpr int PER = (1 << kFcCornerBits) / kFcThreads;
      uint32_t key[kFcLambdas][PER];  // 0: not feasible, not in the range, no such option
#pragma unroll
      for (int u = 0; u < PER; ++u) {
        uint32_t c = tid + u * kFcThreads;
        bool in = true;
        float2 sum[kFcLambdas];
        uint64_t idx[kFcLambdas];
#pragma unroll
        for (int g = 0; g < kFcLambdas; ++g) { sum[g] = make_float2(0.f, 0.f); idx[g] = 0; }
#pragma unroll
        for (int i = 0; i < NMAX; ++i)
          if (i < N) {
            const uint32_t d = c & ((1u << S.bits[i]) - 1u);
            c >>= S.bits[i];
            in = in && d < (uint32_t)s_span[i].n;
            if (in) {
#pragma unroll
              for (int g = 0; g < kFcLambdas; ++g) {
                const int r = order[(g * MF_MAX_MODELS + i) * kFcCornerOpts + d];
                sum[g] = __fadd2_rn(sum[g], tab[r]);
                if (!whole) idx[g] += (uint64_t)(r - P.off[i]) * P.stride[i];
              }
            }
          }
        in = in && c == 0;  // (a corner of fewer configurations: the rest are repeats)
#pragma unroll
        for (int g = 0; g < kFcLambdas; ++g)
          key[g][u] = in && sum[g].y <= cap && sum[g].x == sum[g].x && (whole || idx[g] - R.base < R.len) ? order_key(sum[g].x) : 0u;
      }
      // the first lambda with k feasible configurations, and their k-th best score
      uint32_t mine[PER] = {};
      bool found = false;
#pragma unroll
      for (int g = 0; g < kFcLambdas; ++g) {
        if (found) continue;  // (uniform)
        int c = 0;
#pragma unroll
        for (int u = 0; u < PER; ++u) c += __syncthreads_count(key[g][u] > 0u);
        found = c >= R.k;
#pragma unroll
        for (int u = 0; u < PER; ++u) mine[u] = key[g][u];
      }
      if (found) {
        uint32_t v = 0u;
        for (int b = 31; b >= 0; --b) {
          const uint32_t t = v | (1u << b);
          int n = 0;
#pragma unroll
          for (int u = 0; u < PER; ++u) n += __syncthreads_count(mine[u] >= t);
          if (n >= R.k) v = t;
          if (n >= R.k && n <= R.k + (R.k >> 2)) break;  // (any bar that k scores reach holds)
        }
        const float b = from_key(v);
        if (b > thr0_s) { thr0_s = b; thr0_i = kEmptyIdx; }
      }
    }
  }
  const FcSpan sb = REG ? s_span[last] : FcSpan{}, spa = REG && last >= 1 ? s_span[last - 1] : FcSpan{};
  float thr_s = thr0_s;
  uint64_t thr_i = thr0_i;
  // Thread g of the grid takes units u0 + g, u0 + g + T, ..; the range's ends cut the first
  // unit and the last.  BIG (lead = N - 2): the unit's configurations run over models N - 2
  // and N - 1.
  const int lead = S.lead;
  const bool big = lead < last;
  const int na = big ? kprev : 1;
  const uint64_t unit = (uint64_t)klast * na;
  const uint64_t end = R.base + R.len, u0 = R.base / unit;
  const uint64_t nu = R.len == 0 ? 0 : (end - 1) / unit - u0 + 1;  // units of the range
  const uint64_t nthreads = (uint64_t)gridDim.x * blockDim.x;
  // this lane's unit, from u0 (where most are looked at they go round the warps, which look at
  // their units one after another)
  uint64_t my = !S.corner && nu < nthreads ? (uint64_t)lane * (nthreads / 32) + (uint64_t)warp * gridDim.x + blockIdx.x
                                           : (uint64_t)blockIdx.x * blockDim.x + tid;
  int row[NMAX];  // option rows of models 0 .. lead - 1
  {
    uint64_t v = my < nu ? u0 + my : 0;
#pragma unroll
    for (int i = NMAX - 1; i >= 0; --i)
      if (i < lead) {
        const uint32_t K = (uint32_t)P.K[i];
        uint32_t d;
        if (v <= 0xffffffffull) {
          const uint32_t q32 = (uint32_t)v / K;
          d = (uint32_t)v - q32 * K;
          v = q32;
        } else {
          const uint64_t q64 = v / K;
          d = (uint32_t)(v - q64 * K);
          v = q64;
        }
        row[i] = P.off[i] + (int)d;
      }
  }
  unsigned long long my_count = 0;
  // look-at state of the warp: the lanes whose units wait, the current unit's row of 32 of
  // model N - 2's options, those of the row still to do (when `open`), and the next row of
  // 32 of the last model's options
  unsigned waiting = 0u, todo = 0u;
  int at_a = 0, at_b = 0;
  bool open = false;
  float pJ2 = 0.f, pV2 = 0.f;  // this lane's unit: sums over models 0 .. lead - 1, in order
  bool count_there = false;    // it is counted when it is looked at
  auto merge_warp = [&]() {
    __syncwarp();
    if (*(volatile int*)wt.qn > 32) topk_merge_sorted(wt, lane, 32, [] __device__() { __syncwarp(); });
    else if (*(volatile int*)wt.qn > 0) topk_merge(wt, lane, 32, [] __device__() { __syncwarp(); });
  };
  auto raise_bar = [&]() {  // the list's k-th entry where it is the better bar (none while not full)
    const float ks = wt.ls[R.k - 1];
    const uint64_t ki = wt.li[R.k - 1];
    if (ki != kEmptyIdx && precedes(ks, ki, thr_s, thr_i)) { thr_s = ks; thr_i = ki; }
  };
  for (;;) {  // rounds; WL needs one only
    for (;;) {
      if (!waiting) {
        // ---- every lane settles its next unit ----
        if (!__any_sync(0xffffffffu, my < nu)) break;
        bool look = false;
        if (my < nu) {
          pJ2 = 0.f;
          pV2 = 0.f;
#pragma unroll
          for (int i = 0; i < NMAX; ++i)
            if (i < lead) { const float2 e = tab[row[i]]; pJ2 += e.x; pV2 += e.y; }
          const uint64_t t0 = (u0 + my) * unit;
          if (!REG || t0 < R.base || end - t0 < unit) {
            look = count_there = true;  // looked at one by one
          } else if (big) {
            const bool none = !((pV2 + spa.vmin) + sb.vmin <= cap);
            look = !none && (pJ2 + spa.jmax) + sb.jmax >= thr_s;
            count_there = false;
            if ((pV2 + spa.vmax) + sb.vmax <= cap) {
              my_count += (unsigned)(spa.n * sb.n);
            } else if (!none) {
              // each step moves one pointer: no lane waits in an inner loop for another
              int c = sb.n, a = 0;
              unsigned n = 0;
              while (a < spa.n && c > 0) {
                const bool fits = (pV2 + sa[a]) + sv[c - 1] <= cap;
                n += fits ? (unsigned)c : 0u;
                a += fits ? 1 : 0;
                c -= fits ? 0 : 1;
              }
              my_count += n;
            }
          } else {
            int lo = 0, hi = sb.n;
            while (lo < hi) {
              const int mid = (lo + hi) >> 1;
              if (pV2 + sv[mid] <= cap) lo = mid + 1; else hi = mid;
            }
            my_count += (unsigned)lo;
            look = lo > 0 && pJ2 + sb.jmax >= thr_s;
            count_there = false;
          }
        }
        waiting = __ballot_sync(0xffffffffu, look);
      }
      // ---- the warp looks at the waiting units, one after another ----
      bool full = false;
      while (waiting && !full) {
        const int src = __ffs(waiting) - 1;
        const float bJ = __shfl_sync(0xffffffffu, pJ2, src), bV = __shfl_sync(0xffffffffu, pV2, src);
        const bool cnt = __shfl_sync(0xffffffffu, count_there ? 1 : 0, src) != 0;
        const uint64_t t0 = (u0 + __shfl_sync(0xffffffffu, my, src)) * unit;
        const bool later = t0 > thr_i;  // (all of the unit comes after the bar's entry)
        for (; at_a < na; at_a += 32) {
          // this lane's option of model N - 2, and the options of the row worth a look
          float aJ = bJ, aV = bV;
          const bool have = at_a + lane < na;
          if (big && have) {
            const float2 e = tab[off_prev + at_a + lane];
            aJ += e.x;
            aV += e.y;
          }
          if (!open) {
            const float top = aJ + sb.jmax;
            todo = __ballot_sync(0xffffffffu, have && (!REG || cnt || (aV + sb.vmin <= cap && (later ? top > thr_s : top >= thr_s))));
            open = true;
          }
          for (; todo; todo &= todo - 1u) {
            const int ua = __ffs(todo) - 1;
            const float uJ = __shfl_sync(0xffffffffu, aJ, ua), uV = __shfl_sync(0xffffffffu, aV, ua);
            const uint64_t t1 = t0 + (uint64_t)(at_a + ua) * klast;
            for (; at_b < klast; at_b += 32) {
              // room for this row of 32 (in a CTA's queue: for a row of every warp)
              if (WL) {
                if (*(volatile int*)wt.qn > kFcWarpQ - 32) {
                  merge_warp();
                  raise_bar();
                }
              } else {
                // (one lane reads the queue's length, which other warps move, for all)
                full = __shfl_sync(0xffffffffu, *(volatile int*)wt.qn, 0) > QCAP - 32 * kFcWarps;
                if (full) break;
              }
              const int o = at_b + lane;
              const uint64_t idx = t1 + o;
              const bool in = o < klast && idx >= R.base && idx < end;
              const float2 e = in ? tab[off_last + o] : make_float2(0.f, 0.f);
              const float J = uJ + e.x;
              const bool feas = in && uV + e.y <= cap;  // NaN compares false
              my_count += cnt && feas ? 1u : 0u;
              const bool push = feas && J >= thr_s && precedes(J, idx, thr_s, thr_i);
              const unsigned m = __ballot_sync(0xffffffffu, push);
              if (m) {
                int pos = 0;
                if (lane == 0) pos = atomicAdd(wt.qn, __popc(m));
                pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(m & ((1u << lane) - 1u));
                if (push) { wt.qs[pos] = J; wt.qi[pos] = idx; }
                __syncwarp();
              }
            }
            if (full) break;  // (resumed at this row after the merge)
            at_b = 0;
          }
          if (full) break;
          open = false;
        }
        if (full) break;
        at_a = 0;
        waiting &= waiting - 1u;
      }
      if (full) break;
      // ---- the lane's next unit: the thread count added to the leading models' digits ----
      my += nthreads;
      uint32_t carry = 0;
#pragma unroll
      for (int i = NMAX - 1; i >= 0; --i)
        if (i < lead) {
          const int off = P.off[i];
          uint32_t d = (uint32_t)(row[i] - off) + S.step[i] + carry;
          carry = d >= (uint32_t)P.K[i];
          if (carry) d -= (uint32_t)P.K[i];
          row[i] = off + (int)d;
        }
    }
    if (WL) {
      merge_warp();
      break;
    }
    const bool more = __syncthreads_or(waiting != 0u);
    // a long queue (the first merges of a search) is sorted first
    if (*(volatile int*)tk.qn > 64) topk_merge_sorted(tk, tid, blockDim.x, [] __device__() { __syncthreads(); });
    else if (*(volatile int*)tk.qn > 0) topk_merge(tk, tid, blockDim.x, [] __device__() { __syncthreads(); });
    if (!more) break;
    raise_bar();
  }
  if (WL) {  // the warps' lists join the CTA's
    __syncthreads();
    for (int e = lane; e < R.k; e += 32)
      if (wt.li[e] != kEmptyIdx) {
        const int pos = atomicAdd(tk.qn, 1);
        tk.qs[pos] = wt.ls[e];
        tk.qi[pos] = wt.li[e];
      }
    __syncthreads();
    if (*(volatile int*)tk.qn > 0) {
      if (*(volatile int*)tk.qn > 64) topk_merge_sorted(tk, tid, blockDim.x, [] __device__() { __syncthreads(); });
      else topk_merge(tk, tid, blockDim.x, [] __device__() { __syncthreads(); });
    }
  }
  for (int e = tid; e < R.k; e += blockDim.x) {
    R.lists_s[gl + e] = tk.ls[e];
    R.lists_i[gl + e] = tk.li[e];
  }
  unsigned long long c = my_count;
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) c += __shfl_xor_sync(0xffffffffu, c, w);
  if (lane == 0 && c) atomicAdd(R.count, c);
}

// ---------------------------------------------------------------------------
// VRAM-feasible space as an ascending index list.  A thread takes one setting of the leading
// N - 1 models, whose demand it sums once for all options of the last model.  k_vram_count
// counts the feasible configurations of each CTA's contiguous segment of settings;
// k_vram_write (same segments) starts at the sum of the counts before its own and writes:
// per step of 512 settings a block-wide scan of the threads' counts gives each warp its
// place.  Where the last model has at most 32 options, each lane lists its setting's
// configurations in shared memory (16-bit offsets, in order) and the warp streams the list
// out in whole rows; above that, the warp writes one setting after another, a lane per option.
// Bound by issue, then by the writes for long lists.  48 M configurations, 15 M indices written: 78 us; one candidate a thread,
// N lookups each and two block barriers per 512 candidates took 773 us.
// ---------------------------------------------------------------------------
constexpr int kVramThreads = 512;

struct VramArgs {
  uint64_t lo, hi;                // the range
  uint64_t first, n, seg;         // settings: the range's first, their number, a CTA's share
  uint32_t step[MF_MAX_MODELS];   // mixed-radix digits of kVramThreads in models 0 .. N - 2
  unsigned long long* counts;     // [grid]
  uint64_t* out;
  uint64_t cap;
  unsigned long long* total;      // pinned host memory
};

// A thread's settings of the leading N - 1 models, from setting p on in steps of kVramThreads.
// NMAX: a bound on N.
template <int NMAX>
struct VramRows {
  int row[NMAX];
  __device__ __forceinline__ void start(const Params& P, uint64_t p) {
#pragma unroll
    for (int i = NMAX - 1; i >= 0; --i)
      if (i < P.n_models - 1) {
        const uint32_t K = (uint32_t)P.K[i];
        uint32_t d;
        if (p <= 0xffffffffull) {
          d = (uint32_t)p % K;
          p = (uint32_t)p / K;
        } else {
          d = (uint32_t)(p % K);
          p /= K;
        }
        row[i] = P.off[i] + (int)d;
      }
  }
  __device__ __forceinline__ float sum(const Params& P, const float* vr) const {
    float V = 0.f;
#pragma unroll
    for (int i = 0; i < NMAX; ++i)
      if (i < P.n_models - 1) V += vr[row[i]];
    return V;
  }
  __device__ __forceinline__ void advance(const Params& P, const uint32_t (&step)[MF_MAX_MODELS]) {
    uint32_t carry = 0;
#pragma unroll
    for (int i = NMAX - 1; i >= 0; --i)
      if (i < P.n_models - 1) {
        const int off = P.off[i];
        uint32_t d = (uint32_t)(row[i] - off) + step[i] + carry;
        carry = d >= (uint32_t)P.K[i];
        if (carry) d -= (uint32_t)P.K[i];
        row[i] = off + (int)d;
      }
  }
};

// Feasible options of the last model for a setting whose leading models need V: those of
// [o0, o1) (the whole row but at the range's ends).
__device__ __forceinline__ unsigned vram_row_count(const float* vl, float V, float cap, int o0, int o1) {
  unsigned c = 0;
#pragma unroll 8
  for (int o = o0; o < o1; ++o) c += V + vl[o] <= cap ? 1u : 0u;
  return c;
}

// Counts of the segments.  PAIR: a thread takes one setting of models 0 .. N - 3 at a time
// (segments cut them) and runs over the options of models N - 2 and N - 1, whose settings it
// decodes once; else one setting of models 0 .. N - 2.
template <int NMAX, bool PAIR>
__global__ void __launch_bounds__(kVramThreads, 2)
k_vram_count(const Params P, const VramArgs A) {
  extern __shared__ __align__(16) float vr[];  // [sumK] VRAM of each option
  __shared__ unsigned long long s_sum;
  const int N = P.n_models, K = pick(P.K, N - 1), KA = PAIR ? pick(P.K, N - 2) : 1;
  const int sumK = pick(P.off, N - 1) + K;
  const int tid = threadIdx.x;
  if (tid == 0) s_sum = 0ull;
  for (int e = tid; e < sumK; e += kVramThreads) vr[e] = P.dem[e].y;
  __syncthreads();
  const float* vl = vr + (sumK - K);
  const float cap = P.vram_cap;
  // this segment's first and last setting
  const uint64_t s0 = A.first + (uint64_t)blockIdx.x * A.seg;
  const uint64_t s1 = s0 + A.seg < A.first + A.n ? s0 + A.seg : A.first + A.n;
  unsigned long long mine = 0;
  auto count = [&](uint64_t s, float V) {
    const uint64_t i0 = s * (uint64_t)K;
    const int o0 = i0 < A.lo ? (int)(A.lo - i0) : 0, o1 = A.hi - i0 < (uint64_t)K ? (int)(A.hi - i0) : K;
    mine += vram_row_count(vl, V, cap, o0, o1);
  };
  if constexpr (PAIR) {
    const float* va = vl - KA;
    const uint64_t u1 = (s1 + KA - 1) / KA;
    for (uint64_t u = s0 / KA + tid; u < u1; u += kVramThreads) {
      int row[NMAX];
      uint64_t p = u;
#pragma unroll
      for (int i = NMAX - 1; i >= 0; --i)
        if (i < N - 2) {
          const uint32_t Ki = (uint32_t)P.K[i];
          uint32_t d;
          if (p <= 0xffffffffull) {
            d = (uint32_t)p % Ki;
            p = (uint32_t)p / Ki;
          } else {
            d = (uint32_t)(p % Ki);
            p /= Ki;
          }
          row[i] = P.off[i] + (int)d;
        }
      float V2 = 0.f;
#pragma unroll
      for (int i = 0; i < NMAX; ++i)
        if (i < N - 2) V2 += vr[row[i]];
      for (int a = 0; a < KA; ++a) {
        const uint64_t s = u * KA + a;
        if (s >= s0 && s < s1) count(s, V2 + va[a]);
      }
    }
  } else {
    VramRows<NMAX> rows;
    uint64_t s = s0 + tid;
    if (s < s1) rows.start(P, s);
    for (; s < s1; s += kVramThreads) {
      count(s, rows.sum(P, vr));
      rows.advance(P, A.step);
    }
  }
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, w);
  if ((tid & 31) == 0 && mine) atomicAdd(&s_sum, mine);
  __syncthreads();
  if (tid == 0) A.counts[blockIdx.x] = s_sum;
}

template <int NMAX>
__global__ void __launch_bounds__(kVramThreads, 2)
k_vram_write(const Params P, const VramArgs A) {
  extern __shared__ __align__(16) float vr[];  // [sumK] VRAM of each option
  __shared__ uint16_t s_list[kVramThreads / 32][32 * 32];
  __shared__ unsigned int s_warp[kVramThreads / 32];
  __shared__ unsigned long long s_base;
  const int N = P.n_models, K = pick(P.K, N - 1);
  const int sumK = pick(P.off, N - 1) + K;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) s_base = 0ull;
  for (int e = tid; e < sumK; e += kVramThreads) vr[e] = P.dem[e].y;
  __syncthreads();
  // where this CTA's indices start; the last CTA knows the total
  unsigned long long before_me = 0;
  for (int b = tid; b < (int)blockIdx.x; b += kVramThreads) before_me += A.counts[b];
#pragma unroll
  for (int w = 16; w > 0; w >>= 1) before_me += __shfl_xor_sync(0xffffffffu, before_me, w);
  if (lane == 0 && before_me) atomicAdd(&s_base, before_me);
  __syncthreads();
  if (blockIdx.x + 1 == gridDim.x && tid == 0) *A.total = s_base + A.counts[blockIdx.x];
  if (s_base >= A.cap) return;
  __syncthreads();
  const float* vl = vr + (sumK - K);
  const float cap = P.vram_cap;
  const uint64_t s0 = (uint64_t)blockIdx.x * A.seg;
  const uint64_t s1 = s0 + A.seg < A.n ? s0 + A.seg : A.n;
  VramRows<NMAX> rows;
  rows.start(P, A.first + (s0 + tid < s1 ? s0 + tid : 0));
  for (uint64_t b = s0; b < s1; b += kVramThreads) {
    const uint64_t p = b + tid;
    const bool in = p < s1;
    const float V = rows.sum(P, vr);
    const uint64_t i0 = (A.first + p) * (uint64_t)K;  // the setting's first configuration
    const int o0 = i0 < A.lo ? (int)(A.lo - i0) : 0, o1 = in ? (A.hi - i0 < (uint64_t)K ? (int)(A.hi - i0) : K) : 0;
    const unsigned c = vram_row_count(vl, V, cap, o0, o1);
    unsigned sum = c;  // the warp's total
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, w);
    if (lane == 0) s_warp[warp] = sum;
    __syncthreads();
    unsigned before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < kVramThreads / 32; ++w) {
      const unsigned v = s_warp[w];
      before += w < warp ? v : 0u;
      total += v;
    }
    uint64_t pos = s_base + before;
    const uint64_t w0 = (A.first + b + (uint64_t)warp * 32) * (uint64_t)K;  // the warp's first configuration
    if (sum > 0 && pos < A.cap) {
      if (K <= 32) {
        unsigned at = c;  // this lane's place in the warp's list: an exclusive scan
#pragma unroll
        for (int w = 1; w < 32; w <<= 1) {
          const unsigned left = __shfl_up_sync(0xffffffffu, at, w);
          at += lane >= w ? left : 0u;
        }
        at -= c;
        uint16_t* list = s_list[warp];
#pragma unroll 8
        for (int o = o0; o < o1; ++o)
          if (V + vl[o] <= cap) list[at++] = (uint16_t)(lane * K + o);
        __syncwarp();
        const unsigned room = A.cap - pos < sum ? (unsigned)(A.cap - pos) : sum;
        uint64_t* out = A.out + pos;
#pragma unroll 4
        for (unsigned e = lane; e < room; e += 32) out[e] = w0 + list[e];
        __syncwarp();
      } else {
        // (the settings that list anything; four rows of 32 options in flight)
        for (unsigned rest = __ballot_sync(0xffffffffu, c > 0); rest; rest &= rest - 1u) {
          const int u = __ffs(rest) - 1;
          const float Vu = __shfl_sync(0xffffffffu, V, u);
          const int a0 = __shfl_sync(0xffffffffu, o0, u), a1 = __shfl_sync(0xffffffffu, o1, u);
          for (int c0 = 0; c0 < K; c0 += 128) {
            unsigned m[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const int o = c0 + 32 * j + lane;
              m[j] = __ballot_sync(0xffffffffu, o >= a0 && o < a1 && Vu + vl[o] <= cap);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint64_t to = pos + __popc(m[j] & ((1u << lane) - 1u));
              if (((m[j] >> lane) & 1u) && to < A.cap) A.out[to] = w0 + (uint64_t)u * K + (c0 + 32 * j + lane);
              pos += __popc(m[j]);
            }
          }
        }
      }
    }
    __syncthreads();
    if (tid == 0) s_base += total;
    rows.advance(P, A.step);
  }
}

// ---------------------------------------------------------------------------
// The paper's GA (Sec. IV-C) on the fixed-context landscape, one CTA; fitness is the table
// sum of fc mode.  Operators and draws follow the GA of k_ga.cu with two more: crossover
// applied with probability crossover_p (draw kGaCrossDo, else the first parent is copied)
// and repair of an infeasible individual by rejection sampling from the uniform
// distribution over Lambda (draws kGaRepair, j = a * N + i, at most 256 / N attempts, the
// first feasible one kept).  The block has 1024 threads whatever the population: LPC lanes
// breed an individual (tournament entries and genes shared out over them), and lanes share
// the repairs (see repair).  LPC is the most that holds the population in one round (8 up to
// 128 individuals, 4 up to 256, 2 up to 512, else 1): the lanes cut a generation's chain, but
// rounds of them one after another cost more than a thread per individual (population 908, 11
// generations, with its table: 137 us with one thread each, 224 with eight).  Bound by the
// latency of a generation's chain: draws, fitness reads, the two tournaments, genes, their
// terms in model order, one block barrier.  Population 100, 30 generations, N = 5: 66 us without
// repairs, up to 93 with; one thread per individual, its draws one after another, took 180 us.
// ---------------------------------------------------------------------------
struct FcGaArgs {
  const float2* tab;
  int pop, gens, tournament, elitism, repair;
  uint32_t mut_thr, cross_thr;     // 24-bit thresholds
  uint64_t seed;
  int32_t* out_genome;
  float* out_fit;
};

// Shared memory of k_fc_ga: the table, then two generations' fitness and genes.
constexpr size_t fc_ga_bytes(int sumK, int pop, int n) {
  return sizeof(float2) * (size_t)sumK + 2 * (size_t)pop * (sizeof(float) + (size_t)n);
}

// (fitness, slot) as one word that orders by fitness, then by lower slot.
__device__ __forceinline__ unsigned long long fc_rank(float f, int slot) {
  return ((unsigned long long)order_key(f) << 32) | (0xFFFFFFFFu - (uint32_t)slot);
}
__device__ __forceinline__ int fc_slot(unsigned long long r) { return (int)(0xFFFFFFFFu - (uint32_t)r); }

// LPC: lanes per individual (a power of two); NG: genes a lane holds (N <= NG LPC).
template <int NG, int LPC>
__global__ void __launch_bounds__(1024)
k_fc_ga(const Params P, const FcGaArgs A) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ unsigned long long s_best[3];  // the fittest of generation g in s_best[g % 3]
  const int N = P.n_models, pop = A.pop;
  const int sumK = pick(P.off, N - 1) + pick(P.K, N - 1);
  float2* tab = reinterpret_cast<float2*>(sm);
  float* fit0 = reinterpret_cast<float*>(tab + sumK);
  float* fit1 = fit0 + pop;
  uint8_t* g0 = reinterpret_cast<uint8_t*>(fit1 + pop);
  uint8_t* g1 = g0 + (size_t)pop * N;
  const int c = threadIdx.x;
  for (int e = c; e < sumK; e += blockDim.x) tab[e] = A.tab[e];
  if (c < 3) s_best[c] = 0ull;
  __syncthreads();
  // Does any configuration meet the floors and the VRAM bound?  Exactly when every model
  // has an option with a finite term and the smallest such VRAM demands, summed in model
  // order as the fitness sums them, fit the cap (fp32 rounding is monotone, so no other
  // configuration sums to less).  If none does, every repair would draw all its attempts
  // in vain; its draws come from their own stream, so skipping it changes nothing else.
  __shared__ int s_any_feasible;
  if (c < 32) {
    float V = 0.f;
    bool every = true;
    for (int i = 0; i < N; ++i) {
      const int off = pick(P.off, i), K = pick(P.K, i);
      float m = INFINITY;
      for (int o = c; o < K; o += 32) {
        const float2 e = tab[off + o];
        if (e.x > -INFINITY && e.y < m) m = e.y;
      }
#pragma unroll
      for (int w = 16; w > 0; w >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, w));
      every = every && m < INFINITY;
      V += m;
    }
    if (c == 0) s_any_feasible = every && V <= P.vram_cap ? 1 : 0;
  }
  __syncthreads();
  const bool repairable = A.repair && s_any_feasible;
  const uint64_t sd = A.seed;
  const int attempts = 256 / N;
  const int lane = c & 31;
  // LPC lanes per individual: lane gl of a group holds genes gl, gl + LPC, ..
  const int gl = lane % LPC, group = c / LPC, g0l = lane - gl;  // (g0l: the group's first lane)
  int off[NG], K[NG];
#pragma unroll
  for (int q = 0; q < NG; ++q) {
    const int i = gl + LPC * q;
    off[q] = i < N ? pick(P.off, i) : 0;
    K[q] = i < N ? pick(P.K, i) : 1;
  }
  // a group's individual: its genes and its fitness, the terms summed in model order
  auto place = [&](int child, const int (&gene)[NG], uint8_t* genes, float* fit) {
    float2 e[NG];
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      e[q] = tab[off[q] + gene[q]];
      if (gl + LPC * q < N && child < pop) genes[(size_t)child * N + gl + LPC * q] = (uint8_t)gene[q];
    }
    float J = 0.f, V = 0.f;
#pragma unroll
    for (int q = 0; q < NG; ++q)
#pragma unroll
      for (int i = 0; i < LPC; ++i)
        if (i + LPC * q < N) {
          J += LPC == 1 ? e[q].x : __shfl_sync(0xffffffffu, e[q].x, g0l + i);
          V += LPC == 1 ? e[q].y : __shfl_sync(0xffffffffu, e[q].y, g0l + i);
        }
    const bool ok = V <= P.vram_cap && J > -INFINITY;
    if (gl == 0 && child < pop) fit[child] = ok ? J : -INFINITY;
    return ok ? J : -INFINITY;
  };
  // Attempts for the infeasible child `who` (done: none) of the lane's set of gs lanes (gmask):
  // they try the child's attempts in order, so many at a time; the lowest feasible attempt of
  // the first successful round is the sequential search's result.  The winning lane writes the
  // child's genes and fitness over the unrepaired ones.
  auto attempt = [&](uint32_t G, int who, bool done, int gs, unsigned gmask, uint8_t* genes, float* fit) {
    for (int a0 = 0; a0 < attempts && __any_sync(0xffffffffu, !done); a0 += gs) {
      const int a = a0 + lane % gs;
      float Jc = -INFINITY;
      uint32_t cand[(NG * LPC + 3) / 4] = {};
      if (!done && a < attempts) {  // the fitness' sums, with the draws kept in registers
        float Js = 0.f, Vs = 0.f;
#pragma unroll
        for (int i = 0; i < LPC * NG; ++i)
          if (i < N) {
            const int o = ga_unif(ga_rng(sd, G, (uint32_t)who, kGaRepair, (uint32_t)(a * N + i)), (uint32_t)P.K[i]);
            cand[i >> 2] |= (uint32_t)o << (8 * (i & 3));
            const float2 e = tab[P.off[i] + o];
            Js += e.x;
            Vs += e.y;
          }
        Jc = (Vs <= P.vram_cap && Js > -INFINITY) ? Js : -INFINITY;
      }
      const unsigned ok = __ballot_sync(0xffffffffu, Jc != -INFINITY) & gmask;
      if (!done && ok) {
        if (lane == __ffs(ok) - 1) {
#pragma unroll
          for (int i = 0; i < LPC * NG; ++i)  // (unrolled: an index known at run time would put `cand` in memory)
            if (i < N) genes[(size_t)who * N + i] = (uint8_t)(cand[i >> 2] >> (8 * (i & 3)));
          fit[who] = Jc;
        }
        done = true;
      }
    }
  };
  // Repair of the infeasible children (`bad`: this lane's group has one, child `child`): lanes
  // are shared out over them, 32, 16, 8, .. each.  With lanes to spare for each individual the
  // warp's lanes go to its own; with one lane each (half of a warp or more can need repair, and
  // warps past the population have nothing else to do) the block's lanes go to all of them, at
  // two barriers (600 individuals, N = 12, most of them infeasible, 30 generations: 530 us, by
  // the warp 751).
  auto repair = [&](uint32_t G, bool bad, int child, uint8_t* genes, float* fit) {
    const unsigned bal = __ballot_sync(0xffffffffu, bad && gl == 0);
    auto mask = [&](int gs, int mine) { return gs == 32 ? 0xffffffffu : ((1u << gs) - 1u) << (mine * gs); };
    if constexpr (LPC > 1) {
      if (!bal) return;
      __syncwarp();
      const int cnt = __popc(bal);
      int gs = 32;
      while (gs * cnt > 32) gs >>= 1;
      const int mine = lane / gs;  // this lane works for the mine-th of them
      unsigned rest = bal;
      for (int j = 0; j < mine; ++j) rest &= rest - 1u;
      const int who = __shfl_sync(0xffffffffu, child, rest ? __ffs(rest) - 1 : 0);
      attempt(G, who, rest == 0u, gs, mask(gs, mine), genes, fit);
      __syncwarp();
    } else {
      __shared__ uint16_t s_who[1024];
      __shared__ int s_bad[2];  // their number: of generation G in s_bad[G & 1]
      if (G == 0u) {
        if (c < 2) s_bad[c] = 0;
        __syncthreads();
      }
      int at = 0;
      if (lane == 0 && bal) at = atomicAdd(&s_bad[G & 1u], __popc(bal));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & ((1u << lane) - 1u));
      if (bad) s_who[at] = (uint16_t)child;
      __syncthreads();
      const int cnt = s_bad[G & 1u];
      if (c == 0) s_bad[(G + 1u) & 1u] = 0;  // (read before the last generation's end, used after this one's)
      if (cnt == 0) return;
      int gs = 32;
      while (gs * cnt > 1024) gs >>= 1;
      const int mine = c / gs;
      attempt(G, mine < cnt ? s_who[mine] : 0, mine >= cnt, gs, mask(gs, lane / gs), genes, fit);
      __syncthreads();
    }
  };
  // the fittest of the warp's individuals joins the population's (gl: one lane of a group)
  auto rank_in = [&](int child, const float* fit, unsigned long long* best) {
    unsigned long long r = gl == 0 && child < pop ? fc_rank(fit[child], child) : 0ull;
#pragma unroll
    for (int w = LPC; w < 32; w <<= 1) r = max(r, __shfl_xor_sync(0xffffffffu, r, w));
    if (lane == 0 && r) atomicMax(best, r);
  };
  // (LPC is chosen so that every individual has a group; a warp whose individuals all lie past
  // the population has nothing to draw)
  const int child = group;
  const bool breeds = (c - lane) / LPC < pop;
  {  // initial population: uniform over Lambda, repaired
    float J = 0.f;
    if (breeds) {
      int gene[NG] = {};
#pragma unroll
      for (int q = 0; q < NG; ++q)
        if (gl + LPC * q < N) gene[q] = ga_unif(ga_rng(sd, 0, (uint32_t)child, kGaInit, (uint32_t)(gl + LPC * q)), (uint32_t)K[q]);
      J = place(child, gene, g0, fit0);
    }
    if (repairable) repair(0u, child < pop && J == -INFINITY, child, g0, fit0);
    rank_in(child, fit0, &s_best[0]);
  }
  __syncthreads();
  uint8_t* gc = g0;
  uint8_t* gn = g1;
  float* fc_ = fit0;
  float* fn = fit1;
  for (int gen = 0; gen + 1 < A.gens; ++gen) {
    const uint32_t G = (uint32_t)gen + 1u;
    // (three words in turn: the one for the generation after this is cleared now, which no
    // warp reads or writes before the barrier)
    if (c == 0) s_best[(gen + 2) % 3] = 0ull;
    float J = 0.f;
    const bool elite = A.elitism && child == 0;  // slot 0 keeps the fittest (lowest slot among equals)
    if (breeds) {
      const uint32_t cu = (uint32_t)child;
      // the draws that do not depend on fitness
      bool take_b[NG] = {}, mutate[NG] = {};
      int mval[NG] = {};
      const bool cross = (uint32_t)(ga_rng(sd, G, cu, kGaCrossDo, 0u) >> 40) < A.cross_thr;
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        const uint32_t i = (uint32_t)(gl + LPC * q);
        if (i >= (uint32_t)N) continue;
        take_b[q] = cross && (ga_rng(sd, G, cu, kGaCross, i) >> 63);
        mutate[q] = (uint32_t)(ga_rng(sd, G, cu, kGaMut, i) >> 40) < A.mut_thr;
        mval[q] = ga_unif(ga_rng(sd, G, cu, kGaMutVal, i), (uint32_t)K[q]);
      }
      // the two tournaments
      int parent[2];
      if constexpr (LPC == 1) {
        // (nothing to exchange: a comparison of floats an entry takes a third less to issue than
        // the ranks; 1024 individuals, 256 entries, 30 generations: 3.14 ms, with ranks 4.70)
        for (int w = 0; w < 2; ++w) {
          float best = -INFINITY;
          int slot = 0x7fffffff;
          for (int t = 0; t < A.tournament; ++t) {
            const int s2 = ga_unif(ga_rng(sd, G, cu, w ? kGaTourB : kGaTourA, (uint32_t)t), (uint32_t)pop);
            const float f = fc_[s2];
            if (f > best || (f == best && s2 < slot)) { best = f; slot = s2; }
          }
          parent[w] = slot;
        }
      } else {  // entries shared out over the group's lanes
        unsigned long long win[2] = {0ull, 0ull};
        for (int d = gl; d < 2 * A.tournament; d += LPC) {
          const int w = d < A.tournament ? 0 : 1;
          const int s2 = ga_unif(ga_rng(sd, G, cu, w ? kGaTourB : kGaTourA, (uint32_t)(d - w * A.tournament)), (uint32_t)pop);
          const unsigned long long r = fc_rank(fc_[s2], s2);
          if (w) win[1] = max(win[1], r); else win[0] = max(win[0], r);
        }
#pragma unroll
        for (int w = LPC / 2; w > 0; w >>= 1) {
          win[0] = max(win[0], __shfl_xor_sync(0xffffffffu, win[0], w));
          win[1] = max(win[1], __shfl_xor_sync(0xffffffffu, win[1], w));
        }
        parent[0] = fc_slot(win[0]);
        parent[1] = fc_slot(win[1]);
      }
      if (elite) parent[0] = parent[1] = fc_slot(s_best[gen % 3]);
      int gene[NG];
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        const int i = gl + LPC * q;
        gene[q] = i < N ? gc[(size_t)(take_b[q] ? parent[1] : parent[0]) * N + i] : 0;
        if (mutate[q] && !elite && i < N) gene[q] = mval[q];
      }
      J = place(child, gene, gn, fn);
    }
    if (repairable) repair(G, child < pop && !elite && J == -INFINITY, child, gn, fn);
    rank_in(child, fn, &s_best[(gen + 1) % 3]);
    __syncthreads();
    uint8_t* tg = gc; gc = gn; gn = tg;
    float* tf = fc_; fc_ = fn; fn = tf;
  }
  {
    const int e = fc_slot(s_best[(A.gens - 1) % 3]);
    if (c < N) A.out_genome[c] = gc[(size_t)e * N + c];
    if (c == 0) *A.out_fit = fc_[e];
  }
}

// Whether the corners are worth their ranking: where the range's share of their configurations
// can hold k.
static bool fc_corner(const mf_ctx* c, uint64_t len, int k) {
  return c->sumK <= kFcCornerRows && (double)len * (1 << kFcCornerBits) >= (double)k * (double)c->P.total;
}

// One CTA per SM, fewer where the range has fewer settings of the leading N - 1 models than
// they have threads (a short list of lists to merge), or, without a bar from the corners, four
// settings a warp, since it looks at most of them.
int fc_grid(const mf_ctx* c, uint64_t len, int k) {
  const uint64_t units = len / (uint64_t)c->P.K[c->P.n_models - 1] + 2;
  const uint64_t per = fc_corner(c, len, k) ? kFcThreads : 4 * kFcWarps;
  const uint64_t ctas = (units + per - 1) / per;
  return (int)(ctas < (uint64_t)c->num_sms ? ctas : (uint64_t)c->num_sms);
}

mf_status fc_search_chunk(mf_ctx* c, const RangeArgs& a, int grid, cudaStream_t s) {
  FcLayout L;
  fc_bytes(c->sumK, &L, (char*)c->d_fc);
  const Params& P = c->P;
  const int N = P.n_models;
  FcScan S{};
  S.tab = L.tab;
  const bool reg = !c->vram_minus_inf && (!c->vram_plus_inf || P.vram_cap < INFINITY);
  if (reg && fc_corner(c, a.len, a.k)) {
    // one bit of the corner for each model in turn, while it has options for it
    int left = kFcCornerBits;
    for (bool grew = true; grew && left > 0;) {
      grew = false;
      for (int i = 0; i < N && left > 0; ++i)
        if ((1 << S.bits[i]) < P.K[i] && (2 << S.bits[i]) <= kFcCornerOpts) {
          ++S.bits[i];
          --left;
          grew = true;
        }
    }
    S.corner = 1;
  }
  // units of N - 2 models' settings where every thread gets one, else of N - 1 models'
  const uint64_t threads = (uint64_t)grid * kFcThreads;
  const uint64_t bigunit = (uint64_t)P.K[N - 1] * (N >= 2 ? P.K[N - 2] : 1);
  S.lead = N >= 2 && a.len / bigunit >= threads ? N - 2 : N - 1;
  uint64_t v = threads;
  for (int i = S.lead - 1; i >= 0; --i) {
    S.step[i] = (uint32_t)(v % (uint64_t)P.K[i]);
    v /= (uint64_t)P.K[i];
  }
  const bool wl = a.k <= kFcWarpK;  // per-warp lists
  const size_t smem = fc_scan_table_bytes(c->sumK) + fc_scan_list_bytes(a.k, wl);
  if (smem > kFcScanSmem) {
    set_error("fixed-context search: top-k lists do not fit shared memory; use a smaller k");
    return MF_EUNSUPPORTED;
  }
  using ScanFn = void (*)(const Params, const FcScan, const RangeArgs);
  const bool n8 = P.n_models <= 8;
  ScanFn fn;
  if (reg)
    fn = wl ? (n8 ? k_fc_scan<8, true, true> : k_fc_scan<MF_MAX_MODELS, true, true>)
            : (n8 ? k_fc_scan<8, false, true> : k_fc_scan<MF_MAX_MODELS, false, true>);
  else
    fn = wl ? (n8 ? k_fc_scan<8, true, false> : k_fc_scan<MF_MAX_MODELS, true, false>)
            : (n8 ? k_fc_scan<8, false, false> : k_fc_scan<MF_MAX_MODELS, false, false>);
  // (the maximum, whatever this launch takes: another context's call may be in between)
  MF_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFcScanSmem));
  fn<<<grid, kFcThreads, smem, s>>>(P, S, a);
  MF_CUDA(cudaGetLastError());
  return MF_OK;
}

}  // namespace mf

using namespace mf;

static mf_status fc_einval(const std::string& m) {
  set_error(m);
  return MF_EINVAL;
}

mf_status mf_fc_set(mf_ctx* ctx, const mf_fc_params* p, void* stream) {
  set_error("");
  if (!ctx || !p) return fc_einval("NULL argument");
  if (!p->obs || !p->variant || !p->quality || !p->f_min || !p->f_max || !p->omega || !p->tau ||
      !p->reload_cost || !p->prev_variant)
    return fc_einval("mf_fc_params: every array is required");
  const int N = ctx->P.n_models, sumK = ctx->sumK;
  for (int r = 0; r < sumK; ++r) {
    if (!(p->f_max[r] > p->f_min[r])) return fc_einval("mf_fc_params: f_max must exceed f_min for every option");
    if (p->variant[r] < 0) return fc_einval("mf_fc_params: variants must be >= 0");
  }
  for (int i = 0; i < N; ++i)
    if (p->prev_variant[i] < -1) return fc_einval("mf_fc_params: prev_variant must be >= -1");
  if (!std::isfinite(p->alpha) || !std::isfinite(p->beta) || !std::isfinite(p->delta))
    return fc_einval("mf_fc_params: alpha, beta and delta must be finite");
  DeviceGuard guard(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  const size_t bytes = fc_bytes(sumK, nullptr, nullptr);
  if (!ctx->d_fc) MF_CUDA(cudaMalloc(&ctx->d_fc, bytes));
  FcLayout L;
  fc_bytes(sumK, &L, (char*)ctx->d_fc);
  // (every call of a context that uses the staging buffer waits for its work)
  mf_status st = ensure_host_stage(ctx, fc_input_bytes(sumK, N, nullptr, nullptr));
  if (st != MF_OK) return st;
  FcInputs I;
  fc_input_bytes(sumK, N, &I, (char*)ctx->h_stage);
  std::memcpy(I.obs, p->obs, sizeof(float) * 4);
  std::memcpy(I.variant, p->variant, sizeof(int32_t) * sumK);
  std::memcpy(I.quality, p->quality, sizeof(float) * sumK);
  std::memcpy(I.f_min, p->f_min, sizeof(float) * sumK);
  std::memcpy(I.f_max, p->f_max, sizeof(float) * sumK);
  std::memcpy(I.omega, p->omega, sizeof(float) * N);
  std::memcpy(I.tau, p->tau, sizeof(float) * N);
  std::memcpy(I.cost, p->reload_cost, sizeof(float) * N);
  std::memcpy(I.prev, p->prev_variant, sizeof(int32_t) * N);
  const FcConst C{p->alpha, p->beta, p->delta};
  const size_t wbytes = sizeof(float) * (size_t)ctx->P.per_model;
  if (wbytes <= kFcStage) {
    MF_CUDA(cudaFuncSetAttribute(k_fc_local<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFcStage));
    k_fc_local<true><<<sumK, 256, wbytes, s>>>(ctx->P, L, I, C);
  } else {
    k_fc_local<false><<<sumK, 256, 0, s>>>(ctx->P, L, I, C);
  }
  MF_CUDA(cudaGetLastError());
  MF_CUDA(cudaStreamSynchronize(s));
  ctx->fc_ready = 1;
  return MF_OK;
}

mf_status mf_fc_table(mf_ctx* ctx, float* d_fhat, float* d_f, float* d_u, uint8_t* d_ok, void* stream) {
  set_error("");
  if (!ctx) return fc_einval("NULL argument");
  if (!ctx->fc_ready) return fc_einval("mf_fc_set has not been called on this context");
  DeviceGuard guard(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  FcLayout L;
  fc_bytes(ctx->sumK, &L, (char*)ctx->d_fc);
  const size_t n = (size_t)ctx->sumK;
  if (d_fhat) MF_CUDA(cudaMemcpyAsync(d_fhat, L.fhat, sizeof(float) * n, cudaMemcpyDeviceToDevice, s));
  if (d_f) MF_CUDA(cudaMemcpyAsync(d_f, L.f, sizeof(float) * n, cudaMemcpyDeviceToDevice, s));
  if (d_u) MF_CUDA(cudaMemcpyAsync(d_u, L.u, sizeof(float) * n, cudaMemcpyDeviceToDevice, s));
  if (d_ok) MF_CUDA(cudaMemcpyAsync(d_ok, L.ok, n, cudaMemcpyDeviceToDevice, s));
  return MF_OK;
}

mf_status mf_vram_feasible(mf_ctx* ctx, uint64_t lo, uint64_t hi, uint64_t* d_out, uint64_t cap,
                           uint64_t* count, void* stream) {
  set_error("");
  if (!ctx || !count) return fc_einval("NULL argument");
  if (lo > hi || hi > ctx->P.total) return fc_einval("need lo <= hi <= |Lambda|");
  if (cap > 0 && !d_out) return fc_einval("d_out is NULL");
  DeviceGuard guard(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  if (lo == hi) {
    *count = 0;
    return MF_OK;
  }
  const int N = ctx->P.n_models;
  const uint64_t K = (uint64_t)ctx->P.K[N - 1];
  VramArgs A{};
  A.lo = lo;
  A.hi = hi;
  A.first = lo / K;
  A.n = (hi - 1) / K - A.first + 1;
  // segments of whole steps, two rounds of the two CTAs an SM holds
  const uint64_t steps = (A.n + kVramThreads - 1) / kVramThreads;
  const uint64_t most = 4ull * ctx->num_sms;
  A.seg = (steps + most - 1) / most * kVramThreads;
  // (fewer steps than SMs: shorter ones, in warps, so that every SM takes part)
  const uint64_t sms = (uint64_t)ctx->num_sms;
  if (steps < sms) A.seg = ((A.n + sms - 1) / sms + 31) / 32 * 32;
  const unsigned grid = (unsigned)((A.n + A.seg - 1) / A.seg);
  mf_status st = ensure_scratch(ctx, sizeof(unsigned long long) * grid);
  if (st != MF_OK) return st;
  st = ensure_host_stage(ctx, sizeof(unsigned long long));
  if (st != MF_OK) return st;
  uint64_t v = kVramThreads;
  for (int i = N - 2; i >= 0; --i) {
    A.step[i] = (uint32_t)(v % (uint64_t)ctx->P.K[i]);
    v /= (uint64_t)ctx->P.K[i];
  }
  A.counts = (unsigned long long*)ctx->d_scratch;
  A.out = d_out;
  A.cap = cap;
  A.total = (unsigned long long*)ctx->h_stage;
  const size_t smem = sizeof(float) * (size_t)ctx->sumK;
  // Settings of N - 2 models where a segment holds one for a quarter of its threads: with 43 units
  // (24^5) the call takes 71 us by them and 57 by settings of N - 1, with one or two (255^2, 255^3)
  // 581 and 593 against 58 and 65; with 128 (40^3 x 8 x 16) 56 and 55; with 331 (48 M
  // configurations) 110 and 117, with 554 (24^6) 199 and 221.
  const bool pair = N >= 2 && A.seg >= (uint64_t)ctx->P.K[N - 2] * (kVramThreads / 4);
  const auto count_fn = pair ? (N <= 8 ? k_vram_count<8, true> : k_vram_count<MF_MAX_MODELS, true>)
                             : (N <= 8 ? k_vram_count<8, false> : k_vram_count<MF_MAX_MODELS, false>);
  count_fn<<<grid, kVramThreads, smem, s>>>(ctx->P, A);
  MF_CUDA(cudaGetLastError());
  (N <= 8 ? k_vram_write<8> : k_vram_write<MF_MAX_MODELS>)<<<grid, kVramThreads, smem, s>>>(ctx->P, A);
  MF_CUDA(cudaGetLastError());
  MF_CUDA(cudaStreamSynchronize(s));
  *count = *A.total;
  return MF_OK;
}

mf_status mf_fc_ga_run(mf_ctx* ctx, const mf_fc_ga_params* g, uint64_t seed, int32_t* best_genome,
                       float* best_fitness, void* stream) {
  set_error("");
  if (!ctx || !g || !best_genome || !best_fitness) return fc_einval("NULL argument");
  if (!ctx->fc_ready) return fc_einval("mf_fc_set has not been called on this context");
  if (g->pop < 2 || g->pop > 1024) return fc_einval("pop must be in 2..1024");
  if (g->gens < 1) return fc_einval("gens must be >= 1");
  if (g->tournament < 1 || g->tournament > 256) return fc_einval("tournament must be in 1..256");
  if (!(g->crossover_p >= 0.0 && g->crossover_p <= 1.0) || !(g->mutation_p >= 0.0 && g->mutation_p <= 1.0))
    return fc_einval("crossover_p and mutation_p must be in [0, 1]");
  if ((g->elitism != 0 && g->elitism != 1) || (g->repair != 0 && g->repair != 1))
    return fc_einval("elitism and repair must be 0 or 1");
  DeviceGuard guard(ctx->device);
  cudaStream_t s = (cudaStream_t)stream;
  const int N = ctx->P.n_models;
  FcLayout L;
  fc_bytes(ctx->sumK, &L, (char*)ctx->d_fc);
  // result, written by the kernel itself to pinned host memory: genome (16 ints), fitness
  mf_status st = ensure_host_stage(ctx, sizeof(int32_t) * 17);
  if (st != MF_OK) return st;
  int32_t* h = (int32_t*)ctx->h_stage;
  FcGaArgs A{};
  A.tab = L.tab;
  A.pop = g->pop;
  A.gens = g->gens;
  A.tournament = g->tournament;
  A.elitism = g->elitism;
  A.repair = g->repair;
  A.mut_thr = (uint32_t)std::floor(g->mutation_p * 16777216.0 + 0.5);
  A.cross_thr = (uint32_t)std::floor(g->crossover_p * 16777216.0 + 0.5);
  A.seed = seed;
  A.out_genome = h;
  A.out_fit = (float*)(h + 16);
  const size_t smem = fc_ga_bytes(ctx->sumK, g->pop, N);
  const bool n8 = N <= 8;
  const auto fn = g->pop <= 128   ? (n8 ? k_fc_ga<1, 8> : k_fc_ga<2, 8>)
                  : g->pop <= 256 ? (n8 ? k_fc_ga<2, 4> : k_fc_ga<4, 4>)
                  : g->pop <= 512 ? (n8 ? k_fc_ga<4, 2> : k_fc_ga<8, 2>)
                                  : (n8 ? k_fc_ga<8, 1> : k_fc_ga<16, 1>);
  // (the maximum, whatever this launch takes: another context's call may be in between)
  constexpr size_t kMost = fc_ga_bytes(MF_MAX_MODELS * MF_MAX_OPTIONS, 1024, MF_MAX_MODELS);
  MF_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMost));
  fn<<<1, 1024, smem, s>>>(ctx->P, A);
  MF_CUDA(cudaGetLastError());
  MF_CUDA(cudaStreamSynchronize(s));
  std::memcpy(best_genome, h, sizeof(int32_t) * N);
  std::memcpy(best_fitness, h + 16, sizeof(float));
  return MF_OK;
}
