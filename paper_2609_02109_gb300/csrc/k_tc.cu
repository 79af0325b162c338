// Tensor-core scorer, host side: operand images, tensor-memory and shared-memory layout,
// weight passes, launches, and the run-time instantiations of the kernel of k_tc.cuh.
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "k_tc.cuh"

namespace mf {

// ---------------------------------------------------------------------------
// Host side: operand images, layout, launches
// ---------------------------------------------------------------------------
namespace {

uint16_t f2bf(float f) {  // round to nearest even
  uint32_t u;
  std::memcpy(&u, &f, 4);
  if ((u & 0x7FFFFFFFu) > 0x7F800000u) return 0x7FC0;
  u += 0x7FFFu + ((u >> 16) & 1u);
  return (uint16_t)(u >> 16);
}

// fp16 bits of |f| < 65504 (nearest even); `rounded`: the value they stand for.  Without a
// branch, so that loops over it vectorise.
inline uint16_t f2half(float f, float& rounded) {
  uint32_t u, m, r;
  std::memcpy(&u, &f, 4);
  const uint32_t sign = u & 0x80000000u;
  u ^= sign;
  // from 2^-14 on: the mantissa rounded to 10 bits
  const uint32_t un = (u + 0xFFFu + ((u >> 13) & 1u)) & ~0x1FFFu;
  // below: multiples of 2^-24, which the sum with 1/2 rounds to
  float a;
  std::memcpy(&a, &u, 4);
  const float v = a + 0.5f, vs = v - 0.5f;
  std::memcpy(&m, &v, 4);
  std::memcpy(&r, &vs, 4);
  const uint32_t small = u < 0x38800000u ? 0xFFFFFFFFu : 0u;
  const uint32_t bits = (small & (m - 0x3F000000u)) | (~small & ((un - 0x38000000u) >> 13));
  const uint32_t val = ((small & r) | (~small & un)) | sign;
  std::memcpy(&rounded, &val, 4);
  return (uint16_t)((sign >> 16) | bits);
}

// Hi and lo parts of n <= 8 values.
inline void split_half(const float* v, int n, uint16_t* hi, uint16_t* lo) {
  for (int k = 0; k < n; ++k) {
    float r, rest;
    hi[k] = f2half(v[k], r);
    lo[k] = f2half(v[k] - r, rest);
  }
}

float bf2f(uint16_t b) {
  const uint32_t u = (uint32_t)b << 16;
  float f;
  std::memcpy(&f, &u, 4);
  return f;
}

// Byte offset of element (r, k) of a K-major no-swizzle UMMA operand with kdim columns:
// 8-row x 16-byte core matrices, K-adjacent cores 128 B apart, 8-row groups kdim*16 B apart.
size_t umma_off(int r, int k, int kdim) {
  return (size_t)(r >> 3) * (size_t)(kdim / 8) * 128u + (size_t)(k >> 3) * 128u + (size_t)(r & 7) * 16u +
         (size_t)(k & 7) * 2u;
}

// The same for 4-byte (tf32) elements: 4 per 16-byte core-matrix row.
size_t umma_off4(int r, int k, int kdim) {
  return (size_t)(r >> 3) * (size_t)(kdim / 4) * 128u + (size_t)(k >> 2) * 128u + (size_t)(r & 7) * 16u +
         (size_t)(k & 3) * 4u;
}

// v rounded to tf32 (nearest, ties away from zero), as an fp32 value.
float tf32_round(double v) {
  const float f = (float)v;
  uint32_t u;
  std::memcpy(&u, &f, 4);
  if ((u & 0x7F800000u) != 0x7F800000u) u = (u + 0x1000u) & 0xFFFFE000u;  // (inf and NaN as they are)
  float r;
  std::memcpy(&r, &u, 4);
  return r;
}

int round_up(int v, int a) { return (v + a - 1) / a * a; }

size_t topk_bytes_pipe(int kcap, int qcap) {
  return (sizeof(uint64_t) + sizeof(float)) * (2 * (size_t)kcap + qcap) + 16;
}

size_t image_bytes(const Params& P, int k1, int n3) {
  const int hl = P.h2 > 0 ? P.h2 : P.h1;
  const size_t per = (size_t)P.h1 * k1 * 2 + (size_t)P.h2 * (P.h1 + 16) * 2 + (size_t)n3 * hl * 2;
  return per * P.n_models;
}

constexpr uint32_t kSmemLimit = 227 * 1024 - 1024;  // static shared variables take the rest

// Shared-memory layout for a launch with per-pipeline lists of kcap entries.
void layout_smem(const Params& P, TcArgs& T, int kcap) {
  const int sumK = P.off[P.n_models - 1] + P.K[P.n_models - 1];
  uint32_t o = round_up((int)T.img_bytes, 1024);
  T.sm_xw = o; o += round_up(sumK * T.kw * 4, 16);
  T.sm_dem = o; o += sumK * 16;
  T.sm_rows = o; o += T.pipes * tc_row_bytes(T.ew);
  // the candidate queue: 512 entries (a merge every few tiles) where shared memory allows,
  // else one tile's 128 (a merge after every tile that queued a candidate)
  const uint32_t rest = o + 16 + 8 * (3 + 2 * kTcMaxPipes);
  T.qcap = 128;
  if (kcap > 0 && rest + T.pipes * topk_bytes_pipe(kcap, 512) <= kSmemLimit) T.qcap = 512;
  T.sm_topk = o; o += kcap > 0 ? (uint32_t)(T.pipes * topk_bytes_pipe(kcap, T.qcap)) : 0u;
  o = round_up((int)o, 16);
  T.sm_bar = o; o += 8 * (3 + 2 * kTcMaxPipes);
  T.sm_total = o;
  T.kcap = kcap;
}

constexpr size_t kPassImageBudget = 160 * 1024;      // weights staged per pass

// The 20 -> 128 -> 128 -> 2 shape (up to 8 models), with an instantiation of its own.
bool tc_wide(const TcArgs& T) { return T.kw == 16 && T.dle == 16 && T.h1 == 128 && T.h2 == 128 && T.n3 == 16; }

// Instantiations: the two benchmark shapes (d_L 8, 64-64 and d_L 16, 128-128, up to 8
// models) with all counts fixed at compile time, and a run-time fallback per A1 row width.
template <int MODE, bool MP, bool UT>
TcFn tc_kernel_mode(const TcArgs& T, int n_models) {
  if (T.tf != kXmBf16) return tc_kernel_exact(T.tf, MODE, MP, UT);
  // S1 = k1 / 16, S2 = h1 / 16 + 1 (the b2 step), S3 = hl / 16
  if (T.kw == 8 && T.dle == 8 && T.h1 == 64 && T.h2 == 64 && T.n3 == 16) {
    // The model loop unrolled with register digits, where a pass holds all models and their
    // digits fit seven bytes (one or two models have nothing to unroll): 435 cycles a model
    // and tile against 577 with the run-time loop (N = 6 and 7, 24^6 and 13^7), lists of 8 M candidates 541 against 681.
    if constexpr (!MP && !UT) {
      if (n_models >= 3 && n_models <= 7) return MODE == kTcRange ? tc_kernel_nm_range(n_models, T.sb != 0) : tc_kernel_nm_list(n_models);
    }
    return k_score_tc<MODE, 8, 4, 1, 5, 4, 16, MP, UT, 0, kXmBf16>;
  }
  if (tc_wide(T))
    return k_score_tc<MODE, 16, 8, 2, 9, 8, 16, MP, UT, 0, kXmBf16>;
  if (T.kw == 8) return k_score_tc<MODE, 8, -1, 0, 0, 0, 0, MP, UT, 0, kXmBf16>;
  return k_score_tc<MODE, 16, -1, 0, 0, 0, 0, MP, UT, 0, kXmBf16>;
}

template <bool UT>
TcFn tc_kernel_ut(int mode, const TcArgs& T, int n) {
  if (T.npasses > 1)
    return mode == kTcRange ? tc_kernel_mode<kTcRange, true, UT>(T, n) : tc_kernel_mode<kTcList, true, UT>(T, n);
  return mode == kTcRange ? tc_kernel_mode<kTcRange, false, UT>(T, n) : tc_kernel_mode<kTcList, false, UT>(T, n);
}

TcFn tc_kernel(int mode, const TcArgs& T, bool util, int n) {
  return util ? tc_kernel_ut<true>(mode, T, n) : tc_kernel_ut<false>(mode, T, n);
}
constexpr uint32_t kSmemFloor = 120 * 1024;          // keeps one CTA (one TMEM owner) per SM

}  // namespace

namespace {

// Candidates per launch when the models run in several passes (the partial records of
// one launch: 16 B each, 256 MiB).
constexpr uint64_t kPassSpan = 1ull << 24;

// Per-launch fields of pass p.
void set_pass(TcArgs& T, int p, float4* partial) {
  T.m0 = T.pass_m[p];
  T.m1 = T.pass_m[p + 1];
  T.pass_first = p == 0;
  T.pass_last = p + 1 == T.npasses;
  T.img_lo = T.off_b1[T.m0];
  T.img_copy = (p + 1 < T.npasses ? T.off_b1[T.m1] : T.img_total) - T.img_lo;
  T.partial = partial;
}

mf_status ensure_partial(mf_ctx* c, int npasses, uint64_t n, cudaStream_t s, float4** out) {
  *out = nullptr;
  if (npasses == 1) return MF_OK;
  const size_t need = sizeof(float4) * (size_t)(n < kPassSpan ? (n > 0 ? n : 1) : kPassSpan);
  if (need > c->partial_bytes) {
    MF_CUDA(cudaStreamSynchronize(s));
    cudaFree(c->d_partial);
    c->d_partial = nullptr;
    c->partial_bytes = 0;
    MF_CUDA(cudaMalloc(&c->d_partial, need));
    c->partial_bytes = need;
  }
  *out = static_cast<float4*>(c->d_partial);
  return MF_OK;
}

}  // namespace

bool tc_supported(const Params& P, std::string* why) {
  auto no = [&](const char* m) { if (why) *why = m; return false; };
  if (P.h1 % 32 || P.h1 > 256) return no("hidden1 must be a multiple of 32 up to 256");
  if (P.h2 % 32 || P.h2 > 256) return no("hidden2 must be 0 or a multiple of 32 up to 256");
  if (P.d_local > 24) return no("d_local must be <= 24");
  const int hmax = P.h1 > P.h2 ? P.h1 : P.h2;
  const int dle = P.d_local + (P.d_local & 1);
  const int k1 = round_up(dle + 8, 16);
  const int n3 = 2 * P.n_models <= 16 ? 16 : 32;
  const int col_a = hmax + hmax / 2 + 8;
  const int col_d3 = round_up(col_a + k1 / 2, 16);
  if (round_up(col_d3 + n3, 32) > 512) return no("tensor-memory footprint above 512 columns");
  if (image_bytes(P, k1, n3) / P.n_models > kPassImageBudget)
    return no("one model's bf16 weights exceed the shared-memory budget");
  return true;
}

bool tc_exact_supported(const Params& P) {
  return P.d_local == 8 && P.h1 == 64 && P.h2 == 64 && P.n_models <= 8;
}

// Passes of consecutive models whose images fit `budget` together.
static void set_passes(const Params& P, TcArgs& T, size_t budget) {
  const int N = P.n_models;
  auto end = [&](int j) { return j < N ? T.off_b1[j] : T.img_total; };  // of model j - 1's image
  T.npasses = 0;
  T.pass_m[0] = 0;
  T.img_bytes = 0;
  for (int i = 0; i < N;) {
    int j = i + 1;
    while (j < N && (size_t)(end(j + 1) - T.off_b1[i]) <= budget) ++j;
    T.pass_m[++T.npasses] = j;
    if (end(j) - T.off_b1[i] > T.img_bytes) T.img_bytes = end(j) - T.off_b1[i];
    i = j;
  }
}

// The shared-memory layout for lists of kcap entries: in the fp16 variant (three pipelines'
// lists), and where two epilogue warps share a lane quarter (their rows take more), with
// fewer models per pass if the lists would not fit next to a full pass's weights.
static bool layout_for(const Params& P, TcArgs& T, int kcap) {
  layout_smem(P, T, kcap);
  if (T.sm_total > kSmemLimit && (T.tf == kXmHalf || T.ew == 2)) {
    set_passes(P, T, 2 * kPassImageBudget / 3);
    set_pass(T, 0, nullptr);
    layout_smem(P, T, kcap);
  }
  return T.sm_total <= kSmemLimit;
}

bool tc_fits(const mf_ctx* c, int kcap) {
  TcArgs T = c->tc;
  return layout_for(c->P, T, kcap);
}

int tc_grid(const mf_ctx* c) { return c->num_sms * c->tc.pipes; }

namespace {

// The exact fp32 variant's layout and operand images (d_L 8, 12 -> 64 -> 64 -> 2): every
// operand as a tf32 hi part and the rest (a lo part, also tf32), so that hi.hi + hi.lo +
// lo.hi carries about 22 bits of each product.
mf_status tc_prepare_exact(mf_ctx* c, const TcHost& h) {
  const Params& P = c->P;
  TcArgs& T = c->tc;
  const int N = P.n_models, dl = P.d_local, h1 = P.h1, h2 = P.h2, hl = h2, din = P.d_in;
  T.tf = kXmTf32;
  T.ew = 1;
  T.dle = dl;
  T.k1 = 16;   // [x (8) | aggregate (3) | 1 | 0 0 0 0]
  T.kw = 16;   // words per option: x hi (8), x lo (8)
  T.h1 = h1;
  T.h2 = h2;
  T.hl = hl;
  T.n3 = 16;
  // TMEM columns of a pipeline: D (64 fp32) | H hi (64) | ones (8) | H lo (64) | A1 hi (16), A1 lo (16) | D3 (16)
  T.col_d = 0;
  T.col_h = h1;
  T.col_ones = 2 * h1;
  T.col_hlo = T.col_ones + 8;
  T.col_a = T.col_hlo + h1;
  T.col_d3 = round_up(T.col_a + 32, 16);
  T.pipe_stride = T.ps_d = T.ps_d3 = round_up(T.col_d3 + T.n3, 32);
  T.pipes = 512 / T.pipe_stride;
  if (T.pipes > 2) T.pipes = 2;
  // per model: B1 [h1 x 16], B2 [h2 x (h1 + 8)] (its last K-step holds b2 hi, lo against
  // the ones block), B3 [16 x hl], each as a hi image followed by a lo image
  const int k2 = h1 + 8;
  const size_t b1 = (size_t)h1 * T.k1 * 4, b2 = (size_t)h2 * k2 * 4, b3 = (size_t)T.n3 * hl * 4;
  T.img_lo1 = (uint32_t)b1;
  T.img_lo2 = (uint32_t)b2;
  T.img_lo3 = (uint32_t)b3;
  std::vector<unsigned char> img;
  auto put = [&](size_t base, size_t lo_off, int r, int k, int kdim, double v) {
    const float hi = tf32_round(v), lo = tf32_round(v - (double)hi);
    std::memcpy(img.data() + base + umma_off4(r, k, kdim), &hi, 4);
    std::memcpy(img.data() + base + lo_off + umma_off4(r, k, kdim), &lo, 4);
  };
  const double s3 = P.agg_scale[3];
  for (int i = 0; i < N; ++i) {
    const float* W1 = h.w + (size_t)i * P.per_model;
    const float* bb1 = W1 + (size_t)h1 * din;
    const float* W2 = bb1 + h1;
    const float* bb2 = W2 + (size_t)h2 * h1;
    const float* W3 = bb2 + h2;
    T.off_b1[i] = (uint32_t)img.size();
    img.resize(img.size() + 2 * b1, 0);
    for (int j = 0; j < h1; ++j) {
      for (int k = 0; k < dl + 3; ++k) put(T.off_b1[i], b1, j, k, T.k1, W1[(size_t)j * din + k]);
      // the constant-1 column: b1 plus the weight of the constant feature N * s_3
      put(T.off_b1[i], b1, j, dl + 3, T.k1, (double)bb1[j] + (double)W1[(size_t)j * din + dl + 3] * s3 * N);
    }
    T.off_b2[i] = (uint32_t)img.size();
    img.resize(img.size() + 2 * b2, 0);
    for (int j = 0; j < h2; ++j) {
      for (int k = 0; k < h1; ++k) put(T.off_b2[i], b2, j, k, k2, W2[(size_t)j * h1 + k]);
      // b2 as two tf32 values (hi, then the rest) in the hi image, against the ones (1, 1)
      const float bh = tf32_round(bb2[j]), bl = tf32_round((double)bb2[j] - (double)bh);
      std::memcpy(img.data() + T.off_b2[i] + umma_off4(j, h1, k2), &bh, 4);
      std::memcpy(img.data() + T.off_b2[i] + umma_off4(j, h1 + 1, k2), &bl, 4);
    }
    T.off_b3[i] = (uint32_t)img.size();
    img.resize(img.size() + 2 * b3, 0);
    T.img_model = (uint32_t)(2 * (b1 + b2 + b3));
    for (int k = 0; k < hl; ++k) {
      put(T.off_b3[i], b3, i, k, hl, W3[k]);
      put(T.off_b3[i], b3, T.n3 / 2 + i, k, hl, W3[hl + k]);
    }
  }
  img.resize(round_up((int)img.size(), 16), 0);
  T.img_total = (uint32_t)img.size();
  set_passes(P, T, kPassImageBudget);
  set_pass(T, 0, nullptr);
  if (T.npasses == 1) { T.pass_last = 1; }
  // option words: x hi (8), x lo (8)
  const int sumK = c->sumK;
  const float* x = h.x;
  std::vector<float> xw((size_t)sumK * T.kw, 0.f);
  for (int r = 0; r < sumK; ++r)
    for (int k = 0; k < dl; ++k) {
      const float v = x[(size_t)r * dl + k], hi = tf32_round(v);
      xw[(size_t)r * T.kw + k] = hi;
      xw[(size_t)r * T.kw + 8 + k] = tf32_round((double)v - (double)hi);
    }
  const size_t o_xw = round_up((int)img.size(), 256);
  const size_t total = o_xw + round_up((int)(xw.size() * 4), 256);
  MF_CUDA(cudaMalloc(&c->d_tc, total));
  c->tc_bytes = total;
  unsigned char* base = static_cast<unsigned char*>(c->d_tc);
  MF_CUDA(cudaMemcpy(base, img.data(), img.size(), cudaMemcpyHostToDevice));
  MF_CUDA(cudaMemcpy(base + o_xw, xw.data(), xw.size() * 4, cudaMemcpyHostToDevice));
  c->stats.h2d_bytes_create += img.size() + xw.size() * 4;
  T.img = base;
  T.xw = reinterpret_cast<const uint32_t*>(base + o_xw);
  for (int u = 0; u < 2; ++u) {
    MF_CUDA(cudaFuncSetAttribute(tc_kernel(kTcRange, T, u, P.n_models), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit));
    MF_CUDA(cudaFuncSetAttribute(tc_kernel(kTcList, T, u, P.n_models), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit));
  }
  layout_smem(P, T, 0);
  if (T.sm_total > kSmemLimit) {
    set_error("exact tensor-core path: tables and weights exceed shared memory");
    return MF_EUNSUPPORTED;
  }
  return MF_OK;
}

// The powers of two of the fp16 variant (all exact in fp32).
struct HalfScales {
  float cagg[3];                    // aggregate columns (shared by the models)
  std::vector<float> cx, t, u, v;   // [N][dl] features, [N][h1], [N][h2] units, [N][2] outputs
};

// 2^e with m 2^e in (2^(top - 1), 2^top]; 1 for m = 0.
float pow2_to(float m, int top) {
  if (m == 0.f) return 1.f;
  int e;
  const float f = std::frexp(m, &e);
  return std::ldexp(1.f, top - (f == 0.5f ? e - 1 : e));
}

// sum of |w_k| x_k, in eight partial sums (so that it vectorises)
float abs_dot(const float* w, const float* x, int n) {
  float s[8] = {};
  int k = 0;
  for (; k + 8 <= n; k += 8)
    for (int j = 0; j < 8; ++j) s[j] += std::fabs(w[k + j]) * x[k + j];
  for (; k < n; ++k) s[0] += std::fabs(w[k]) * x[k];
  return ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
}

// Scales from the largest value that each feature column, the aggregate and each unit can
// take over the option tables (|W| times the inputs' maxima, plus |b|): inputs to 2^4, the
// first hidden layer to 2^9, the second to 2^14, below fp16's 65504 whatever the candidate.
// Weights then are of order 1 to 2^6.  A part below 2^-3 loses lo bits (fp16's spacing ends
// at 2^-24): an absolute error of 2^-25, which is below what the split itself leaves as long
// as a unit's inputs and weights have products of order 1 (2^-22 of them) to sum.  So the
// rule: everything finite, and for every first-layer unit and option the sum of |products|
// (b1 and the least aggregate among them) is at least 1, 2^-9 of its largest; the second
// layer inherits errors of that size.  Option tables whose features differ by more, outliers
// for instance, run on tf32, whose exponent needs no scaling.
bool half_ranges(const Params& P, const TcHost& host, HalfScales& S) {
  const float *w = host.w, *x = host.x, *dem4 = host.dem4;
  const int N = P.n_models, dl = P.d_local, h1 = P.h1, h2 = P.h2, din = P.d_in;
  // (NaN fails every comparison; the bounds carry a margin for their own rounding)
  auto fits = [](float m) { return m == 0.f || (m > 1e-15f && m < 1e15f); };
  constexpr float kMargin = 1.0001f;
  float amax[3], amin[3];
  for (int q = 0; q < 3; ++q) {
    float hi = 0.f, lo = 0.f;
    bool positive = true;
    for (int i = 0; i < N; ++i) {
      float m = 0.f, l = INFINITY;
      for (int o = 0; o < P.K[i]; ++o) {
        const float d = dem4[(size_t)(P.off[i] + o) * 4 + q];
        if (!std::isfinite(d)) return false;
        m = std::fmax(m, std::fabs(d));
        l = std::fmin(l, d);
      }
      hi += m;
      lo += l;
      positive = positive && l >= 0.f;
    }
    amax[q] = hi * std::fabs(P.agg_scale[q]) * kMargin;
    amin[q] = positive ? lo * std::fabs(P.agg_scale[q]) : 0.f;
    if (!fits(amax[q])) return false;
    S.cagg[q] = pow2_to(amax[q], 4);
  }
  S.cx.resize((size_t)N * dl);
  S.t.resize((size_t)N * h1);
  S.u.resize((size_t)N * h2);
  S.v.resize((size_t)N * 2);
  float hb[MF_MAX_HIDDEN], in[MF_MAX_D_LOCAL + 4];
  std::vector<float> xs;  // |x| scaled
  for (int i = 0; i < N; ++i) {
    const float* W1 = w + (size_t)i * P.per_model;
    const float* b1 = W1 + (size_t)h1 * din;
    const float* W2 = b1 + h1;
    const float* b2 = W2 + (size_t)h2 * h1;
    const float* W3 = b2 + h2;
    const float* xi = x + (size_t)P.off[i] * dl;
    for (int k = 0; k < dl; ++k) {
      in[k] = 0.f;
      for (int o = 0; o < P.K[i]; ++o) {
        const float v = std::fabs(xi[(size_t)o * dl + k]);
        if (!std::isfinite(v)) return false;
        in[k] = std::fmax(in[k], v);
      }
      if (!fits(in[k])) return false;
      S.cx[(size_t)i * dl + k] = pow2_to(in[k], 4);
    }
    for (int q = 0; q < 3; ++q) in[dl + q] = amax[q];
    xs.clear();
    for (int j = 0; j < h1; ++j) {
      const float* wj = W1 + (size_t)j * din;
      const float bb = std::fabs(b1[j]) + std::fabs(wj[dl + 3] * P.agg_scale[3] * (float)N);
      const float m = (abs_dot(wj, in, dl + 3) + bb) * kMargin;
      if (!fits(m)) return false;
      hb[j] = m;
      const float t = S.t[(size_t)i * h1 + j] = pow2_to(m, 9);
      const float cst = std::fabs(b1[j] + wj[dl + 3] * P.agg_scale[3] * (float)N);
      const float least = (cst + abs_dot(wj + dl, amin, 3)) * t;
      if (m == 0.f || least >= 1.f) continue;
      if (xs.empty()) {
        xs.resize((size_t)P.K[i] * dl);
        for (size_t e = 0; e < xs.size(); ++e) xs[e] = std::fabs(xi[e]) * S.cx[(size_t)i * dl + e % dl];
      }
      float aw[MF_MAX_D_LOCAL];
      for (int k = 0; k < dl; ++k) aw[k] = wj[k] * t / S.cx[(size_t)i * dl + k];
      for (int o = 0; o < P.K[i]; ++o)
        if (!(least + abs_dot(aw, xs.data() + (size_t)o * dl, dl) >= 1.f)) return false;
    }
    float top[2] = {0.f, 0.f};
    for (int j = 0; j < h2; ++j) {
      const float m = (abs_dot(W2 + (size_t)j * h1, hb, h1) + std::fabs(b2[j])) * kMargin;
      if (!fits(m)) return false;
      const float u = S.u[(size_t)i * h2 + j] = pow2_to(m, 14);
      for (int r = 0; r < 2; ++r) {
        const float v = std::fabs(W3[(size_t)r * h2 + j]) / u;
        if (!std::isfinite(v)) return false;
        top[r] = std::fmax(top[r], v);
      }
    }
    for (int r = 0; r < 2; ++r) {
      if (!fits(top[r]) || !std::isfinite(W3[2 * h2 + r])) return false;
      S.v[(size_t)i * 2 + r] = pow2_to(top[r], 6);
    }
  }
  return true;
}

// The fp16 variant's layout and operand images; MF_EUNSUPPORTED (nothing changed) where
// half_ranges rules it out.
mf_status tc_prepare_half(mf_ctx* c, const TcHost& h) {
  const Params& P = c->P;
  TcArgs& T = c->tc;
  const int N = P.n_models, dl = P.d_local, h1 = P.h1, h2 = P.h2, hl = h2, din = P.d_in, sumK = c->sumK;
  const float *w = h.w, *x = h.x;
  HalfScales S;
  if (!half_ranges(P, h, S)) return MF_EUNSUPPORTED;
  T.tf = kXmHalf;
  T.dle = dl;
  T.k1 = 16;  // [x (8) | aggregate (3) | 1 | 0 0 0 0]
  T.kw = 8;   // words per option: x hi pairs (4), x lo pairs (4)
  T.h1 = h1;
  T.h2 = h2;
  T.hl = hl;
  T.n3 = 16;
  // TMEM columns: the pipelines' D (64 each), their D3 (16 each), then per pipeline
  // H hi (32) | ones (8) | H lo (32) | A1 hi (8), A1 lo (8): 504 of 512 for three pipelines
  T.pipes = tc_pipes(kXmHalf);
  T.ew = 1;
  T.ps_d = h1;
  T.ps_d3 = T.n3;
  T.col_d = 0;
  T.col_d3 = T.pipes * h1;
  T.col_h = T.col_d3 + T.pipes * T.n3;
  T.col_ones = T.col_h + h1 / 2;
  T.col_hlo = T.col_ones + 8;
  T.col_a = T.col_hlo + h1 / 2;
  T.pipe_stride = T.col_a + 16 - T.col_h;
  for (int q = 0; q < 3; ++q) T.cagg[q] = S.cagg[q];
  // per model: B1 [h1 x 16] hi, lo; B2 [h2 x (h1 + 16)] hi (its last K-step holds b2 hi, lo
  // against the ones block), [h2 x h1] lo; B3 [16 x hl] hi, lo
  const int k2 = h1 + 16;
  const size_t b1 = (size_t)h1 * T.k1 * 2, b2 = (size_t)h2 * k2 * 2, b2lo = (size_t)h2 * h1 * 2, b3 = (size_t)T.n3 * hl * 2;
  T.img_lo1 = (uint32_t)b1;
  T.img_lo2 = (uint32_t)b2;
  T.img_lo3 = (uint32_t)b3;
  T.img_model = (uint32_t)(2 * b1 + b2 + b2lo + 2 * b3);
  std::vector<unsigned char> img(round_up((int)(T.img_model * N), 16), 0);
  // n columns (a multiple of 8) of row r of an image with kdim columns, hi and lo image apart
  auto put_row = [&](size_t at, int kdim, size_t at_lo, int kdim_lo, int r, const float* v, int n) {
    unsigned char* ph = img.data() + at + umma_off(r, 0, kdim);
    unsigned char* pl = img.data() + at_lo + umma_off(r, 0, kdim_lo);
    for (int k = 0; k < n; k += 8, ph += 128, pl += 128) {
      uint16_t hi[8], lo[8];
      split_half(v + k, 8, hi, lo);
      std::memcpy(ph, hi, 16);
      std::memcpy(pl, lo, 16);
    }
  };
  const double s3 = P.agg_scale[3];
  float row[MF_MAX_HIDDEN], it[MF_MAX_HIDDEN], iu[MF_MAX_HIDDEN];  // a row; 1 / t, 1 / u
  for (int i = 0; i < N; ++i) {
    const float* W1 = w + (size_t)i * P.per_model;
    const float* bb1 = W1 + (size_t)h1 * din;
    const float* W2 = bb1 + h1;
    const float* bb2 = W2 + (size_t)h2 * h1;
    const float* W3 = bb2 + h2;
    const float *cx = &S.cx[(size_t)i * dl], *t = &S.t[(size_t)i * h1], *u = &S.u[(size_t)i * h2], *v = &S.v[(size_t)i * 2];
    for (int k = 0; k < h1; ++k) it[k] = 1.f / t[k];
    for (int k = 0; k < h2; ++k) iu[k] = 1.f / u[k];
    T.off_b1[i] = T.img_model * i;
    T.off_b2[i] = T.off_b1[i] + (uint32_t)(2 * b1);
    T.off_b3[i] = T.off_b2[i] + (uint32_t)(b2 + b2lo);
    for (int j = 0; j < h1; ++j) {
      const float* wj = W1 + (size_t)j * din;
      std::memset(row, 0, sizeof(float) * 16);
      for (int k = 0; k < dl; ++k) row[k] = wj[k] * t[j] / cx[k];
      for (int q = 0; q < 3; ++q) row[dl + q] = wj[dl + q] * t[j] / S.cagg[q];
      // the constant-1 column: b1 plus the weight of the constant feature N * s_3
      row[dl + 3] = (float)(((double)bb1[j] + (double)wj[dl + 3] * s3 * N) * t[j]);
      put_row(T.off_b1[i], T.k1, T.off_b1[i] + b1, T.k1, j, row, 16);
    }
    for (int j = 0; j < h2; ++j) {
      for (int k = 0; k < h1; ++k) row[k] = W2[(size_t)j * h1 + k] * u[j] * it[k];
      put_row(T.off_b2[i], k2, T.off_b2[i] + b2, h1, j, row, h1);
      uint16_t hi, lo;
      row[0] = bb2[j] * u[j];
      split_half(row, 1, &hi, &lo);
      std::memcpy(img.data() + T.off_b2[i] + umma_off(j, h1, k2), &hi, 2);
      std::memcpy(img.data() + T.off_b2[i] + umma_off(j, h1 + 1, k2), &lo, 2);
    }
    for (int r = 0; r < 2; ++r) {
      T.back[i][r] = 1.f / v[r];
      for (int k = 0; k < hl; ++k) row[k] = W3[(size_t)r * hl + k] * v[r] * iu[k];
      put_row(T.off_b3[i], hl, T.off_b3[i] + b3, hl, r * (T.n3 / 2) + i, row, hl);
    }
  }
  T.img_total = (uint32_t)img.size();
  set_passes(P, T, kPassImageBudget);
  set_pass(T, 0, nullptr);
  std::vector<uint32_t> xw((size_t)sumK * T.kw, 0u);
  for (int i = 0; i < N; ++i)
    for (int r = P.off[i]; r < P.off[i] + P.K[i]; ++r) {
      uint16_t hi[8], lo[8];  // (d_L 8)
      for (int k = 0; k < dl; ++k) row[k] = x[(size_t)r * dl + k] * S.cx[(size_t)i * dl + k];
      split_half(row, dl, hi, lo);
      std::memcpy(&xw[(size_t)r * T.kw], hi, 16);
      std::memcpy(&xw[(size_t)r * T.kw + 4], lo, 16);
    }
  layout_smem(P, T, 0);
  if (T.sm_total > kSmemLimit) return MF_EUNSUPPORTED;
  const size_t o_xw = round_up((int)img.size(), 256);
  const size_t total = o_xw + round_up((int)(xw.size() * 4), 256);
  MF_CUDA(cudaMalloc(&c->d_tc, total));
  c->tc_bytes = total;
  unsigned char* base = static_cast<unsigned char*>(c->d_tc);
  MF_CUDA(cudaMemcpy(base, img.data(), img.size(), cudaMemcpyHostToDevice));
  MF_CUDA(cudaMemcpy(base + o_xw, xw.data(), xw.size() * 4, cudaMemcpyHostToDevice));
  c->stats.h2d_bytes_create += img.size() + xw.size() * 4;
  T.img = base;
  T.xw = reinterpret_cast<const uint32_t*>(base + o_xw);
  for (int u = 0; u < 2; ++u) {
    MF_CUDA(cudaFuncSetAttribute(tc_kernel(kTcRange, T, u, N), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit));
    MF_CUDA(cudaFuncSetAttribute(tc_kernel(kTcList, T, u, N), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit));
  }
  return MF_OK;
}

}  // namespace

mf_status tc_prepare(mf_ctx* c, bool exact, const TcHost& h) {
  const Params& P = c->P;
  TcArgs& T = c->tc;
  std::memset(&T, 0, sizeof(T));
  if (exact) {
    const mf_status st = tc_prepare_half(c, h);
    if (st != MF_EUNSUPPORTED) return st;
    std::memset(&T, 0, sizeof(T));
    return tc_prepare_exact(c, h);
  }
  const int N = P.n_models, dl = P.d_local, h1 = P.h1, h2 = P.h2, hl = h2 > 0 ? h2 : h1;
  const int din = P.d_in;
  T.dle = dl + (dl & 1);
  T.k1 = round_up(T.dle + 8, 16);
  T.kw = T.k1 / 2;
  T.h1 = h1;
  T.h2 = h2;
  T.hl = hl;
  T.n3 = 2 * N <= 16 ? 16 : 32;
  const int hmax = h1 > h2 ? h1 : h2;
  T.col_d = 0;
  T.col_h = hmax;
  T.col_ones = hmax + hmax / 2;
  T.col_a = T.col_ones + 8;
  T.col_d3 = round_up(T.col_a + T.kw, 16);
  T.pipe_stride = T.ps_d = T.ps_d3 = round_up(T.col_d3 + T.n3, 32);
  T.pipes = 512 / T.pipe_stride;
  if (T.pipes > kTcMaxPipes) T.pipes = kTcMaxPipes;
  T.ew = tc_wide(T) ? 2 : 1;

  // B operand images (K-major): B1 [h1 x k1], B2 [h2 x (h1 + 16)], B3 [n3 x hl]
  const int k2 = h1 + 16, k3 = hl;
  const size_t b1_bytes = (size_t)h1 * T.k1 * 2, b2_bytes = (size_t)h2 * k2 * 2, b3_bytes = (size_t)T.n3 * k3 * 2;
  std::vector<unsigned char> img;
  const double s3 = P.agg_scale[3];
  auto put = [&](uint32_t base, int r, int k, int kdim, double v) {
    const uint16_t b = f2bf((float)v);
    std::memcpy(img.data() + base + umma_off(r, k, kdim), &b, 2);
  };
  // a bias as a bf16 pair (hi, lo) whose sum carries ~16 mantissa bits
  auto put_bias = [&](uint32_t base, int r, int k, int kdim, float v) {
    const uint16_t hi = f2bf(v);
    put(base, r, k, kdim, bf2f(hi));
    put(base, r, k + 1, kdim, (double)v - (double)bf2f(hi));
  };
  for (int i = 0; i < N; ++i) {
    const float* src = h.w + (size_t)i * P.per_model;
    const float* W1 = src;
    const float* b1 = W1 + (size_t)h1 * din;
    const float* W2 = b1 + h1;
    const float* b2 = W2 + (size_t)h2 * h1;
    const float* W3 = h2 > 0 ? b2 + h2 : W2;
    T.off_b1[i] = (uint32_t)img.size();
    img.resize(img.size() + b1_bytes, 0);
    for (int j = 0; j < h1; ++j) {
      for (int k = 0; k < dl; ++k) put(T.off_b1[i], j, k, T.k1, W1[(size_t)j * din + k]);
      // A1 carries the scaled aggregate (hi and lo parts), so these columns hold W1 as is;
      // the constant-1 column carries b1 plus the weight of the constant feature N * s_3
      for (int q = 0; q < 3; ++q) {
        put(T.off_b1[i], j, T.dle + q, T.k1, W1[(size_t)j * din + dl + q]);
        put(T.off_b1[i], j, T.dle + 4 + q, T.k1, W1[(size_t)j * din + dl + q]);
      }
      put(T.off_b1[i], j, T.dle + 3, T.k1, (double)b1[j] + (double)W1[(size_t)j * din + dl + 3] * s3 * N);
    }
    T.off_b2[i] = (uint32_t)img.size();
    img.resize(img.size() + b2_bytes, 0);
    for (int j = 0; j < h2; ++j) {
      for (int k = 0; k < h1; ++k) put(T.off_b2[i], j, k, k2, W2[(size_t)j * h1 + k]);
      put_bias(T.off_b2[i], j, h1, k2, b2[j]);
    }
    T.off_b3[i] = (uint32_t)img.size();
    img.resize(img.size() + b3_bytes, 0);
    T.img_model = (uint32_t)(b1_bytes + b2_bytes + b3_bytes);  // the kernel steps descriptors by it
    for (int k = 0; k < hl; ++k) {
      put(T.off_b3[i], i, k, k3, W3[k]);
      put(T.off_b3[i], T.n3 / 2 + i, k, k3, W3[hl + k]);
    }
  }
  img.resize(round_up((int)img.size(), 16), 0);
  T.img_total = (uint32_t)img.size();
  set_passes(P, T, kPassImageBudget);
  set_pass(T, 0, nullptr);  // single-pass defaults (a pass-0 image of all models)
  if (T.npasses == 1) { T.pass_last = 1; }

  // local-feature words
  const int sumK = c->sumK;
  const float* x = h.x;
  std::vector<uint32_t> xw((size_t)sumK * T.kw, 0u);
  for (int r = 0; r < sumK; ++r)
    for (int k = 0; k < dl; ++k)
      xw[(size_t)r * T.kw + k / 2] |= (uint32_t)f2bf(x[(size_t)r * dl + k]) << (16 * (k & 1));
  const size_t o_xw = round_up((int)img.size(), 256);
  const size_t total = o_xw + round_up((int)(xw.size() * 4), 256);
  MF_CUDA(cudaMalloc(&c->d_tc, total));
  c->tc_bytes = total;
  unsigned char* base = static_cast<unsigned char*>(c->d_tc);
  MF_CUDA(cudaMemcpy(base, img.data(), img.size(), cudaMemcpyHostToDevice));
  MF_CUDA(cudaMemcpy(base + o_xw, xw.data(), xw.size() * 4, cudaMemcpyHostToDevice));
  c->stats.h2d_bytes_create += img.size() + xw.size() * 4;
  T.img = base;
  T.xw = reinterpret_cast<const uint32_t*>(base + o_xw);
  for (int u = 0; u < 2; ++u) {
    MF_CUDA(cudaFuncSetAttribute(tc_kernel(kTcRange, T, u, P.n_models), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit));
    MF_CUDA(cudaFuncSetAttribute(tc_kernel(kTcList, T, u, P.n_models), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit));
  }
  layout_smem(P, T, 0);
  if (T.sm_total > kSmemLimit) {
    set_error("tensor-core path: tables and weights exceed shared memory");
    return MF_EUNSUPPORTED;
  }
  return MF_OK;
}


mf_status tc_search_chunk(mf_ctx* c, const RangeArgs& a, cudaStream_t s, int* nlaunch) {
  TcArgs T = c->tc;
  T.sb = a.tops != nullptr;
  if (!layout_for(c->P, T, a.k)) {
    set_error("tensor-core path: top-k lists do not fit shared memory; use a smaller k");
    return MF_EUNSUPPORTED;
  }
  if (T.npasses != c->tc.npasses || T.sb)  // (another kernel than the one prepared)
    MF_CUDA(cudaFuncSetAttribute(tc_kernel(kTcRange, T, c->P.objective == MF_OBJ_UTILITY, c->P.n_models),
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit));
  // digits of the per-tile index stride (grid x pipes x 128), modulo |Lambda|
  const uint64_t stride = ((uint64_t)c->num_sms * T.pipes * 128) % c->P.total;
  uint64_t v = stride;
  T.dstep = 0;
  T.dbias = 0;
  for (int i = c->P.n_models - 1; i >= 0; --i) {
    T.step[i] = (uint32_t)(v % (uint64_t)c->P.K[i]);
    v /= (uint64_t)c->P.K[i];
    if (c->P.n_models <= 7) {
      const int sh = 8 * (c->P.n_models - 1 - i);
      T.dstep |= (uint64_t)(T.step[i] + 256u - (uint32_t)c->P.K[i]) << sh;
      T.dbias |= (uint64_t)(256u - (uint32_t)c->P.K[i]) << sh;
    }
  }
  const uint32_t smem = T.sm_total > kSmemFloor ? T.sm_total : kSmemFloor;
  TcList L{};
  float4* partial = nullptr;
  mf_status st = ensure_partial(c, T.npasses, a.len, s, &partial);
  if (st != MF_OK) return st;
  // one launch per pass and span of candidates; the lists and the count belong to the
  // last pass only
  const uint64_t span = T.npasses == 1 ? (a.len > 0 ? a.len : 1) : kPassSpan;
  int launches = 0;
  RangeArgs r = a;
  for (uint64_t b = 0; b == 0 || b < a.len; b += span) {
    r.base = a.base + b;
    r.len = a.len - b < span ? a.len - b : span;
    r.first = a.first && b == 0;
    for (int p = 0; p < T.npasses; ++p) {
      set_pass(T, p, partial);
      tc_kernel(kTcRange, T, c->P.objective == MF_OBJ_UTILITY, c->P.n_models)<<<c->num_sms, T.pipes * tc_pipe_threads(T.ew), smem, s>>>(c->P, T, r, L);
      MF_CUDA(cudaGetLastError());
      ++launches;
    }
  }
  *nlaunch = launches;
  return MF_OK;
}

mf_status tc_score_list(mf_ctx* c, const uint64_t* idx, uint64_t n, float* score, uint8_t* feas, float* pred,
                        cudaStream_t s) {
  if (n == 0) return MF_OK;
  TcArgs T = c->tc;
  layout_smem(c->P, T, 0);
  const uint32_t smem = T.sm_total > kSmemFloor ? T.sm_total : kSmemFloor;
  float4* partial = nullptr;
  mf_status st = ensure_partial(c, T.npasses, n, s, &partial);
  if (st != MF_OK) return st;
  const uint64_t span = T.npasses == 1 ? n : kPassSpan;
  const int N = c->P.n_models;
  RangeArgs R{};
  for (uint64_t b = 0; b < n; b += span) {
    const uint64_t m = n - b < span ? n - b : span;
    const uint64_t tiles = (m + 127) / 128;
    const uint64_t grid = tiles < (uint64_t)c->num_sms ? tiles : (uint64_t)c->num_sms;
    TcList L{idx + b, m, score + b, feas ? feas + b : nullptr, pred ? pred + b * N * 2 : nullptr};
    for (int p = 0; p < T.npasses; ++p) {
      set_pass(T, p, partial);
      tc_kernel(kTcList, T, c->P.objective == MF_OBJ_UTILITY, c->P.n_models)<<<(unsigned)grid, T.pipes * tc_pipe_threads(T.ew), smem, s>>>(c->P, T, R, L);
      MF_CUDA(cudaGetLastError());
    }
  }
  return MF_OK;
}

}  // namespace mf
