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
  if (T.tf != kXmBf16) return tc_kernel_exact(MODE, MP, UT);
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

// The shared-memory layout for lists of kcap entries: in the shape with two epilogue warps per
// lane quarter (48 KB of weights a model), with fewer models per pass if the lists would not
// fit next to a full pass's weights.
static bool layout_for(const Params& P, TcArgs& T, int kcap) {
  layout_smem(P, T, kcap);
  if (T.sm_total > kSmemLimit && T.ew == 2) {
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

}  // namespace

mf_status tc_prepare(mf_ctx* c, bool exact, const TcHost& h) {
  const Params& P = c->P;
  TcArgs& T = c->tc;
  std::memset(&T, 0, sizeof(T));
  if (exact) return tc_prepare_exact(c, h);
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
