// Reductions of the exhaustive search (the argmax of Sec. II extended to a
// top-k): merging the running lists, and the top-k of a re-scored shortlist.
// Order: J descending, index ascending.
#include "mf_internal.cuh"

namespace mf {

namespace {

constexpr int kMergeThreads = 1024;
constexpr int kMergeLane = 20;                       // list entries a lane holds: up to 640 lists
constexpr int kMergeMaxLists = 32 * kMergeLane;
static_assert(kMergeMaxLists == kMaxTops, "one bound for both");
constexpr size_t kPair = sizeof(uint64_t) + sizeof(float);

// Entries of a sorted row of 32 ahead of (s, id), where scores tie with s: by index too.  Out of
// line (ties are rare and the kernels' instructions are read once a launch).  (One after
// another, the ties of 18 lists of 32 equal scores took 45 us.)
__device__ __noinline__ int row_rank(const float* rs, const uint64_t* ri, float s, uint64_t id) {
  int lo = 0;
#pragma unroll
  for (int step = 16; step > 0; step >>= 1) lo += precedes(rs[lo + step - 1], ri[lo + step - 1], s, id) ? step : 0;
  return lo + (precedes(rs[lo], ri[lo], s, id) ? 1 : 0);
}

// The part of a warp's bound (see k_merge_lists) that ties need: of the lists whose entry at
// position p has the score key v, the last index that is wanted so that `need` lists come up to
// (v, that index).  `tied`: room for kMergeMaxLists indices.  Out of line, as above.
__device__ __noinline__ uint64_t tied_index(const float* in_s, const uint64_t* in_i, int nlists, int k, int p, uint32_t v,
                                            int need, uint64_t* tied) {
  const int lane = threadIdx.x & 31;
  int above = 0;
  uint32_t hi = 0u;
  for (int l = lane; l < kMergeMaxLists; l += 32) {
    const uint32_t key = l < nlists ? order_key(in_s[(size_t)l * k + p]) : 0u;
    const uint64_t id = key == v ? in_i[(size_t)l * k + p] : kEmptyIdx;
    above += key > v ? 1 : 0;
    tied[l] = id;
    if (id != kEmptyIdx) hi |= (uint32_t)(id >> 32);
  }
  const int want = need - __reduce_add_sync(0xffffffffu, above);
  hi = __reduce_or_sync(0xffffffffu, hi);
  uint64_t x = 0ull;  // the largest bound with fewer than `want` indices below it
  for (int b = hi ? 63 - __clz(hi) : 31; b >= 0; --b) {
    const uint64_t t = x | (1ull << b);
    int c = 0;
#pragma unroll 4
    for (int j = 0; j < kMergeLane; ++j) c += tied[lane + 32 * j] < t ? 1 : 0;
    if (__reduce_add_sync(0xffffffffu, c) < want) x = t;
  }
  return x;
}

// The gather of k_merge_lists where the bar cuts equal scores by index: the entries of the
// lists `which` up to (bar, the least of the lanes' bound_i).  Out of line, as above.
__device__ __noinline__ void gather_cut(const float* in_s, const uint64_t* in_i, int k, const int* which, int n, uint32_t bar,
                                        uint64_t bound_i, int cap, float* ss, uint64_t* si, int* count) {
  const int lane = threadIdx.x & 31;
  for (int w = 16; w > 0; w >>= 1) bound_i = min(bound_i, __shfl_xor_sync(0xffffffffu, bound_i, w));
  for (int q = threadIdx.x >> 5; q < n; q += blockDim.x >> 5) {
    const size_t l = (size_t)which[q] * k;
    unsigned m = 0xffffffffu;  // the lanes whose entry stays: a prefix (the lists are sorted)
    for (int pos = lane; m == 0xffffffffu; pos += 32) {
      const float sc = pos < k ? in_s[l + pos] : -INFINITY;
      const uint64_t ix = pos < k ? in_i[l + pos] : kEmptyIdx;
      const uint32_t key = order_key(sc);
      const bool keep = ix != kEmptyIdx && (key > bar || (key == bar && ix <= bound_i));
      m = __ballot_sync(0xffffffffu, keep);
      int at = 0;
      if (lane == 0 && m) at = atomicAdd(count, __popc(m));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
      if (keep && at < cap) { ss[at] = sc; si[at] = ix; }
    }
  }
}

// Sorts n distinct entries (ss, si) of shared memory best first and writes the first k
// to the output, empty slots after them.  Up to one entry per thread: each warp sorts its
// 32 in registers (shuffles), then an entry's position is its place in its own row of 32
// plus, by binary search, the entries of every other row ahead of it.  The sorted entries
// leave in whole rows: the output may be host memory, where each scattered word costs a
// transaction.  More entries: a bitonic network over the next power of two.  The arrays
// hold n rounded up to whole rows of 32, or that power of two (at least 1024).
__device__ void sort_out(float* ss, uint64_t* si, int n, int k, const ResultOut& out) {
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, row = tid >> 5;
  const int rows = (n + 31) >> 5;
  if (n <= nthr) {
    float s = -INFINITY;
    uint64_t id = kEmptyIdx;
    if (tid < n) { s = ss[tid]; id = si[tid]; }
    if (row < rows) {
#pragma unroll
      for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
          const float os = __shfl_xor_sync(0xffffffffu, s, stride);
          const uint64_t oid = __shfl_xor_sync(0xffffffffu, id, stride);
          const bool keep_better = ((lane & stride) == 0) == ((lane & size) == 0);
          if (precedes(s, id, os, oid) != keep_better) { s = os; id = oid; }
        }
      ss[tid] = s;
      si[tid] = id;
    }
    __syncthreads();
    int rank = lane;
    if (row < rows) {
#pragma unroll 4
      for (int r = 0; r < rows; ++r) {
        const float* rs = ss + 32 * r;
        int lo = 0;  // entries with a better score: no branch in the search
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) lo += rs[lo + step - 1] > s ? step : 0;
        lo += rs[lo] > s ? 1 : 0;
        if (r == row) continue;
        if (lo < 32 && rs[lo] == s) lo = row_rank(rs, si + 32 * r, s, id);
        rank += lo;
      }
    }
    __syncthreads();
    if (row < rows && id != kEmptyIdx) { ss[rank] = s; si[rank] = id; }
    __syncthreads();
    for (int j = tid; j < k && j < n; j += nthr) { out.score[j] = ss[j]; out.idx[j] = si[j]; }
  } else {
    int n2 = 1024;
    while (n2 < n) n2 <<= 1;
    for (int e = n + tid; e < n2; e += nthr) { ss[e] = -INFINITY; si[e] = kEmptyIdx; }
    __syncthreads();
    for (int size = 2; size <= n2; size <<= 1)
      for (int stride = size >> 1; stride > 0; stride >>= 1) {
        for (int i = tid; i < (n2 >> 1); i += nthr) {
          const int a = 2 * i - (i & (stride - 1)), b = a + stride;
          const float sa = ss[a], sb = ss[b];
          const uint64_t ia = si[a], ib = si[b];
          const bool best_first = (a & size) == 0;
          if (best_first ? precedes(sb, ib, sa, ia) : precedes(sa, ia, sb, ib)) {
            ss[a] = sb; si[a] = ib;
            ss[b] = sa; si[b] = ia;
          }
        }
        __syncthreads();
      }
    for (int e = tid; e < k && e < n; e += nthr) { out.score[e] = ss[e]; out.idx[e] = si[e]; }
  }
  for (int e = n + tid; e < k; e += nthr) { out.score[e] = -INFINITY; out.idx[e] = kEmptyIdx; }
}

// The count, the times and the status word beside the lists (nothing where the caller copies
// what it wants).
__device__ __forceinline__ void pass_on(const ResultOut& out) {
  if (threadIdx.x == 0 && out.tail) {
    out.tail->count = out.words->count;
    out.tail->t[0] = out.words->t[0];
    out.tail->t[1] = out.words->t[1];
    out.tail->status = *out.status;
    out.words->count = 0ull;
    out.tail->t[2] = device_ns();
  }
}

// Pairwise merge tree over `nlists` sorted lists of length k through the buffers a and b.
// Each element's output position is its position in its own list plus the number of
// elements of the partner list that precede it (binary search); elements at positions
// >= k are dropped.  Indices are distinct, so positions never collide.
__device__ __noinline__ void merge_tree(const float* in_s, const uint64_t* in_i, int nlists, int k, float* a_s,
                                        uint64_t* a_i, float* b_s, uint64_t* b_i, const ResultOut& out) {
  const float* src_s = in_s;
  const uint64_t* src_i = in_i;
  float* dst_s = a_s;
  uint64_t* dst_i = a_i;
  int n = nlists;
  while (n > 1) {
    const int m = (n + 1) / 2;
    for (int e = threadIdx.x; e < m * k; e += blockDim.x) { dst_s[e] = -INFINITY; dst_i[e] = kEmptyIdx; }
    __syncthreads();
    for (int e = threadIdx.x; e < 2 * m * k; e += blockDim.x) {
      const int p = e / (2 * k);
      const int r = e - p * 2 * k;
      const int which = r / k;
      const int pos = r - which * k;
      const int mine = 2 * p + which;
      if (mine >= n) continue;
      const float s = src_s[(size_t)mine * k + pos];
      const uint64_t id = src_i[(size_t)mine * k + pos];
      if (id == kEmptyIdx) continue;
      int cnt = 0;
      const int other = 2 * p + 1 - which;
      if (other < n) {
        const float* os = src_s + (size_t)other * k;
        const uint64_t* oi = src_i + (size_t)other * k;
        int lo = 0, hi = k;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (precedes(os[mid], oi[mid], s, id)) lo = mid + 1; else hi = mid;
        }
        cnt = lo;
      }
      const int rank = pos + cnt;
      if (rank < k) { dst_s[(size_t)p * k + rank] = s; dst_i[(size_t)p * k + rank] = id; }
    }
    __syncthreads();
    src_s = dst_s;
    src_i = dst_i;
    dst_s = (dst_s == a_s) ? b_s : a_s;
    dst_i = (dst_i == a_i) ? b_i : a_i;
    n = m;
  }
  for (int e = threadIdx.x; e < k; e += blockDim.x) { out.score[e] = src_s[e]; out.idx[e] = src_i[e]; }
}

}  // namespace

// Merge of `nlists` sorted lists of length k into one, by one CTA.
//
// Only k of the nlists * k entries survive, so the entries that cannot are dropped before
// anything is sorted.  If T lists have an entry of score >= x at position p, at least
// T (p + 1) entries reach x; so for T = ceil(k / (p + 1)) the T-th largest score at
// position p bounds the k-th best entry from below.  Warp j takes the bound of position
// p = 4^j - 1 (bisection over the score keys, each lane holding up to kMergeLane lists),
// and the largest bound is the bar: at most k / 4^j lists then hold more than 4^j - 1
// entries above it, so one to two k entries remain, and 4 k (log4(k) + 1) at most.  Where more
// than T lists reach the bound, some only tie with it: a bisection over the tied entries'
// indices then tells which T come first, so that entries equal to the bar in score are cut by
// index.  What remains is gathered into shared memory (`cap` entries) and sorted there.  Where
// that is more than the room, and above kMergeMaxLists lists, a merge tree through global memory
// takes over.
//
// Bound by latency (a few dependent L2 reads and block barriers).  608 lists of 256
// entries: 14 us, where the tree alone took 380-560; 304 lists of 32: 9 (tree: 35).  608 lists of
// 800 equal scores, with the re-scoring that follows: 94 us (by the tree 2.15 ms).
__global__ void __launch_bounds__(kMergeThreads)
k_merge_lists(const float* __restrict__ in_s, const uint64_t* __restrict__ in_i, int nlists, int k, int cap,
              float* a_s, uint64_t* a_i, float* b_s, uint64_t* b_i, const ResultOut out) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ uint32_t s_bar[32];      // a warp's bound: score key, and the last index among equals
  __shared__ uint64_t s_bar_i[32];
  __shared__ int s_lists[kMergeMaxLists];
  __shared__ int s_nlist, s_n;
  uint64_t* si = reinterpret_cast<uint64_t*>(smem);
  float* ss = reinterpret_cast<float*>(si + cap);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < 32) {
    s_bar[tid] = 0u;
    s_bar_i[tid] = kEmptyIdx;
  }
  if (tid == 0) {
    s_nlist = 0;
    s_n = 0;
    if (out.words) out.words->t[1] = device_ns();
  }
  if (out.words && tid < kMaxTops) out.words->tops[tid] = 0u;  // (for the next search)
  __syncthreads();
  bool few = nlists <= kMergeMaxLists;
  if (few) {
    const int p = (1 << (warp < 10 ? 2 * warp : 20)) - 1;
    const int need = (k + p) / (p + 1);  // T
    if (p < k && need <= nlists) {
      uint32_t key[kMergeLane];
#pragma unroll
      for (int j = 0; j < kMergeLane; ++j) {
        const int l = lane + 32 * j;
        key[j] = l < nlists ? order_key(in_s[(size_t)l * k + p]) : 0u;
      }
      uint32_t v = 0u;
      bool exact = false;  // `need` lists reach v, no more
      for (int b = 31; b >= 0; --b) {
        const uint32_t t = v | (1u << b);
        int c[4] = {0, 0, 0, 0};  // (short chains of dependent adds)
#pragma unroll
        for (int j = 0; j < kMergeLane; ++j) c[j & 3] += key[j] >= t ? 1 : 0;
        const int reach = __reduce_add_sync(0xffffffffu, (c[0] + c[1]) + (c[2] + c[3]));
        if (reach >= need) v = t;
        exact = reach == need;
        if (exact) break;  // (lower bits would only tighten the bar past ties)
      }
      // (the gather's room is not in use yet)
      const uint64_t x = exact || v <= kKeyMinusInf
                             ? kEmptyIdx
                             : tied_index(in_s, in_i, nlists, k, p, v, need, si + (size_t)warp * kMergeMaxLists);
      if (lane == 0) {
        s_bar[warp] = v;
        s_bar_i[warp] = x;
      }
    }
    __syncthreads();
    const uint32_t bar = __reduce_max_sync(0xffffffffu, s_bar[lane]);
    const uint64_t bound_i = s_bar[lane] == bar ? s_bar_i[lane] : kEmptyIdx;
    const bool cut = __any_sync(0xffffffffu, bound_i != kEmptyIdx);  // equal scores by index
    // the lists whose best entry reaches the bar, then their entries that do
    for (int l = tid; l < nlists; l += kMergeThreads)
      if (order_key(in_s[(size_t)l * k]) >= bar)
        s_lists[atomicAdd(&s_nlist, 1)] = l;
    __syncthreads();
    const int nl = s_nlist;
    if (cut) gather_cut(in_s, in_i, k, s_lists, nl, bar, bound_i, cap, ss, si, &s_n);
    constexpr int kBatch = 8;  // lists a warp has in flight
    for (int q0 = warp; q0 < nl && !cut; q0 += (kMergeThreads / 32) * kBatch) {
      float v[kBatch];
      uint64_t id[kBatch];
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        const int q = q0 + j * (kMergeThreads / 32);
        const bool in = q < nl && lane < k;
        const size_t at = in ? (size_t)s_lists[q] * k + lane : 0;
        v[j] = in ? in_s[at] : -INFINITY;
        id[j] = in ? in_i[at] : kEmptyIdx;
      }
      auto place = [&](bool keep, unsigned m, int at, float sc, uint64_t ix) {
        at += __popc(m & ((1u << lane) - 1u));
        if (keep && at < cap) { ss[at] = sc; si[at] = ix; }
      };
      unsigned m[kBatch];  // the lanes whose entry stays: a prefix (the lists are sorted)
      int total = 0;
      unsigned more = 0u;  // the lists whose first 32 entries all stay
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        m[j] = __ballot_sync(0xffffffffu, id[j] != kEmptyIdx && order_key(v[j]) >= bar);
        total += __popc(m[j]);
        more |= m[j] == 0xffffffffu ? 1u << j : 0u;
      }
      int at = 0;
      if (lane == 0 && total) at = atomicAdd(&s_n, total);
      at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
      for (int j = 0; j < kBatch; ++j) {
        place((m[j] >> lane) & 1u, m[j], at, v[j], id[j]);
        at += __popc(m[j]);
      }
      for (; more; more &= more - 1u) {
        const size_t l = (size_t)s_lists[q0 + (__ffs(more) - 1) * (kMergeThreads / 32)] * k;
        unsigned whole = 0xffffffffu;
        for (int pos = lane + 32; whole == 0xffffffffu; pos += 32) {
          const float sc = pos < k ? in_s[l + pos] : -INFINITY;
          const uint64_t ix = pos < k ? in_i[l + pos] : kEmptyIdx;
          const bool keep = ix != kEmptyIdx && order_key(sc) >= bar;
          whole = __ballot_sync(0xffffffffu, keep);
          int to = 0;
          if (lane == 0 && whole) to = atomicAdd(&s_n, __popc(whole));
          place(keep, whole, __shfl_sync(0xffffffffu, to, 0), sc, ix);
        }
      }
    }
    __syncthreads();
    few = s_n <= cap;
  }
  if (few) sort_out(ss, si, s_n, k, out);
  else merge_tree(in_s, in_i, nlists, k, a_s, a_i, b_s, b_i, out);
  pass_on(out);
}

// The end of a bf16 search: objective and constraints of the shortlist's n entries from
// their fp32 predictions (pred [n][N][2]; an empty entry stays empty), and the best k of
// them.  One CTA: n is 8 k or 256, and what it costs is latency.  NMAX: a bound on N.
template <int NMAX>
__global__ void __launch_bounds__(512)
k_finish(const Params P, const uint64_t* __restrict__ idx, const float* __restrict__ pred, int n, int n2, int k,
         const ResultOut out) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_n;
  uint64_t* si = reinterpret_cast<uint64_t*>(smem);
  float* ss = reinterpret_cast<float*>(si + n2);
  if (threadIdx.x == 0) s_n = 0;
  __syncthreads();
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const uint64_t id = idx[e];
    if (id >= P.total) continue;
    // every operand is read before the first is used: one L2 round trip, not one per model
    int row[NMAX];
    float2 pr[NMAX];
    float vr[NMAX];
    float4 ut[NMAX];
#pragma unroll
    for (int i = 0; i < NMAX; ++i) {
      if (i < P.n_models) {
        row[i] = P.off[i] + digit_of(P, id, i);
        pr[i] = *reinterpret_cast<const float2*>(pred + ((size_t)e * P.n_models + i) * 2);
        vr[i] = __ldg(&P.dem[row[i]].y);
        if (P.objective == MF_OBJ_UTILITY) ut[i] = __ldg(&P.util[row[i]]);
      }
    }
    Acc acc;
    acc.init();
    float vram = 0.f;
#pragma unroll
    for (int i = 0; i < NMAX; ++i) {
      if (i < P.n_models) {
        vram += vr[i];
        acc.add_util(P, i, pr[i].x, pr[i].y, ut[i]);
      }
    }
    acc.finish(P, vram);
    if (acc.J == -INFINITY) continue;  // infeasible in fp32
    const int at = atomicAdd(&s_n, 1);
    ss[at] = acc.J;
    si[at] = id;
  }
  __syncthreads();
  sort_out(ss, si, s_n, k, out);
  pass_on(out);
}

mf_status merge_lists(const float* ls, const uint64_t* li, int nlists, int k, float* tmp_s, uint64_t* tmp_i,
                      const ResultOut& out, cudaStream_t s) {
  // tmp holds two buffers of ceil(nlists / 2) * k entries each
  const size_t half = (size_t)((nlists + 1) / 2) * k;
  // room for 4096 survivors in short lists (k <= 256), else 16384.  (The attribute belongs to
  // the function, not to the launch: always the maximum, or a call of another context in
  // another thread could lower it in between.)
  constexpr int kCapMax = 16384;
  const int cap = k <= 256 ? 4096 : kCapMax;
  const size_t smem = (size_t)cap * kPair;
  MF_CUDA(cudaFuncSetAttribute(k_merge_lists, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kCapMax * kPair)));
  k_merge_lists<<<1, kMergeThreads, smem, s>>>(ls, li, nlists, k, cap, tmp_s, tmp_i, tmp_s + half, tmp_i + half,
                                               out);
  MF_CUDA(cudaGetLastError());
  return MF_OK;
}

mf_status finish_shortlist(const Params& P, const uint64_t* idx, const float* pred, int n, int k,
                           const ResultOut& out, cudaStream_t s) {
  constexpr int kMost = 8192;
  int n2 = 32;
  while (n2 < n) n2 <<= 1;
  if (n2 > kMost) {
    set_error("finish_shortlist: more than 8192 entries");
    return MF_EINVAL;
  }
  const size_t smem = (size_t)n2 * kPair;
  const auto fn = P.n_models <= 8 ? k_finish<8> : k_finish<MF_MAX_MODELS>;
  MF_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kMost * kPair)));  // (the maximum: see merge_lists)
  fn<<<1, 512, smem, s>>>(P, idx, pred, n, n2, k, out);
  MF_CUDA(cudaGetLastError());
  return MF_OK;
}

}  // namespace mf
