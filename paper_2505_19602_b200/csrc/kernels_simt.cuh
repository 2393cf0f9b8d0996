// Kernels of the ScaleKV hot path beside the attention: append, observation-window scoring, per-slice top-k, in-place gather-compaction and the offline layer statistics.
#pragma once
#include <cfloat>

#include "common.cuh"

namespace scalekv {

// Window description handed to the select / score kernels by value.
struct WindowArg {
  int w;                 // number of window rows
  int all;               // 1: the whole current map is the window
  int n_prev;            // N_{k-1}: original position of the current map's first token
  int n_k;               // tokens of the current map
  int pos[kMaxWindow];   // ascending raster indices (unused when all = 1)
};

__device__ __forceinline__ bool is_window_pos(const WindowArg &wa, int p) {
  int r = p - wa.n_prev;
  if (r < 0) return false;
  if (wa.all) return true;
  int lo = 0, hi = wa.w;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (wa.pos[mid] < r) lo = mid + 1; else hi = mid;
  }
  return lo < wa.w && wa.pos[lo] == r;
}

// ------------------------------------------------------------------------------------------
// append: rows of the current map are copied behind the slice's history (Sec. 1; Sec. 3.3).
// grid (ceil(n_k / 64), n_slices), 256 threads, one 16-byte piece per thread per step.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) append_kernel(LayerView lv, TensorView K, TensorView V, int n_k, int n_prev,
                                                      int elem_bytes) {
  const int slice = blockIdx.y;
  const int b = slice / lv.n_heads, h = slice % lv.n_heads;
  const int ppr = lv.row_bytes >> 4;  // 16-byte pieces per row
  const int hist = lv.hist_len[slice];
  if (outgrown(lv, hist + n_k)) return;
  const int rows_per_step = 256 / ppr;
  const int r_in = threadIdx.x / ppr, c = threadIdx.x % ppr;
  const int i0 = blockIdx.x * 64;
  if (r_in >= rows_per_step) return;
  for (int r = r_in; r < 64; r += rows_per_step) {
    const int i = i0 + r;
    if (i >= n_k) break;
    const size_t row = slot_row(lv, slice, hist + i);
    const char *ks = K.ptr + ((long long)b * K.sb + (long long)h * K.sh + (long long)i * K.st) * elem_bytes;
    const char *vs = V.ptr + ((long long)b * V.sb + (long long)h * V.sh + (long long)i * V.st) * elem_bytes;
    uint4 kv = __ldg(reinterpret_cast<const uint4 *>(ks) + c);
    uint4 vv = __ldg(reinterpret_cast<const uint4 *>(vs) + c);
    reinterpret_cast<uint4 *>(lv.k_pool + row * lv.row_bytes)[c] = kv;
    reinterpret_cast<uint4 *>(lv.v_pool + row * lv.row_bytes)[c] = vv;
    if (c == 0) lv.pos_pool[row] = n_prev + i;
  }
}

// The length after a current map that was neither attended nor compressed (attend writes it itself).
__global__ void commit_kernel(LayerView lv, int n_k) {
  int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < lv.n_slices) lv.next_len[s] = lv.hist_len[s] + n_k;
}

constexpr float kNoMax = -FLT_MAX;       // a finite stand-in for -inf, so that differences of maxima are numbers; no finite score lies below

template <typename T, int D>
__device__ __forceinline__ void load_tile_rows(float *dst, int ld, const LayerView &lv, const char *pool, int slice,
                                               int j0, int L) {
  constexpr int CH = D * (int)sizeof(T) / 16;
  constexpr int VN = Vec16<T>::N;
  for (int idx = threadIdx.x; idx < 64 * CH; idx += 256) {
    const int r = idx / CH, c = idx % CH;
    float v[VN];
    if (j0 + r < L) {
      const size_t row = slot_row(lv, slice, j0 + r);
      Vec16<T>::load(reinterpret_cast<const T *>(pool + row * lv.row_bytes) + c * VN, v);
    } else {
#pragma unroll
      for (int e = 0; e < VN; ++e) v[e] = 0.f;
    }
#pragma unroll
    for (int e = 0; e < VN; ++e) dst[r * ld + c * VN + e] = v[e];
  }
}

// The base-2 logits of w window rows (Qs, 64 rows of D + 4 columns) against the 64 entries from j0 on (Ks alike): every one a chain of
// multiply-adds in the order of the columns, whichever kernel asks.  256 threads; `out`: the rows' logits by slot.
template <int D>
__device__ __forceinline__ void tile_logits(const float *Qs, const float *Ks, int w, int j0, int L, float *out, int ld_l, float scale) {
  constexpr int LD = D + 4;
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  const int ni = (w + 15) >> 4;  // active 16-row groups
  float s[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) s[i][j] = 0.f;
  for (int c = 0; c < D; c += 4) {
    float4 k[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) k[j] = *reinterpret_cast<const float4 *>(&Ks[(tx + 16 * j) * LD + c]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (i < ni) {
        const float4 q = *reinterpret_cast<const float4 *>(&Qs[(ty + 16 * i) * LD + c]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          s[i][j] = fmaf(q.x, k[j].x, s[i][j]);
          s[i][j] = fmaf(q.y, k[j].y, s[i][j]);
          s[i][j] = fmaf(q.z, k[j].z, s[i][j]);
          s[i][j] = fmaf(q.w, k[j].w, s[i][j]);
        }
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = ty + 16 * i;
    if (r >= w) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int col = j0 + tx + 16 * j;
      if (col < L) out[(size_t)r * ld_l + col] = s[i][j] * (scale * 1.4426950408889634f);
    }
  }
}

// ------------------------------------------------------------------------------------------
// score, step 1 (only when attend did not record them): logits of the window rows against a tile of
// 64 cache entries (Eq. 5), in base-2 units: y = scale * log2(e) * <q, k>.
// grid (ceil(L_max / 64), n_slices), 256 threads.  logits is [n_slices][w][ld_l] fp32.
// ------------------------------------------------------------------------------------------
template <typename T, int D>
__global__ void __launch_bounds__(256) score_logits_kernel(LayerView lv, TensorView Qw, WindowArg wa, int full_map,
                                                           float *logits, int ld_l, float scale) {
  constexpr int LD = D + 4;
  constexpr int CH = D * (int)sizeof(T) / 16;
  constexpr int VN = Vec16<T>::N;
  extern __shared__ float smem[];
  float *Qs = smem;             // [64][LD], rows >= w zero
  float *Ks = Qs + 64 * LD;     // [64][LD]
  const int tid = threadIdx.x;
  const int slice = blockIdx.y;
  const int b = slice / lv.n_heads, h = slice % lv.n_heads;
  const int L = lv.hist_len[slice] + wa.n_k;
  const int j0 = blockIdx.x * 64;
  if (outgrown(lv, L) || j0 >= L) return;
  for (int idx = tid; idx < 64 * CH; idx += 256) {
    const int r = idx / CH, c = idx % CH;
    float v[VN];
    if (r < wa.w) {
      const int qi = full_map ? (wa.all ? r : wa.pos[r]) : r;
      Vec16<T>::load(row_ptr<T>(Qw, b, h, qi) + c * VN, v);
    } else {
#pragma unroll
      for (int e = 0; e < VN; ++e) v[e] = 0.f;
    }
#pragma unroll
    for (int e = 0; e < VN; ++e) Qs[r * LD + c * VN + e] = v[e];
  }
  load_tile_rows<T, D>(Ks, LD, lv, lv.k_pool, slice, j0, L);
  __syncthreads();
  tile_logits<D>(Qs, Ks, wa.w, j0, L, logits + (size_t)slice * wa.w * ld_l, ld_l, scale);
}

// ------------------------------------------------------------------------------------------
// score, step 2 (Sec. 3.3, Eq. 5): from the base-2 logits y[w][L] of the window rows to the importance
// s_i = (1/w) sum_j 2^(y_ji - lse_j), lse_j the base-2 log-sum-exp of row j (recorded by attend, or
// computed by row_lse_kernel).  Streaming and embarrassingly parallel: grid (ceil(L_max / 256),
// n_slices), one entry per thread, the w loads of a thread independent and coalesced across the warp.
// Besides the score (kept for inspection) it writes the entry's key: the bit pattern of the
// non-negative float, or a sentinel for window entries, which never take part in the selection.
// ------------------------------------------------------------------------------------------
constexpr uint32_t kWindowKey = 0xFFFFFFFFu;

// logit_scale: what turns a stored logit into a base-2 logit (1 when the logits kernel wrote them, softmax scale *
// log2(e) when attend recorded raw products).  tile_padded: attend recorded them while the current map was
// not in the store yet, so its entries sit behind the history rounded up to a multiple of 128 columns.
__global__ void __launch_bounds__(256) score_kernel(LayerView lv, WindowArg wa, const float *logits, const float *lse,
                                                    int ld_l, float logit_scale, int tile_padded, float *scores, uint32_t *keys,
                                                    int ld_s) {
  __shared__ float lse_row[kMaxWindow];
  const int slice = blockIdx.y;
  const int hist = lv.hist_len[slice];
  const int L = hist + wa.n_k;
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (outgrown(lv, L) || blockIdx.x * 256 >= L) return;
  const int w = wa.w;
  if (threadIdx.x < w) lse_row[threadIdx.x] = lse[(size_t)slice * w + threadIdx.x];
  __syncthreads();
  if (i >= L) return;
  const int col = (tile_padded && i >= hist) ? (((hist + 127) >> 7) << 7) + (i - hist) : i;
  const float *y = logits + (size_t)slice * w * ld_l + col;
  float sc = 0.f;
  int j = 0;
  for (; j + 8 <= w; j += 8) {
    float t[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) t[e] = __ldg(y + (size_t)(j + e) * ld_l);
#pragma unroll
    for (int e = 0; e < 8; ++e) sc += exp2f(fmaf(t[e], logit_scale, -lse_row[j + e]));
  }
  for (; j < w; ++j) sc += exp2f(fmaf(__ldg(y + (size_t)j * ld_l), logit_scale, -lse_row[j]));
  sc *= 1.f / (float)w;
  scores[(size_t)slice * ld_s + i] = sc;
  const bool win = is_window_pos(wa, lv.pos_pool[slot_row(lv, slice, i)]);
  keys[(size_t)slice * ld_s + i] = win ? kWindowKey : (__float_as_uint(sc) & 0x7FFFFFFFu);
}

// Head-shared importance (Sec. 3.3, "a unified importance metric" read as shared between the heads of a
// batch element): every entry's importance becomes the mean over the heads, summed in head order, and
// the keys follow.  The heads must hold the same entries: equal lengths and equal original positions,
// else the device status is raised and the selection that follows does not run.
// grid (ceil(L_max / 256), B), 256 threads; scores and keys are [n_slices][ld_s].
__global__ void __launch_bounds__(256) head_mean_kernel(LayerView lv, WindowArg wa, float *scores, uint32_t *keys, int ld_s) {
  const int H = lv.n_heads;
  const int s0 = blockIdx.y * H;
  const int L = lv.hist_len[s0] + wa.n_k;
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (blockIdx.x == 0 && threadIdx.x < H && lv.hist_len[s0 + threadIdx.x] + wa.n_k != L) atomicExch(lv.status, kDevCheck);
  if (outgrown(lv, L) || i >= L) return;
  const int pos = lv.pos_pool[slot_row(lv, s0, i)];
  float sum = 0.f;
  bool same = true;
  for (int h = 0; h < H; ++h) {
    sum += scores[(size_t)(s0 + h) * ld_s + i];
    same = same && (lv.hist_len[s0 + h] + wa.n_k <= i || lv.pos_pool[slot_row(lv, s0 + h, i)] == pos);
  }
  if (!same) atomicExch(lv.status, kDevCheck);
  const float mean = sum * (1.f / (float)H);
  const uint32_t key = is_window_pos(wa, pos) ? kWindowKey : (__float_as_uint(mean) & 0x7FFFFFFFu);
  for (int h = 0; h < H; ++h) {
    scores[(size_t)(s0 + h) * ld_s + i] = mean;
    keys[(size_t)(s0 + h) * ld_s + i] = key;
  }
}

// Keys of the positional keep rule (the comparison policies of Sec. 4.1: sliding window, sinks + recent
// tokens): entries whose original position is below n_sink carry the sentinel (always kept), every
// other entry competes on its position, most recent first.  grid (ceil(L_max / 256), n_slices).
__global__ void __launch_bounds__(256) recent_keys_kernel(LayerView lv, int n_k, int n_sink, uint32_t *keys, int ld_s) {
  const int slice = blockIdx.y;
  const int L = lv.hist_len[slice] + n_k;
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (outgrown(lv, L) || i >= L) return;
  const int pos = lv.pos_pool[slot_row(lv, slice, i)];
  keys[(size_t)slice * ld_s + i] = pos < n_sink ? kWindowKey : (uint32_t)pos + 1u;
}

// Base-2 log-sum-exp of every window row of y[w][L] when attend did not record it: a CTA of 1024 threads per slice and four
// rows, a maximum sweep and a sum sweep.  What bounds it is the latency of its reductions: 16 slices behind 92 to 772 entries, us per layer and
// step of the f32 attention with 16 rows per CTA -> so: 64 queries 20.5 -> 19.5, 576: 55.3 -> 53.8.  lse is [n_slices][w].
// grid (n_slices, ceil(w / 4)).
__global__ void __launch_bounds__(1024) row_lse_kernel(LayerView lv, WindowArg wa, const float *logits, int ld_l, float *lse) {
  constexpr int R = 4;
  __shared__ float part[32][R];
  __shared__ float m_row[R];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");      // (the compress comes up and waits)
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int slice = blockIdx.x;
  const int L = lv.hist_len[slice] + wa.n_k;
  if (outgrown(lv, L)) return;
  const int w = wa.w;
  const float *y = logits + (size_t)slice * w * ld_l;
  for (int g0 = R * (int)blockIdx.y; g0 < w; g0 += R * (int)gridDim.y) {
    const int nr = w - g0 < R ? w - g0 : R;
    float acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = -INFINITY;
    for (int i = tid; i < L; i += 1024) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (r < nr) acc[r] = fmaxf(acc[r], y[(size_t)(g0 + r) * ld_l + i]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float v = acc[r];
      for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
      if (lane == 0) part[wid][r] = v;
    }
    __syncthreads();
    if (tid < R) {
      float v = part[0][tid];
      for (int k = 1; k < 32; ++k) v = fmaxf(v, part[k][tid]);
      m_row[tid] = v;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0.f;
    for (int i = tid; i < L; i += 1024) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (r < nr) acc[r] += exp2f(y[(size_t)(g0 + r) * ld_l + i] - m_row[r]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float v = acc[r];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) part[wid][r] = v;
    }
    __syncthreads();
    if (tid < R) {
      float v = 0.f;
      for (int k = 0; k < 32; ++k) v += part[k][tid];     // fixed order: deterministic
      if (tid < nr) lse[(size_t)slice * w + g0 + tid] = m_row[tid] + log2f(v);
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------------------
// select: per-slice top-k' of the non-window entries by key (Sec. 3.3), one CTA of 1024 threads per
// slice with the slice's keys in shared memory (with pool > 1 a candidate's key is first replaced by
// its importance averaged over the neighbouring entries); see select_and_emit.  Ties at the threshold go to the lowest
// slots = lowest original positions.  Deterministic.
// Dynamic shared memory: 4 * ld_s bytes of keys.
// ------------------------------------------------------------------------------------------
constexpr int kMaxHeadBudgets = 128;
struct HeadBudgets {     // per-head budgets of one compress call
  int v[kMaxHeadBudgets];
};
// Spreads the per-head budgets of a compress call over the slices (slice = b * n_heads + h), so that the
// select kernel reads its budget with one load instead of indexing a by-value table.
__global__ void head_budget_kernel(HeadBudgets hb, int n_heads, int n_slices, int *slice_budget) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < n_slices) slice_budget[s] = hb.v[s % n_heads];
}
// Shared state of one selection (static shared memory of the calling kernel).
constexpr int kSelectBins = 2048;
struct SelectShared {
  int hist[kSelectBins];
  int warp_sums[32];
  union { uint32_t lowest[32]; int keeps[32]; };           // bounds first, counts behind several barriers (every byte here is one that a
  union { uint32_t highest[32]; int ties[32]; };           // slice's keys and keep list cannot have)
  int first_gap;
  int bin, need, in_bin, n_cand, n_ties;
  uint32_t tie_key;
};

// The selection proper, run by a whole CTA of NT threads: key[0 .. L) (shared or global memory) -> out[] = the
// ascending slots of the survivors (the `budget` largest keys, equal keys by lowest slot, plus every sentinel
// entry).  Returns the number of survivors; *kprime_plus_win receives the count the rule demands, sh.first_gap the lowest slot that
// does not survive (L: all do).  lowest / highest: bounds of the keys, other than the sentinel, that this thread has seen; every key has
// been seen by one.  Its first barrier ends its callers' writes of keys; out has room for L entries and serves as scratch before it is
// written.
//   Up to kRankAll entries: every key is ranked against all.
//   More: a histogram of 2 048 bins between the lowest and the highest key says in which bin the budget runs out; when the bin
//   holds no more keys than there are threads they are gathered and every one is ranked against all, else the next 11 bits
//   decide in the same way.  The emit gives every warp a run of consecutive entries and orders them by ballots, twice: to count, and
//   behind one exclusive sum over the warps to write.
// What bounds it is the latency of its rounds of block barriers, and updates of one bin, which take turns.  512 threads, 56 / 224 /
// 785 / 1 233 / 4 248 entries: 1 870 / 3 170 / 3 930 / 5 400 / 8 900 cycles.  (Bins of the keys' upper 11 bits, eight to an octave of importance,
// and no ranking of all: 4 050 / 4 140 / 5 370 / 6 240 / 13 870.  Ranking 144 entries against all takes 3 900, hence the line at 128.)
constexpr int kRankAll = 128;
template <int NT>
__device__ __forceinline__ int select_and_emit(const uint32_t *key, int L, int budget, uint32_t lowest, uint32_t highest, int *out,
                                                SelectShared &sh, int *kprime_plus_win) {
  constexpr int NW = NT / 32, PER = kSelectBins / NT;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  lowest = __reduce_min_sync(0xffffffffu, lowest);
  highest = __reduce_max_sync(0xffffffffu, highest);
  if (lane == 0) { sh.lowest[wid] = lowest; sh.highest[wid] = highest; }
  for (int i = tid; i < kSelectBins; i += NT) sh.hist[i] = 0;
  if (tid == 0) { sh.n_cand = 0; sh.first_gap = L; }
  __syncthreads();
  const uint32_t lower = (1u << lane) - 1u;
  if (L <= kRankAll) {
    // entry i by the threads i, i + 128, ..: how many candidates of their share of the entries stand before it (sentinels are
    // zeros here, and stand before nothing)
    constexpr int kParts = NT / kRankAll;
    const int i = tid % kRankAll, part = tid / kRankAll, share = (L + kParts - 1) / kParts, lo = part * share, hi = min(lo + share, L);
    const uint32_t k = i < L ? key[i] + 1u : 0u;
    int before = 0;
    if ((i & ~31) < L) {
#pragma unroll 8
      for (int j = lo; j < hi; ++j) {
        const uint32_t o = key[j] + 1u;
        before += o > k || (o == k && j < i);
      }
    }
    if (part > 0) sh.hist[tid] = before;
    const int all = __syncthreads_count(part == 0 && k != 0u);
    kprime_plus_win[0] = (budget < 0 || budget > all ? all : budget) + (L - all);
    bool keep = false;
    if (part == 0) {
#pragma unroll
      for (int p = 1; p < kParts; ++p) before += sh.hist[p * kRankAll + i];
      keep = i < L && (k == 0u || budget < 0 || before < budget);
      const uint32_t kept = __ballot_sync(0xffffffffu, keep), gaps = __ballot_sync(0xffffffffu, i < L && !keep);
      if (lane == 0) {
        sh.keeps[wid] = __popc(kept);
        if (gaps) atomicMin(&sh.first_gap, wid * 32 + __ffs(gaps) - 1);
      }
    }
    __syncthreads();
    const int keeps = lane < kRankAll / 32 ? sh.keeps[lane] : 0;
    const uint32_t kept = __ballot_sync(0xffffffffu, keep);
    const int at = __reduce_add_sync(0xffffffffu, lane < wid ? keeps : 0) + __popc(kept & lower);
    if (keep) out[at] = i;
    return __reduce_add_sync(0xffffffffu, keeps);
  }
  lowest = __reduce_min_sync(0xffffffffu, lane < NW ? sh.lowest[lane] : 0xffffffffu);
  highest = __reduce_max_sync(0xffffffffu, lane < NW ? sh.highest[lane] : 0u);
  if (lowest > highest) lowest = highest = 0;          // nothing but sentinels
  const int shift = max(21 - __clz((highest - lowest) | 1u), 0);       // the range of keys in 11 bits
  int kprime = 0;
  uint32_t above_min = kWindowKey, tie_key = kWindowKey;     // the smallest key of which every entry stays; the key of which
  int n_ties = 0;                                            // the first n_ties entries stay as well
  // (keys less the lowest from here on)
  uint32_t prefix = 0;                                       // the keys in question: those with key >> above_shift == prefix
  for (int above_shift = shift + 11, s = shift, need = 0;; above_shift = s, s = s > 11 ? s - 11 : 0) {
    const bool first = above_shift == shift + 11;
    if (!first) {
      for (int i = tid; i < kSelectBins; i += NT) sh.hist[i] = 0;
      __syncthreads();
    }
    for (int i = tid; i < L; i += NT) {
      const uint32_t k = key[i];
      if (k != kWindowKey && ((k - lowest) >> above_shift) == prefix) atomicAdd(&sh.hist[((k - lowest) >> s) - (prefix << (above_shift - s))], 1);
    }
    __syncthreads();
    // thread t counts the bins 2047 - PER t, .. downwards, so that the exclusive sum is what lies above them
    int c[PER], mine = 0, all;
#pragma unroll
    for (int e = 0; e < PER; ++e) { c[e] = sh.hist[kSelectBins - 1 - (tid * PER + e)]; mine += c[e]; }
    int above = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, above, o);
      if (lane >= o) above += x;
    }
    if (lane == 31) sh.warp_sums[wid] = above;
    __syncthreads();
    {
      const int sums = lane < NW ? sh.warp_sums[lane] : 0;
      all = __reduce_add_sync(0xffffffffu, sums);
      above += __reduce_add_sync(0xffffffffu, lane < wid ? sums : 0) - mine;
    }
    if (first) {
      kprime = (budget < 0 || budget > all) ? all : budget;
      *kprime_plus_win = kprime + (L - all);
      if (kprime == all) above_min = 0;
      if (kprime == 0 || kprime == all) break;
      need = kprime;
    }
    if (above < need && above + mine >= need) {
      int r = need - above;
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        if (r > 0) {
          if (c[e] >= r) { sh.bin = kSelectBins - 1 - (tid * PER + e); sh.need = r; sh.in_bin = c[e]; r = 0; }
          else r -= c[e];
        }
      }
    }
    __syncthreads();
    prefix = (prefix << (above_shift - s)) + (uint32_t)sh.bin;
    need = sh.need;
    const int m = sh.in_bin;
    if (m == need) {                             // the whole bin stays
      above_min = (prefix << s) + lowest;
      break;
    }
    if (s == 0) {                                // equal keys
      tie_key = prefix + lowest;
      n_ties = need;
      above_min = tie_key + 1;
      break;
    }
    if (m <= NT) {
      for (int i = tid; i < L; i += NT) {
        const uint32_t k = key[i];
        if (k != kWindowKey && ((k - lowest) >> s) == prefix) out[atomicAdd(&sh.n_cand, 1)] = (int)k;
      }
      __syncthreads();
      const int v = tid < m ? out[tid] : -1;     // (keys are below 2^31)
      int gt = 0, ge = 0;
      if (wid * 32 < m) {
#pragma unroll 8
        for (int i = 0; i < m; ++i) {
          const int o = out[i];
          gt += o > v;
          ge += o >= v;
        }
      }
      if (tid < m && gt < need && ge >= need) { sh.tie_key = (uint32_t)v; sh.n_ties = need - gt; }   // (equal keys write the same)
      __syncthreads();                           // (and the candidates have been read: out may be written)
      tie_key = sh.tie_key;
      n_ties = sh.n_ties;
      above_min = tie_key + 1;
      break;
    }
  }

  // ordered emit: warp w owns entries [w * run, (w + 1) * run)
  const int run = ((L + NW - 1) / NW + 31) & ~31, lo = wid * run, hi = min(lo + run, L);
  int n_keep = 0, n_tie = 0;
  for (int i0 = lo; i0 < hi; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t k = i < hi ? key[i] : 0u;
    n_keep += __popc(__ballot_sync(0xffffffffu, i < hi && (k >= above_min || k == kWindowKey)));
    n_tie += __popc(__ballot_sync(0xffffffffu, i < hi && k == tie_key && k != kWindowKey));
  }
  if (lane == 0) { sh.keeps[wid] = n_keep; sh.ties[wid] = n_tie; }
  __syncthreads();
  const int keeps = lane < NW ? sh.keeps[lane] : 0, ties = lane < NW ? sh.ties[lane] : 0;
  const int total = __reduce_add_sync(0xffffffffu, keeps) + min(__reduce_add_sync(0xffffffffu, ties), n_ties);
  int tie_at = __reduce_add_sync(0xffffffffu, lane < wid ? ties : 0);
  int at = __reduce_add_sync(0xffffffffu, lane < wid ? keeps : 0) + min(tie_at, n_ties), gap = L;
  for (int i0 = lo; i0 < hi; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t k = i < hi ? key[i] : 0u;
    const bool tie = i < hi && k == tie_key && k != kWindowKey;
    const uint32_t tied = __ballot_sync(0xffffffffu, tie);
    const bool keep = (i < hi && (k >= above_min || k == kWindowKey)) || (tie && tie_at + __popc(tied & lower) < n_ties);
    const uint32_t kept = __ballot_sync(0xffffffffu, keep), gaps = __ballot_sync(0xffffffffu, i < hi && !keep);
    if (keep) out[at + __popc(kept & lower)] = i;
    if (gap == L && gaps) gap = i0 + __ffs(gaps) - 1;
    at += __popc(kept);
    tie_at += __popc(tied);
  }
  if (lane == 0 && gap < L) atomicMin(&sh.first_gap, gap);
  return total;
}

// The importance averaged over `pool` neighbouring entries (zeros beyond both ends), summed in slot order.
__device__ __forceinline__ uint32_t pooled_key(const float *sc, int i, int L, int pool) {
  const int r = pool >> 1;
  float acc = 0.f;
  for (int d = -r; d <= r; ++d)
    if (i + d >= 0 && i + d < L) acc += sc[i + d];
  return __float_as_uint(acc / (float)pool) & 0x7FFFFFFFu;
}

// slice_budget: per-slice budgets (nullptr: every slice takes `budget`).
// in_smem != 0: the slice's keys are staged in dynamic shared memory (4 * ld_s bytes); 0: a slice too long for
// that is selected from the global key array as it stands (with pool > 1 the pooled keys are first written back
// there), every pass streaming the keys through L2.
__global__ void __launch_bounds__(1024) select_kernel(LayerView lv, WindowArg wa, int budget, const int *slice_budget, uint32_t *keys,
                                                      const float *scores, int pool, int ld_s, int in_smem, int *keep_list,
                                                      int *kept_count) {
  extern __shared__ uint32_t key_sm[];         // [L] when in_smem
  __shared__ SelectShared sh;
  const int tid = threadIdx.x;
  const int slice = blockIdx.x;
  const int dev_status = *reinterpret_cast<volatile int *>(lv.status);   // both loads in flight before the test
  const int L = lv.hist_len[slice] + wa.n_k;
  if (dev_status != 0 || outgrown(lv, L)) return;   // a failed check, an earlier kernel's or this one's: leave the store alone
  int *out = keep_list + (size_t)slice * ld_s;
  uint32_t *gkey = keys + (size_t)slice * ld_s;
  const float *sc = scores + (size_t)slice * ld_s;
  uint32_t lowest = 0xffffffffu, highest = 0u;
  for (int i = tid; i < L; i += 1024) {
    uint32_t k = gkey[i];
    if (pool > 1 && k != kWindowKey) k = pooled_key(sc, i, L, pool);
    if (k != kWindowKey) { lowest = min(lowest, k); highest = max(highest, k); }
    if (in_smem) key_sm[i] = k;
    else if (pool > 1) gkey[i] = k;
  }
  if (slice_budget != nullptr) budget = slice_budget[slice];
  int want;
  const int keep_total = select_and_emit<1024>(in_smem ? key_sm : gkey, L, budget, lowest, highest, out, sh, &want);
  if (tid == 0) {
    kept_count[slice] = keep_total;
    // the count rule of the selection: k' candidates and every sentinel entry survive
    if (keep_total != want) atomicExch(lv.status, kDevCheck);
  }
}

// ------------------------------------------------------------------------------------------
// compact: slot j <- old slot keep[j], in place (Sec. 3.3, pruning).  grid (n_slices, 2, 4):
// blockIdx.y = 0 moves K (and, in column block 0, pos), 1 moves V; blockIdx.z picks a quarter of
// the row's 16-byte pieces, so that a slice's move is spread over 8 CTAs that touch disjoint bytes.
// The slice's page table and keep list are staged in shared memory first, so that the row moves
// depend on no further global look-up.  keep is ascending, so keep[j] >= j: within a chunk every
// source is read before any destination is written, and the sources of later chunks lie beyond
// every earlier destination.  256 threads, chunks of 2048 / ppq rows (ppq = pieces per row
// quarter), 8 pieces in flight per thread.  Dynamic shared memory: 4 * (pages_per_slice [+ ld_s]) B.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) compact_kernel(LayerView lv, const int *keep_list, int ld_s, int list_in_smem,
                                                      const int *kept_count) {
  extern __shared__ int csm[];
  int *pt = csm;                   // [pages_per_slice]
  const int slice = blockIdx.x;
  const int which = blockIdx.y;
  const int quarter = blockIdx.z;
  char *pool = which == 0 ? lv.k_pool : lv.v_pool;
  const int dev_status = *reinterpret_cast<volatile int *>(lv.status);   // both loads in flight before the test
  const int kept = kept_count[slice];
  if (dev_status != 0) return;                 // the selection did not run: nothing to move
  // the keep list is staged in shared memory when it fits ([kept] behind the page table), else read where it is
  const int *list = keep_list + (size_t)slice * ld_s;
  if (list_in_smem) {
    int *ls = csm + lv.pages_per_slice;
    for (int i = threadIdx.x; i < kept; i += 256) ls[i] = __ldg(list + i);
    list = ls;
  }
  for (int i = threadIdx.x; i < lv.pages_per_slice; i += 256) pt[i] = __ldg(lv.page_table + (size_t)slice * lv.pages_per_slice + i);
  __syncthreads();
  auto row_of = [&](int slot) { return ((size_t)pt[slot >> lv.page_shift] << lv.page_shift) + (size_t)(slot & lv.page_mask); };
  const int ppr = lv.row_bytes >> 4;       // 16-byte pieces per row
  const int ppq = ppr >> 2;                // pieces of this CTA's quarter (row_bytes is a multiple of 64)
  const int C = 2048 / ppq;                // rows per chunk
  int lo = 0, hi = kept;                   // first j with keep[j] != j (the untouched prefix is skipped)
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (list[mid] == mid) lo = mid + 1; else hi = mid;
  }
  const bool do_pos_cta = which == 0 && quarter == 0;
  const int r_in = threadIdx.x / ppq, c = quarter * ppq + threadIdx.x % ppq;   // piece u of a thread: row r_in + u * 256 / ppq
  const int r_step = 256 / ppq;
  const bool pos_thread = do_pos_cta && (threadIdx.x % ppq == 0);
  for (int c0 = lo; c0 < kept; c0 += C) {
    uint4 buf[8];
    int pv[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = c0 + r_in + u * r_step;
      if (j < kept) {
        const size_t row = row_of(list[j]);
        buf[u] = reinterpret_cast<const uint4 *>(pool + row * lv.row_bytes)[c];
        if (pos_thread) pv[u] = lv.pos_pool[row];
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int j = c0 + r_in + u * r_step;
      if (j < kept) {
        const size_t row = row_of(j);
        reinterpret_cast<uint4 *>(pool + row * lv.row_bytes)[c] = buf[u];
        if (pos_thread) lv.pos_pool[row] = pv[u];
      }
    }
  }
  if (do_pos_cta && threadIdx.x == 0) lv.next_len[slice] = kept;
}

// ------------------------------------------------------------------------------------------
// compress in one launch (Sec. 3.3, "KV Cache Selection"): importance, selection and pruning of one slice by one
// CTA of 512 threads, the phases separated by block barriers - what score_kernel, select_kernel and
// compact_kernel do in three launches, for every slice whose keys and keep list fit in shared memory.
//   phase 1  policy 0: s_i = (1/w) sum_j 2^(y_ji * logit_scale - lse_j) from the window rows' logits (see
//            score_kernel), two neighbouring columns per thread -> scores (global, kept for inspection) and keys
//            (shared); the window entries, whose slots follow from the map's place behind the history, get the sentinel.
//            policy 1: keys from the original positions (see recent_keys_kernel).
//   phase 2  select_and_emit, ascending keep list in shared memory.
//   phase 3  slot j <- old slot keep[j] for K, V and pos, in chunks: every thread loads its 8 16-byte pieces of
//            the chunk, block barrier, stores them.  keep is ascending and keep[j] >= j: within a chunk every source is read
//            before any destination is written, and the sources of later chunks lie beyond every earlier destination.  The
//            untouched prefix is skipped.
// ext.on: the current map has not been copied into the pages (a one-call step whose attend left it in the caller's
// tensors): entries hist .. L-1 are rows of those tensors, phase 3 reads the survivors among them there and every kept
// row of the map is written, whatever its index.
// What bounds it: for short keep lists the latency of the phases, which 512 threads (so that two slices can share an SM) and
// fewer rounds of barriers cut; for long ones the memory system: an SM stores 32 bytes per cycle (17 cycles per row, 22
// measured for loads and stores of 16 slices), and 128 slices at once move at the HBM's rate (42 cycles per row = 5.9 TB/s).
// Dynamic shared memory: 4 * (2 * ld_s + pages_per_slice) bytes.  grid (n_slices).
// ------------------------------------------------------------------------------------------
constexpr int kCompressThreads = 512;
constexpr int kSumsInCompress = 512;      // entries of a slice up to which it can take the window rows' log-sum-exps itself: a warp's lanes hold a row

__global__ void __launch_bounds__(kCompressThreads, 2) compress_fused_kernel(LayerView lv, WindowArg wa, int policy, int n_sink,
                                                                          const float *logits, const float *lse, int ld_l,
                                                                          float logit_scale, int tile_padded, int budget,
                                                                          const int *slice_budget, int pool, float *scores, int ld_s,
                                                                          int *kept_count, ExternalMap ext) {
  constexpr int NT = kCompressThreads;
  extern __shared__ __align__(16) uint32_t fsm[];
  int *list = reinterpret_cast<int *>(fsm);              // [ld_s]
  uint32_t *key = fsm + ld_s;                            // [ld_s]
  int *pt = list + 2 * ld_s;                             // [pages_per_slice]
  __shared__ SelectShared sh;
  __shared__ float lse_row[kMaxWindow];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int slice = blockIdx.x;
  const int w = wa.w;
  // All of this is under way before any of it is needed.  (Behind a kernel of the same call the CTA comes up while that ends: only the page
  // table is there before the wait.)
  const int *pages = lv.page_table + (size_t)slice * lv.pages_per_slice;
  const int page = tid < lv.pages_per_slice ? __ldg(pages + tid) : 0;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int dev_status = *reinterpret_cast<volatile int *>(lv.status);
  const int hist = *reinterpret_cast<volatile int *>(lv.hist_len + slice);
  if (slice_budget != nullptr) budget = slice_budget[slice];
  const float row_lse = policy == 0 && lse != nullptr && tid < w ? lse[(size_t)slice * w + tid] : 0.f;
  if (tid < lv.pages_per_slice) pt[tid] = page;
  for (int i = tid + NT; i < lv.pages_per_slice; i += NT) pt[i] = __ldg(pages + i);
  if (policy == 0 && lse != nullptr && tid < w) lse_row[tid] = row_lse;
  const int L = hist + wa.n_k;
  if (dev_status != 0 || outgrown(lv, L)) return;   // a failed check, an earlier kernel's or this one's: leave the store alone
  __syncthreads();
  if (policy == 0 && lse == nullptr) {
    if (L > kSumsInCompress) {                 // (no caller asks for it)
      if (tid == 0) atomicExch(lv.status, kDevCheck);
      return;
    }
    // The rows' log-sum-exps, a warp a row at a time, to the bit those of row_lse_kernel: there a thread takes the exponential of one entry (of
    // up to 1 024), a warp adds its threads' crosswise and one thread the warps' in turn.
    const int mine = L - lane;                 // (this lane's entries are 32 u, 32 u below it)
    for (int j = wid; j < w; j += NT / 32) {
      const float *y = logits + ((size_t)slice * w + j) * ld_l + lane;
      float x[kSumsInCompress / 32], top = -INFINITY, sum = 0.f;
#pragma unroll
      for (int u = 0; u < kSumsInCompress / 32; ++u) x[u] = 32 * u < mine ? __ldg(y + 32 * u) : -INFINITY;
#pragma unroll
      for (int u = 0; u < kSumsInCompress / 32; ++u) top = fmaxf(top, x[u]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
#pragma unroll
      for (int u0 = 0; u0 < kSumsInCompress / 32; u0 += 4) {
        if (32 * u0 >= L) break;
#pragma unroll
        for (int u = u0; u < u0 + 4; ++u) x[u] = 32 * u < mine ? exp2f(x[u] - top) : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int u = u0; u < u0 + 4; ++u) x[u] += __shfl_xor_sync(0xffffffffu, x[u], o);
#pragma unroll
        for (int u = u0; u < u0 + 4; ++u) sum += x[u];
      }
      if (lane == 0) lse_row[j] = top + log2f(sum);
    }
    __syncthreads();
  }
  auto row_of = [&](int slot) { return ((size_t)pt[slot >> lv.page_shift] << lv.page_shift) + (size_t)(slot & lv.page_mask); };
  const long long ext_base = ext.on ? (long long)(slice / lv.n_heads) * ext.sb + (long long)(slice % lv.n_heads) * ext.sh : 0;

  // ---- phase 1: keys
  uint32_t lowest = 0xffffffffu, highest = 0u;
  if (policy == 0) {
    float *sc_out = scores + (size_t)slice * ld_s;
    // columns of a logit row: the history's, then the current map's from map_col on
    const int map_col = tile_padded ? (hist + 127) & ~127 : hist, cols = map_col + wa.n_k;
    const float inv_w = 1.f / (float)w;
    const float *y = logits + (size_t)slice * w * ld_l;
    for (int c0 = tid * 2; c0 < cols; c0 += NT * 2) {
      float s0 = 0.f, s1 = 0.f;
      int j = 0;
      for (; j + 16 <= w; j += 16) {             // (a window of 16: one round of loads)
        float2 t[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) t[e] = __ldg(reinterpret_cast<const float2 *>(y + (size_t)(j + e) * ld_l + c0));
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          s0 += exp2f(fmaf(t[e].x, logit_scale, -lse_row[j + e]));
          s1 += exp2f(fmaf(t[e].y, logit_scale, -lse_row[j + e]));
        }
      }
#pragma unroll 4
      for (; j < w; ++j) {
        const float2 t = __ldg(reinterpret_cast<const float2 *>(y + (size_t)j * ld_l + c0));
        s0 += exp2f(fmaf(t.x, logit_scale, -lse_row[j]));
        s1 += exp2f(fmaf(t.y, logit_scale, -lse_row[j]));
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int col = c0 + e;
        const int i = col < hist ? col : (col >= map_col && col < cols ? col - map_col + hist : -1);   // (the padding between them is nobody's)
        if (i >= 0) {
          const float sc = (e == 0 ? s0 : s1) * inv_w;
          const uint32_t k = __float_as_uint(sc) & 0x7FFFFFFFu;
          sc_out[i] = sc;
          key[i] = k;
          lowest = min(lowest, k);
          highest = max(highest, k);
        }
      }
    }
    __syncthreads();
    if (pool > 1) {
      lowest = 0xffffffffu; highest = 0u;
      for (int i = tid; i < L; i += NT) {
        const uint32_t k = pooled_key(reinterpret_cast<const float *>(key), i, L, pool);
        list[i] = (int)k;
        lowest = min(lowest, k);
        highest = max(highest, k);
      }
      __syncthreads();
      for (int i = tid; i < L; i += NT) key[i] = (uint32_t)list[i];
      __syncthreads();
    }
    if (tid < w) key[hist + (wa.all ? tid : wa.pos[tid])] = kWindowKey;
  } else {
    for (int i = tid; i < L; i += NT) {
      const int pos = i >= hist ? wa.n_prev + (i - hist) : lv.pos_pool[row_of(i)];
      key[i] = pos < n_sink ? kWindowKey : (uint32_t)pos + 1u;
      if (pos >= n_sink) { lowest = min(lowest, (uint32_t)pos + 1u); highest = max(highest, (uint32_t)pos + 1u); }
    }
  }

  // ---- phase 2: selection
  int want;
  const int kept = select_and_emit<NT>(key, L, budget, lowest, highest, list, sh, &want);
  if (kept != want) {                          // the count rule of the selection (block-uniform)
    if (tid == 0) atomicExch(lv.status, kDevCheck);
    return;
  }
  __syncthreads();

  // ---- phase 3: in-place gather of K, V and pos (a row of K or V is 256 bytes for either data type)
  int lo = min(sh.first_gap, kept);            // first j with keep[j] != j
  if (ext.on && lo > hist) lo = hist;          // kept rows of the current map are not where they belong yet, whatever their index
  const int piece = lane;                      // of a row's 32 16-byte pieces (16 of K, 16 of V)
  const char *ext_ptr = (piece < 16 ? ext.k : ext.v) + (piece & 15) * 16;
  char *pool_ptr = (piece < 16 ? lv.k_pool : lv.v_pool) + (piece & 15) * 16;
  // Chunks of 128 rows, eight to a warp; a lane looks up where one row of four chunks comes from and goes, and the warp learns it
  // by shuffles (16 slices, 1 944 rows: 61 700 -> 51 100 cycles, 26 a row; look-ups by every lane for every row cost as many issue slots
  // as the copies take).  Copies of the next chunk under the stores of this one, in registers or by cp.async, gave nothing: loads
  // queue behind the stores.
  constexpr int kUnits = 8, C = kUnits * NT / 32;
  for (int j0 = lo; j0 < kept; j0 += NT) {
    const int mine = j0 + (lane / kUnits) * C + wid * kUnits + lane % kUnits;
    unsigned long long from = 0;               // offset of the row in its array; odd: in the caller's
    unsigned to = 0;
    int pos = 0;
    if (mine < kept) {
      const int src = list[mine];
      to = (unsigned)row_of(mine);
      if (ext.on && src >= hist) {
        from = (unsigned long long)((ext_base + (long long)(src - hist) * ext.st) * ext.esize) + 1;
        pos = wa.n_prev + (src - hist);
      } else {
        const size_t row = row_of(src);
        from = (unsigned long long)row * 256;
        pos = lv.pos_pool[row];
      }
    }
#pragma unroll 1
    for (int e = 0; e < 32 / kUnits && j0 + e * C < kept; ++e) {
      const int n = kept - (j0 + e * C + wid * kUnits);      // rows of this warp in the chunk, if less than kUnits
      uint4 buf[kUnits];
#pragma unroll
      for (int u = 0; u < kUnits; ++u) {
        const unsigned long long f = __shfl_sync(0xffffffffu, from, e * kUnits + u);
        if (u < n) buf[u] = __ldcg(reinterpret_cast<const uint4 *>(f & 1 ? ext_ptr + (f - 1) : pool_ptr + f));
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < kUnits; ++u) {
        const unsigned t = __shfl_sync(0xffffffffu, to, e * kUnits + u);
        if (u < n) *reinterpret_cast<uint4 *>(pool_ptr + (size_t)t * 256) = buf[u];
      }
      if (e == 0 && mine < kept) lv.pos_pool[to] = pos;      // (of all four chunks: their sources have been read)
    }
  }
  if (tid == 0) {
    lv.next_len[slice] = kept;
    kept_count[slice] = kept;
  }
}

// ------------------------------------------------------------------------------------------
// layer statistics (Eq. 2): for sampled query rows i of the current map, alpha_i = softmax row over all L
// entries, c_i = mass on the current map, t_i = sum of the K' largest alpha_ij over the history.
// A CTA of 256 threads owns 64 sampled rows of one slice and streams a range of the slice's keys in tiles of
// 64, so a key tile is read once for 64 rows.  Per tile: logits by fp32 FMA (thread (ty, tx) owns rows
// ty + 16 i, columns tx + 16 j), staged in shared memory; then four threads per row, 16 columns each, fold the
// tile into the row's running maximum, normaliser and current-map mass (online softmax statistics) and into
// their own descending list of the K' largest history logits seen in their columns (the K' largest weights
// are the K' largest logits).  Nothing of length L is kept.  At the end one thread per row merges the four
// lists (K' steps of a four-way merge).
// The calibration runs few slices (one image), so the keys of a slice are split over gridDim.z CTAs to fill
// the GPU: with one split the block adds its rows' c_i and t_i to the accumulators itself; with several every
// CTA writes, per row, (maximum, normaliser, current mass, K' largest logits) to `partial` and
// layer_stats_merge_kernel combines the splits.
// acc: per slice the sums of c_i and t_i over the sampled rows, and the slice's length.
// (This kernel serves f32 and K' > 16; see stats_mma_kernel.)
// grid (ceil(n_rows / 64), n_slices, n_split); dynamic shared memory: layer_stats_smem_bytes<D>(K').
// ------------------------------------------------------------------------------------------
template <int D> __host__ __device__ constexpr size_t layer_stats_smem_bytes(int topk) {
  return (size_t)(2 * 64 * (D + 4) + 64 * 65 + 64 + 256 * (topk > 0 ? topk : 1)) * 4;
}
constexpr int kStatsRec = 4 + 64;        // floats per (split, row) record: m, z, cur, unused, then up to 64 logits

__device__ __forceinline__ void stats_block_accumulate(float c_i, float t_i, double *acc, float *red_c, float *red_t) {
  const int tid = threadIdx.x;
  for (int o = 16; o > 0; o >>= 1) {
    c_i += __shfl_xor_sync(0xffffffffu, c_i, o);
    t_i += __shfl_xor_sync(0xffffffffu, t_i, o);
  }
  if ((tid & 31) == 0) { red_c[tid >> 5] = c_i; red_t[tid >> 5] = t_i; }
  __syncthreads();
  if (tid == 0) {
    float cs = 0.f, ts = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { cs += red_c[w]; ts += red_t[w]; }   // fixed order
    atomicAdd(&acc[3 * blockIdx.y], (double)cs);
    atomicAdd(&acc[3 * blockIdx.y + 1], (double)ts);
  }
}

template <typename T, int D>
__global__ void __launch_bounds__(256) layer_stats_kernel(LayerView lv, TensorView Q, int n_k, int n_prev, int stride, int n_rows,
                                                          int topk_prime, float scale, double *acc, float *partial) {
  constexpr int LD = D + 4, LDS = 65;
  constexpr int CH = D * (int)sizeof(T) / 16;
  constexpr int VN = Vec16<T>::N;
  extern __shared__ float smem[];
  float *Qs = smem;                    // [64][LD]
  float *Ks = Qs + 64 * LD;            // [64][LD]
  float *Ss = Ks + 64 * LD;            // [64][LDS] scaled logits of the tile
  int *is_cur = reinterpret_cast<int *>(Ss + 64 * LDS);   // [64] the tile's entries that belong to the current map
  float *top = reinterpret_cast<float *>(is_cur + 64);    // [256][K'] per-thread descending lists
  __shared__ float red_c[8], red_t[8];
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int slice = blockIdx.y;
  const int b = slice / lv.n_heads, h = slice % lv.n_heads;
  const int L = lv.hist_len[slice] + n_k;
  if (outgrown(lv, L)) return;
  if (tid == 0 && blockIdx.x == 0 && blockIdx.z == 0) acc[3 * slice + 2] = (double)L;
  const int r0 = blockIdx.x * 64;
  const int Kp = topk_prime;
  const int n_split = gridDim.z;
  const int tiles = (L + 63) >> 6;
  const int t_lo = (int)((long long)tiles * blockIdx.z / n_split), t_hi = (int)((long long)tiles * (blockIdx.z + 1) / n_split);
  for (int idx = tid; idx < 64 * CH; idx += 256) {
    const int r = idx / CH, c = idx % CH;
    float v[VN];
    if (r0 + r < n_rows) {
      Vec16<T>::load(row_ptr<T>(Q, b, h, (r0 + r) * stride) + c * VN, v);
    } else {
#pragma unroll
      for (int e = 0; e < VN; ++e) v[e] = 0.f;
    }
#pragma unroll
    for (int e = 0; e < VN; ++e) Qs[r * LD + c * VN + e] = v[e];
  }
  const int Ks_ = Kp > 0 ? Kp : 1;
  float *mine = top + (size_t)tid * Ks_;
  for (int e = 0; e < Kp; ++e) mine[e] = -INFINITY;
  // row statistics of the 4 threads that share a row (row = tid >> 2): kept redundantly in each of them
  const int row = tid >> 2, part = tid & 3;
  float m_run = -INFINITY, z_run = 0.f, cur_run = 0.f;
  float thr = Kp > 0 ? -INFINITY : INFINITY;           // the smallest member of this thread's list (nothing enters when K' = 0)
  // the next key tile (and its positions) travels from global memory into registers while the current one is worked on
  constexpr int PIECES = 64 * CH / 256;                // 16-byte pieces of a tile per thread
  uint4 nxt[PIECES];
  int nxt_pos = 0;
  auto fetch = [&](int t) {
    const int j0 = t << 6;
#pragma unroll
    for (int u = 0; u < PIECES; ++u) {
      const int idx = tid + u * 256, r = idx / CH, c = idx % CH;
      nxt[u] = make_uint4(0u, 0u, 0u, 0u);
      if (j0 + r < L) nxt[u] = reinterpret_cast<const uint4 *>(lv.k_pool + slot_row(lv, slice, j0 + r) * lv.row_bytes)[c];
    }
    if (tid < 64) nxt_pos = (j0 + tid < L) ? lv.pos_pool[slot_row(lv, slice, j0 + tid)] : -1;
  };
  if (t_lo < t_hi) fetch(t_lo);
  for (int t = t_lo; t < t_hi; ++t) {
    const int j0 = t << 6;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < PIECES; ++u) {
      const int idx = tid + u * 256, r = idx / CH, c = idx % CH;
      float v[VN];
      Vec16<T>::load(reinterpret_cast<const T *>(&nxt[u]), v);
#pragma unroll
      for (int e = 0; e < VN; e += 4)                  // 16-byte stores (LD and VN are multiples of 4)
        *reinterpret_cast<float4 *>(&Ks[r * LD + c * VN + e]) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
    }
    if (tid < 64) is_cur[tid] = nxt_pos >= n_prev ? 1 : 0;
    __syncthreads();
    if (t + 1 < t_hi) fetch(t + 1);
    float s[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) s[i][j] = 0.f;
#pragma unroll 4
    for (int c = 0; c < D; c += 4) {
      float4 q[4], k[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) q[i] = *reinterpret_cast<const float4 *>(&Qs[(ty + 16 * i) * LD + c]);
#pragma unroll
      for (int j = 0; j < 4; ++j) k[j] = *reinterpret_cast<const float4 *>(&Ks[(tx + 16 * j) * LD + c]);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          s[i][j] = fmaf(q[i].x, k[j].x, s[i][j]);
          s[i][j] = fmaf(q[i].y, k[j].y, s[i][j]);
          s[i][j] = fmaf(q[i].z, k[j].z, s[i][j]);
          s[i][j] = fmaf(q[i].w, k[j].w, s[i][j]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        Ss[(ty + 16 * i) * LDS + tx + 16 * j] = (j0 + tx + 16 * j < L) ? s[i][j] * scale : -INFINITY;
    __syncthreads();
    {
      const float *srow = Ss + row * LDS + part * 16;
      float mx = -INFINITY;
#pragma unroll
      for (int e = 0; e < 16; ++e) mx = fmaxf(mx, srow[e]);
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      const float m_new = fmaxf(m_run, mx);            // finite: every tile holds at least one entry
      float sum = 0.f, cur = 0.f;
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        const float v = srow[e];
        const float pe = expf(v - m_new);              // 0 for the padding beyond L
        sum += pe;
        if (is_cur[part * 16 + e]) {
          cur += pe;
        } else if (v > thr) {                          // a history logit that enters this thread's K' largest
          int at = Kp - 1;
          while (at > 0 && mine[at - 1] < v) { mine[at] = mine[at - 1]; --at; }
          mine[at] = v;
          thr = mine[Kp - 1];
        }
      }
      sum += __shfl_xor_sync(0xffffffffu, sum, 1);
      sum += __shfl_xor_sync(0xffffffffu, sum, 2);
      cur += __shfl_xor_sync(0xffffffffu, cur, 1);
      cur += __shfl_xor_sync(0xffffffffu, cur, 2);
      const float a = expf(m_run - m_new);             // 0 at the first tile
      z_run = z_run * a + sum;
      cur_run = cur_run * a + cur;
      m_run = m_new;
    }
  }
  __syncthreads();
  float c_i = 0.f, t_i = 0.f;
  if (part == 0) {
    // four-way merge of the row's four descending lists: the K' largest history logits of this key range
    const float *l0 = top + (size_t)(tid + 0) * Ks_, *l1 = top + (size_t)(tid + 1) * Ks_;
    const float *l2 = top + (size_t)(tid + 2) * Ks_, *l3 = top + (size_t)(tid + 3) * Ks_;
    float *rec = nullptr;
    if (n_split > 1) {
      rec = partial + ((((size_t)slice * gridDim.x + blockIdx.x) * n_split + blockIdx.z) * 64 + row) * kStatsRec;
      rec[0] = m_run; rec[1] = z_run; rec[2] = cur_run;
    }
    int i0 = 0, i1 = 0, i2 = 0, i3 = 0;
    float tsum = 0.f;
    for (int e = 0; e < Kp; ++e) {
      const float v0 = i0 < Kp ? l0[i0] : -INFINITY, v1 = i1 < Kp ? l1[i1] : -INFINITY;
      const float v2 = i2 < Kp ? l2[i2] : -INFINITY, v3 = i3 < Kp ? l3[i3] : -INFINITY;
      const float best = fmaxf(fmaxf(v0, v1), fmaxf(v2, v3));
      if (rec) rec[4 + e] = best;                      // (-inf once the range's history is exhausted)
      if (best == -INFINITY) { if (!rec) break; else continue; }
      tsum += expf(best - m_run);
      if (best == v0) ++i0; else if (best == v1) ++i1; else if (best == v2) ++i2; else ++i3;
    }
    if (r0 + row < n_rows) { c_i = cur_run / z_run; t_i = tsum / z_run; }
  }
  if (n_split == 1) stats_block_accumulate(c_i, t_i, acc, red_c, red_t);
}

// Combines the key-range splits of layer_stats_kernel: per row the maxima, normalisers and current masses by
// the usual rescaling, the K' largest history logits by an n_split-way merge of the splits' descending lists.
// grid (ceil(n_rows / 64), n_slices), 64 threads, one row per thread.
__global__ void __launch_bounds__(64) layer_stats_merge_kernel(const float *partial, int n_split, int n_rows, int topk_prime,
                                                               double *acc) {
  __shared__ float red_c[2], red_t[2];
  const int row = threadIdx.x;
  const float *base = partial + (((size_t)blockIdx.y * gridDim.x + blockIdx.x) * n_split * 64 + row) * kStatsRec;
  const size_t step = (size_t)64 * kStatsRec;          // from one split's record of this row to the next
  float m = -INFINITY;
  for (int s = 0; s < n_split; ++s) m = fmaxf(m, base[s * step]);
  float z = 0.f, cur = 0.f;
  for (int s = 0; s < n_split; ++s) {
    const float a = expf(base[s * step] - m);
    z += base[s * step + 1] * a;
    cur += base[s * step + 2] * a;
  }
  int head[16];
  for (int s = 0; s < 16; ++s) head[s] = 0;
  float tsum = 0.f;
  for (int e = 0; e < topk_prime; ++e) {
    float best = -INFINITY;
    int who = -1;
    for (int s = 0; s < n_split; ++s) {
      const float v = head[s] < topk_prime ? base[s * step + 4 + head[s]] : -INFINITY;
      if (v > best) { best = v; who = s; }
    }
    if (who < 0) break;                                // history exhausted
    tsum += expf(best - m);
    ++head[who];
  }
  float c_i = 0.f, t_i = 0.f;
  if (blockIdx.x * 64 + row < n_rows) { c_i = cur / z; t_i = tsum / z; }
  stats_block_accumulate(c_i, t_i, acc, red_c, red_t);
}

// ------------------------------------------------------------------------------------------
// layer statistics, bf16 x 128 and K' <= 16.  The same quantities as above; a CTA of 256 threads owns 64 sampled rows of one
// slice and a range of its keys in tiles of 64.  Warp (wr, wc) takes rows 16 wr .. and keys 32 wc .. of a tile by tensor-core
// products (m16n8k16), and every thread keeps, for the two rows of which it holds scores, its own maximum, normaliser,
// current-map mass and descending list of the 16 largest history logits in registers: nothing is exchanged before the end,
// when the four lanes and two warps of a row, and in the CTA that finishes last the key ranges, merge their lists pair by pair.
// Entries hist .. L-1 of a slice are the current map.  Logits are kept in base 2.
// The work is small (a calibration pass of one image: 70 GF, 0.3 G weights); what bounds it is the instructions per weight - an
// exponential, an insertion where a list grows - and, at the small scales, the latency of a call.  Tensor-core products by
// m16n8k16 leave the scores in registers and are a tenth of that time, so a TMEM pipeline would not shorten it.
// One layer's 13 scales, one image, 16 slices: 2 048 us with the kernels above, 485 us here (4 096 queries, every 16th of them,
// 10 521 keys: 921 + 19 -> 111 + 16 us); a call at the small scales 67 -> 32 us, sums in page-locked memory among the causes. A pass of four layers 2 708 -> 2 145 us
// since small maps are read where they are and the sums are watched (see the launch).
// map_outside: the current map is still in the caller's tensors.  Its keys are read there, and CTAs of their own (blockIdx.z >=
// n_split) copy its rows into the pages meanwhile.
// sums (host memory, which the caller watches): per slice and block of rows the sums of c_i and t_i, then the slices' lengths, then a
// word per copying CTA.  counters: one per slice and block of rows, zero before and after.
// grid (ceil(n_rows / 64), n_slices, n_split <= 16 and as many again as copy); static shared memory: two K tiles and the query tile.
// ------------------------------------------------------------------------------------------
constexpr int kTop = 16;

__device__ __forceinline__ float pow2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void order(float &a, float &b) {
  const float hi = fmaxf(a, b);
  b = fminf(a, b);
  a = hi;
}
// eight values into descending order (odd-even merge sort)
__device__ __forceinline__ void sort8(float *v) {
#pragma unroll
  for (int i = 0; i < 8; i += 2) order(v[i], v[i + 1]);
#pragma unroll
  for (int i = 0; i < 8; i += 4) { order(v[i], v[i + 2]); order(v[i + 1], v[i + 3]); order(v[i + 1], v[i + 2]); }
#pragma unroll
  for (int i = 0; i < 4; ++i) order(v[i], v[i + 4]);
  order(v[2], v[4]); order(v[3], v[5]);
  order(v[1], v[2]); order(v[3], v[4]); order(v[5], v[6]);
}
// a bitonic list into descending order
__device__ __forceinline__ void order_bitonic(float *a) {
#pragma unroll
  for (int d = kTop / 2; d > 0; d >>= 1)
#pragma unroll
    for (int i = 0; i < kTop; ++i)
      if ((i & d) == 0) order(a[i], a[i + d]);
}
// the kTop largest of two descending lists, descending
__device__ __forceinline__ void merge_top(float *a, const float *b) {
#pragma unroll
  for (int i = 0; i < kTop; ++i) a[i] = fmaxf(a[i], b[kTop - 1 - i]);
  order_bitonic(a);
}
struct RowStats {
  float m, z, cur, top[kTop];
  __device__ __forceinline__ void clear() {
    m = kNoMax; z = 0.f; cur = 0.f;
#pragma unroll
    for (int i = 0; i < kTop; ++i) top[i] = -INFINITY;
  }
  __device__ __forceinline__ void merge(float m2, float z2, float cur2, const float *top2) {
    const float mm = fmaxf(m, m2), f = pow2(m - mm), f2 = pow2(m2 - mm);
    z = z * f + z2 * f2;
    cur = cur * f + cur2 * f2;
    m = mm;
    merge_top(top, top2);
  }
  // with the lane `mask` away
  __device__ __forceinline__ void merge_lane(int mask) {
    float t[kTop];
#pragma unroll
    for (int i = 0; i < kTop; ++i) t[i] = __shfl_xor_sync(0xffffffffu, top[i], mask);
    const float m2 = __shfl_xor_sync(0xffffffffu, m, mask), z2 = __shfl_xor_sync(0xffffffffu, z, mask);
    const float cur2 = __shfl_xor_sync(0xffffffffu, cur, mask);
    merge(m2, z2, cur2, t);
  }
};
// Rows part, part + parts, .. (in blocks of 128) of a bf16 map: K, V and positions to the pages.  256 threads, 16 pieces of 16 bytes in
// flight per thread.
__device__ __forceinline__ void copy_map_rows(const LayerView &lv, const TensorView &K, const TensorView &V, int slice, int hist, int n_k,
                                              int n_prev, int part, int parts) {
  const int b = slice / lv.n_heads, h = slice % lv.n_heads, c = threadIdx.x & 15, r = threadIdx.x >> 4;
  for (int r0 = part * 128; r0 < n_k; r0 += parts * 128) {
    uint4 x[2][8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = r0 + u * 16 + r;
      if (i >= n_k) continue;
      x[0][u] = __ldcs(reinterpret_cast<const uint4 *>(row_ptr<__nv_bfloat16>(K, b, h, i)) + c);
      x[1][u] = __ldcs(reinterpret_cast<const uint4 *>(row_ptr<__nv_bfloat16>(V, b, h, i)) + c);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int i = r0 + u * 16 + r;
      if (i >= n_k) continue;
      const size_t row = slot_row(lv, slice, hist + i);
      reinterpret_cast<uint4 *>(lv.k_pool + row * 256)[c] = x[0][u];
      reinterpret_cast<uint4 *>(lv.v_pool + row * 256)[c] = x[1][u];
      if (c == 0) lv.pos_pool[row] = n_prev + i;
    }
  }
}
constexpr int kStatsRec16 = 4 + kTop;    // floats per (split, row) record: m, z, cur, unused, the list

__global__ void __launch_bounds__(256, 2) stats_mma_kernel(LayerView lv, TensorView Q, int n_k, int stride, int n_rows, int topk_prime,
                                                           float scale_log2e, float *partial, int *counters, double *sums, int n_split,
                                                           TensorView mapK, TensorView mapV, int map_outside, int n_prev) {
  __shared__ __align__(128) uint8_t sm[3 * 64 * 256];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wr = warp & 3, wc = warp >> 2;
  const int slice = blockIdx.y, b = slice / lv.n_heads, h = slice % lv.n_heads;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int hist = lv.hist_len[slice], L = hist + n_k;
  const bool copies = (int)blockIdx.z >= n_split;
  const int parts = ((int)gridDim.z - n_split) * gridDim.x, part = ((int)blockIdx.z - n_split) * (int)gridDim.x + (int)blockIdx.x;
  double *copied = sums + ((size_t)2 * gridDim.x + 1) * gridDim.y + (size_t)slice * parts + part;
  if (outgrown(lv, L)) {
    // (an answer all the same, and every word of it by one CTA: behind the last of them the host may prepare the words for another call)
    if (tid < 2 && blockIdx.z == 0) sums[((size_t)slice * gridDim.x + blockIdx.x) * 2 + tid] = NAN;
    if (tid == 2 && blockIdx.z == 0 && blockIdx.x == 0) sums[(size_t)2 * gridDim.x * gridDim.y + slice] = NAN;
    if (tid == 3 && copies) *copied = NAN;
    return;
  }
  if (copies) {
    copy_map_rows(lv, mapK, mapV, slice, hist, n_k, n_prev, part, parts);
    __syncthreads();
    if (tid == 0) {                      // (the caller may change the tensors when the call returns: what the CTA has done comes first)
      __threadfence_system();
      *copied = 0.0;
    }
    return;
  }
  const int r0 = blockIdx.x * 64;
  const int tiles = (L + 63) >> 6;
  const int t_lo = (int)((long long)tiles * blockIdx.z / n_split), t_hi = (int)((long long)tiles * (blockIdx.z + 1) / n_split);
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(sm);
  // 16-byte piece c of row r of a 64 x 256-byte tile
  auto at = [&](int tile, int r, int c) { return base + (uint32_t)(tile * 16384 + r * 256 + ((c ^ (r & 7)) << 4)); };
  auto fetch = [&](int t) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = u * 16 + (tid >> 4), c = tid & 15, slot = t * 64 + r;
      if (slot < L) {
        const char *src = map_outside && slot >= hist ? reinterpret_cast<const char *>(row_ptr<__nv_bfloat16>(mapK, b, h, slot - hist))
                                                      : lv.k_pool + slot_row(lv, slice, slot) * 256;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(at(t & 1, r, c)), "l"(src + c * 16) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = u * 16 + (tid >> 4), c = tid & 15;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (r0 + r < n_rows) v = reinterpret_cast<const uint4 *>(row_ptr<__nv_bfloat16>(Q, b, h, (r0 + r) * stride))[c];
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at(2, r, c)), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
  }
  if (t_lo < t_hi) fetch(t_lo);
  // What the next scale finds.  It is read by kernels of this device behind this one, and stored here so that the fences around the counter below
  // lie between it and the length's word for the host; a fence of its own for the whole system cost a call 1.2 us here and 4.4 us behind the sums.
  if (tid == 0 && blockIdx.x == 0 && blockIdx.z == 0) lv.next_len[slice] = L;
  __syncthreads();
  uint32_t qa[8][4];                     // the warp's 16 query rows, 8 steps of 16 columns
#pragma unroll
  for (int k = 0; k < 8; ++k)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(qa[k][0]), "=r"(qa[k][1]), "=r"(qa[k][2]), "=r"(qa[k][3])
                 : "r"(at(2, wr * 16 + (lane & 15), 2 * k + (lane >> 4))));
  RowStats st[2];
  st[0].clear();
  st[1].clear();
  const bool idle = r0 + wr * 16 >= n_rows;            // (such a warp only helps to load)
  for (int t = t_lo; t < t_hi; ++t) {
    if (t + 1 < t_hi) fetch(t + 1); else asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    if (idle) { __syncthreads(); continue; }
    float acc[4][4];
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
#pragma unroll
      for (int n = 0; n < 4; n += 2) {
        uint32_t kb[4];                  // two groups of 8 keys, each with both halves of the 16 columns
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(kb[0]), "=r"(kb[1]), "=r"(kb[2]), "=r"(kb[3])
                     : "r"(at(t & 1, wc * 32 + n * 8 + (lane & 7) + ((lane >> 4) << 3), 2 * k + ((lane >> 3) & 1))));
#pragma unroll
        for (int g = 0; g < 2; ++g)
          asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                       : "+f"(acc[n + g][0]), "+f"(acc[n + g][1]), "+f"(acc[n + g][2]), "+f"(acc[n + g][3])
                       : "r"(qa[k][0]), "r"(qa[k][1]), "r"(qa[k][2]), "r"(qa[k][3]), "r"(kb[2 * g]), "r"(kb[2 * g + 1]));
      }
    }
    // acc[n][2 i + e] belongs to row lane / 4 + 8 i and key 8 n + 2 (lane % 4) + e of the warp's part
    const int j0 = t * 64 + wc * 32 + 2 * (lane & 3);
    const bool ragged = t * 64 + 64 > L, any_hist = t * 64 < hist, any_cur = t * 64 + 64 > hist;     // (the same for all threads)
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      RowStats &s = st[i];
      float y[8], mx = kNoMax;
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float v = acc[n][2 * i + e] * scale_log2e;
          if (ragged && j0 + 8 * n + e >= L) v = -INFINITY;
          y[2 * n + e] = v;
          mx = fmaxf(mx, v);
        }
      const float m_new = fmaxf(s.m, mx), f = pow2(s.m - m_new);
      float sum = 0.f, cur = 0.f;
#pragma unroll
      for (int n = 0; n < 4; ++n)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float p = pow2(y[2 * n + e] - m_new);
          sum += p;
          if (any_cur && j0 + 8 * n + e >= hist) cur += p;
        }
      s.z = s.z * f + sum;
      s.cur = s.cur * f + cur;
      s.m = m_new;
      if (any_hist) {
        float top = -INFINITY;
#pragma unroll
        for (int n = 0; n < 4; ++n)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            if (any_cur && j0 + 8 * n + e >= hist) y[2 * n + e] = -INFINITY;
            top = fmaxf(top, y[2 * n + e]);
          }
        if (__any_sync(0xffffffffu, top > s.top[kTop - 1])) {        // eight at a time: 14 operations a weight, 32 one by one
          sort8(y);
#pragma unroll
          for (int q = 0; q < 8; ++q) s.top[8 + q] = fmaxf(s.top[8 + q], y[7 - q]);
          order_bitonic(s.top);
        }
      }
    }
    __syncthreads();                     // the tile has been read: its buffer is the next but one's
  }
  // the four lanes of a row, then its two warps
  float *ex = reinterpret_cast<float *>(sm);           // [64][kStatsRec16]: the K tiles are done with
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    st[i].merge_lane(1);
    st[i].merge_lane(2);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    float *e = ex + (wr * 16 + 8 * i + (lane >> 2)) * kStatsRec16;
    if (wc == 1 && (lane & 3) == 0) {
      e[0] = st[i].m; e[1] = st[i].z; e[2] = st[i].cur;
#pragma unroll
      for (int q = 0; q < kTop; ++q) e[4 + q] = st[i].top[q];
    }
  }
  __syncthreads();
  if (wc == 0) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int row = wr * 16 + 8 * i + (lane >> 2);
      const float *e = ex + row * kStatsRec16;
      float t2[kTop];
#pragma unroll
      for (int q = 0; q < kTop; ++q) t2[q] = e[4 + q];
      st[i].merge(e[0], e[1], e[2], t2);
      if ((lane & 3) == 0 && r0 + row < n_rows) {
        float4 *rec = reinterpret_cast<float4 *>(partial + (((size_t)slice * n_rows + r0 + row) * n_split + blockIdx.z) * kStatsRec16);
        rec[0] = make_float4(st[i].m, st[i].z, st[i].cur, 0.f);
#pragma unroll
        for (int q = 0; q < kTop / 4; ++q) rec[1 + q] = make_float4(st[i].top[4 * q], st[i].top[4 * q + 1], st[i].top[4 * q + 2], st[i].top[4 * q + 3]);
      }
    }
  }
  // The CTA that finishes a block of rows last merges the key ranges' records, sixteen lanes per row, a record each, and sums
  // c_i and t_i over the rows in a fixed order.
  int *last = reinterpret_cast<int *>(sm);
  __threadfence();
  __syncthreads();
  if (n_split > 1) {
    if (tid == 0) {
      int *count = counters + (size_t)slice * gridDim.x + blockIdx.x;
      const int before = atomicAdd(count, 1);
      *last = before == n_split - 1;
      if (before == n_split - 1) *count = 0;           // as the next launch wants to find it
    }
    __syncthreads();
    if (!*last) return;
    __threadfence();
  }
  const int l = tid & 15, n_here = min(64, n_rows - r0);
  double c_sum = 0.0, t_sum = 0.0;
  for (int row0 = 0; row0 < n_here; row0 += 16) {
    const int row = row0 + (tid >> 4);
    RowStats &s = st[0];
    s.clear();
    if (row < n_here && l < n_split) {
      const float4 *rec = reinterpret_cast<const float4 *>(partial + (((size_t)slice * n_rows + r0 + row) * n_split + l) * kStatsRec16);
      const float4 r = __ldcg(rec);
      s.m = r.x; s.z = r.y; s.cur = r.z;
#pragma unroll
      for (int q = 0; q < kTop / 4; ++q) {
        const float4 v = __ldcg(rec + 1 + q);
        s.top[4 * q] = v.x; s.top[4 * q + 1] = v.y; s.top[4 * q + 2] = v.z; s.top[4 * q + 3] = v.w;
      }
    }
    for (int d = 1; d < n_split; d <<= 1) s.merge_lane(d);
    if (l == 0 && row < n_here) {
      float t = 0.f;
#pragma unroll
      for (int q = 0; q < kTop; ++q)
        if (q < topk_prime) t += pow2(s.top[q] - s.m);
      c_sum += (double)(s.cur / s.z);
      t_sum += (double)(t / s.z);
    }
  }
  double *red = reinterpret_cast<double *>(sm + 64);   // [2][16]
  if (l == 0) { red[tid >> 4] = c_sum; red[16 + (tid >> 4)] = t_sum; }
  __syncthreads();
  // (A word stands for itself and for inputs that have been read, by loads whose values are in it.  The length above has its fence behind it.)
  if (tid < 32) {                        // half a warp sums the c_i, half the t_i
    double v = red[tid];
    for (int d = 8; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    double *out = sums + ((size_t)slice * gridDim.x + blockIdx.x) * 2;
    if (l == 0) out[tid >> 4] = v;
    __threadfence_system();              // (on its way at once: the host is watching)
  }
  if (blockIdx.x == 0 && tid == 32) {
    sums[(size_t)2 * gridDim.x * gridDim.y + slice] = (double)L;
    __threadfence_system();
  }
}

}  // namespace scalekv
