// Per-(request, head) top-k with the window appended (Algorithm 1 (k, TopK and window append)).
//
// Radix select on an order-preserving 32-bit image of the fp32 score, 11+11+10
// bits from the top: the exact k-th largest key is found; every token with a
// larger key is kept, and of the tokens equal to it the lowest-indexed fill the
// remainder.  Two forms.  Segments of up to 256 K scores go to one CTA each in a
// single launch (second half of this file) wherever an estimate of both forms' times
// says so (one_cta_is_faster).  The others are cut into tiles of 4096 scores,
// one 256-thread CTA per tile with its 16 scores per thread in registers, and
// into five short kernels that meet only through global memory:
//
//   digit 1 histogram -> pick + digit 2 histogram -> pick + digit 3 histogram
//   -> pick + per-tile counts of larger / equal keys -> ordered emit
//
// Every CTA of a kernel repeats the (cheap) pick of the previous digit from the
// segment's global histogram, so no kernel waits for another CTA, and no CTA
// needs a neighbour on a particular SM: the kernels run on whatever SMs a
// concurrently running persistent kernel leaves free.  The emit writes the kept
// indices in ascending order, followed by T .. n-1.
#include <math.h>

#include "asl_internal.cuh"

namespace {

constexpr int THREADS = 256;
constexpr int PER_THREAD = 16;
constexpr int TILE = THREADS * PER_THREAD;    // scores per CTA
constexpr int BINS = 2048;
constexpr int STATE_INTS = 8;                 // per segment: prefix/remaining after each digit
constexpr int SEG_INTS = 3 * BINS + STATE_INTS;

__device__ __forceinline__ uint32_t asc_key(float s) {
  uint32_t u = __float_as_uint(s);
  if (u == 0x80000000u) u = 0;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

struct TopkArgs {
  const float* scores;
  const AslReq* req;
  int32_t* scratch;      // [segments][SEG_INTS]
  int32_t* counts;       // [segments][max_tiles][2]
  int32_t* idx_out;
  int64_t sum_T, sum_kept;
  int32_t n_heads, max_tiles, max_T;
  const asl_stat* gate;  // null, or: only requests whose statistic selected at layer `gate_layer` are worked on
  int32_t gate_layer;
  const asl_stat* latch; // null, or: requests that finished before layer `cur_layer` are left alone
  int32_t cur_layer;
};

struct Segment {
  const float* row;
  int32_t* hist;         // three tables of BINS
  int32_t* state;
  int32_t* counts;
  int32_t* out;
  int T, k, kept, tile;
  bool open;             // false: the gate keeps this request's list as it is
};

__device__ __forceinline__ Segment segment_of(const TopkArgs& a) {
  const int b = blockIdx.z, h = blockIdx.y;
  const AslReq rq = a.req[b];
  const int64_t seg = (int64_t)b * a.n_heads + h;
  Segment s;
  s.open = !a.gate || (a.gate[b].selected && a.gate[b].layer_idx == a.gate_layer);
  if (a.latch && asl_finished(a.latch + b, a.cur_layer)) s.open = false;
  s.row = a.scores + (int64_t)h * a.sum_T + rq.t_off;
  s.hist = a.scratch + seg * SEG_INTS;
  s.state = s.hist + 3 * BINS;
  s.counts = a.counts + seg * a.max_tiles * 2;
  s.out = a.idx_out + (int64_t)h * a.sum_kept + rq.kept_off;
  s.T = rq.T; s.k = rq.k; s.kept = rq.kept; s.tile = blockIdx.x;
  return s;
}

__device__ __forceinline__ void load_keys(const Segment& s, uint32_t (&key)[PER_THREAD]) {
  const int i0 = s.tile * TILE + threadIdx.x * PER_THREAD;
  if (i0 + PER_THREAD <= s.T && ((reinterpret_cast<uintptr_t>(s.row + i0) & 15) == 0)) {
#pragma unroll
    for (int q = 0; q < PER_THREAD / 4; ++q) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(s.row + i0) + q);
      key[4 * q] = asc_key(v.x); key[4 * q + 1] = asc_key(v.y); key[4 * q + 2] = asc_key(v.z); key[4 * q + 3] = asc_key(v.w);
    }
  } else {
#pragma unroll
    for (int e = 0; e < PER_THREAD; ++e) key[e] = (i0 + e < s.T) ? asc_key(__ldg(s.row + i0 + e)) : 0u;
  }
}

// The bin (counted from the top) that holds the `remaining`-th largest key of a
// table of `bins` counts, and how many keys of that bin are still wanted.
// Thread t owns the bins/THREADS bins just below bins-1-t*(bins/THREADS).
template <int PER>
__device__ __forceinline__ void pick(const int32_t* __restrict__ table, int remaining, int& bin, int& rem_out) {
  __shared__ int warp_tot[THREADS / 32];
  __shared__ int found[2];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int top = PER * THREADS - 1 - PER * tid;       // highest bin of this thread
  int c[PER];
  int sum = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) { c[j] = __ldcg(table + top - j); sum += c[j]; }
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  int above = incl - sum;                              // keys in bins above this thread's
  for (int w2 = 0; w2 < wid; ++w2) above += warp_tot[w2];
  if (above < remaining && remaining <= above + sum) {
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      if (above < remaining && remaining <= above + c[j]) { found[0] = top - j; found[1] = remaining - above; }
      above += c[j];
    }
  }
  __syncthreads();
  bin = found[0];
  rem_out = found[1];
  __syncthreads();
}

// counts the digit (key >> shift) & dmask of the keys whose bits under `mask` equal `prefix`
__device__ __forceinline__ void tile_histogram(const Segment& s, const uint32_t (&key)[PER_THREAD], uint32_t mask,
                                               uint32_t prefix, int shift, uint32_t dmask, int32_t* __restrict__ table) {
  __shared__ int hist[BINS];
  const int tid = threadIdx.x;
  for (int i = tid; i < BINS; i += THREADS) hist[i] = 0;
  __syncthreads();
  const int i0 = s.tile * TILE + tid * PER_THREAD;
  int run_bin = -1, run = 0;                           // neighbouring scores often share a digit: one atomic per run
#pragma unroll
  for (int e = 0; e < PER_THREAD; ++e) {
    const bool in = (i0 + e < s.T) && ((key[e] & mask) == prefix);
    const int d = (int)((key[e] >> shift) & dmask);
    if (in && d == run_bin) { ++run; continue; }
    if (run) atomicAdd(&hist[run_bin], run);
    run_bin = in ? d : -1;
    run = in ? 1 : 0;
  }
  if (run) atomicAdd(&hist[run_bin], run);
  __syncthreads();
  for (int i = tid; i < BINS; i += THREADS) {
    const int v = hist[i];
    if (v) atomicAdd(table + i, v);
  }
}

// stage 0: digit 1 histogram; stage 1 / 2: pick the previous digit, histogram the next
template <int STAGE>
__global__ void __launch_bounds__(THREADS) topk_digit_kernel(TopkArgs a) {
  pdl_release_successor();
  const Segment s = segment_of(a);
  if (!s.open || s.k == 0 || s.tile * TILE >= s.T) return;
  uint32_t key[PER_THREAD];
  load_keys(s, key);                      // the scores were complete before the first of these kernels started
  pdl_wait_predecessor();
  if (STAGE == 0) {
    tile_histogram(s, key, 0u, 0u, 21, 2047u, s.hist);
  } else if (STAGE == 1) {
    int bin, rem;
    pick<8>(s.hist, s.k, bin, rem);
    if (s.tile == 0 && threadIdx.x == 0) { s.state[0] = bin; s.state[1] = rem; }
    tile_histogram(s, key, 2047u << 21, (uint32_t)bin << 21, 10, 2047u, s.hist + BINS);
  } else {
    const int bin1 = __ldcg(s.state + 0), rem1 = __ldcg(s.state + 1);
    int bin, rem;
    pick<8>(s.hist + BINS, rem1, bin, rem);
    if (s.tile == 0 && threadIdx.x == 0) { s.state[2] = bin; s.state[3] = rem; }
    const uint32_t prefix = ((uint32_t)bin1 << 21) | ((uint32_t)bin << 10);
    tile_histogram(s, key, 0xfffffc00u, prefix, 0, 1023u, s.hist + 2 * BINS);
  }
}

// the k-th largest key and the number of keys equal to it that are kept; per-tile counts
__global__ void __launch_bounds__(THREADS) topk_count_kernel(TopkArgs a) {
  __shared__ int w_gt[THREADS / 32], w_eq[THREADS / 32];
  pdl_release_successor();
  const Segment s = segment_of(a);
  if (!s.open || s.k == 0 || s.tile * TILE >= s.T) return;
  uint32_t key[PER_THREAD];
  load_keys(s, key);
  pdl_wait_predecessor();
  const int bin1 = __ldcg(s.state + 0), bin2 = __ldcg(s.state + 2), rem2 = __ldcg(s.state + 3);
  int bin, need;
  pick<4>(s.hist + 2 * BINS, rem2, bin, need);
  const uint32_t thr = ((uint32_t)bin1 << 21) | ((uint32_t)bin2 << 10) | (uint32_t)bin;
  if (s.tile == 0 && threadIdx.x == 0) { s.state[4] = (int32_t)thr; s.state[5] = need; }
  const int i0 = s.tile * TILE + threadIdx.x * PER_THREAD;
  int gt = 0, eq = 0;
#pragma unroll
  for (int e = 0; e < PER_THREAD; ++e) {
    if (i0 + e < s.T) { gt += key[e] > thr; eq += key[e] == thr; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    gt += __shfl_down_sync(0xffffffffu, gt, o);
    eq += __shfl_down_sync(0xffffffffu, eq, o);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) { w_gt[wid] = gt; w_eq[wid] = eq; }
  __syncthreads();
  if (threadIdx.x == 0) {
    int g = 0, q = 0;
    for (int w2 = 0; w2 < THREADS / 32; ++w2) { g += w_gt[w2]; q += w_eq[w2]; }
    s.counts[2 * s.tile] = g;
    s.counts[2 * s.tile + 1] = q;
  }
}

// ordered emit (Algorithm 1 (TopK and window append))
__global__ void __launch_bounds__(THREADS) topk_emit_kernel(TopkArgs a) {
  __shared__ int w_gt[THREADS / 32], w_eq[THREADS / 32];
  const Segment s = segment_of(a);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int tiles = max(1, (s.T + TILE - 1) / TILE);
  if (!s.open || s.tile >= tiles) return;
  uint32_t key[PER_THREAD];
  if (s.k) load_keys(s, key);
  pdl_wait_predecessor();
  for (int t = s.tile * THREADS + tid; t < s.kept - s.k; t += tiles * THREADS) s.out[s.k + t] = s.T + t;   // the window
  if (s.k == 0) return;
  const uint32_t thr = (uint32_t)__ldcg(s.state + 4);
  const int need = __ldcg(s.state + 5);
  // larger / equal keys in the tiles before this one
  int run_gt = 0, run_eq = 0;
  for (int t = tid; t < s.tile; t += THREADS) { run_gt += __ldcg(s.counts + 2 * t); run_eq += __ldcg(s.counts + 2 * t + 1); }
  const int i0 = s.tile * TILE + tid * PER_THREAD;
  int gt = 0, eq = 0;
#pragma unroll
  for (int e = 0; e < PER_THREAD; ++e) {
    if (i0 + e < s.T) { gt += key[e] > thr; eq += key[e] == thr; }
  }
  // block totals of the look-behind sums, block-exclusive scans of this tile's counts
  int tg = run_gt, te = run_eq, ig = gt, ie = eq;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    tg += __shfl_xor_sync(0xffffffffu, tg, o);
    te += __shfl_xor_sync(0xffffffffu, te, o);
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int vg = __shfl_up_sync(0xffffffffu, ig, o), ve = __shfl_up_sync(0xffffffffu, ie, o);
    if (lane >= o) { ig += vg; ie += ve; }
  }
  __shared__ int b_gt[THREADS / 32], b_eq[THREADS / 32];
  if (lane == 31) { w_gt[wid] = ig; w_eq[wid] = ie; }
  if (lane == 0) { b_gt[wid] = tg; b_eq[wid] = te; }
  __syncthreads();
  int gt_before = ig - gt, eq_before = ie - eq;
  for (int w2 = 0; w2 < THREADS / 32; ++w2) {
    gt_before += b_gt[w2];
    eq_before += b_eq[w2];
    if (w2 < wid) { gt_before += w_gt[w2]; eq_before += w_eq[w2]; }
  }
#pragma unroll
  for (int e = 0; e < PER_THREAD; ++e) {
    const int i = i0 + e;
    if (i < s.T) {
      if (key[e] > thr) {
        s.out[gt_before + min(eq_before, need)] = i;
        ++gt_before;
      } else if (key[e] == thr) {
        if (eq_before < need) s.out[gt_before + eq_before] = i;
        ++eq_before;
      }
    }
  }
}

// ---------------------------------------------------------------------------
// One CTA per segment (up to 256 K scores; which calls take it: one_cta_is_faster): one launch, no scratch in global memory.
//
//   2048 sampled scores -> two keys L <= H that hold the k-th largest key between them with a wide margin (segments of up
//   to 12288 scores: their smallest and largest key) -> ONE pass over the segment: a bitmap of the keys above H, and a
//   list in shared memory of the keys in [L, H] -> exact radix select of the remaining rank in the list, digits taken
//   from the top of the range H - L -> the list's larger keys into the bitmap, the keys equal to the k-th into a second
//   one, the lowest-indexed of which fill the remainder -> ordered emit from the bitmap.
//
// The bounds are only a way to look at few keys: the pass counts, and if the k-th key is not between them or the list
// overflows (long runs of equal scores), the CTA takes the same radix select over the whole segment (four more passes).
// Both ways end in the exact k-th key and the same tie rule, so the kept list does not depend on which ran.
//
// A lane reads 16-byte vectors, eight in flight; bit p of the bitmaps is score p - mis, mis scores lying between the
// 16-byte boundary before the row and the row, so that a vector is a nibble of a word.  (One score per lane and a ballot
// per word takes six times the instructions: 40 us for the pass over 131008 scores instead of 8.)  Bound by what one SM
// pulls from L2 and by the chain of passes:
// one segment of 96K scores, k = 3.8K, 18.8 us; 32 segments of 24K scores, k half of them, 13.7 us (back to back).
// ---------------------------------------------------------------------------
constexpr int SEG_THREADS = 1024;
constexpr int SEG_WARPS = SEG_THREADS / 32;
constexpr int SEG_CAP = 12288;                 // (key, index) pairs the shared-memory list holds
constexpr int SEG_SAMPLE = 2048;
constexpr int SEG_MAX_T = 262144;              // the bitmaps cover this many scores
constexpr int SEG_UNROLL = 8;                  // 16-byte loads in flight per lane
constexpr int SEG_DENSE = 16, SEG_DENSE_WORDS = 8;  // bits of a word that the whole warp writes; such words of 32 at most
constexpr int SEG_FEW = 128;                   // keys of one bin that are ranked by comparing each with all (their square: 512 cost more than a digit)

struct __align__(16) SegSmem {
  int hist[BINS];
  uint32_t cand_key[SEG_CAP];
  int32_t cand_idx[SEG_CAP];
  int warp_a[SEG_WARPS];
  uint32_t lo[SEG_WARPS], hi[SEG_WARPS];
  int found[2][3];
  int n_cand, n_above, n_few;
  uint32_t few[SEG_FEW];
  // behind this struct, sized for the plan's longest segment: two bitmaps over the segment
};
__host__ __device__ inline int seg_words(int max_T) { return ((max_T + 3 + 31) / 32 + 3) & ~3; }
inline size_t seg_smem_bytes(int max_T) { return sizeof(SegSmem) + (size_t)seg_words(max_T) * 2 * sizeof(uint32_t); }

// exclusive prefix over the block of v, in thread order
__device__ __forceinline__ int seg_block_prefix(SegSmem& sm, int v) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  __syncthreads();
  if (lane == 31) sm.warp_a[wid] = incl;
  __syncthreads();
  const int t = sm.warp_a[lane];
  int w = t;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, w, o);
    if (lane >= o) w += u;
  }
  return incl - v + __shfl_sync(0xffffffffu, w - t, wid);
}

// The bin of the shared table (counted from the top) that holds the `remaining`-th largest key, how many keys of that
// bin are still wanted and how many it has; `par` alternates between consecutive calls.
__device__ __forceinline__ void seg_pick(SegSmem& sm, int remaining, int par, uint32_t& bin, int& rem_out, int& in_bin) {
  constexpr int PER = BINS / SEG_THREADS;
  const int top = BINS - 1 - PER * (int)threadIdx.x;
  int c[PER];
  int sum = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) { c[j] = sm.hist[top - j]; sum += c[j]; }
  int above = seg_block_prefix(sm, sum);
  if (above < remaining && remaining <= above + sum) {
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      if (above < remaining && remaining <= above + c[j]) { sm.found[par][0] = top - j; sm.found[par][1] = remaining - above; sm.found[par][2] = c[j]; }
      above += c[j];
    }
  }
  __syncthreads();
  bin = sm.found[par][0];
  rem_out = sm.found[par][1];
  in_bin = sm.found[par][2];
}

// The `rank`-th largest of keys[0..n) in shared memory (all of them in [lo, hi]), how many equal to it are wanted and how
// many there are.  Digits from the top of the range, until the bin that counts holds few keys: after one digit of 2048 bins
// as a rule.  (Few: 128.  Comparing up to 512 with one another took several digits' time where scores are heavy tailed.)  128K
// tokens, eight heads, k = 4032, call by call: the benchmark's scores 28.7 us with all digits counted and now, behind a
// scorer that has swept L2, 28.7 -> 26.6 where a top-k ran shortly before; log-normal ones 31.8 -> 27.1, smooth 30.7 -> 25.6.
__device__ __forceinline__ void seg_select(SegSmem& sm, int n, uint32_t lo, uint32_t hi, int rank, uint32_t& thr, int& need, int& equal) {
  int shift = 32 - __clz((int)((hi - lo) | 1u));            // bits of the range still open
  uint32_t base = lo;                                        // keys in [base, base + 2^shift) are still candidates
  need = rank;
  for (int par = 0;; par ^= 1) {
    const int bits = shift < 11 ? shift : 11;
    for (int i = threadIdx.x; i < BINS; i += SEG_THREADS) sm.hist[i] = 0;
    if (threadIdx.x == 0) sm.n_few = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += SEG_THREADS) {
      const uint32_t d = sm.cand_key[i] - base;
      if (shift == 32 || (d >> shift) == 0u) atomicAdd(&sm.hist[d >> (shift - bits)], 1);
    }
    __syncthreads();
    seg_pick(sm, need, par, lo, need, equal);
    shift -= bits;
    base += lo << shift;
    if (shift == 0) { thr = base; return; }
    if (equal > SEG_FEW) continue;
    for (int i = threadIdx.x; i < n; i += SEG_THREADS) {
      const uint32_t key = sm.cand_key[i];
      if (((key - base) >> shift) == 0u) sm.few[atomicAdd(&sm.n_few, 1)] = key;
    }
    __syncthreads();
    if ((int)threadIdx.x < equal) {
      const uint32_t key = sm.few[threadIdx.x];
      int larger = 0, same = 0;
      for (int i = 0; i < equal; ++i) { larger += sm.few[i] > key; same += sm.few[i] == key; }
      if (larger < need && need <= larger + same) {          // the same by every equal key
        sm.found[par ^ 1][0] = (int)key; sm.found[par ^ 1][1] = need - larger; sm.found[par ^ 1][2] = same;
      }
    }
    __syncthreads();
    thr = (uint32_t)sm.found[par ^ 1][0];
    need = sm.found[par ^ 1][1];
    equal = sm.found[par ^ 1][2];
    return;
  }
}

__global__ void __launch_bounds__(SEG_THREADS, 1) topk_segment_kernel(TopkArgs a) {
  extern __shared__ __align__(16) uint8_t seg_smem_raw[];
  SegSmem& sm = *reinterpret_cast<SegSmem*>(seg_smem_raw);
  uint32_t* const bm_gt = reinterpret_cast<uint32_t*>(seg_smem_raw + sizeof(SegSmem));
  uint32_t* const bm_eq = bm_gt + seg_words(a.max_T);
  pdl_wait_predecessor();
  const Segment s = segment_of(a);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  if (!s.open) return;
  for (int t = tid; t < s.kept - s.k; t += SEG_THREADS) s.out[s.k + t] = s.T + t;   // the window
  if (s.k == 0) return;
  const int mis = (int)((reinterpret_cast<uintptr_t>(s.row) >> 2) & 3);
  const float4* const row4 = reinterpret_cast<const float4*>(s.row - mis);
  const int nv = (s.T + mis + 3) >> 2, words = (nv + 7) >> 3;      // vectors; bitmap words
  // A warp takes blocks of SEG_UNROLL x 32 vectors.  bits of vector v (score bits); m: which of its elements are scores.
  auto load_block = [&](int v0, uint4 (&x)[SEG_UNROLL], uint32_t (&m)[SEG_UNROLL]) {
#pragma unroll
    for (int u = 0; u < SEG_UNROLL; ++u) {
      const int v = v0 + 32 * u + lane;
      m[u] = v < nv ? 15u : 0u;
      if (v == 0) m[u] &= 15u << mis;
      if (v == nv - 1) m[u] &= 15u >> (4 * nv - mis - s.T);
      x[u] = make_uint4(0u, 0u, 0u, 0u);
      if (m[u] == 15u) x[u] = __ldcg(reinterpret_cast<const uint4*>(row4) + v);
    }
#pragma unroll
    for (int u = 0; u < SEG_UNROLL; ++u) {
      if (m[u] != 15u && m[u] != 0u) {                       // the ends of a row off a 16-byte boundary
        const uint32_t* e = reinterpret_cast<const uint32_t*>(row4 + v0 + 32 * u + lane);
        if (m[u] & 1u) x[u].x = __ldcg(e);
        if (m[u] & 2u) x[u].y = __ldcg(e + 1);
        if (m[u] & 4u) x[u].z = __ldcg(e + 2);
        if (m[u] & 8u) x[u].w = __ldcg(e + 3);
      }
    }
  };
  // a nibble per lane -> the bitmap word of eight lanes, stored by one of them
  auto put_word = [&](uint32_t* bm, int v, uint32_t nibble) {
    uint32_t w = nibble << (4 * (lane & 7));
    w |= __shfl_xor_sync(0xffffffffu, w, 1);
    w |= __shfl_xor_sync(0xffffffffu, w, 2);
    w |= __shfl_xor_sync(0xffffffffu, w, 4);
    if ((lane & 7) == 0 && (v >> 3) < words) bm[v >> 3] = w;
  };
  auto nibble_of = [](const uint4& x, auto test) {
    return (test(x.x) ? 1u : 0u) | (test(x.y) ? 2u : 0u) | (test(x.z) ? 4u : 0u) | (test(x.w) ? 8u : 0u);
  };

  // ---- bounds on the k-th largest key
  uint32_t L = 0u, H = 0xffffffffu;
  const bool whole = s.T <= SEG_CAP;                        // the list takes every key
  if (tid == 0) { sm.n_cand = 0; sm.n_above = 0; }
  if (!whole) {
    float x[SEG_SAMPLE / SEG_THREADS];
    uint32_t mn = 0xffffffffu, mx = 0u;
#pragma unroll
    for (int j = 0; j < SEG_SAMPLE / SEG_THREADS; ++j) x[j] = __ldcg(s.row + (int)(((long long)(tid + j * SEG_THREADS) * s.T) / SEG_SAMPLE));
#pragma unroll
    for (int j = 0; j < SEG_SAMPLE / SEG_THREADS; ++j) {
      const uint32_t key = asc_key(x[j]);
      sm.cand_key[tid + j * SEG_THREADS] = key;
      mn = min(mn, key);
      mx = max(mx, key);
    }
    mn = __reduce_min_sync(0xffffffffu, mn);
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) { sm.lo[wid] = mn; sm.hi[wid] = mx; }
    __syncthreads();
    mn = __reduce_min_sync(0xffffffffu, sm.lo[lane]);
    mx = __reduce_max_sync(0xffffffffu, sm.hi[lane]);
    // sample ranks four standard deviations and two to either side of the expected one; their bins in a histogram of the
    // sample's range are bound enough
    const float mean = (float)SEG_SAMPLE * (float)s.k / (float)s.T;
    const float dev = 4.f * sqrtf(mean * (1.f - (float)s.k / (float)s.T)) + 2.f;
    const int r_lo = (int)ceilf(mean + dev), r_hi = (int)floorf(mean - dev);
    const int open = 32 - __clz((int)((mx - mn) | 1u)), shift = open > 11 ? open - 11 : 0;
    for (int i = tid; i < BINS; i += SEG_THREADS) sm.hist[i] = 0;
    __syncthreads();
    for (int i = tid; i < SEG_SAMPLE; i += SEG_THREADS) atomicAdd(&sm.hist[(sm.cand_key[i] - mn) >> shift], 1);
    __syncthreads();
    uint32_t bin;
    int rest, count;
    if (r_lo <= SEG_SAMPLE) { seg_pick(sm, r_lo, 0, bin, rest, count); L = mn + (bin << shift); }
    // an upper bound costs the pass as much as the lower one: only where the keys above L would not fit the list
    if (r_hi >= 1 && 1.2f * (float)s.T * (float)min(r_lo, SEG_SAMPLE) > (float)SEG_CAP * (float)SEG_SAMPLE) {
      seg_pick(sm, r_hi, 1, bin, rest, count);
      const uint32_t top = mn + (bin << shift) + ((1u << shift) - 1u);
      H = top < mn ? 0xffffffffu : top;
    }
    __syncthreads();
  }

  // ---- one pass: the bitmap of keys above H, the list of keys in [L, H]
  uint32_t mn = 0xffffffffu, mx = 0u;                       // of the listed keys
  for (int i = tid; i < words; i += SEG_THREADS) { bm_eq[i] = 0u; bm_gt[i] = 0u; }
  if (!whole) __syncthreads();
  if (whole) {
    for (int i0 = tid; i0 < s.T; i0 += 4 * SEG_THREADS) {
      float x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = i0 + u * SEG_THREADS < s.T ? __ldcg(s.row + i0 + u * SEG_THREADS) : 0.f;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * SEG_THREADS;
        if (i >= s.T) break;
        const uint32_t key = asc_key(x[u]);
        sm.cand_key[i] = key;
        mn = min(mn, key);
        mx = max(mx, key);
      }
    }
  } else {
    // Bounds above zero are compared on the raw bits: a score reaches L unless its sign bit or that of bits - lo is set; the
    // sign is shifted into a mask, three instructions per score.
    const bool raw = L > 0x80000000u;
    const uint32_t lo = L & 0x7fffffffu, hi = H == 0xffffffffu ? 0x7fffffffu : (H & 0x7fffffffu) + 1u;
    const bool none_above = H == 0xffffffffu;
    auto below = [](uint32_t bits, uint32_t bound, uint32_t mask) { return __funnelshift_l(bits | (bits - bound), mask, 1); };
    int above = 0;
    for (int v0 = wid * 32 * SEG_UNROLL; v0 < nv; v0 += SEG_WARPS * 32 * SEG_UNROLL) {
      uint32_t hit, gt;                                     // bit 4u + c: element c of the lane's u-th vector reaches L / is above H
      if (raw && v0 > 0 && v0 + 32 * SEG_UNROLL < nv) {     // (not the first or the last vector of the row)
        uint4 x[SEG_UNROLL];
#pragma unroll
        for (int u = 0; u < SEG_UNROLL; ++u) x[u] = __ldcg(reinterpret_cast<const uint4*>(row4) + v0 + 32 * u + lane);
        uint32_t not_hit = 0u, not_gt = 0u;
#pragma unroll
        for (int u = SEG_UNROLL - 1; u >= 0; --u)
          not_hit = below(x[u].x, lo, below(x[u].y, lo, below(x[u].z, lo, below(x[u].w, lo, not_hit))));
        if (!none_above) {
#pragma unroll
          for (int u = SEG_UNROLL - 1; u >= 0; --u)
            not_gt = below(x[u].x, hi, below(x[u].y, hi, below(x[u].z, hi, below(x[u].w, hi, not_gt))));
        }
        hit = ~not_hit;
        gt = none_above ? 0u : ~not_gt;
      } else {
        uint4 x[SEG_UNROLL];
        uint32_t m[SEG_UNROLL];
        load_block(v0, x, m);
        hit = gt = 0u;
#pragma unroll
        for (int u = 0; u < SEG_UNROLL; ++u) {
          hit |= (nibble_of(x[u], [&](uint32_t b) { return asc_key(__uint_as_float(b)) >= L; }) & m[u]) << (4 * u);
          gt |= (nibble_of(x[u], [&](uint32_t b) { return asc_key(__uint_as_float(b)) > H; }) & m[u]) << (4 * u);
        }
      }
      if (__any_sync(0xffffffffu, gt != 0u)) {
        above += __popc(gt);
#pragma unroll
        for (int u = 0; u < SEG_UNROLL; ++u) put_word(bm_gt, v0 + 32 * u + lane, (gt >> (4 * u)) & 15u);
      }
      hit &= ~gt;
      const int cnt = __popc(hit);
      int incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      const int total = __shfl_sync(0xffffffffu, incl, 31);
      if (total == 0) continue;                             // the same for the whole warp
      int at = 0;
      if (lane == 31) at = atomicAdd(&sm.n_cand, total);
      int slot = __shfl_sync(0xffffffffu, at, 31) + incl - cnt;
      while (hit) {
        const int bpos = __ffs(hit) - 1;
        hit &= hit - 1;
        if (slot < SEG_CAP) sm.cand_idx[slot] = 4 * (v0 + 32 * (bpos >> 2) + lane) + (bpos & 3) - mis;
        ++slot;
      }
    }
    above = __reduce_add_sync(0xffffffffu, above);
    if (lane == 0 && above) atomicAdd(&sm.n_above, above);
    __syncthreads();
    const int listed = min(sm.n_cand, SEG_CAP);
    for (int i0 = tid; i0 < listed; i0 += 4 * SEG_THREADS) {         // their keys
      float x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = i0 + u * SEG_THREADS < listed ? __ldcg(s.row + sm.cand_idx[i0 + u * SEG_THREADS]) : 0.f;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * SEG_THREADS;
        if (i >= listed) break;
        const uint32_t key = asc_key(x[u]);
        sm.cand_key[i] = key;
        mn = min(mn, key);
        mx = max(mx, key);
      }
    }
  }
  mn = __reduce_min_sync(0xffffffffu, mn);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) { sm.lo[wid] = mn; sm.hi[wid] = mx; }
  __syncthreads();
  mn = __reduce_min_sync(0xffffffffu, sm.lo[lane]);
  mx = __reduce_max_sync(0xffffffffu, sm.hi[lane]);
  const int n = whole ? s.T : sm.n_cand, n_above = sm.n_above;
  const bool listed = n <= SEG_CAP && n_above < s.k && s.k <= n_above + n;

  // ---- the exact k-th largest key, how many keys equal to it are kept, and the two bitmaps
  uint32_t thr;
  int need, equal;                                          // keys equal to it: kept, and in all
  if (listed) {
    seg_select(sm, n, mn, mx, s.k - n_above, thr, need, equal);
    for (int i = tid; i < n; i += SEG_THREADS) {
      const uint32_t key = sm.cand_key[i];
      const int e = (whole ? i : sm.cand_idx[i]) + mis;
      if (key > thr || (key == thr && need == equal)) atomicOr(&bm_gt[e >> 5], 1u << (e & 31));
      else if (key == thr) atomicOr(&bm_eq[e >> 5], 1u << (e & 31));
    }
  } else {
    uint32_t base = 0u;
    int shift = 32;
    need = s.k;
    for (int par = 0; shift > 0; par ^= 1) {
      const int bits = shift < 11 ? shift : 11;
      for (int i = tid; i < BINS; i += SEG_THREADS) sm.hist[i] = 0;
      __syncthreads();
      for (int v0 = wid * 32 * SEG_UNROLL; v0 < nv; v0 += SEG_WARPS * 32 * SEG_UNROLL) {
        uint4 x[SEG_UNROLL];
        uint32_t m[SEG_UNROLL];
        load_block(v0, x, m);
        int run_bin = -1, run = 0;                           // neighbouring scores often share a digit: one atomic per run
#pragma unroll
        for (int u = 0; u < SEG_UNROLL; ++u)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint32_t b = c == 0 ? x[u].x : (c == 1 ? x[u].y : (c == 2 ? x[u].z : x[u].w));
            const uint32_t d = asc_key(__uint_as_float(b)) - base;
            const bool in = ((m[u] >> c) & 1u) && (shift == 32 || (d >> shift) == 0u);
            const int bin = in ? (int)(d >> (shift - bits)) : -1;
            if (in && bin == run_bin) { ++run; continue; }
            if (run) atomicAdd(&sm.hist[run_bin], run);
            run_bin = bin;
            run = in ? 1 : 0;
          }
        if (run) atomicAdd(&sm.hist[run_bin], run);
      }
      __syncthreads();
      uint32_t bin;
      seg_pick(sm, need, par, bin, need, equal);
      shift -= bits;
      base += bin << shift;
    }
    thr = base;
    for (int v0 = wid * 32 * SEG_UNROLL; v0 < nv; v0 += SEG_WARPS * 32 * SEG_UNROLL) {
      uint4 x[SEG_UNROLL];
      uint32_t m[SEG_UNROLL];
      load_block(v0, x, m);
#pragma unroll
      for (int u = 0; u < SEG_UNROLL; ++u) {
        put_word(bm_gt, v0 + 32 * u + lane, nibble_of(x[u], [&](uint32_t b) { return asc_key(__uint_as_float(b)) > thr; }) & m[u]);
        put_word(bm_eq, v0 + 32 * u + lane, nibble_of(x[u], [&](uint32_t b) { return asc_key(__uint_as_float(b)) == thr; }) & m[u]);
      }
    }
  }
  __syncthreads();

  // ---- of the equal keys the first `need`; thread t owns a run of words
  const int wpt = (words + SEG_THREADS - 1) / SEG_THREADS;
  const int w0 = min(words, tid * wpt), w1 = min(words, w0 + wpt);
  int kept = 0;
  if (listed && need == equal) {                             // no tie to cut: they are all in the bitmap
    for (int i = w0; i < w1; ++i) kept += __popc(bm_gt[i]);
  } else {
    int eq = 0;
    for (int i = w0; i < w1; ++i) eq += __popc(bm_eq[i]);
    int left = need - seg_block_prefix(sm, eq);
    for (int i = w0; i < w1; ++i) {
      uint32_t q = bm_eq[i];
      const int cnt = __popc(q);
      if (left < cnt) {                                      // keep the lowest `left` of them
        uint32_t some = 0u;
        for (int c = 0; c < left; ++c) { some |= q & (0u - q); q &= q - 1; }
        q = some;
      }
      left -= cnt;
      const uint32_t word = bm_gt[i] | q;
      bm_gt[i] = word;
      kept += __popc(word);
    }
  }
  // ---- ordered emit (Algorithm 1 (TopK and window append)): in shared memory first where the kept indices fit there (the
  // list is done with), so that the copy out is coalesced
  int32_t* const ordered = reinterpret_cast<int32_t*>(sm.cand_key);
  const bool staged = s.k <= 2 * SEG_CAP;
  int32_t* const to = staged ? ordered : s.out;
  int at = seg_block_prefix(sm, kept);
  for (int j = 0; j < wpt; ++j) {                            // a word with many bits (kept tokens come in passages): by the whole warp
    const int i = tid * wpt + j;
    const uint32_t word = i < words ? bm_gt[i] : 0u;
    uint32_t dense = __ballot_sync(0xffffffffu, __popc(word) >= SEG_DENSE);
    if (__popc(dense) > SEG_DENSE_WORDS) dense = 0u;         // (nearly all words are: each lane its own takes no longer)
    if (!((dense >> lane) & 1u)) {
      int32_t* p = to + at;
      for (uint32_t bits = word; bits; bits &= bits - 1) *p++ = i * 32 + __ffs(bits) - 1 - mis;
    }
    for (; dense; dense &= dense - 1) {
      const int from = __ffs(dense) - 1;
      const uint32_t w = __shfl_sync(0xffffffffu, word, from);
      const int p = __shfl_sync(0xffffffffu, at, from);
      if ((w >> lane) & 1u) to[p + __popc(w & ((1u << lane) - 1u))] = (i + (from - lane) * wpt) * 32 + lane - mis;
    }
    at += __popc(word);
  }
  if (staged) {
    __syncthreads();
    for (int i = tid; i < s.k; i += SEG_THREADS) s.out[i] = ordered[i];
  }
}

}  // namespace

size_t asl_topk_scratch_bytes(int64_t segments, int64_t max_T) {
  const int64_t tiles = (max_T + TILE - 1) / TILE > 0 ? (max_T + TILE - 1) / TILE : 1;
  return (size_t)(segments * SEG_INTS + segments * tiles * 2) * sizeof(int32_t);
}

// Whether the one-CTA kernel can take the plan's segments: the longest fits its bitmaps, and the keys expected between the
// two sampled bounds (above the lower one where that is all the list needs) fit the list with a quarter to spare (bins are coarse); where they
// do not, the kernel would select over whole segments: 130 us and more.  Called with the context's device current.
bool asl_topk_plan(asl_ctx* c) {
  c->topk_one_cta = c->max_T <= SEG_MAX_T;
  for (const AslReq& r : c->req) {
    if (r.T <= SEG_CAP) continue;
    const double mean = (double)SEG_SAMPLE * r.k / r.T, dev = 4.0 * sqrt(mean * (1.0 - (double)r.k / r.T)) + 2.0;
    const double above = (double)r.T * fmin(mean + dev, SEG_SAMPLE) / SEG_SAMPLE;
    if (1.25 * fmin(above, 2.0 * dev * r.T / SEG_SAMPLE) > SEG_CAP) c->topk_one_cta = false;
  }
  if (cudaFuncSetAttribute(topk_segment_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)seg_smem_bytes(SEG_MAX_T)) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

// The faster form, on an idle GPU: one CTA takes as long as the longest segment and the largest k say, for any
// number of segments up to the SM count (172 KB of shared memory a CTA at 256K scores: one to an SM), and 6 us more where k
// is too large for the ordered copy; the tiled kernels take as long as the scores of all segments say.  The constants were
// fitted before kernels were launched ahead of their predecessor's end; both forms have since become 2 to 4 us faster, and
// the line between them holds: measured again on 1, 2, 8, 32 and 64 segments of 4K to 256K smooth and log-normal scores, k of 2 to
// 60 % of them, it takes the faster form or one within 6 %, but for 8 segments of 64K, k = 20K (22.5 / 19.9 us; call by call
// 26.6 both), 8 of 256K, k = 5K (31.4 / 28.7) and one of 64K, k = 6.5K (19.1 / 17.4).  One CTA / tiled, back to back: one segment of
// 128K, k = 2.6K, 18.9 / 17.9 us; 8 of 128K, k = 13K, 28.8 / 22.4; 64 of 64K, k = 20K, 22.7 / 50.7.  An estimate, no
// bound: it takes the longest segment and the largest k for one request's where they are two, and a layer issues the call
// beside a scorer that leaves 16 SMs, where neither form has been measured against the other.
static bool one_cta_is_faster(const asl_ctx* c, int n_heads) {
  const double k = c->max_kept - c->p.window;
  const double one = 10.0 + 0.08e-3 * c->max_T + 0.75e-3 * fmin(k, 6500.0) + 0.3e-3 * c->max_T / 65536.0 * fmax(0.0, k - 6500.0) +
                     (k > 2 * SEG_CAP ? 6.0 : 0.0);
  const double tiled = 20.5 + 7.3e-6 * (double)n_heads * (double)c->sum_T;
  return one <= tiled;
}

asl_status asl_launch_topk(asl_ctx* c, const float* scores, int32_t n_heads, int32_t* idx_out, const asl_stat* gate,
                           int32_t gate_layer, char* ws, cudaStream_t st) {
  if (n_heads > c->p.n_kv_heads) return ASL_ERR_INVALID;      // the scratch is sized for H_k heads
  const int tiles = c->max_T > 0 ? (c->max_T + TILE - 1) / TILE : 1;
  const int64_t segments = (int64_t)c->p.batch * n_heads;
  TopkArgs a;
  a.scores = scores;
  a.req = c->d_req;
  a.scratch = reinterpret_cast<int32_t*>(ws + c->ws.topk_scratch);
  a.counts = a.scratch + segments * SEG_INTS;
  a.idx_out = idx_out;
  a.sum_T = c->sum_T;
  a.sum_kept = c->sum_kept;
  a.n_heads = n_heads;
  a.max_tiles = tiles;
  a.max_T = c->max_T;
  a.gate = gate;
  a.gate_layer = gate_layer;
  a.latch = gate ? nullptr : c->latch_stat;      // the gated call has its own rule
  a.cur_layer = c->cur_layer;
  if (c->topk_one_cta && one_cta_is_faster(c, n_heads)) {
    launch_after_smem(topk_segment_kernel, dim3(1, n_heads, c->p.batch), dim3(SEG_THREADS), seg_smem_bytes(c->max_T), st, a);
    c->launches += 1;
    ASL_CUDA(cudaGetLastError());
    return ASL_OK;
  }
  ASL_CUDA(cudaMemsetAsync(a.scratch, 0, (size_t)segments * SEG_INTS * sizeof(int32_t), st));
  const dim3 grid(tiles, n_heads, c->p.batch);
  topk_digit_kernel<0><<<grid, THREADS, 0, st>>>(a);
  launch_after(topk_digit_kernel<1>, grid, dim3(THREADS), st, a);
  launch_after(topk_digit_kernel<2>, grid, dim3(THREADS), st, a);
  launch_after(topk_count_kernel, grid, dim3(THREADS), st, a);
  launch_after(topk_emit_kernel, grid, dim3(THREADS), st, a);
  c->launches += 5;
  ASL_CUDA(cudaGetLastError());
  return ASL_OK;
}
