// Rank row and rank-variance statistic (Algorithm 1 (RankDesc); Algorithm 2 (stacked rank rows R, k, TopKIndices J, Unique U, RelNormVar, threshold test);
// Section 4.1 "var_top" and "relative variance").
//
// RankDesc: position of every (key, token index) pair in sorted order per request, key = bit pattern that ascends as the
// score descends; equal scores keep ascending index order, so the position is the token's 0-based rank with ties to the
// lower index.  One segment of up to 4096 tokens: every token counts those before it.  Batches of short ones: a block sorts
// a segment (sort_takes).  Up to 256K tokens: split at sampled pairs, then placed bucket by bucket.  Longer ones: a stable
// least-significant-digit radix sort (8-bit digits, one kernel per digit after a first histogram); the last pass scatters
// positions straight into the ring row.
//
// Statistic: a token is in the union iff its smallest rank over the rows is < k
// (the k smallest ranks of a row are exactly ranks 0..k-1).  The numerator
// sum_j (rows*sum r^2 - (sum r)^2) is accumulated in 64-bit integers with
// integer atomics, so it does not depend on the order of accumulation.
#include <mutex>

#include "asl_internal.cuh"

namespace {

constexpr int TILE = ASL_RANK_TILE;      // keys per block
constexpr int SORT_THREADS = 256;
constexpr int WARPS = SORT_THREADS / 32;
constexpr int PER_WARP = TILE / WARPS;   // consecutive keys of one warp
constexpr int ROUNDS = PER_WARP / 32;    // walked 32 at a time, all loads issued up front
static_assert(SORT_THREADS == 256 && TILE % SORT_THREADS == 0, "a thread per digit; whole rounds");

__device__ __forceinline__ uint32_t desc_key(float s) {
  uint32_t u = __float_as_uint(s);
  if (u == 0x80000000u) u = 0;                           // -0 ranks with +0
  u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);        // ascending with the score
  return ~u;                                             // ascending as the score descends
}

// Lanes of the warp whose 8-bit digit equals this lane's (only valid lanes count).  They find one another through an
// atomic OR of their lane bits into the digit's word of `lanes`, which is zero before and after: 11 cycles per warp
// where eight ballots take 27.  One vote catches the digit that every lane has, where the atomics would serialise.
__device__ __forceinline__ uint32_t same_digit(uint32_t* lanes, uint32_t d, bool valid, int lane) {
  if (__all_sync(0xffffffffu, d == __shfl_sync(0xffffffffu, d, 0))) return __ballot_sync(0xffffffffu, valid);
  if (valid) atomicOr(lanes + d, 1u << lane);
  __syncwarp();
  const uint32_t peers = lanes[d];
  __syncwarp();
  lanes[d] = 0;
  __syncwarp();
  return peers;
}

// Adds the digits of a warp's valid lanes to the counts of a shared table.
__device__ __forceinline__ void count_digit(int* counts, uint32_t d, bool valid, int lane) {
  if (__all_sync(0xffffffffu, d == __shfl_sync(0xffffffffu, d, 0))) {         // one digit: the adds would serialise
    const int n = __popc(__ballot_sync(0xffffffffu, valid));
    if (lane == 0) atomicAdd(counts + d, n);
  } else if (valid) {
    atomicAdd(counts + d, 1);
  }
}

// The first pass reads the fp32 scores and forms keys on the fly (token index =
// position); later passes read the (key, index) pairs of the previous pass, which may
// still be running when their blocks become resident: coherent loads, behind the wait.
template <bool FIRST>
__device__ __forceinline__ void load_tile(const float* __restrict__ agg, const uint32_t* __restrict__ keys_in,
                                          const int32_t* __restrict__ idx_in, const AslReq& rq, int wstart, int lane,
                                          uint32_t (&key)[ROUNDS], int32_t (&id)[ROUNDS]) {
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const int i = wstart + r * 32 + lane;
    key[r] = 0u;
    id[r] = i;
    if (i < rq.T) {
      if (FIRST) key[r] = desc_key(agg[rq.t_off + i]);
      else { key[r] = __ldcg(keys_in + rq.t_off + i); id[r] = __ldcg(idx_in + rq.t_off + i); }
    }
  }
}

// hist[0][b][blk][digit]: digit counts of one tile of the scores, lowest digit.  The
// tables of the three later passes are cleared here; each scatter pass counts the
// next digit of what it writes into them.
__global__ void __launch_bounds__(SORT_THREADS) rank_hist_first(const float* __restrict__ agg, const AslReq* __restrict__ req,
                                                                const asl_stat* __restrict__ latch, int nblk, int64_t table,
                                                                int32_t* __restrict__ hist) {
  __shared__ int cnt[256];
  pdl_release_successor();                 // launched the plain way: the scores are complete when it starts
  const int b = blockIdx.y, blk = blockIdx.x;
  const int64_t row = ((int64_t)b * nblk + blk) * 256 + (threadIdx.x & 255);
  if (threadIdx.x < 256) {
#pragma unroll
    for (int t = 1; t < 4; ++t) hist[t * table + row] = 0;
  }
  if (latch && latch[b].selected) return;              // the request's selection is final: no more rank rows
  const AslReq rq = req[b];
  const int start = blk * TILE;
  if (start >= rq.T) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x < 256) cnt[threadIdx.x] = 0;
  uint32_t key[ROUNDS];
  int32_t id[ROUNDS];
  load_tile<true>(agg, nullptr, nullptr, rq, start + wid * PER_WARP, lane, key, id);
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) count_digit(cnt, key[r] & 255u, start + wid * PER_WARP + r * 32 + lane < rq.T, lane);
  __syncthreads();
  if (threadIdx.x < 256) hist[row] = cnt[threadIdx.x];
}

// in place: hist[b][blk][digit] -> first output position of (digit, blk), i.e. the
// exclusive scan in (digit, blk) order.  1024 threads: thread (part, digit) walks a
// quarter of the tiles with its loads batched, the parts are chained through shared memory.
__global__ void __launch_bounds__(1024) rank_scan(int32_t* __restrict__ hist, const AslReq* __restrict__ req,
                                                  const asl_stat* __restrict__ latch, int nblk) {
  __shared__ int part_tot[4][256];
  __shared__ int warp_tot[8];
  pdl_release_successor();
  pdl_wait_predecessor();
  const int b = blockIdx.x;
  if (latch && latch[b].selected) return;
  const int used = (req[b].T + TILE - 1) / TILE;             // tiles of this request
  const int d = threadIdx.x & 255, part = threadIdx.x >> 8;
  const int per = (used + 3) / 4;
  const int b0 = part * per, b1 = min(used, b0 + per);
  int32_t* col = hist + (int64_t)b * nblk * 256 + d;
  int total = 0;
  for (int i0 = b0; i0 < b1; i0 += 8) {
    int v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = (i0 + k < b1) ? col[(int64_t)(i0 + k) * 256] : 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) total += v[k];
  }
  part_tot[part][d] = total;
  __syncthreads();
  int digit_total = 0, before = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int t = part_tot[q][d];
    digit_total += t;
    if (q < part) before += t;
  }
  // exclusive scan of the digit totals over the 256 digits (every part computes it)
  const int lane = threadIdx.x & 31, w8 = d >> 5;
  int incl = digit_total;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (part == 0 && lane == 31) warp_tot[w8] = incl;
  __syncthreads();
  int base = incl - digit_total + before;
  for (int w2 = 0; w2 < w8; ++w2) base += warp_tot[w2];
  for (int i0 = b0; i0 < b1; i0 += 8) {
    int v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = (i0 + k < b1) ? col[(int64_t)(i0 + k) * 256] : 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (i0 + k < b1) col[(int64_t)(i0 + k) * 256] = base;
      base += v[k];
    }
  }
}

// Stable scatter of one tile; the last pass writes rank[token] = position.  A pass that is not the last counts, per
// destination tile, the next digit of every pair it writes (integer atomics: the table does not depend on the order of
// arrival).
template <bool FIRST>
__global__ void __launch_bounds__(SORT_THREADS) rank_scatter(const float* __restrict__ agg,
                                                             const uint32_t* __restrict__ keys_in,
                                                             const int32_t* __restrict__ idx_in,
                                                             uint32_t* __restrict__ keys_out, int32_t* __restrict__ idx_out,
                                                             int32_t* __restrict__ rank_row, const int32_t* __restrict__ counts,
                                                             int32_t* __restrict__ next_counts,
                                                             const AslReq* __restrict__ req,
                                                             const asl_stat* __restrict__ latch, int shift, int nblk) {
  __shared__ int cnt[WARPS][256];
  __shared__ uint32_t lanes[WARPS][256];
  __shared__ int digit_off[256];
  pdl_release_successor();
  const int b = blockIdx.y, blk = blockIdx.x;
  if (latch && latch[b].selected) {                    // (waits, as every request may be final: the tables are still being cleared)
    pdl_wait_predecessor();
    return;
  }
  const AslReq rq = req[b];
  const int start = blk * TILE;
  if (start >= rq.T) return;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int wstart = start + wid * PER_WARP;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t key[ROUNDS];
  int32_t id[ROUNDS];
  // the scores were complete before the first histogram ran: the first pass loads them while that kernel
  // finishes; pairs and counts come from the kernel just before
  if (!FIRST) pdl_wait_predecessor();
  load_tile<FIRST>(agg, keys_in, idx_in, rq, wstart, lane, key, id);
  if (FIRST) pdl_wait_predecessor();
  digit_off[threadIdx.x] = __ldcg(counts + ((int64_t)b * nblk + blk) * 256 + threadIdx.x);
  for (int i = threadIdx.x; i < WARPS * 256; i += SORT_THREADS) { (&cnt[0][0])[i] = 0; (&lanes[0][0])[i] = 0; }
  __syncthreads();
  // per-warp digit counts; the peer masks are kept for the second walk
  uint32_t peers[ROUNDS];
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const bool valid = wstart + r * 32 + lane < rq.T;
    const uint32_t d = (key[r] >> shift) & 255u;
    peers[r] = same_digit(lanes[wid], d, valid, lane);
    if (valid && (peers[r] & lt) == 0) cnt[wid][d] += __popc(peers[r]);
    __syncwarp();
  }
  __syncthreads();
  if (threadIdx.x < 256) {  // digit threadIdx.x: bases of the warps, in warp order, after the tile's global offset
    int run = digit_off[threadIdx.x];
#pragma unroll
    for (int w2 = 0; w2 < WARPS; ++w2) {
      const int v = cnt[w2][threadIdx.x];
      cnt[w2][threadIdx.x] = run;
      run += v;
    }
  }
  __syncthreads();
  int32_t* next_b = next_counts ? next_counts + (int64_t)b * nblk * 256 : nullptr;
  const bool top_next = shift == 16;        // the next digit is the sign/exponent byte: few distinct values
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) {
    const bool valid = wstart + r * 32 + lane < rq.T;
    const uint32_t d = (key[r] >> shift) & 255u;
    int pos = 0;
    if (valid) pos = cnt[wid][d] + __popc(peers[r] & lt);
    __syncwarp();
    if (valid && (peers[r] & lt) == 0) cnt[wid][d] += __popc(peers[r]);
    __syncwarp();
    if (valid) {
      if (rank_row) rank_row[rq.t_off + id[r]] = pos;
      else { keys_out[rq.t_off + pos] = key[r]; idx_out[rq.t_off + pos] = id[r]; }
    }
    if (next_b) {
      const uint32_t slot = valid ? (uint32_t)(pos / TILE) * 256u + ((key[r] >> (shift + 8)) & 255u) : 0xffffffffu;
      if (top_next) {                       // one atomic per distinct counter of the warp
        const uint32_t same = __match_any_sync(0xffffffffu, slot);
        if (valid && (same & lt) == 0) atomicAdd(next_b + slot, __popc(same));
      } else if (valid) {
        atomicAdd(next_b + slot, 1);
      }
    }
  }
}

// the four passes of one rank row; scratch: two key and two index arrays, four tables of tile histograms
int launch_sort(const float* agg, const AslReq* req, const asl_stat* latch, int batch, int max_T, uint32_t* const keys[2],
                int32_t* const idx[2], int32_t* hist, int32_t* rank_row, cudaStream_t st) {
  const int nblk = (max_T + TILE - 1) / TILE;
  const dim3 grid(nblk, batch);
  const int64_t table = (int64_t)batch * nblk * 256;
  rank_hist_first<<<grid, SORT_THREADS, 0, st>>>(agg, req, latch, nblk, table, hist);
  for (int pass = 0; pass < 4; ++pass) {
    const int in = (pass + 1) & 1, out = in ^ 1;           // pass 0 reads the scores, writes buffer 0
    const int shift = pass * 8;
    int32_t* row = pass == 3 ? rank_row : nullptr;
    int32_t* cur = hist + pass * table;
    int32_t* nxt = pass == 3 ? nullptr : hist + (pass + 1) * table;
    launch_after(rank_scan, dim3(batch), dim3(1024), st, cur, req, latch, nblk);
    if (pass == 0) launch_after(rank_scatter<true>, grid, dim3(SORT_THREADS), st, agg, nullptr, nullptr, keys[out], idx[out], row, cur, nxt, req, latch, shift, nblk);
    else launch_after(rank_scatter<false>, grid, dim3(SORT_THREADS), st, nullptr, keys[in], idx[in], keys[out], idx[out], row, cur, nxt, req, latch, shift, nblk);
  }
  return 9;
}


struct StatArgs {
  const int32_t* ring;
  const AslReq* req;
  unsigned long long* acc;   // [B][2]: numerator, union size; then one counter of finished blocks
  asl_stat* stat;
  int64_t sum_T;
  int32_t l_obs, first_layer, n_rows, batch, layer_idx, latch;
  double tau;
};

// Algorithm 2 (threshold test) for request b from the accumulated integers
__device__ void stat_finalize_one(unsigned long long num, unsigned long long m, const AslReq* __restrict__ req, asl_stat* __restrict__ stat, int b,
                                  int layer_idx, int n_rows, int evaluate, double tau, int latch) {
  asl_stat s = stat[b];
  if (latch && s.selected) return;                     // final: the record keeps the selection layer
  s.layer_idx = layer_idx;
  s.k = req[b].k;
  s.rows = n_rows;
  s.evaluated = 0;
  s.selected = 0;
  s.num = 0;
  s.m = 0;
  if (evaluate) {
    s.num = (int64_t)num;
    s.m = (int32_t)m;
    s.evaluated = 1;
    s.var_top = (double)num / ((double)n_rows * (double)n_rows * (double)m);   // empty union (k = 0): NaN, never selects
    if (!s.has_init) { s.init_var = s.var_top; s.has_init = 1; }
    s.rel = s.init_var != 0.0 ? s.var_top / s.init_var : __longlong_as_double(0x7ff8000000000000ll);   // zero first variance: undefined, never selects
    s.selected = (s.rel < tau) ? 1 : 0;
  }
  const int32_t selected = s.selected;
  s.selected = 0;
  stat[b] = s;
  if (selected) {                                      // last, behind a fence: see asl_finished
    __threadfence();
    reinterpret_cast<volatile asl_stat*>(stat + b)->selected = 1;
  }
}

// layers before L_min (or with a single rank row): only the bookkeeping fields change
__global__ void rank_stat_skip(const AslReq* __restrict__ req, asl_stat* __restrict__ stat, int batch, int layer_idx, int n_rows, int latch) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < batch) stat_finalize_one(0, 0, req, stat, b, layer_idx, n_rows, 0, 0.0, latch);
}

// Thread 0 adds its block's share of request b; the block that finishes last sees every block's and closes the statistic.
__device__ void stat_close(const StatArgs& a, int b, unsigned long long num, int m, int evaluate) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    if (m) {
      atomicAdd(&a.acc[2 * b], num);
      atomicAdd(&a.acc[2 * b + 1], (unsigned long long)m);
    }
    __threadfence();
    const unsigned long long blocks = (unsigned long long)gridDim.x * gridDim.y;
    last = atomicAdd(&a.acc[2 * a.batch], 1ull) + 1 == blocks;
  }
  __syncthreads();
  if (last) {
    __threadfence();
    for (int bb = threadIdx.x; bb < a.batch; bb += blockDim.x) {
      const unsigned long long sum = __ldcg(a.acc + 2 * bb), size = __ldcg(a.acc + 2 * bb + 1);
      a.acc[2 * bb] = 0;                                 // for the next layer
      a.acc[2 * bb + 1] = 0;
      stat_finalize_one(sum, size, a.req, a.stat, bb, a.layer_idx, a.n_rows, evaluate, a.tau, a.latch);
    }
    if (threadIdx.x == 0) a.acc[2 * a.batch] = 0;
  }
}

constexpr int STAT_TOKENS = 4;   // tokens per thread: few, fat blocks (one wave on the SMs a persistent scorer leaves free)

__global__ void __launch_bounds__(256) rank_stat_accumulate(StatArgs a) {
  __shared__ unsigned long long s_num[8];
  __shared__ int s_m[8];
  const int b = blockIdx.y;
  const AslReq rq = a.req[b];
  const bool open = !(a.latch && a.stat[b].selected);
  unsigned long long num = 0;
  int m = 0;
  int j[STAT_TOKENS];
  long long s1[STAT_TOKENS], s2[STAT_TOKENS];
  int mn[STAT_TOKENS];
#pragma unroll
  for (int i = 0; i < STAT_TOKENS; ++i) {
    j[i] = (blockIdx.x * STAT_TOKENS + i) * 256 + threadIdx.x;
    s1[i] = 0; s2[i] = 0; mn[i] = 0x7fffffff;
  }
  // the rows of the earlier layers are read (all of a batch's loads in flight) while the sort of this layer's row ends
  for (int r0 = 0; r0 < a.n_rows - 1; r0 += 8) {
    int v[STAT_TOKENS][8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int slot = (a.first_layer + r0 + q) % a.l_obs;
#pragma unroll
      for (int i = 0; i < STAT_TOKENS; ++i)
        v[i][q] = (open && j[i] < rq.T && r0 + q < a.n_rows - 1) ? __ldcg(a.ring + (int64_t)slot * a.sum_T + rq.t_off + j[i]) : -1;
    }
#pragma unroll
    for (int i = 0; i < STAT_TOKENS; ++i)
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (v[i][q] >= 0) { mn[i] = min(mn[i], v[i][q]); s1[i] += v[i][q]; s2[i] += (long long)v[i][q] * v[i][q]; }
  }
  pdl_wait_predecessor();
  {
    const int slot = (a.first_layer + a.n_rows - 1) % a.l_obs;
    int v[STAT_TOKENS];
#pragma unroll
    for (int i = 0; i < STAT_TOKENS; ++i) v[i] = (open && j[i] < rq.T) ? __ldcg(a.ring + (int64_t)slot * a.sum_T + rq.t_off + j[i]) : -1;
#pragma unroll
    for (int i = 0; i < STAT_TOKENS; ++i) {
      if (v[i] < 0) continue;
      mn[i] = min(mn[i], v[i]);
      s1[i] += v[i];
      s2[i] += (long long)v[i] * v[i];
      if (mn[i] < rq.k) {
        m += 1;
        num += (unsigned long long)((long long)a.n_rows * s2[i] - s1[i] * s1[i]);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    num += __shfl_down_sync(0xffffffffu, num, o);
    m += __shfl_down_sync(0xffffffffu, m, o);
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) { s_num[wid] = num; s_m[wid] = m; }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w2 = 1; w2 < 8; ++w2) { num += s_num[w2]; m += s_m[w2]; }
  stat_close(a, b, num, m, 1);
}

struct RowArgs {
  const float* agg;
  int32_t* rank_row;
  const AslReq* req;           // null: one segment of T tokens, no statistic
  int32_t T;
  unsigned long long* pairs;   // the tiles' pairs, bucket after bucket; a request's at its u_off
  unsigned long long* list;    // room of the same size for buckets that do not fit a block
  unsigned long long* splitters;   // [request][S], the first of them unused
  uint16_t* table;             // [request][tile][split_pitch] first place of every bucket in the tile
  int32_t max_tiles;
  StatArgs stat;               // ring, records, rows
  int32_t evaluate;
};

__device__ __forceinline__ AslReq row_request(const RowArgs& a, int b) {
  AslReq rq{};
  rq.T = a.T;
  if (a.req) rq = a.req[b];
  return rq;
}
__device__ __forceinline__ bool row_is_final(const RowArgs& a, int b) { return a.req && a.stat.latch && a.stat.stat[b].selected; }

// ---------------------------------------------------------------------------
// One segment of up to COUNT_MAX_T tokens: a token's rank is the number of tokens that go before it, counted outright.
// A block takes 32 tokens, one per lane; its warps share the others, which lie in shared memory (a broadcast load per
// four).  The statistic of the block's tokens goes with them: one launch.  T^2 compares are 2 us of the whole GPU at 4096
// tokens; bound by the launch and three round trips.  4096 scores: 14.3 us by one block's radix sort, a chain of shared-
// memory passes, -> 4.7 us.  Not for batches, whose compares add up, and not above: at 8192 tokens the compares alone are
// 8 us, and eight times that beside a scorer.
// ---------------------------------------------------------------------------
constexpr int COUNT_MAX_T = 4096;
constexpr int COUNT_THREADS = 1024;
constexpr int COUNT_WARPS = COUNT_THREADS / 32;

__global__ void __launch_bounds__(COUNT_THREADS) rank_count_kernel(RowArgs a) {
  __shared__ __align__(16) uint32_t keys[COUNT_MAX_T];
  __shared__ int part[COUNT_WARPS][32];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  pdl_wait_predecessor();
  const bool open = !row_is_final(a, 0);
  const AslReq rq = row_request(a, 0);
  const int T = rq.T, padded = (T + 127) & ~127;                     // padding goes before nothing
  unsigned long long num = 0;
  int m = 0;
  if (open) {
    const int i0 = blockIdx.x * 32, i = i0 + lane;
    // the earlier rows' ranks of the block's tokens, on their way while it counts
    long long s1 = 0, s2 = 0;
    int mn = 0x7fffffff;
    if (wid == 0 && a.evaluate) {
      for (int r0 = 0; r0 < a.stat.n_rows - 1; r0 += 8) {
        int v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int slot = (a.stat.first_layer + r0 + q) % a.stat.l_obs;
          v[q] = i < T && r0 + q < a.stat.n_rows - 1 ? __ldcg(a.stat.ring + (int64_t)slot * a.stat.sum_T + rq.t_off + i) : -1;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (v[q] >= 0) { mn = min(mn, v[q]); s1 += v[q]; s2 += (long long)v[q] * v[q]; }
      }
    }
#pragma unroll
    for (int q = 0; q < COUNT_MAX_T / COUNT_THREADS; ++q) {
      const int j = tid + q * COUNT_THREADS;
      if (j < padded) keys[j] = j < T ? desc_key(__ldcg(a.agg + rq.t_off + j)) : 0xffffffffu;
    }
    __syncthreads();
    const uint32_t key = keys[min(i, padded - 1)];
    const int per = padded / COUNT_WARPS, j0 = wid * per, j1 = j0 + per;        // (a multiple of four)
    int before = 0;
    for (int j = j0; j < min(j1, i0); j += 4) {                       // earlier tokens go first among equals
      const uint4 k = *reinterpret_cast<const uint4*>(keys + j);
      before += (k.x <= key) + (k.y <= key) + (k.z <= key) + (k.w <= key);
    }
    for (int j = max(j0, i0); j < min(j1, i0 + 32); ++j) before += keys[j] < key || (keys[j] == key && j < i);
    for (int j = max(j0, i0 + 32); j < j1; j += 4) {
      const uint4 k = *reinterpret_cast<const uint4*>(keys + j);
      before += (k.x < key) + (k.y < key) + (k.z < key) + (k.w < key);
    }
    part[wid][lane] = before;
    __syncthreads();
    if (wid == 0) {
      int rank = 0;
#pragma unroll
      for (int w = 0; w < COUNT_WARPS; ++w) rank += part[w][lane];
      if (i < T) {
        a.rank_row[rq.t_off + i] = rank;
        mn = min(mn, rank);
        s1 += rank;
        s2 += (long long)rank * rank;
        if (a.evaluate && mn < rq.k) {
          m = 1;
          num = (unsigned long long)((long long)a.stat.n_rows * s2 - s1 * s1);
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        num += __shfl_down_sync(0xffffffffu, num, o);
        m += __shfl_down_sync(0xffffffffu, m, o);
      }
    }
  }
  if (a.req) stat_close(a.stat, 0, num, m, a.evaluate);
}

// ---------------------------------------------------------------------------
// Batches of short segments: a block a request sorts the whole segment in shared memory (four stable passes of 8-bit digits),
// writes the row and takes the statistic: one launch, which takes as long as one request does while there is an SM for each.
// Bound by what its rounds issue to shared memory and by five block barriers a pass.
//
// The split row (below) ranks a segment sooner, but in three launches, and its blocks add up over a batch: always slower up
// to 1024 tokens, and above where the requests are many (sort_takes; the fit is within 1 us of the figures up to a wave of
// requests).  Rank statistic in us, here / split: 8 of 500 tokens 7.9 / 10.8, 128 of 500 8.0 / 16.0, 1000 of 100 45 / 60,
// 32 of 1000 9.3 / 11.6, 32 of 1500 11.8 / 11.5, 64 of 1500 11.8 / 12.7, 32 of 2000 13.3 / 12.2, 64 of 2000 13.3 / 13.7, 8 of
// 4096 21.3 / 11.5, 64 of 4096 21.4 / 18.1, 96 of 4096 21.4 / 22.0, 200 of 4096 41.9 / 39.3.  (Counted rows for batches of few
// compares: 8 of 500 tokens 6.9, but 128 of 500 22, and in a layer, on the SMs that a scorer leaves, never faster: four
// layers (32q/8kv) of 8 requests of 500 tokens 129 us, here 117, of 4 of 1000 106, here 91.)
// ---------------------------------------------------------------------------
constexpr int SORT_MAX_T = 4096;
constexpr int ROW_THREADS = 1024;
constexpr int ROW_WARPS = ROW_THREADS / 32;

__host__ __device__ constexpr int sort_smem_bytes(int rounds) {     // per warp: lanes per digit, digit counts; keys, token numbers
  return rounds * ROW_THREADS * (int)(sizeof(uint32_t) + sizeof(uint16_t)) + ROW_WARPS * 256 * (int)(sizeof(uint16_t) + sizeof(uint32_t));
}
bool sort_takes(int max_T, int64_t sum_T, int batch, int sms) {
  if (batch == 1 || max_T > SORT_MAX_T) return false;
  const int waves = (batch + sms - 1) / sms;
  return max_T <= 1024 || waves * (6.7 + 3.5e-3 * max_T) <= 10.3 + 0.028e-3 * (double)sum_T;
}

template <int R>
__global__ void __launch_bounds__(ROW_THREADS, 1) rank_sort_kernel(RowArgs a) {
  constexpr int N = R * ROW_THREADS;
  extern __shared__ __align__(16) uint8_t sort_raw[];
  uint32_t (*lanes)[256] = reinterpret_cast<uint32_t (*)[256]>(sort_raw);
  uint32_t (*cnt2)[128] = reinterpret_cast<uint32_t (*)[128]>(lanes + ROW_WARPS);       // two digits' counts per word
  uint32_t* s_key = reinterpret_cast<uint32_t*>(cnt2 + ROW_WARPS);
  uint16_t* s_id = reinterpret_cast<uint16_t*>(s_key + N);
  __shared__ uint32_t part_sum[8][128];
  __shared__ int warp_tot[4];
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  uint16_t* const cnt = reinterpret_cast<uint16_t*>(cnt2[wid]);
  pdl_wait_predecessor();
  if (row_is_final(a, b)) return;
  const AslReq rq = row_request(a, b);
  const uint32_t lt = (1u << lane) - 1u;
  const int w0 = wid * R * 32;                                        // a warp owns consecutive keys
  uint32_t key[R];
  uint32_t id[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = w0 + r * 32 + lane;
    id[r] = i;
    key[r] = i < rq.T ? desc_key(__ldcg(a.agg + rq.t_off + i)) : 0xffffffffu;   // padding sorts last (and stays behind equal keys)
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) lanes[wid][i * 32 + lane] = 0;
#pragma unroll 1
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 8 * pass;
    uint32_t before[R];                                               // keys of the warp with the same digit and a lower place
#pragma unroll
    for (int i = 0; i < 4; ++i) cnt2[wid][i * 32 + lane] = 0;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint32_t d = (key[r] >> shift) & 255u;
      const uint32_t peers = same_digit(lanes[wid], d, true, lane);
      const uint32_t c = cnt[d];
      __syncwarp();
      if ((peers & lt) == 0) cnt[d] = (uint16_t)(c + __popc(peers));
      before[r] = c + __popc(peers & lt);
      __syncwarp();
    }
    __syncthreads();
    {  // the counts become positions, in (digit, warp) order: thread (part, word) has two digits of four warps
      const int w = tid & 127, part = tid >> 7;
      uint32_t v[4], total = 0, mine = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) { v[i] = cnt2[part * 4 + i][w]; mine += v[i]; }
      part_sum[part][w] = mine;
      __syncthreads();
      mine = 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) { const uint32_t s = part_sum[q][w]; total += s; mine += q < part ? s : 0u; }
      const int both = (int)((total & 0xffffu) + (total >> 16));
      int incl = both;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
      }
      if (part == 0 && lane == 31) warp_tot[wid] = incl;
      __syncthreads();
      uint32_t off = (uint32_t)(incl - both);
#pragma unroll
      for (int q = 0; q < 3; ++q) off += q < (w >> 5) ? (uint32_t)warp_tot[q] : 0u;
      uint32_t run = mine + (off | (off + (total & 0xffffu)) << 16);
#pragma unroll
      for (int i = 0; i < 4; ++i) { cnt2[part * 4 + i][w] = run; run += v[i]; }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint32_t pos = cnt[(key[r] >> shift) & 255u] + before[r];
      if (pass == 3) { s_key[id[r]] = pos; continue; }      // the rank row, in token order
      s_key[pos] = key[r];
      s_id[pos] = (uint16_t)id[r];
    }
    __syncthreads();
    if (pass == 3) break;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      key[r] = s_key[w0 + r * 32 + lane];
      id[r] = s_id[w0 + r * 32 + lane];
    }
  }
  // ---- the row, and the statistic over it and the earlier rows
  __shared__ unsigned long long s_num[ROW_WARPS];
  __shared__ int s_m[ROW_WARPS];
  unsigned long long num = 0;
  int m = 0;
#pragma unroll 1
  for (int i = tid; i < rq.T; i += ROW_THREADS) {
    const int mine = (int)s_key[i];
    a.rank_row[rq.t_off + i] = mine;
    if (a.evaluate) {
      long long s1 = mine, s2 = (long long)mine * mine;
      int mn = mine;
      for (int r0 = 0; r0 < a.stat.n_rows - 1; r0 += 8) {
        int v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int slot = (a.stat.first_layer + r0 + q) % a.stat.l_obs;
          v[q] = r0 + q < a.stat.n_rows - 1 ? __ldcg(a.stat.ring + (int64_t)slot * a.stat.sum_T + rq.t_off + i) : -1;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (v[q] >= 0) { mn = min(mn, v[q]); s1 += v[q]; s2 += (long long)v[q] * v[q]; }
      }
      if (mn < rq.k) {
        m += 1;
        num += (unsigned long long)((long long)a.stat.n_rows * s2 - s1 * s1);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    num += __shfl_down_sync(0xffffffffu, num, o);
    m += __shfl_down_sync(0xffffffffu, m, o);
  }
  if (lane == 0) { s_num[wid] = num; s_m[wid] = m; }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < ROW_WARPS; ++w) { num += s_num[w]; m += s_m[w]; }
    stat_finalize_one(num, (unsigned long long)m, a.req, a.stat.stat, b, a.stat.layer_idx, a.stat.n_rows, a.evaluate, a.stat.tau, a.stat.latch);
  }
}

// ---------------------------------------------------------------------------
// Segments of up to SPLIT_MAX_T tokens: (key, token) pairs are all different, so S pairs sampled across the segment, once
// sorted, cut it into S buckets of about the same size whatever the scores are, long runs of equal ones included.
//
//   rank_split_kernel   a block takes a tile of 4 S scores: sorts the sample (all blocks the same one), finds each score's
//                       bucket in the sorted sample, writes the tile's pairs bucket after bucket, and where each begins
//   rank_place_kernel   a block takes a few buckets: the pairs that go before them are the sum of their first places over
//                       the tiles; its own are dealt to bins (two to four of them a pair on average) by where they lie
//                       between their bucket's splitters, and a pair is compared with those of its bin only; where
//                       pairs crowd into a bucket or a bin, the block sorts them digit by digit (place_by_digits)
//
// Neither waits for another block, and the row does not depend on the order in which pairs arrive.  Bound by latency: the
// first takes 4 to 6 us (the sample's round trip, its sort, 8 to 10 steps of search), the second 7 (three round trips).
// 100003 tokens with the statistic: five radix passes 34.8 us -> 16.7.  32768 tokens beside a scorer that leaves 16 SMs:
// sorted tiles of 4096 and their merge, whose searches grow with the square of the length, 35 us -> 23; eight layers
// 471 -> 460 us.  Longer segments would need a larger sample, whose sort every block repeats.
// ---------------------------------------------------------------------------
constexpr int SPLIT_MAX_T = 262144;
constexpr int SPLIT_MAX_TILES = 64;
__host__ __device__ constexpr int split_pitch(int S) { return S + 8; }
__host__ __device__ constexpr int split_max_T(int S) { return S == 256 ? 32768 : (S == 512 ? 131072 : SPLIT_MAX_T); }
static_assert(split_max_T(256) <= 4 * 256 * SPLIT_MAX_TILES && split_max_T(512) <= 4 * 512 * SPLIT_MAX_TILES && SPLIT_MAX_T <= 4 * 1024 * SPLIT_MAX_TILES, "tiles of a segment");

__device__ __forceinline__ unsigned long long pair_of(uint32_t key, int token) { return (unsigned long long)key << 32 | (uint32_t)token; }

template <int S>
__global__ void __launch_bounds__(S) rank_split_kernel(RowArgs a) {
  constexpr int PER = 4, TILE_N = PER * S, LEVELS = S == 256 ? 8 : (S == 512 ? 9 : 10);
  static_assert(1 << LEVELS == S, "a thread per sampled pair");
  extern __shared__ __align__(16) uint8_t split_raw[];
  unsigned long long* const stage = reinterpret_cast<unsigned long long*>(split_raw);     // [TILE_N]; the sample's sort uses it first
  unsigned long long* const tree = stage + TILE_N;                                        // [S] the splitters in the order of a search, from 1 on
  int* const count = reinterpret_cast<int*>(tree + S);                                    // [S]
  __shared__ int warp_tot[S / 32];
  const int b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const AslReq rq = row_request(a, b);
  pdl_wait_predecessor();
  if (row_is_final(a, b)) return;
  const int start = blockIdx.x * TILE_N;
  if (start >= rq.T) return;
  const int n = min(TILE_N, rq.T - start);
  // a sampled token lies somewhere in its S-th of the segment, so that no period of the scores can meet the sample's
  const int s_lo = (int)((long long)tid * rq.T / S), s_hi = (int)((long long)(tid + 1) * rq.T / S);
  const int s_at = min(rq.T - 1, s_lo + (int)(((uint32_t)tid * 2654435761u >> 8) % (uint32_t)max(1, s_hi - s_lo)));
  const float s_score = __ldcg(a.agg + rq.t_off + s_at);
  float score[PER];
#pragma unroll
  for (int r = 0; r < PER; ++r) score[r] = r * S + tid < n ? __ldcg(a.agg + rq.t_off + start + r * S + tid) : 0.f;
  count[tid] = 0;
  // bitonic sort, a pair per thread: exchanges within a warp by shuffles, across warps through two buffers in turn
  unsigned long long v = pair_of(desc_key(s_score), s_at);
  int flip = 0;
#pragma unroll
  for (int k = 2; k <= S; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      unsigned long long o;
      if (j >= 32) {
        stage[flip * S + tid] = v;
        __syncthreads();
        o = stage[flip * S + (tid ^ j)];
        flip ^= 1;
      } else {
        o = __shfl_xor_sync(0xffffffffu, v, j);
      }
      v = (((tid & k) == 0) == ((tid & j) == 0)) == (o < v) ? o : v;
    }
  }
  __syncthreads();
  stage[tid] = v;
  __syncthreads();
  if (tid) {                                           // node `tid` of the search tree: the middle of what its path leaves
    const int level = 31 - __clz(tid);
    tree[tid] = stage[(2 * (tid - (1 << level)) + 1) * (S >> (level + 1))];
  }
  __syncthreads();
  unsigned long long pair[PER];
  int node[PER];
#pragma unroll
  for (int r = 0; r < PER; ++r) { pair[r] = pair_of(desc_key(score[r]), start + r * S + tid); node[r] = 1; }
#pragma unroll
  for (int l = 0; l < LEVELS; ++l)
#pragma unroll
    for (int r = 0; r < PER; ++r) node[r] = 2 * node[r] + (pair[r] >= tree[node[r]] ? 1 : 0);
  int place[PER];
#pragma unroll
  for (int r = 0; r < PER; ++r) place[r] = r * S + tid < n ? atomicAdd(&count[node[r] - S], 1) : 0;
  __syncthreads();
  int mine = count[tid], incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  int before = incl - mine;
  {
    int t = lane < S / 32 && lane < wid ? warp_tot[lane] : 0;
    before += __reduce_add_sync(0xffffffffu, t);
  }
  count[tid] = before;
  if (blockIdx.x == 0) a.splitters[b * S + tid] = v;
  uint16_t* const row = a.table + ((int64_t)b * a.max_tiles + blockIdx.x) * split_pitch(S);
  row[tid] = (uint16_t)before;
  if (tid == 0) row[S] = (uint16_t)n;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < PER; ++r)
    if (r * S + tid < n) stage[count[node[r] - S] + place[r]] = pair[r];
  __syncthreads();
  unsigned long long* const out = a.pairs + rq.u_off + start;
#pragma unroll
  for (int r = 0; r < PER; ++r)
    if (r * S + tid < n) out[r * S + tid] = stage[r * S + tid];
}

constexpr int PLACE_THREADS = 512;
template <int S>
struct PlaceSmem {
  static constexpr int PER = S == 256 ? 6 : (S == 512 ? 8 : 12);        // pairs of a thread that stay on the SM
  static constexpr int HELD = PER * PLACE_THREADS, BINS = 4 * PLACE_THREADS;
  static constexpr int MIN_GROUP = S == 512 ? 2 : 4, MAX_GROUP = 64;  // buckets of a block
  unsigned long long held[HELD];
  unsigned long long split[MAX_GROUP], least[MAX_GROUP], most[MAX_GROUP];
  float scale[MAX_GROUP];
  int bin[BINS + 4];
  int first_of[SPLIT_MAX_TILES + 1], from[SPLIT_MAX_TILES];       // the tiles' parts in the buckets, and in their tiles
  int warp_tot[PLACE_THREADS / 32], base;
  // buckets of a block: as many (a power of two) as give a block a sixth of the pairs that it can hold, so that nearly every
  // block has room for its own (eight ragged requests, blocks of four buckets whatever their lengths: 39 us, not 31); fewer
  // of a longer request, so that the longest one says how many blocks a request may need
  __host__ __device__ static int group_of(int T) {
    int group = MIN_GROUP;
    while (group < MAX_GROUP && (long long)T * group * 2 <= (long long)S * (HELD / 6)) group *= 2;
    return group;
  }
  __device__ __forceinline__ int slot_of(int e) const {           // the block's e-th pair, tile after tile
    int t = 0;
#pragma unroll
    for (int h = SPLIT_MAX_TILES / 2; h; h >>= 1) t += first_of[t + h] <= e ? h : 0;
    return from[t] + (e - first_of[t]);
  }
};

// The block's m pairs sorted, whatever they are: stable passes over the 8-bit digits in which they differ, lowest first, to and
// fro between the pairs' own slots in the tiles and the list; the last one writes the ranks.  For blocks that have no room for
// their pairs, and for bins of more than BIN_MAX pairs (a bucket's ends far apart and the rest nearly
// alike: the border of two long runs of equal scores, scores on both sides of zero), whose compares grow with their square.
// One SM's seven passes, 9 to 13 ns a pair, are what a row costs whose tokens, but for the sampled ones, lie in one bucket:
// 131072 tokens of one value 1.6 s -> 1.3 ms, of random values 5.6 -> 1.7 ms, 5000 of one value 870 -> 66 us.  Rows that the
// sample stands for do not get here, or with few pairs: 131072 tokens in runs of a dozen values 42 -> 30 us.  (512: with 256
// the passes take over from compares that are still faster, 65536 tokens in runs 17.8 -> 22.1 us; with 1024 too late, 131072 tokens 50 us.)
constexpr int BIN_MAX = 512;
template <int S>
__device__ __noinline__ void place_by_digits(PlaceSmem<S>& sm, unsigned long long* pairs, unsigned long long* list,
                                             int32_t* rank_row, int m, int base) {
  constexpr int THREADS = PLACE_THREADS, W = THREADS / 32, STEPS = 4;
  uint32_t* const lanes = reinterpret_cast<uint32_t*>(sm.held);             // [W][256], see same_digit
  uint16_t* const cnt = reinterpret_cast<uint16_t*>(lanes + W * 256);       // [W][256]
  static_assert(sizeof(sm.held) >= W * 256 * 6 && PlaceSmem<S>::BINS == 8 * 256 && W * 256 == 8 * THREADS, "eight tables of digits, two of warps");
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const uint32_t lt = (1u << lane) - 1u;
  *reinterpret_cast<int4*>(sm.bin + 4 * tid) = make_int4(0, 0, 0, 0);
  for (int i = tid; i < W * 256; i += THREADS) lanes[i] = 0;
  __syncthreads();
  for (int e0 = 0; e0 < m; e0 += THREADS) {             // every digit's counts: no pass changes them
    const bool valid = e0 + tid < m;
    const unsigned long long p = valid ? __ldcg(pairs + sm.slot_of(e0 + tid)) : 0ull;
#pragma unroll
    for (int d = 0; d < 8; ++d) count_digit(sm.bin + 256 * d, (uint32_t)(p >> 8 * d) & 255u, valid, lane);
  }
  __syncthreads();
  uint32_t differ = 0;                                  // (pairs are all different: not zero)
  for (int d = 0; d < 8; ++d)
    if (!__syncthreads_or(tid < 256 && sm.bin[256 * d + tid] == m)) differ |= 1u << d;
  bool in_list = false;
  for (; differ; differ &= differ - 1) {
    const int d = __ffs(differ) - 1;
    const bool last = (differ & (differ - 1)) == 0;
    int* const start = sm.bin + 256 * d;
    const int c = tid < 256 ? start[tid] : 0;
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    if (lane == 31) sm.warp_tot[wid] = incl;
    __syncthreads();
    const int before = __reduce_add_sync(0xffffffffu, lane < wid ? sm.warp_tot[lane] : 0);
    if (tid < 256) start[tid] = before + incl - c;
    for (int c0 = 0; c0 < m; c0 += STEPS * THREADS) {
      const int w0 = c0 + wid * STEPS * 32 + lane;
      unsigned long long p[STEPS];
      uint32_t peers[STEPS];
#pragma unroll
      for (int r = 0; r < STEPS; ++r) {
        const int e = w0 + 32 * r;
        p[r] = e < m ? __ldcg(in_list ? list + e : pairs + sm.slot_of(e)) : 0ull;
      }
      *reinterpret_cast<uint4*>(cnt + 8 * tid) = make_uint4(0u, 0u, 0u, 0u);
      __syncthreads();
#pragma unroll
      for (int r = 0; r < STEPS; ++r) {
        const bool valid = w0 + 32 * r < m;
        const uint32_t v = (uint32_t)(p[r] >> 8 * d) & 255u;
        peers[r] = same_digit(lanes + 256 * wid, v, valid, lane);
        if (valid && (peers[r] & lt) == 0) cnt[256 * wid + v] += (uint16_t)__popc(peers[r]);
        __syncwarp();
      }
      __syncthreads();
      int total = 0;
      if (tid < 256) {
        uint16_t of[W];
#pragma unroll
        for (int w = 0; w < W; ++w) of[w] = cnt[256 * w + tid];
#pragma unroll
        for (int w = 0; w < W; ++w) { cnt[256 * w + tid] = (uint16_t)total; total += of[w]; }
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < STEPS; ++r) {
        const bool valid = w0 + 32 * r < m;
        const uint32_t v = (uint32_t)(p[r] >> 8 * d) & 255u;
        const int pos = start[v] + cnt[256 * wid + v] + __popc(peers[r] & lt);
        __syncwarp();
        if (valid && (peers[r] & lt) == 0) cnt[256 * wid + v] += (uint16_t)__popc(peers[r]);
        __syncwarp();
        if (valid && last) rank_row[(int)(uint32_t)p[r]] = base + pos;
        else if (valid) *(in_list ? pairs + sm.slot_of(pos) : list + pos) = p[r];
      }
      __syncthreads();
      if (tid < 256) start[tid] += total;
    }
    in_list = !in_list;
    __syncthreads();
  }
}

template <int S>
__global__ void __launch_bounds__(PLACE_THREADS, S == 1024 ? 2 : 3) rank_place_kernel(RowArgs a) {
  using M = PlaceSmem<S>;
  constexpr int TILE_N = 4 * S, THREADS = PLACE_THREADS, PER = M::PER, HELD = M::HELD, BINS = M::BINS;
  extern __shared__ __align__(16) uint8_t place_raw[];
  M& sm = *reinterpret_cast<M*>(place_raw);
  const int b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  pdl_release_successor();
  const AslReq rq = row_request(a, b);
  pdl_wait_predecessor();
  if (row_is_final(a, b)) return;
  const int tiles = (rq.T + TILE_N - 1) / TILE_N;
  const int group = M::group_of(rq.T);
  const int b0 = blockIdx.x * group, own = BINS / group;
  if (b0 >= S) return;
  *reinterpret_cast<int4*>(sm.bin + 4 * tid) = make_int4(0, 0, 0, 0);
  if (wid == 0) {
    int lo[2] = {0, 0}, n[2] = {0, 0};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int t = 2 * lane + q;
      if (t < tiles) {
        const uint16_t* row = a.table + ((int64_t)b * a.max_tiles + t) * split_pitch(S) + b0;
        lo[q] = __ldcg(row);
        n[q] = __ldcg(row + group) - lo[q];
      }
    }
    int incl = n[0] + n[1];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    sm.first_of[2 * lane] = incl - n[1] - n[0];
    sm.first_of[2 * lane + 1] = incl - n[1];
    sm.from[2 * lane] = 2 * lane * TILE_N + lo[0];
    sm.from[2 * lane + 1] = (2 * lane + 1) * TILE_N + lo[1];
    if (lane == 31) sm.first_of[SPLIT_MAX_TILES] = incl;
    const int base = __reduce_add_sync(0xffffffffu, lo[0] + lo[1]);
    if (lane == 0) sm.base = base;
  } else if (tid < 32 + group) {
    // a bucket's bins lie between its two splitters; the first and the last bucket have one only (below)
    const int g = tid - 32, q = b0 + g;
    const unsigned long long* split = a.splitters + b * S;
    const unsigned long long x0 = __ldcg(split + max(q, 1)), x1 = __ldcg(split + min(q + 1, S - 1));
    sm.split[g] = sm.least[g] = x0;
    sm.scale[g] = (float)own / __ull2float_rz(max(1ull, x1 - x0));
  }
  __syncthreads();
  const int m = sm.first_of[SPLIT_MAX_TILES], base = sm.base;
  if (m == 0) return;
  const unsigned long long* const pairs = a.pairs + rq.u_off;
  auto bucket_of = [&](unsigned long long pair) {
    int g = 0;
    for (int h = group / 2; h; h >>= 1) g += pair >= sm.split[g + h] ? h : 0;
    return g;
  };
  auto bin_of = [&](unsigned long long pair) {         // no pair gets a lower one than a smaller pair
    const int g = bucket_of(pair);
    const unsigned long long least = sm.least[g];
    return g * own + (pair > least ? min(own - 1, (int)(__ull2float_rz(pair - least) * sm.scale[g])) : 0);
  };
  unsigned long long pair[PER];
  // a pair's place among those of its bin, in the order of arrival; then where the bins begin
  uint32_t at[PER];                              // bin << 16 | place
  bool sort = m > HELD;
  if (!sort) {
#pragma unroll
    for (int r = 0; r < PER; ++r)
      if (r * THREADS < m) pair[r] = __ldcg(pairs + sm.slot_of(min(r * THREADS + tid, m - 1)));
    if (b0 == 0 || b0 + group == S) {                  // the segment's first pair, or its last one, is the bound that lacks
      unsigned long long end = pair[0];
#pragma unroll
      for (int r = 1; r < PER; ++r)
        if (r * THREADS < m) end = b0 == 0 ? min(end, pair[r]) : max(end, pair[r]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, end, o);
        end = b0 == 0 ? min(end, other) : max(end, other);
      }
      if (lane == 0) sm.most[wid] = end;
      __syncthreads();
      if (tid == 0) {
        for (int w = 1; w < THREADS / 32; ++w) end = b0 == 0 ? min(end, sm.most[w]) : max(end, sm.most[w]);
        const int g = b0 == 0 ? 0 : group - 1;
        const unsigned long long low = b0 == 0 ? end : sm.least[g], high = b0 == 0 ? sm.least[0] : end;
        sm.least[g] = min(low, high);                  // (an empty bucket's is not used)
        sm.scale[g] = (float)own / __ull2float_rz(max(1ull, high - min(low, high)));
      }
      __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < PER; ++r)
      if (r * THREADS + tid < m) {
        const int q = bin_of(pair[r]), place = atomicAdd(&sm.bin[q], 1);
        at[r] = (uint32_t)q << 16 | (uint32_t)place;
        sort |= place >= BIN_MAX;
      }
  }
  if (__syncthreads_or(sort)) {
    place_by_digits(sm, a.pairs + rq.u_off, a.list + rq.u_off + base, a.rank_row + rq.t_off, m, base);
    return;
  }
  {
    const int4 c = *reinterpret_cast<int4*>(sm.bin + 4 * tid);
    const int mine = c.x + c.y + c.z + c.w;
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    if (lane == 31) sm.warp_tot[wid] = incl;
    __syncthreads();
    int run = incl - mine + __reduce_add_sync(0xffffffffu, lane < wid ? sm.warp_tot[lane] : 0);
    int4 s;
    s.x = run; s.y = s.x + c.x; s.z = s.y + c.y; s.w = s.z + c.z;
    *reinterpret_cast<int4*>(sm.bin + 4 * tid) = s;
    if (tid == THREADS - 1) sm.bin[BINS] = m;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < PER; ++r)
    if (r * THREADS + tid < m) sm.held[sm.bin[at[r] >> 16] + (int)(at[r] & 0xffffu)] = pair[r];
  __syncthreads();
#pragma unroll
  for (int r = 0; r < PER; ++r)
    if (r * THREADS + tid < m) {
      const int q = (int)(at[r] >> 16), begin = sm.bin[q], end = sm.bin[q + 1];
      int rank = base + begin;
#pragma unroll 4
      for (int i = begin; i < end; ++i) rank += sm.held[i] < pair[r] ? 1 : 0;
      a.rank_row[rq.t_off + (int)(uint32_t)pair[r]] = rank;
    }
}

template <int S>
constexpr int split_smem_bytes() { return (int)(5 * S * sizeof(unsigned long long) + S * sizeof(int)); }

void launch_count(const RowArgs& r, int T, cudaStream_t st) { launch_after(rank_count_kernel, dim3((T + 31) / 32), dim3(COUNT_THREADS), st, r); }

void launch_row_sort(const RowArgs& r, int max_T, int batch, cudaStream_t st) {
  const int rounds = max_T <= 1024 ? 1 : max_T <= 2048 ? 2 : 4;
  const auto kernel = rounds == 1 ? rank_sort_kernel<1> : rounds == 2 ? rank_sort_kernel<2> : rank_sort_kernel<4>;
  launch_after_smem(kernel, dim3(batch), dim3(ROW_THREADS), sort_smem_bytes(rounds), st, r);
}

template <int S>
void launch_split_of(RowArgs r, int max_T, int batch, cudaStream_t st) {
  r.max_tiles = (max_T + 4 * S - 1) / (4 * S);
  r.table = reinterpret_cast<uint16_t*>(r.splitters + (size_t)batch * S);
  launch_after_smem(rank_split_kernel<S>, dim3(r.max_tiles, batch), dim3(S), split_smem_bytes<S>(), st, r);
  launch_after_smem(rank_place_kernel<S>, dim3(S / PlaceSmem<S>::group_of(max_T), batch), dim3(PLACE_THREADS), sizeof(PlaceSmem<S>), st, r);
}

// Buckets of up to 128 pairs on average to 32K tokens, 256 above.  (A block of one bucket each, bins between its smallest and
// its largest pair: 100003 tokens 25.8 us, and eight layers of 32K no faster than by merging; the blocks' fixed costs count.)
int launch_split(const RowArgs& r, int max_T, int batch, cudaStream_t st) {
  if (max_T <= split_max_T(256)) launch_split_of<256>(r, max_T, batch, st);
  else if (max_T <= split_max_T(512)) launch_split_of<512>(r, max_T, batch, st);
  else launch_split_of<1024>(r, max_T, batch, st);
  return 2;
}

}  // namespace

// once per device, with that device current
asl_status asl_rank_ready() {
  ASL_CUDA(cudaFuncSetAttribute(rank_sort_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, sort_smem_bytes(1)));
  ASL_CUDA(cudaFuncSetAttribute(rank_sort_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, sort_smem_bytes(2)));
  ASL_CUDA(cudaFuncSetAttribute(rank_sort_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, sort_smem_bytes(4)));
  ASL_CUDA(cudaFuncSetAttribute(rank_split_kernel<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, split_smem_bytes<1024>()));
  ASL_CUDA(cudaFuncSetAttribute(rank_place_kernel<512>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PlaceSmem<512>)));
  ASL_CUDA(cudaFuncSetAttribute(rank_place_kernel<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PlaceSmem<1024>)));
  return ASL_OK;
}

asl_status asl_launch_rank(asl_ctx* c, const float* agg, int32_t layer_idx, int32_t n_rows, int32_t* ring,
                           asl_stat* stat, char* ws, cudaStream_t st) {
  const asl_params& p = c->p;
  uint32_t* keys[2] = {reinterpret_cast<uint32_t*>(ws + c->ws.rank_keys[0]),
                       reinterpret_cast<uint32_t*>(ws + c->ws.rank_keys[1])};
  int32_t* idx[2] = {reinterpret_cast<int32_t*>(ws + c->ws.rank_idx[0]),
                     reinterpret_cast<int32_t*>(ws + c->ws.rank_idx[1])};
  int32_t* hist = reinterpret_cast<int32_t*>(ws + c->ws.rank_hist);
  int32_t* row = ring + (int64_t)(layer_idx % p.l_obs) * c->sum_T;
  const asl_stat* latch = c->controller == ASL_CONTROLLER_LATCH ? stat : nullptr;
  const int evaluate = (layer_idx >= p.l_min && n_rows >= 2) ? 1 : 0;
  const StatArgs a{ring, c->d_req, c->d_acc, stat, c->sum_T, p.l_obs, layer_idx - n_rows + 1, n_rows, p.batch, layer_idx,
                   latch ? 1 : 0, p.tau};
  RowArgs r{agg, row, c->d_req, 0, reinterpret_cast<unsigned long long*>(keys[0]), reinterpret_cast<unsigned long long*>(idx[0]),
            reinterpret_cast<unsigned long long*>(hist), nullptr, 0, a, evaluate};
  const bool counted = p.batch == 1 && c->max_T <= COUNT_MAX_T;
  if (counted || sort_takes(c->max_T, c->sum_T, p.batch, c->sm_count)) {         // the statistic goes with the row
    if (counted) launch_count(r, c->max_T, st);
    else launch_row_sort(r, c->max_T, p.batch, st);
    c->launches += 1;
    ASL_CUDA(cudaGetLastError());
    return ASL_OK;
  }
  if (c->max_T <= SPLIT_MAX_T) c->launches += launch_split(r, c->max_T, p.batch, st);
  else c->launches += launch_sort(agg, c->d_req, latch, p.batch, c->max_T, keys, idx, hist, row, st);
  if (evaluate) {
    launch_after(rank_stat_accumulate, dim3((c->max_T + 256 * STAT_TOKENS - 1) / (256 * STAT_TOKENS), p.batch), dim3(256), st, a);
  } else {
    rank_stat_skip<<<(p.batch + 63) / 64, 64, 0, st>>>(c->d_req, stat, p.batch, layer_idx, n_rows, latch ? 1 : 0);
  }
  c->launches += 1;
  ASL_CUDA(cudaGetLastError());
  return ASL_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free rank row.
//
// Some hosts of this library are not allowed to allocate device memory while
// they run: a serving engine that hands its whole memory pool to its own
// allocator at start-up, a plugin called from inside another runtime's
// execution callback, code running under a "no cudaMalloc after init" rule.
// For them the scratch (two arrays of pairs and the table of bucket starts)
// lives in this file-scope device array; nothing in it has to start from a known
// value: every call writes what it reads.  Every device that loads the library carries these
// bytes until the process exits, which is why the segment length is capped.
//
// In host code `g_rank_static` is only a handle: the device address is asked
// for once per device with cudaGetSymbolAddress and that pointer is what the
// kernels get.
// ---------------------------------------------------------------------------
namespace {

constexpr int STATIC_MAX_T = ASL_RANK_STATIC_MAX_T;
constexpr int STATIC_MAX_DEVICES = 64;
static_assert(STATIC_MAX_T <= SPLIT_MAX_T, "the radix passes need a request table");

struct RankStaticScratch {
  unsigned long long pairs[STATIC_MAX_T], list[STATIC_MAX_T];
  unsigned long long table[1024 + SPLIT_MAX_TILES * split_pitch(1024) / 4];       // splitters, then the tiles' bucket starts
};

static __device__ __align__(256) unsigned char g_rank_static[sizeof(RankStaticScratch)];

struct RankStaticDevices {
  RankStaticScratch* ptr[STATIC_MAX_DEVICES] = {};
  asl_status status[STATIC_MAX_DEVICES] = {};
  bool done[STATIC_MAX_DEVICES] = {};
  std::mutex lock;
};

RankStaticDevices& rank_static_devices() {
  static RankStaticDevices d;
  return d;
}

// Once per device, with that device current: architecture check and the
// device address of the scratch array.
asl_status rank_static_setup(int device, RankStaticScratch** out) {
  RankStaticDevices& d = rank_static_devices();
  std::lock_guard<std::mutex> guard(d.lock);
  if (!d.done[device]) {
    asl_status st = ASL_OK;
    int major = 0;
    void* p = nullptr;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess) st = ASL_ERR_CUDA;
    else if (major != 10) st = ASL_ERR_ARCH;
    else if (cudaGetSymbolAddress(&p, g_rank_static) != cudaSuccess || !p || asl_rank_ready() != ASL_OK) st = ASL_ERR_CUDA;
    d.ptr[device] = static_cast<RankStaticScratch*>(p);
    d.status[device] = st;
    d.done[device] = st == ASL_OK || st == ASL_ERR_ARCH;     // a failed CUDA call is tried again by the next call
    if (st == ASL_ERR_CUDA) cudaGetLastError();
  }
  *out = d.ptr[device];
  return d.status[device];
}

}  // namespace

extern "C" asl_status asl_rank_desc_static(const float* scores, int32_t T, int32_t* rank_out, void* stream) {
  if (!scores || !rank_out || T < 1) return ASL_ERR_INVALID;
  if (T > STATIC_MAX_T) return ASL_ERR_WORKSPACE;      // the fixed scratch cannot hold this segment
  int device = -1;
  ASL_CUDA(cudaGetDevice(&device));
  if (device < 0 || device >= STATIC_MAX_DEVICES) return ASL_ERR_UNSUPPORTED;
  RankStaticScratch* s = nullptr;
  const asl_status ready = rank_static_setup(device, &s);
  if (ready != ASL_OK) return ready;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const RowArgs r{scores, rank_out, nullptr, T, s->pairs, s->list, s->table, nullptr, 0, StatArgs{}, 0};
  if (T <= COUNT_MAX_T) launch_count(r, T, st);
  else launch_split(r, T, 1, st);
  ASL_CUDA(cudaGetLastError());
  return ASL_OK;
}
