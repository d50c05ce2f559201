// 1-D pooling, GQA group sum and all-head aggregate (Algorithm 1 (1-D pooling, SumGroups) and
// the "scores" sum of Section 4.1).  A thread walks all heads of its tokens, so the
// aggregate needs no atomics and is bit-reproducible.  A "unit" is what gets pooled as one
// row: a kv head's group-summed sums (average pooling) or one query head's sums (max
// pooling); the scorer stores it as `nrows` consecutive partial rows that are added first.
//   average pooling: pooling is linear, so summing the group first is the same up to
//                    rounding; zero padding, divisor always S.
//   max pooling:     each head is pooled over its in-range taps, then the group is summed.
// Taps never cross a request's past segment [0, T_b).
#include "asl_internal.cuh"

namespace {

constexpr int PT = 256;          // threads of a block / tokens per block of the general kernel
constexpr int MAX_HALO = 16;     // pooling kernels up to 33 taps
constexpr int HB = 8;            // general kernel: staged units per round
constexpr int PV_ROWS = 8;       // vector kernel: partial rows in flight per lane, where a head has few
constexpr int PV_THREADS = 128;

struct PoolArgs {
  const float* u;                // [rows][u_stride], every request from a 16-byte boundary on
  const AslReq* req;
  int64_t u_stride, sum_T;
  int32_t Hk, G, S, mode, nrows; // nrows: partial rows per unit
  const asl_stat* latch;
  int32_t cur_layer, vec_out;    // vec_out: every request starts on 16 bytes in the outputs too
  float* scores_kv;
  float* scores_agg;
};

// Windows of up to 9 taps, units of 1, 2, 4, 8 or 16 partial rows.  A lane owns 4 consecutive tokens: one 16-byte load per
// partial row, the rows of a unit added in order, the neighbours' sums fetched by warp shuffles; the
// first and the last lane of a warp only supply the halo, so a warp pools 120 tokens.  No shared memory and no
// block-wide barrier.  Bound by the round trips for the rows.  In flight at a time: eight rows where a kv head has few (with
// sixteen the registers leave room for half as many warps on the SMs that a scorer leaves: eight layers of 32K tokens
// 434.3 -> 431.7 us), sixteen or two units where there are many.  The loads of a single unit in flight the compiler spreads
// among its adds, those ahead of the test for a second unit it issues together.  Us at 8 / 16 / 32 in flight: 65536 tokens,
// average of 8 kv heads with 8 rows each 7.8 / 4.2 (16 before), of 4 with 16 rows - / 10.0 / 3.5 (7.3 before), max of 64
// query heads with 4 rows each 18.7 / 15.2, with 2 9.5 / 8.7, with one 7.4 / 8.8; average of 8 with 4 rows 3.4 / 4.7.
// 128K tokens of 8 heads, two rows each, 3.3.
template <bool MAX, int R, int NR>
__global__ void __launch_bounds__(PV_THREADS) pool_vec4_kernel(PoolArgs a) {
  constexpr int IN_FLIGHT = NR >= 8 ? 2 * NR : MAX && NR >= 2 ? 16 : PV_ROWS;
  constexpr bool ALL_LANES = !MAX && NR >= 8;                          // lanes outside load too, from the segment's first tokens
  pdl_wait_predecessor();
  const int b = blockIdx.y;
  if (a.latch && asl_finished(a.latch + b, a.cur_layer)) return;       // the request's scores stay as its selection layer left them
  const AslReq rq = a.req[b];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int warp_of_segment = blockIdx.x * (PV_THREADS / 32) + wid;
  if (warp_of_segment * 120 >= rq.T) return;                           // the whole warp is past the segment
  const int j0 = 4 * (warp_of_segment * 30 + lane - 1);                // lanes 0 and 31: halo only
  const bool inside = j0 >= 0 && j0 < rq.T;
  const bool owner = inside && lane >= 1 && lane <= 30;
  const int live = rq.T - j0;                                          // tokens from j0 on (4 or more: all of the lane's)
  const float outside = MAX ? -INFINITY : 0.f;
  const float inv = 1.0f / (float)a.S;
  const float* base = a.u + rq.u_off + (ALL_LANES && !inside ? 0 : j0);
  const int per_head = MAX ? a.G : 1, units = a.Hk * per_head, rows = units * NR;
  auto store = [&](float* dst, const float (&p)[4]) {
    if (a.vec_out && live >= 4) *reinterpret_cast<float4*>(dst) = make_float4(p[0], p[1], p[2], p[3]);
    else
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (t < live) dst[t] = p[t];
  };
  float agg[4] = {0.f, 0.f, 0.f, 0.f}, head[4] = {0.f, 0.f, 0.f, 0.f};
  int in_head = 0, h = 0;
  for (int r0 = 0; r0 < rows; r0 += IN_FLIGHT) {
    float4 x[IN_FLIGHT];
#pragma unroll
    for (int e = 0; e < IN_FLIGHT; ++e)
      x[e] = ((ALL_LANES || inside) && r0 + e < rows) ? __ldcg(reinterpret_cast<const float4*>(base + (int64_t)(r0 + e) * a.u_stride)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int q = 0; q < IN_FLIGHT / NR; ++q) {
      if (r0 + q * NR >= rows) break;
      float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int e = 0; e < NR; ++e) { sum.x += x[q * NR + e].x; sum.y += x[q * NR + e].y; sum.z += x[q * NR + e].z; sum.w += x[q * NR + e].w; }
      float v[12];                                                     // tokens j0-4 .. j0+7
      v[4] = live > 0 && inside ? sum.x : outside; v[5] = live > 1 && inside ? sum.y : outside;
      v[6] = live > 2 && inside ? sum.z : outside; v[7] = live > 3 && inside ? sum.w : outside;
#pragma unroll
      for (int d = 0; d < R; ++d) {
        v[3 - d] = __shfl_up_sync(0xffffffffu, v[7 - d], 1);
        v[8 + d] = __shfl_down_sync(0xffffffffu, v[4 + d], 1);
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        float p = MAX ? v[4 + t - R] : 0.f;
#pragma unroll
        for (int d = -R; d <= R; ++d) p = MAX ? fmaxf(p, v[4 + t + d]) : p + v[4 + t + d];
        head[t] = MAX ? head[t] + p : p * inv;
      }
      if (++in_head == per_head) {
        if (owner) store(a.scores_kv + (int64_t)h * a.sum_T + rq.t_off + j0, head);
#pragma unroll
        for (int t = 0; t < 4; ++t) { agg[t] += head[t]; head[t] = 0.f; }
        in_head = 0;
        ++h;
      }
    }
  }
  if (owner) store(a.scores_agg + rq.t_off + j0, agg);
}

// Everything else: one block pools PT consecutive past tokens of one request, one thread per column of the tile (the
// last 2 * MAX_HALO threads load the halo); HB units are staged per round in shared memory and pooled from there.
__global__ void __launch_bounds__(PT + 2 * MAX_HALO) pool_group_kernel(PoolArgs a) {
  __shared__ float tile[HB][PT + 2 * MAX_HALO];
  pdl_wait_predecessor();
  const int b = blockIdx.y;
  if (a.latch && asl_finished(a.latch + b, a.cur_layer)) return;
  const AslReq rq = a.req[b];
  const int j0 = blockIdx.x * PT;
  if (j0 >= rq.T) return;
  const int r = a.S / 2;
  const int j = j0 + threadIdx.x;
  const bool live = threadIdx.x < PT && j < rq.T;
  const int lo = max(0, j - r), hi = min(rq.T - 1, j + r);
  const float inv = 1.0f / (float)a.S;
  const bool avg = a.mode == ASL_POOL_AVG;
  const int per_head = avg ? 1 : a.G, units = a.Hk * per_head;
  float agg = 0.f, p = 0.f;
  for (int u0 = 0; u0 < units; u0 += HB) {
    const int nb = min(HB, units - u0);
    const int tot = nb * a.nrows;                     // rows u0*nrows .. u0*nrows + tot - 1 of u
    __syncthreads();
    if (threadIdx.x < PT + 2 * r) {                     // one column of the tile per thread, halo included
      const int i = threadIdx.x;
      const int t = j0 - r + i;
      const bool inside = t >= 0 && t < rq.T;
      const float* src = a.u + (int64_t)u0 * a.nrows * a.u_stride + rq.u_off + t;
#pragma unroll
      for (int q = 0; q < HB; ++q) tile[q][i] = 0.f;
      for (int e0 = 0; e0 < tot; e0 += 16) {            // sixteen loads in flight
        float x[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) x[k] = (inside && e0 + k < tot) ? __ldcg(src + (int64_t)(e0 + k) * a.u_stride) : 0.f;
#pragma unroll
        for (int k = 0; k < 16; ++k)
          if (e0 + k < tot) tile[(e0 + k) / a.nrows][i] += x[k];
      }
    }
    __syncthreads();
    for (int q = 0; q < nb; ++q) {
      if (live) {
        if (avg) {
          float s = 0.f;
          for (int i = lo; i <= hi; ++i) s += tile[q][i - j0 + r];
          p = s * inv;
        } else {
          float mx = tile[q][lo - j0 + r];
          for (int i = lo + 1; i <= hi; ++i) mx = fmaxf(mx, tile[q][i - j0 + r]);
          p += mx;
        }
      }
      const int unit = u0 + q;
      if ((unit + 1) % per_head == 0) {
        if (live) a.scores_kv[(int64_t)(unit / per_head) * a.sum_T + rq.t_off + j] = p;
        agg += p;
        p = 0.f;
      }
    }
  }
  if (live) a.scores_agg[rq.t_off + j] = agg;
}

using PoolKernel = void (*)(PoolArgs);
template <bool MAX, int R>
PoolKernel pool_vec4_rows(int nrows) {
  switch (nrows) {
    case 1: return pool_vec4_kernel<MAX, R, 1>;
    case 2: return pool_vec4_kernel<MAX, R, 2>;
    case 4: return pool_vec4_kernel<MAX, R, 4>;
    case 8: return pool_vec4_kernel<MAX, R, 8>;
    case 16: return pool_vec4_kernel<MAX, R, 16>;
  }
  return nullptr;
}
template <bool MAX>
PoolKernel pool_vec4_of(int r, int nrows) {
  switch (r) {
    case 0: return pool_vec4_rows<MAX, 0>(nrows);
    case 1: return pool_vec4_rows<MAX, 1>(nrows);
    case 2: return pool_vec4_rows<MAX, 2>(nrows);
    case 3: return pool_vec4_rows<MAX, 3>(nrows);
    case 4: return pool_vec4_rows<MAX, 4>(nrows);
  }
  return nullptr;
}

}  // namespace

asl_status asl_launch_pool(asl_ctx* c, const float* u, float* scores_kv, float* scores_agg, cudaStream_t st) {
  const asl_params& p = c->p;
  const int r = p.pool_kernel / 2;
  if (r > MAX_HALO) return ASL_ERR_UNSUPPORTED;
  const bool max = p.pool_mode == ASL_POOL_MAX;
  const int nrows = max ? c->u_parts : c->u_rows_per_kv;
  bool vec_out = c->sum_T % 4 == 0 && ((reinterpret_cast<uintptr_t>(scores_kv) | reinterpret_cast<uintptr_t>(scores_agg)) & 15) == 0;
  for (const AslReq& q : c->req) vec_out = vec_out && q.t_off % 4 == 0;
  const PoolArgs a{u, c->d_req, c->u_stride, c->sum_T, p.n_kv_heads, p.n_q_heads / p.n_kv_heads, p.pool_kernel, p.pool_mode, nrows,
                   c->latch_stat, c->cur_layer, vec_out, scores_kv, scores_agg};
  if (const PoolKernel vec4 = max ? pool_vec4_of<true>(r, nrows) : pool_vec4_of<false>(r, nrows)) {
    const int warps = (c->max_T + 119) / 120;
    launch_after(vec4, dim3((warps + PV_THREADS / 32 - 1) / (PV_THREADS / 32), p.batch), dim3(PV_THREADS), st, a);
  } else {
    launch_after(pool_group_kernel, dim3((c->max_T + PT - 1) / PT, p.batch), dim3(PT + 2 * MAX_HALO), st, a);
  }
  c->launches += 1;
  ASL_CUDA(cudaGetLastError());
  return ASL_OK;
}
