// K/V compaction (Algorithm 1 (K[I], V[I])): out[h][r][:] = x[tok_off + idx[h][r]][h][:].
// 16 threads move one row (256 bytes of bf16, 128 bytes of FP8 codes) as 16-byte vectors; K and V in one launch, four
// rows per thread with all eight loads in flight.  Bound by HBM's rate for scattered 256-byte rows: half of four 24K-token
// prompts' rows (223 MB moved) 50.5 us one row per thread -> 44.6 us (5.0 TB/s).
#include "asl_internal.cuh"

namespace {

constexpr int ROWS = 4;                   // rows per thread
constexpr int BLOCK_ROWS = 16 * ROWS;     // rows per 256-thread block

__global__ void __launch_bounds__(256) compact_kv_kernel(const uint8_t* __restrict__ k, const uint8_t* __restrict__ v,
                                                         const int32_t* __restrict__ idx, const AslReq* __restrict__ req,
                                                         int64_t ks_t, int64_t ks_h, int64_t vs_t, int64_t vs_h,
                                                         int64_t sum_kept, int k_vec, int v_vec, const asl_stat* __restrict__ latch,
                                                         int cur_layer, uint8_t* __restrict__ k_out,
                                                         uint8_t* __restrict__ v_out) {
  // strides in bytes; a row is k_vec (v_vec) 16-byte vectors; 16 threads per kept row
  pdl_wait_predecessor();
  const int b = blockIdx.z, h = blockIdx.y;
  if (latch && asl_finished(latch + b, cur_layer)) return;       // finished request: its compacted cache is final
  const AslReq rq = req[b];
  const int r0 = blockIdx.x * BLOCK_ROWS + threadIdx.x / 16;
  const int c = threadIdx.x % 16;
  if (blockIdx.x * BLOCK_ROWS >= rq.kept) return;
  const int64_t orow = (int64_t)h * sum_kept + rq.kept_off + r0;
  int64_t tok[ROWS];
#pragma unroll
  for (int i = 0; i < ROWS; ++i) tok[i] = r0 + 16 * i < rq.kept ? (int64_t)rq.tok_off + __ldcg(idx + orow + 16 * i) : -1;
  uint4 kv[ROWS], vv[ROWS];
#pragma unroll
  for (int i = 0; i < ROWS; ++i) {
    if (tok[i] >= 0 && c < k_vec) kv[i] = __ldcs(reinterpret_cast<const uint4*>(k + tok[i] * ks_t + (int64_t)h * ks_h + c * 16));
    if (tok[i] >= 0 && c < v_vec) vv[i] = __ldcs(reinterpret_cast<const uint4*>(v + tok[i] * vs_t + (int64_t)h * vs_h + c * 16));
  }
#pragma unroll
  for (int i = 0; i < ROWS; ++i) {
    if (tok[i] >= 0 && c < k_vec) __stcs(reinterpret_cast<uint4*>(k_out + ((orow + 16 * i) * k_vec + c) * 16), kv[i]);
    if (tok[i] >= 0 && c < v_vec) __stcs(reinterpret_cast<uint4*>(v_out + ((orow + 16 * i) * v_vec + c) * 16), vv[i]);
  }
}

// Row gather of one tensor with rows of `row_bytes` (a multiple of 16): out[kept_off_b + r] = x[tok_off_b + idx[r]].
// A warp moves one row, 16 bytes per lane, up to eight loads in flight (as written: they are not moved above the stores before
// them).  Bound by HBM where rows are long: 3.9K rows of 8 KB (64 MB moved) behind their top-k 37.6 -> 32.0 us for both.
// Rows of up to 2 KB take as many loads as they have, the registers of eight cost short rows their warps, and no streaming
// hint, which sends rows out of L2 that the next gather may find there.  30000 rows, us with eight / as many: of 64 bytes 5.5 /
// 3.9, 400 6.7 / 4.4, 528 7.1 / 4.9, 1040 8.1 / 7.7; 20000 of 2 KB with the hint 9.4, without 8.8.
template <int VECS>                       // vectors in flight per lane
__global__ void __launch_bounds__(256) compact_rows_kernel(const uint4* __restrict__ x, const int32_t* __restrict__ idx,
                                                           const AslReq* __restrict__ req, int vec_per_row,
                                                           uint4* __restrict__ out) {
  pdl_wait_predecessor();
  const int b = blockIdx.y;
  const AslReq rq = req[b];
  const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= rq.kept) return;
  const int64_t src = ((int64_t)rq.tok_off + __ldcg(idx + rq.kept_off + r)) * vec_per_row;
  const int64_t dst = ((int64_t)rq.kept_off + r) * vec_per_row;
  for (int c0 = lane; c0 < vec_per_row; c0 += 32 * VECS) {
    uint4 v[VECS];
#pragma unroll
    for (int q = 0; q < VECS; ++q)
      if (c0 + 32 * q < vec_per_row) v[q] = VECS == 8 ? __ldcs(x + src + c0 + 32 * q) : __ldcg(x + src + c0 + 32 * q);
#pragma unroll
    for (int q = 0; q < VECS; ++q)
      if (c0 + 32 * q < vec_per_row) out[dst + c0 + 32 * q] = v[q];
  }
}

}  // namespace

asl_status asl_launch_compact_rows(asl_ctx* c, const void* x, const int32_t* idx, void* out, int64_t row_bytes,
                                   cudaStream_t st) {
  dim3 grid((c->max_kept + 7) / 8, c->p.batch);
  const int vec_per_row = (int)(row_bytes / 16);
  const auto kernel = vec_per_row > 128 ? compact_rows_kernel<8> : vec_per_row > 64 ? compact_rows_kernel<4>
                      : vec_per_row > 32 ? compact_rows_kernel<2> : compact_rows_kernel<1>;
  launch_after(kernel, grid, dim3(256), st, static_cast<const uint4*>(x), idx, c->d_req, vec_per_row, static_cast<uint4*>(out));
  c->launches += 1;
  ASL_CUDA(cudaGetLastError());
  return ASL_OK;
}

asl_status asl_launch_compact(asl_ctx* c, const void* k, const void* v, const int32_t* idx, void* k_out, void* v_out,
                              cudaStream_t st) {
  const asl_params& p = c->p;
  const int kb = c->k_elem_bytes;                          // K elements are 2 bytes (bf16) or 1 (FP8 codes), V is bf16
  const int k_vec = p.head_dim * kb / 16, v_vec = p.head_dim * 2 / 16;
  dim3 grid((c->max_kept + BLOCK_ROWS - 1) / BLOCK_ROWS, p.n_kv_heads, p.batch);
  launch_after(compact_kv_kernel, grid, dim3(256), st, static_cast<const uint8_t*>(k), static_cast<const uint8_t*>(v), idx, c->d_req,
                                          p.k_stride[0] * kb, p.k_stride[1] * kb, p.v_stride[0] * 2, p.v_stride[1] * 2,
                                          c->sum_kept, k_vec, v_vec, c->latch_stat, c->cur_layer,
                                          static_cast<uint8_t*>(k_out), static_cast<uint8_t*>(v_out));
  c->launches += 1;
  ASL_CUDA(cudaGetLastError());
  return ASL_OK;
}
