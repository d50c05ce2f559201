// Plan of the tensor-core scorer: how the query rows of a kv head are cut into chunks, and the work lists built at
// plan time (or ahead of a launch that leaves finished requests out).
#pragma once
#include <stdint.h>
#include <vector>

constexpr int ASL_TC_KEY_TILE = 128;

#ifdef __CUDACC__
#define ASL_HD __host__ __device__
#else
#define ASL_HD
#endif

// A run: the tiles of one segment = (request, kv head, row chunk) that one CTA takes in one pass; `next`: the CTA's next
// run (-1: none).  (T, u_off, tok_off: the request's past length, offset in the rows of column sums and first token, copied here so that one
// record is all a role needs; rows: query rows of the chunk that exist; kscale: factor between the accumulator and q.k,
// 1 for bf16 keys and k_scale[h] / 16 for FP8 keys, whose queries are scaled by 16 before they are split into two E4M3
// terms; slot: number of the run among its pass's; group of segments; cta:
// whom the plan gave it)
struct __align__(16) TcRun { int32_t tile0, ntiles, pass, seg, b, h, chunk, next, T, u_off, tok_off, rows; float kscale; int32_t slot, group, cta; };

// A group of segments: seg0 .. seg0 + nseg - 1.
struct __align__(16) TcStage { int32_t seg0, nseg, pad0, pad1; };

// What the fold of a segment's softmax denominators needs: the pass-1 runs that publish, in slot order.
struct __align__(16) TcFold { int32_t slot0, nruns, rows, b; };

struct TcList {                  // a work list on the device: runs of pass 1, then of pass 2
  int32_t grid = 0;              // CTAs it is dealt to
  int32_t n1 = 0, n2 = 0, n_groups = 0;
  int32_t most = 0;              // tiles of the largest group
  TcRun* d_runs = nullptr;
  int32_t* d_first = nullptr;    // [grid] first run of every CTA
  TcStage* d_stages = nullptr;
  TcFold* d_folds = nullptr;     // [segments]
};

struct AslTcPlan {
  int NC = 0;           // rows of a chunk's buffer (halves of HR)
  int HR = 0;           // rows of a half: one accumulator of pass 1 (lanes) or pass 2 (columns), a multiple of 32, at most 128
  bool wide = false;    // two halves
  int Wp = 0;           // buffer rows from one query head to the next (the window, padded under max pooling; 256 if longer)
  int m = 0;            // query heads of a chunk
  int pieces = 0;       // chunks per query head (windows of more than 256 rows), else 1
  int nchunk = 0;       // chunks per kv head
  int nseg = 0;         // segments
  // [0]: a call on its own; [1]: a call that other kernels should find room beside (asl_score_columns).  The same where
  // the caller gives the number of CTAs.  [][0]: both passes; [][1]: pass 2 alone (a supplied log-sum-exp).
  TcList lists[2][2];
  void* d_blob = nullptr;       // the device side of the lists below and above, one allocation
  uint32_t* d_sync = nullptr;   // two sets of publish counters, launch number, ticket of arrived CTAs, two sets of offsets
  // device-side controller: the next launch's list without the finished requests' phases, written ahead of it
  TcRun* d_live_runs = nullptr;
  int32_t* d_live_first = nullptr;
  TcFold* d_live_folds = nullptr;
  int32_t* d_live_hdr = nullptr;
  int32_t* d_live_scratch = nullptr;
  int64_t partial_slots = 0;    // pass-1 runs of the longest list
};
