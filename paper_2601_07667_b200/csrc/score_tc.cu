// Observation-window scorer on the 5th-generation tensor cores (Algorithm 1 (window softmax A, past-only column sum U)).
//
// One persistent kernel, one CTA per SM, does both softmax passes of every
// (request, kv head, row chunk) "segment":
//
//   pass 1  D[row][key] = Q_chunk . K_tile^T  (query rows in TMEM lanes): each
//           epilogue thread keeps, for its row, the sum of 2^(x - ref) over the
//           keys it meets (ref: its first logit of the run); at the
//           end of a CTA's run of tiles each epilogue group publishes (ref, sum) per
//           row.  Once every group has published, a helper warp per CTA folds the
//           partials of "their" rows, in a fixed order, into offset[row] = log2 of
//           the row's softmax denominator, off the epilogue's critical path.
//   pass 2  D[key][row] = K_tile . Q_chunk^T  (keys in TMEM lanes): exp2(x -
//           offset[row]) summed over the chunk's rows: the key's column sum U,
//           already summed over the GQA group.
//
// All arithmetic is in the log2 domain x = (q.k) * log2(e)/sqrt(d).  A "chunk" is
// up to 256 of the G*W query rows that share a kv head.  Work is dealt in "runs": the
// contiguous tiles that one CTA takes of one segment in one pass.  Segments form groups;
// a CTA does its runs of pass 1 of group i, then those of pass 2 of group i - 1: it
// meets one or two segments at a time and keeps a Q chunk for a whole run, and the
// offsets that pass 2 needs were folded while other tiles were worked on.  Between the two
// reads of a tile lie up to two groups (up to 140 MB each): of 268 MB of K (128K
// tokens, 8 kv heads) pass 2 finds a quarter in L2 (464 MB are read from DRAM; in groups of 70 MB 438).  Dealing every segment's tiles round-robin
// to all CTAs cost 3 us per segment and pass (64 KB of Q reloaded per CTA, a hand-off each):
// 32K tokens, 8 kv heads 64 -> 48 us, eight ragged requests with W = 32 350 -> 184 us,
// W = 128 with 64 query heads at 64K 374 -> 288 us, 128K tokens 163 -> 153 us.
//
// What bounds it: two exponentials per logit, and power.  Of every 16 column pairs 3
// take a degree-4 polynomial on the FMA pipe, the others the MUFU unit (16 per clock and
// SM): a tile of 128 keys x 256 rows is 32768 of them, 1664 clk of MUFU, and the loop
// takes about 1950 in the kernel.  Kept up for more than some
// ten milliseconds the kernel runs at the 1000 W limit: at 128K tokens a layer takes 193 to
// 204 us (two boards, at 1.62 and 1.55 GHz, 990 W: 191 to 201 mJ; one pass over K 108 to 113
// us), and 166 to 170 us in a burst at 1.97 GHz.
//
// Inside a CTA: warp 0 streams K tiles through a TMA ring (128B-swizzled) and keeps the Q
// chunks of two runs resident; warp 1 issues tcgen05.mma from a warp-uniform loop (under
// a one-thread branch an MMA of 128 columns takes 90-110 clk instead of 64-73) into four
// 128-column accumulators; warp 2 folds, warp 3 fetches offsets; four groups of four
// epilogue warps own one accumulator each, so that up to three groups compute while one
// accumulator fills.  The accumulator is read 16 registers at a time, double buffered.
// Pass 2 reads it in the 16x256b shape, in which a thread meets only every fourth column
// pair and can keep its rows' offsets in registers: broadcast loads of the offsets from
// shared memory (131 KB per tile) cost 400 clk.
//
// Every wait (mbarrier, counter) is bounded: when the limit is reached the thread
// records a code in the context's error word and the CTA drains: producers stop,
// the epilogue keeps walking its barrier sequence without waiting or computing,
// in-flight copies are waited for with the same bound and tensor memory is freed.
#include <cuda.h>
#include <cuda_fp8.h>
#include <string.h>

#include "asl_internal.cuh"

namespace {

constexpr int KT = ASL_TC_KEY_TILE;          // keys per tile
constexpr int MAX_ROWS = 256;                // query rows of a chunk at most
constexpr int THREADS = 640;                 // warp 0: TMA, 1: MMA, 2-3: partial folding, 4-19: four epilogue groups
constexpr int GROUPS = 4;
constexpr unsigned long long OFFSET_READY = 1ull << 32;
constexpr int SYNC_STRIDE = 8;               // words from one segment's counter to the next: a sector each
constexpr unsigned long long WAIT_LIMIT_NS = 2000000000ull;   // every wait gives up after 2 s

// Shared-memory layout of one CTA (offsets from the 1024-aligned base).  WIDE: a chunk of more than 128 rows.
template <bool FP8, bool WIDE>
struct Smem {
  static constexpr int Q_ROWS = WIDE ? 256 : 128;
  static constexpr int Q_BLOCK = Q_ROWS * 128;              // a 64-channel block (FP8: an E4M3 term) of a Q chunk
  static constexpr int Q_BUF = 2 * Q_BLOCK;
  static constexpr int HALF = KT * 128;                     // a 64-channel block of a K tile: 128 rows x 128 B
  static constexpr int STAGE = FP8 ? HALF : 2 * HALF;
  static constexpr int NSTAGE = (WIDE ? 98304 : 163840) / STAGE;
  static constexpr int K = 2 * Q_BUF;                       // two Q chunks, then the ring of K tiles
  static constexpr int BARS = K + NSTAGE * STAGE;
  static constexpr int FULL = 0, EMPTY = NSTAGE, TFULL = 2 * NSTAGE, TEMPTY = TFULL + GROUPS, QFULL = TEMPTY + GROUPS,
                       QEMPTY = QFULL + 2, OFULL = QEMPTY + 2, OEMPTY = OFULL + 2, DRAIN = OEMPTY + 2, N_BARS = DRAIN + 1;
  static constexpr int MISC = BARS + 384;                   // tmem base, abort flag, launch number and its parity
  static constexpr int OFFS = MISC + 64;                    // float[2][256]: -offset of the rows of two pass-2 runs
  static constexpr int BYTES = OFFS + 2048;
  static_assert(N_BARS * 8 <= 384 && BYTES <= 232448, "shared memory budget of one CTA");
};

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long now;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
  return now;
}
// Looks once, without suspending the thread.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait.  `watch_abort`: also give up when another role raised the flag.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int code,
                                          bool watch_abort, unsigned long long limit_ns = WAIT_LIMIT_NS) {
  unsigned long long t0 = 0;
  for (uint32_t it = 0;; ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 15u) == 15u) {
      if (watch_abort && *abort_flag) return false;
      const unsigned long long now = global_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) break;
    }
  }
  *abort_flag = code;
  return false;
}
__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
// Bounded wait until the 32-bit word at p equals `want` (acquire).  Lane 0 polls.
__device__ __forceinline__ bool word_wait(const uint32_t* p, uint32_t want, volatile int* abort_flag, int code, int lane,
                                          uint32_t nap_max, unsigned long long limit_ns = WAIT_LIMIT_NS) {
  int gave_up = 0;
  if (lane == 0) {
    unsigned long long t0 = 0;
    uint32_t nap = 64;
    for (uint32_t it = 0;; ++it) {
      uint32_t v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
      if (v == want) break;
      if ((it & 7u) == 7u) {
        const unsigned long long now = global_ns();
        if (t0 == 0) t0 = now;
        else if (now - t0 > limit_ns || *abort_flag) { gave_up = 1; if (!*abort_flag) *abort_flag = code; break; }
      }
      if (it >= 16) {                    // the first looks follow one another at once: what is waited for is about to come
        __nanosleep(nap);
        if (nap < nap_max) nap <<= 1;
      }
    }
  }
  return __shfl_sync(0xffffffffu, gave_up, 0) == 0;
}

// L2 eviction policies for the K stream: pass 1 asks L2 to keep what pass 2 will read again, pass 2
// (and a launch that has only pass 2) marks what it reads as the first to go.
__device__ __forceinline__ uint64_t l2_policy_keep() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint64_t l2_policy_stream() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1, int c2,
                                            uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;" ::"r"(dst),
      "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1, int c2,
                                            int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(
          dst),
      "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}

__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1, int c2,
                                            int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(
          dst),
      "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem], bf16 x bf16 -> fp32
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accum)
      : "memory");
}
// the same with 8-bit operands (E4M3 x E4M3 -> fp32), 32 channels per instruction
__device__ __forceinline__ void tc_mma_f8(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accum)
      : "memory");
}
// 16 registers of an accumulator: issue only; they hold the data after tc_ld_wait on the same array.
// Shape 32x32b: 16 consecutive columns of this thread's lane.
__device__ __forceinline__ void tc_ld_lane(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// Shape 16x256b: 16 lanes x 32 columns; registers 4i..4i+3 of thread t hold columns 8i + 2(t%4) + {0, 1} of lanes
// t/4 and t/4 + 8.
__device__ __forceinline__ void tc_ld_quad(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// Waits for every tcgen05.ld this thread has issued.  The array is an in/out
// operand so that no use of its registers can be scheduled above the wait.
__device__ __forceinline__ void tc_ld_wait(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void bar_sync(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// ---- two fp32 values in one 64-bit register: the FMA pipe takes fma on such pairs as
//      one instruction, which halves the issue slots of the softmax arithmetic ----
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ f32x2 pku(uint32_t lo, uint32_t hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
  return r;
}
__device__ __forceinline__ void upk(f32x2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ void upku(f32x2 v, uint32_t& lo, uint32_t& hi) { asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(v)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float hsum(f32x2 v) {
  float lo, hi;
  upk(v, lo, hi);
  return lo + hi;
}
// 2^x of a pair on the MUFU unit
__device__ __forceinline__ f32x2 ex2_pair_mufu(f32x2 x) {
  float a, b;
  upk(x, a, b);
  return pk(ex2(a), ex2(b));
}
// 2^x of a pair on the FMA pipe: clamp at -125, round to the nearest
// integer n with the 1.5*2^23 trick, degree-4 minimax polynomial of 2^f on
// f = x - n in [-0.5, 0.5] (relative error 2.6e-6), n added into the exponent field.
// Packed additions are written as such, not as fma(a, 1, b): as fast, and six constant registers fewer.
// ABOVE: x may lie above the fp32 range, and then comes out as infinity or NaN, as a sum that looks for an overflow
// needs it: n = 129 fills the exponent field.  Without the upper clamp n runs into the sign bit there (2^130 as
// -1.2e-38, 2^300 as -1.8e13).  Pass 2 has no such x: a logit is not above the log2 of its row's softmax denominator.
// (The two more instructions a pair: eight layers of 32K tokens 466 -> 470 us, 0.9 to 1.5 % over the runs, four of 128K
// 820 -> 821, 0.2 to 0.7 %, two prompts with W = 24 31.2 -> 31.7.  Tried: the largest x kept by one three-way maximum a pair, 1.3 to 1.5 and 0.7 to 1.9 %; 2 or 1
// of 16 pairs polynomial in pass 1, 1.8 and 1.5 to 2.5 %.)
template <bool ABOVE>
__device__ __forceinline__ f32x2 ex2_pair_poly(f32x2 x) {
  float a, b;
  upk(x, a, b);
  if (ABOVE) { a = fminf(a, 129.0f); b = fminf(b, 129.0f); }
  const f32x2 xc = pk(fmaxf(a, -125.0f), fmaxf(b, -125.0f));
  const f32x2 magic = pk(12582912.0f, 12582912.0f);
  const f32x2 t = add2(xc, magic);
  const f32x2 f = sub2(xc, sub2(t, magic));
  f32x2 p = fma2(pk(0.00956967473f, 0.00956967473f), f, pk(0.0559182465f, 0.0559182465f));
  p = fma2(p, f, pk(0.240247667f, 0.240247667f));
  p = fma2(p, f, pk(0.693121731f, 0.693121731f));
  p = fma2(p, f, pk(0.999999225f, 0.999999225f));
  uint32_t tl, th, pl, ph;
  upku(t, tl, th);
  upku(p, pl, ph);
  return pku(pl + (tl << 23), ph + (th << 23));
}
// Which of every 16 column pairs take the polynomial, spread out.  3: the loop alone is shortest at 5 (clk per tile,
// pass 1 / pass 2, at 4, 5, 6: 1821 / 1833, 1725 / 1794, 1747 / 1839), but a polynomial takes more
// registers; in the kernel, at 128K tokens: 155.4, 156.9, 160.9 us at 3, 4, 5.
constexpr int POLY_OF_16 = 3;
__device__ __forceinline__ constexpr bool pair_is_poly(int i) { return ((i & 15) * POLY_OF_16) % 16 + POLY_OF_16 >= 16; }

// K-major, 128B-swizzled operand: rows of 128 B, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)64 << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)2 << 61);
}
// kind::f16, A = B = bf16, D = fp32, both operands K-major
__device__ __forceinline__ uint32_t instr_desc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// kind::f8f6f4, A = B = E4M3 (format code 0), D = fp32, both operands K-major
__device__ __forceinline__ uint32_t instr_desc_f8(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}


struct TcWork {
  const TcRun* runs;
  const int32_t* first;    // [grid] first run of every CTA, or -1
  const TcFold* folds;     // [segments]
};
struct TcArgs {
  TcWork list, live;       // the plan's list; the one without finished requests, to be taken where live_hdr[0] is set
  const int32_t* live_hdr; // or null
  const TcStage* stages;   // groups of segments whose rows are folded together
  float2* partials;        // pass 1: [run slot][entry][NC] (reference, sum) of every row
  float* offsets;          // [segment][NC], written by the folding warps, read by pass 2
  const float* lse;        // null, or the rows' natural-log softmax denominators [B][H_q][W]: pass 2 alone
  float* u;                // pass 2 out: column sums
  // [2][segment * SYNC_STRIDE]: epilogue groups of the segment that have published.
  // A launch counts in the set that its number's parity names; the last CTA to arrive clears the other set (whose launch
  // is over), advances the number and resets the ticket.  The number lives on the device so that a launch replayed from
  // a CUDA graph counts like any other, and is switched at entry so that no CTA has anything to do at its end.
  uint32_t* counters;
  // [2][segment][NC], sets as above: a row's offset with OFFSET_READY above it, or zero.  The folding warps write the value
  // and the flag in one word, so that who waits for it has it with the look that finds it there, and nothing is fenced; they
  // clear the same rows of the other set.  (A counter of folded rows behind a fence, then a load of the offsets, were two
  // round trips more in front of pass 2: 4096 tokens 18.3 -> 14.2 us, two prompts with W = 24 23 -> 20, 32K 46.2 -> 45.7,
  // 128K 163.7 -> 164.1.)
  unsigned long long* ready;
  uint32_t* launch;        // launch number, then the ticket of arrived CTAs
  int32_t* err;
  int64_t u_stride;
  int32_t n_stages, nseg, NC, HR, W, Wp, m, pieces, G, Hq, u_rows_per_kv, u_parts;
  float scale_log2;
};

// Row r of chunk ch is row t of query head g of its kv head (under max pooling heads start at multiples of Wp > W and
// rows t >= W do not exist; a window of more than 256 rows is cut into pieces, one per chunk).
struct RowPlace { int g, t; };
__device__ __forceinline__ RowPlace row_place(const TcArgs& a, int ch, int r) {
  if (a.pieces > 1) return {ch / a.pieces, (ch % a.pieces) * MAX_ROWS + r};
  return {ch * a.m + r / a.Wp, r % a.Wp};
}

__device__ __forceinline__ TcRun load_run(const TcRun* runs, int slot) {
  TcRun r;
  const int4* s = reinterpret_cast<const int4*>(runs + slot);
  int4* d = reinterpret_cast<int4*>(&r);
#pragma unroll
  for (int i = 0; i < 4; ++i) d[i] = __ldg(s + i);
  return r;
}
__device__ __forceinline__ void prefetch_run(const TcRun* runs, int slot) {
  if (slot >= 0) asm volatile("prefetch.global.L1 [%0];" ::"l"(runs + slot));
}

// FP8: K tiles hold E4M3 codes (one 128-byte row per key: a tile is one 16 KB box), the query chunk holds
// the two E4M3 terms of every query (term t in the t-th block of the chunk's buffer, where bf16
// queries keep their t-th 64-channel block), and a tile takes 2 terms x 4 k-steps of 32 channels.
// A unit = one accumulator: a 128-key tile x one half of the chunk's rows; units are numbered through all of the
// CTA's runs and group g takes units g, g + 4, ...
// FULL: halves of 128 rows (the block loop of pass 2 then has no branches: 128K tokens 171 -> 163 us).
template <bool PER_Q, bool FP8, bool WIDE, bool FULL>
__global__ void __launch_bounds__(THREADS, 1)
score_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k, const TcArgs a) {
  using S = Smem<FP8, WIDE>;
  constexpr int HV = WIDE ? 2 : 1;
  constexpr int ENTRIES = GROUPS / HV;          // groups that meet a row; entry e: tiles e, e + ENTRIES, ... of the run
  extern __shared__ __align__(1024) uint8_t smem[];
  const uint32_t sbase = smem_u32(smem);
  if (sbase & 1023u) {                       // the swizzled operand layout needs a 1024-byte aligned base
    if (threadIdx.x == 0) atomicCAS(a.err, 0, 901);
    return;
  }
  volatile uint32_t* s_tmem = reinterpret_cast<volatile uint32_t*>(smem + S::MISC);
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + S::MISC + 4);
  volatile uint32_t* s_number = reinterpret_cast<volatile uint32_t*>(smem + S::MISC + 8);     // this launch's number
  volatile uint32_t* s_set = reinterpret_cast<volatile uint32_t*>(smem + S::MISC + 12);     // its parity
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int HR = FULL ? 128 : a.HR;
  auto bar = [&](int i) { return sbase + S::BARS + 8u * (uint32_t)i; };
  const bool dense = a.Wp == a.W || a.pieces > 1;             // one copy brings all rows of a chunk
  const int copies = dense ? 1 : a.m;
  const int box_rows = a.pieces > 1 ? MAX_ROWS : (dense ? a.m * a.W : a.W);

  // ---- set-up: zero the Q buffers (rows that no copy writes feed unused MMA rows), barriers, tensor memory ----
  if (copies * box_rows < S::Q_ROWS)
    for (int i = threadIdx.x; i < 2 * S::Q_BUF / 16; i += THREADS) reinterpret_cast<uint4*>(smem)[i] = make_uint4(0, 0, 0, 0);
  if (threadIdx.x == 32) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_q) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tm_k) : "memory");
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < S::NSTAGE; ++s) { mbar_init(bar(S::FULL + s), 1); mbar_init(bar(S::EMPTY + s), 1); }
    for (int i = 0; i < GROUPS; ++i) { mbar_init(bar(S::TFULL + i), 1); mbar_init(bar(S::TEMPTY + i), 4); }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(S::QFULL + i), 1); mbar_init(bar(S::QEMPTY + i), 1);
      mbar_init(bar(S::OFULL + i), 1); mbar_init(bar(S::OEMPTY + i), 4 * GROUPS);
    }
    mbar_init(bar(S::DRAIN), 1);
    *s_abort = 0;
    pdl_wait_predecessor();                  // (the number may be another launch's to advance)
    uint32_t number = 0;
    if (!a.lse) asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(number) : "l"(a.launch) : "memory");
    *s_set = number & 1u;
    *s_number = number;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(sbase + S::MISC) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *s_tmem;
  pdl_wait_predecessor();                    // all above is the CTA's own; operands, lists and counters may be the work of kernels before
  const TcWork work = a.live_hdr && __ldg(a.live_hdr) ? a.live : a.list;
  const int first = __ldg(work.first + blockIdx.x);
  uint32_t* const published = a.counters + (size_t)*s_set * a.nseg * SYNC_STRIDE;

  if (warp == 0) {
    // =============================== TMA producer ===============================
    // The CTA's l-th run uses Q buffer l%2.
    if (lane == 0 && first >= 0) {
      const uint64_t pol_keep = l2_policy_keep(), pol_stream = l2_policy_stream();
      int s = 0, item = 0;                     // ring stage and number of the next tile
      uint32_t s_par = 1;
      int q_issued = -1;                       // last run whose Q chunk has been requested
      int loaded_seg[2] = {-1, -1};
      bool ok = true;
      // requests the Q chunk of run `l` (record p); `block`: wait for the buffer, else only try
      auto issue_q = [&](int l, const TcRun& p, bool block) -> bool {
        const int b = l & 1, use = l >> 1;
        if (use >= 1) {
          const uint32_t par = (uint32_t)((use - 1) & 1);
          if (block) { if (!mbar_wait(bar(S::QEMPTY + b), par, s_abort, 11, true)) return false; }
          else if (!mbar_test(bar(S::QEMPTY + b), par)) return true;
        }
        if (loaded_seg[b] == p.seg) {
          mbar_arrive(bar(S::QFULL + b));      // same chunk as the buffer holds: nothing to copy
        } else {
          const RowPlace r0 = row_place(a, p.chunk, 0);
          mbar_expect_tx(bar(S::QFULL + b), 2u * 128u * (uint32_t)(copies * box_rows));
          for (int i = 0; i < copies; ++i) {
            const int head = p.h * a.G + r0.g + i;
            const uint32_t dst = sbase + (uint32_t)(b * S::Q_BUF + i * a.Wp * 128);
            if (FP8) {
              tma_load_5d(dst, &tm_q, bar(S::QFULL + b), 0, r0.t, head, p.b, 0);
              tma_load_5d(dst + S::Q_BLOCK, &tm_q, bar(S::QFULL + b), 0, r0.t, head, p.b, 1);
            } else {
              tma_load_4d(dst, &tm_q, bar(S::QFULL + b), 0, r0.t, head, p.b);
              tma_load_4d(dst + S::Q_BLOCK, &tm_q, bar(S::QFULL + b), 64, r0.t, head, p.b);
            }
          }
          loaded_seg[b] = p.seg;
        }
        q_issued = l;
        return true;
      };
      TcRun p = load_run(work.runs, first);
      for (int l = 0; ok; ++l) {
        const TcRun nxt = p.next >= 0 ? load_run(work.runs, p.next) : p;
        if (q_issued < l && !issue_q(l, p, true)) { ok = false; break; }
        const uint64_t pol = p.pass == 1 ? pol_keep : pol_stream;
        for (int i = 0; i < p.ntiles; ++i) {
          if (p.next >= 0 && q_issued == l && !issue_q(l + 1, nxt, false)) { ok = false; break; }   // once its buffer is free
          if (!mbar_wait(bar(S::EMPTY + s), s_par, s_abort, 12, true)) { ok = false; break; }
          mbar_expect_tx(bar(S::FULL + s), S::STAGE);
          const uint32_t dst = sbase + S::K + s * S::STAGE;
          const int tok = p.tok_off + (p.tile0 + i) * KT;
          tma_load_3d(dst, &tm_k, bar(S::FULL + s), 0, p.h, tok, pol);
          if (!FP8) tma_load_3d(dst + S::HALF, &tm_k, bar(S::FULL + s), 64, p.h, tok, pol);
          ++item;
          if (++s == S::NSTAGE) { s = 0; s_par ^= 1u; }
        }
        if (p.next < 0) break;
        p = nxt;
      }
      if (!ok) {
        // let the copies already issued land before the CTA's shared memory is released
        const int armed = item < S::NSTAGE ? item : S::NSTAGE;
        for (int i = 0; i < armed; ++i) {
          const int it = item - 1 - i;
          mbar_wait(bar(S::FULL + it % S::NSTAGE), (it / S::NSTAGE) & 1, s_abort, 13, false);
        }
        for (int l = q_issued; l >= 0 && l > q_issued - 2; --l)
          mbar_wait(bar(S::QFULL + (l & 1)), (l >> 1) & 1, s_abort, 14, false);
      }
    }
  } else if (warp == 1) {
    // =============================== MMA issuer =================================
    // The whole warp walks the units; one elected lane issues.
    int s = 0, slot = first;
    uint32_t s_par = 0, u = 0;
    bool ok = true;
    const uint32_t idesc1 = FP8 ? instr_desc_f8(128, KT) : instr_desc(128, KT);
    const uint32_t idesc2 = FP8 ? instr_desc_f8(KT, HR) : instr_desc(KT, HR);
    for (int l = 0; ok && slot >= 0; ++l) {
      // (shuffled so that the compiler knows them to be the same in all lanes: descriptors stay in uniform registers)
      const int pass = __shfl_sync(0xffffffffu, __ldg(&work.runs[slot].pass), 0), ntiles = __shfl_sync(0xffffffffu, __ldg(&work.runs[slot].ntiles), 0),
                next = __shfl_sync(0xffffffffu, __ldg(&work.runs[slot].next), 0);
      prefetch_run(work.runs, next);
      ok = __all_sync(0xffffffffu, mbar_wait(bar(S::QFULL + (l & 1)), (l >> 1) & 1, s_abort, 21, true));
      const uint32_t qbase = sbase + (uint32_t)((l & 1) * S::Q_BUF);
      for (int i = 0; ok && i < ntiles; ++i) {
        ok = __all_sync(0xffffffffu, mbar_wait(bar(S::FULL + s), s_par, s_abort, 23, true));
        const uint64_t kd = smem_desc(sbase + S::K + s * S::STAGE);
#pragma unroll
        for (int hf = 0; hf < HV; ++hf, ++u) {
          const int acc = (int)(u & 3u);
          ok = ok && __all_sync(0xffffffffu, mbar_wait(bar(S::TEMPTY + acc), ((u >> 2) & 1u) ^ 1u, s_abort, 22, true));
          if (!ok) break;
          tc_fence_after();
          const uint32_t d = tmem + (uint32_t)(acc * 128);
          const uint64_t qd = smem_desc(qbase + (uint32_t)(hf * HR * 128));
          if (elect_one()) {
            // k-step ks: bf16 tiles are two 64-channel blocks, 8-bit tiles one block that both query terms meet
#pragma unroll
            for (int ks = 0; ks < 8; ++ks) {
              const uint64_t ko = kd + (FP8 ? (ks & 3) * 2 : (ks >> 2) * (S::HALF >> 4) + (ks & 3) * 2);
              const uint64_t qo = qd + (ks >> 2) * (S::Q_BLOCK >> 4) + (ks & 3) * 2;
              const uint64_t ad = pass == 2 ? ko : qo, bd = pass == 2 ? qo : ko;
              const uint32_t id = pass == 2 ? idesc2 : idesc1;
              if (FP8) tc_mma_f8(d, ad, bd, id, ks > 0);
              else     tc_mma(d, ad, bd, id, ks > 0);
            }
            tc_commit(bar(S::TFULL + acc));                      // accumulator ready for its group
            if (hf == HV - 1) {
              tc_commit(bar(S::EMPTY + s));                      // ring stage free once these MMAs have read it
              if (i + 1 == ntiles) tc_commit(bar(S::QEMPTY + (l & 1)));
            }
          }
          __syncwarp();
        }
        if (++s == S::NSTAGE) { s = 0; s_par ^= 1u; }
      }
      slot = next;
    }
    if (!ok) {  // make sure nothing is still writing tensor memory before it is freed
      if (elect_one()) {
        tc_commit(bar(S::DRAIN));
        mbar_wait(bar(S::DRAIN), 0, s_abort, 24, false);
      }
      __syncwarp();
    }
  } else if (warp == 2) {
    // =============================== partial folding ==============================
    // For every pass-1 stage: the rows of its segments are dealt to the CTAs in runs of `per`; wait until a row's
    // segment has been published by all its epilogue groups, fold the row's partials in a fixed order (the result does
    // not depend on timing) and write its offset.  Up to eight rows at a time, four or more lanes each, so that a
    // stage costs one round trip for the partials (row after row it was 2 us each, 18 us of waiting in front of pass 2 for
    // a group of four heads).
    unsigned long long* const ready = a.ready + (size_t)*s_set * a.nseg * a.NC;
    for (int si = 0; si < a.n_stages; ++si) {
      const int a0 = __ldg(&a.stages[si].seg0), total = __ldg(&a.stages[si].nseg) * a.NC;
      const int per = (total + (int)gridDim.x - 1) / (int)gridDim.x;
      const int lo = (int)blockIdx.x * per, hi = min(total, lo + per);
      int rpi = 1;                                                            // rows at a time
      while (rpi < 8 && rpi < per) rpi <<= 1;
      const int lpr = 32 / rpi, sub = lane / rpi;                             // lanes per row
      bool ok = true;
      for (int base = lo; ok && base < hi; base += rpi) {
        const int s0 = base / a.NC, s1 = min(base + rpi, hi) - 1;
        const int idx = min(base + lane % rpi, hi - 1);
        const int sg = idx / a.NC, row = idx - sg * a.NC;
        const int4 fo = __ldg(reinterpret_cast<const int4*>(work.folds + a0 + sg));        // slot0, nruns, rows, request
        const bool valid = base + lane % rpi < hi && row < fo.z && fo.y > 0;
        if (sub == 0) __stcg(a.ready + ((size_t)(*s_set ^ 1u) * a.nseg + a0 + sg) * a.NC + row, 0ull);
        for (int q = s0; ok && q <= s1 / a.NC; ++q) {
          const int4 fq = __ldg(reinterpret_cast<const int4*>(work.folds + a0 + q));
          if (fq.y > 0) ok = word_wait(published + (a0 + q) * SYNC_STRIDE, (uint32_t)(GROUPS * fq.y), s_abort, 41, lane, 128);
        }
        if (!ok) break;
        const int n = valid ? fo.y * ENTRIES : 0;
        const int n_max = __reduce_max_sync(0xffffffffu, n);
        const float2* src = a.partials + (int64_t)fo.x * ENTRIES * a.NC + row;
        float M = -INFINITY, L = 0.f;
        for (int e0 = 0; e0 < n_max; e0 += 20 * lpr) {
          float2 v[20];
#pragma unroll
          for (int i = 0; i < 20; ++i) {                                      // all loads in flight
            const int e = e0 + sub + lpr * i;
            v[i] = e < n ? __ldcg(src + (int64_t)e * a.NC) : make_float2(-INFINITY, 0.f);
          }
#pragma unroll
          for (int i = 0; i < 20; ++i) {
            if (v[i].y > 0.f) {
              const float Mn = fmaxf(M, v[i].x);
              L = L * ex2(M - Mn) + v[i].y * ex2(v[i].x - Mn);
              M = Mn;
            }
          }
        }
        for (int o = rpi; o < 32; o <<= 1) {                       // butterfly: every lane of a row ends with the same (M, L)
          const float Mo = __shfl_xor_sync(0xffffffffu, M, o), Lo = __shfl_xor_sync(0xffffffffu, L, o);
          const bool lower = (lane & o) == 0;                      // fold in lane order so both partners agree bitwise
          const float Ma = lower ? M : Mo, La = lower ? L : Lo, Mb = lower ? Mo : M, Lb = lower ? Lo : L;
          const float Mn = fmaxf(Ma, Mb);
          float Ln = 0.f;
          if (La > 0.f) Ln += La * ex2(Ma - Mn);
          if (Lb > 0.f) Ln += Lb * ex2(Mb - Mn);
          M = Mn; L = Ln;
        }
        if (valid && sub == 0) {
          const float offset = M + log2f(L);
          const int64_t at = (int64_t)(a0 + sg) * a.NC + row;
          asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(ready + at), "l"(OFFSET_READY | __float_as_uint(offset)) : "memory");
          __stcg(a.offsets + at, offset);                          // for asl_window_lse
        }
      }
      if (!ok) break;
    }
  } else if (warp == 3) {
    // =============================== row offsets ==================================
    // For every pass-2 run of the CTA: look for the segment's offsets until all are there (one warp per CTA: sixteen on 148
    // SMs would keep the L2 slices busy), then hand them, negated, to the epilogue in shared memory.
    if (!a.lse) {
      uint32_t last = 0;
      if (lane == 0) asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(last) : "l"(a.launch + 1) : "memory");
      if (__shfl_sync(0xffffffffu, last, 0) == gridDim.x - 1u) {       // every CTA has read the number
        uint32_t* other = a.counters + (size_t)(*s_set ^ 1u) * a.nseg * SYNC_STRIDE;
        for (int i = lane; i < a.nseg; i += 32) other[(size_t)i * SYNC_STRIDE] = 0;
        if (lane == 0) { a.launch[0] = *s_number + 1u; a.launch[1] = 0; }
      }
    }
    float* s_off = reinterpret_cast<float*>(smem + S::OFFS);
    int q = 0;
    bool ok = true;
    for (int slot = first; slot >= 0;) {
      const TcRun r = load_run(work.runs, slot);
      prefetch_run(work.runs, r.next);
      slot = r.next;
      if (r.pass != 2) continue;
      const int buf = q & 1;
      if (q >= 2 && !__all_sync(0xffffffffu, mbar_wait(bar(S::OEMPTY + buf), ((q >> 1) & 1) ^ 1, s_abort, 32, true))) break;
      const RowPlace p0 = row_place(a, r.chunk, 0);
      const float* lse = a.lse + ((int64_t)r.b * a.Hq + r.h * a.G + p0.g) * a.W + p0.t;
      const unsigned long long* src = a.ready + ((size_t)*s_set * a.nseg + r.seg) * a.NC;
      float o[MAX_ROWS / 32];
      uint32_t left = 0;                                                // rows of this lane that are not there yet
#pragma unroll
      for (int i = 0; i < MAX_ROWS / 32; ++i) {
        const int row = lane + 32 * i;
        int at = row;
        bool exists = row < r.rows;
        if (!dense) {                                                   // max pooling, heads padded to Wp rows
          const int hd = row / a.Wp, t = row - hd * a.Wp;
          exists = exists && t < a.W;
          at = hd * a.W + t;
        }
        o[i] = -INFINITY;                                               // a padding row: 2^(x - inf) = 0
        if (exists && a.lse) o[i] = __ldcg(lse + at) * -1.4426950408889634f;      // natural log -> log2 domain
        if (exists && !a.lse) left |= 1u << i;
      }
      unsigned long long t0 = 0;
      uint32_t nap = 32;
      for (uint32_t it = 0; __any_sync(0xffffffffu, left != 0u); ++it) {
        unsigned long long v[MAX_ROWS / 32];
        // (a wait that lasts looks at the first rows only until they are there)
        const uint32_t look = it >= 8 && __any_sync(0xffffffffu, left & 1u) ? left & 1u : left;
#pragma unroll
        for (int i = 0; i < MAX_ROWS / 32; ++i) v[i] = (look >> i) & 1u ? ld_relaxed(src + lane + 32 * i) : 0ull;
#pragma unroll
        for (int i = 0; i < MAX_ROWS / 32; ++i)
          if (v[i]) { o[i] = -__uint_as_float((uint32_t)v[i]); left &= ~(1u << i); }
        if ((it & 7u) == 7u) {
          int gave_up = 0;
          if (lane == 0) {
            const unsigned long long now = global_ns();
            if (t0 == 0) t0 = now;
            else if (now - t0 > WAIT_LIMIT_NS || *s_abort) { gave_up = 1; if (!*s_abort) *s_abort = 33; }
          }
          if (__shfl_sync(0xffffffffu, gave_up, 0)) { ok = false; break; }
        }
        if (it >= 8) {                       // the first looks follow one another at once: what is waited for is about to come
          __nanosleep(nap);
          if (nap < 256) nap <<= 1;
        }
      }
      if (!ok) break;
#pragma unroll
      for (int i = 0; i < MAX_ROWS / 32; ++i) s_off[buf * MAX_ROWS + lane + 32 * i] = o[i];
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(S::OFULL + buf));
      ++q;
    }
  } else {
    // =============================== epilogue ===================================
    // Group g owns accumulator g (units u with u%4 == g); WIDE: always half g%2 of the chunk's rows.  Its four warps
    // take a lane quarter each.
    const int g = (warp - 4) >> 2;
    const int quarter = warp & 3;                              // TMEM lanes 32*quarter .. +31 are this warp's
    const int lt = quarter * 32 + lane;                        // TMEM lane of this thread, 0..127
    const int half = WIDE ? (g & 1) : 0;
    const uint32_t acc_addr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(g * 128);
    const int nblk = HR >> 5;                                  // 32-column blocks of a pass-2 accumulator
    uint32_t u0 = 0;                                           // unit number at which the current run starts
    uint32_t mine = 0;                                         // units this group has taken
    int q = 0;                                                 // pass-2 runs so far
    // max pooling: after which 32-column blocks of an accumulator a query head ends
    int head_ends = 1 << (nblk - 1);
    if (PER_Q && a.Wp <= 128)
      for (int i = 1; i < nblk; ++i) head_ends |= (32 * i) % a.Wp == 0 ? 1 << (i - 1) : 0;
    bool dead = false;                                         // a wait expired: keep the barrier sequence, skip the work
    auto release = [&]() {                                     // this warp has read its part of the accumulator
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(S::TEMPTY + g));
    };
    for (int slot = first; slot >= 0;) {
      const TcRun* rp = work.runs + slot;
      const int4 ra = __ldg(reinterpret_cast<const int4*>(rp)), rb = __ldg(reinterpret_cast<const int4*>(rp) + 1),
                 rc = __ldg(reinterpret_cast<const int4*>(rp) + 2);
      const int tile0 = ra.x, ntiles = ra.y, pass = ra.z, seg = ra.w, h = rb.y, chunk = rb.z, next = rb.w;
      const int T = rc.x, u_off = rc.y, rows = rc.w;
      prefetch_run(work.runs, next);
      const float scale = FP8 ? a.scale_log2 * __ldg(&rp->kscale) : a.scale_log2;   // log2(e)/sqrt(d) times the accumulator factor
      const f32x2 scale2 = pk(scale, scale);
      const int nu = ntiles * HV;
      int k = (int)((uint32_t)(g - (int)u0) & 3u);             // first unit of the run that is this group's
      uint32_t bufs[2][16];
      auto wait_unit = [&]() {
        if (!dead) dead = !__all_sync(0xffffffffu, mbar_wait(bar(S::TFULL + g), mine & 1u, s_abort, 31, true));
        ++mine;
        if (!dead) tc_fence_after();
        return !dead;
      };
      if (pass == 1) {
        // ---- pass 1: sum of 2^(x - mref) of row half*HR + lt over the keys of the group's tiles of the run.  mref is
        // the row's first logit; the maximum is not tracked (terms may exceed 1, fp32 has the range) unless a sum
        // overflows, in which case the tile is redone with it.  Which tiles are added together follows from the run
        // alone, so the result does not depend on what else the launch works on.
        const int row = half * HR + lt;
        const bool busy = half * HR + quarter * 32 < rows && quarter * 32 < HR;     // the warp has rows of the chunk
        const int entry = (k / HV) & (ENTRIES - 1);
        float mref = -INFINITY, l = 0.f;
        bool begun = false;
        for (; k < nu; k += GROUPS) {
          if (!wait_unit()) continue;
          if (!busy) { release(); continue; }
          const int j_tile = (tile0 + k / HV) * KT;
          const float keep_m = mref, keep_l = l;
          // every key visible to every row: the fast walk.  It stops before the tile's last 16 keys to look for an
          // overflow while the accumulator is still there.
          bool careful = j_tile + KT - 1 > T, tail_careful = false;
          if (!careful) {
            tc_ld_lane(acc_addr, bufs[0]);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              uint32_t (&cur)[16] = bufs[j & 1];
              tc_ld_wait(cur);
              if (j < 7) tc_ld_lane(acc_addr + (uint32_t)(16 * (j + 1)), bufs[(j + 1) & 1]);
              if (j == 0 && !begun) mref = __uint_as_float(cur[0]) * scale;
              if (j == 7) {
                careful = __any_sync(0xffffffffu, !(l < INFINITY));   // a term beyond fp32 range (a logit 127 above the reference)
                if (careful) break;
                release();
              }
              const f32x2 nm2 = pk(-mref, -mref);
              f32x2 am = pk(0.f, 0.f), ap = pk(0.f, 0.f);
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const f32x2 x = fma2(pku(cur[2 * i], cur[2 * i + 1]), scale2, nm2);
                if (pair_is_poly(i + 8 * (j & 1))) ap = add2(ex2_pair_poly<true>(x), ap);
                else                               am = add2(ex2_pair_mufu(x), am);
              }
              const float s = hsum(add2(am, ap));
              if (j == 7 && __any_sync(0xffffffffu, !(l + s < INFINITY))) tail_careful = true;   // redone below from the registers
              else l += s;
            }
            if (careful) { mref = keep_m; l = keep_l; }
          }
          begun = true;
          if (careful || tail_careful) {
            // running maximum over 16-key blocks, per-row visibility, MUFU only
            const int lastkey = T + row_place(a, chunk, row).t;       // last key this row sees
#pragma unroll 1
            for (int j = careful ? 0 : 7; j < 8; ++j) {
              uint32_t (&cur)[16] = bufs[1];
              if (careful) {
                tc_ld_lane(acc_addr + (uint32_t)(16 * j), cur);
                tc_ld_wait(cur);
              }
              const int j0 = j_tile + 16 * j;
              if (j0 <= lastkey) {
                float c[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                  c[i] = fmaxf((j0 + i <= lastkey) ? __uint_as_float(cur[i]) : -INFINITY, (j0 + i + 8 <= lastkey) ? __uint_as_float(cur[i + 8]) : -INFINITY);
                const float mn = fmaxf(mref, scale * fmaxf(fmaxf(fmaxf(c[0], c[1]), fmaxf(c[2], c[3])), fmaxf(fmaxf(c[4], c[5]), fmaxf(c[6], c[7]))));
                float s0 = 0.f, s1 = 0.f;
#pragma unroll
                for (int i = 0; i < 16; i += 2) {
                  s0 += (j0 + i <= lastkey) ? ex2(fmaf(__uint_as_float(cur[i]), scale, -mn)) : 0.f;
                  s1 += (j0 + i + 1 <= lastkey) ? ex2(fmaf(__uint_as_float(cur[i + 1]), scale, -mn)) : 0.f;
                }
                l = fmaf(l, ex2(mref - mn), s0 + s1);
                mref = mn;
              }
            }
            if (careful) release();
          }
          if (l > 0x1p60f) { l *= 0x1p-60f; mref += 60.f; }     // exact: keeps the running sum far from overflow
        }
        // ---- end of the run: the group publishes (reference, sum) per row ----
        if (lt < HR) __stcg(a.partials + ((int64_t)__ldg(&work.runs[slot].slot) * ENTRIES + entry) * a.NC + row, make_float2(mref, dead ? 0.f : l));
        bar_sync(1 + g, 128);
        if (quarter == 0 && lane == 0) {   // the barrier orders the group's stores before this thread's fence: the release is cumulative
          __threadfence();
          atomicAdd(published + __ldg(&work.runs[slot].seg) * SYNC_STRIDE, 1u);       // (read again: a register less through the tiles)
        }
      } else {
        // ---- pass 2: for every key, exp2(x - offset[row]) summed over the half's rows.  In the 16x256b shape a
        // thread meets rows 8i + 2(lane%4) + {0, 1}: their offsets stay in registers for the run.
        if (!dead) dead = !__all_sync(0xffffffffu, mbar_wait(bar(S::OFULL + (q & 1)), (q >> 1) & 1, s_abort, 34, true));
        f32x2 noff[16];
        {
          const float2* src = reinterpret_cast<const float2*>(smem + S::OFFS) + (q & 1) * (MAX_ROWS / 2) + half * (HR >> 1) + (lane & 3);
#pragma unroll
          for (int i = 0; i < 16; ++i) {                        // rows past the half: read, not used
            const float2 v = 8 * i < HR ? src[4 * i] : make_float2(0.f, 0.f);
            noff[i] = pk(v.x, v.y);
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(S::OEMPTY + (q & 1)));
          ++q;
        }
        for (; k < nu; k += GROUPS) {
          if (!wait_unit()) continue;
          const int j = (tile0 + k / HV) * KT + quarter * 32 + (lane >> 2) + 8 * (lane & 1) + 16 * ((lane >> 1) & 1);
          // max pooling: the query head whose rows come first in this accumulator, and which of its partial sums this is
          int head = chunk * a.m + (a.Wp <= 128 ? half * HR / a.Wp : 0), part = a.Wp <= 128 ? 0 : half;
          if (PER_Q && a.pieces > 1) { head = chunk / a.pieces; part = (chunk % a.pieces) * 2 + half; }
          // sums of four keys (lanes lane/4, +8, +16, +24 of the quarter) over the thread's rows
          f32x2 ac[4] = {pk(0.f, 0.f), pk(0.f, 0.f), pk(0.f, 0.f), pk(0.f, 0.f)};
          tc_ld_quad(acc_addr, bufs[0]);
#pragma unroll
          for (int blk = 0; blk < 4; ++blk) {
            if (blk < nblk) {
#pragma unroll
              for (int up = 0; up < 2; ++up) {                  // lanes 0-15, 16-31 of the quarter
                uint32_t (&cur)[16] = bufs[up];
                tc_ld_wait(cur);
                if (up == 0) tc_ld_quad(acc_addr + (uint32_t)(32 * blk) + (16u << 16), bufs[1]);
                else if (blk + 1 < nblk) tc_ld_quad(acc_addr + (uint32_t)(32 * (blk + 1)), bufs[0]);
                else release();
                f32x2 ap[2] = {pk(0.f, 0.f), pk(0.f, 0.f)};
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                  const f32x2 x = fma2(pku(cur[2 * i], cur[2 * i + 1]), scale2, noff[4 * blk + (i >> 1)]);
                  if (pair_is_poly(i + 8 * up)) ap[i & 1] = add2(ex2_pair_poly<false>(x), ap[i & 1]);
                  else ac[2 * up + (i & 1)] = add2(ex2_pair_mufu(x), ac[2 * up + (i & 1)]);
                }
                ac[2 * up] = add2(ap[0], ac[2 * up]);
                ac[2 * up + 1] = add2(ap[1], ac[2 * up + 1]);
              }
              if (PER_Q ? (head_ends >> blk) & 1 : blk + 1 == nblk) {
                // reduce over the four lanes that share keys: each ends with one key
                const float k0 = hsum(ac[0]), k1 = hsum(ac[1]), k2 = hsum(ac[2]), k3 = hsum(ac[3]);
                const bool odd = lane & 1, upper = lane & 2;
                const float q0 = (odd ? k1 : k0) + __shfl_xor_sync(0xffffffffu, odd ? k0 : k1, 1);
                const float q1 = (odd ? k3 : k2) + __shfl_xor_sync(0xffffffffu, odd ? k2 : k3, 1);
                const float sum = (upper ? q1 : q0) + __shfl_xor_sync(0xffffffffu, upper ? q0 : q1, 2);
                if (PER_Q) {
#pragma unroll
                  for (int q = 0; q < 4; ++q) ac[q] = pk(0.f, 0.f);
                  if (j < T && head < a.G) a.u[((int64_t)(h * a.G + head) * a.u_parts + part) * a.u_stride + u_off + j] = sum;
                  ++head;
                } else {
                  if (j < T) a.u[(int64_t)(h * a.u_rows_per_kv + chunk * HV + half) * a.u_stride + u_off + j] = sum;
                }
              }
            }
          }
        }
      }
      u0 += (uint32_t)nu;
      slot = next;
    }
  }

  // ---- teardown ----
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
  }
  if (threadIdx.x == 0 && *s_abort) atomicCAS(a.err, 0, *s_abort);
}

// One warp runs one of the kernel's two kinds of bounded wait on something that never happens (a barrier
// nobody arrives on, a counter nobody advances) with a short limit, and reports like the scorer does.
__global__ void bounded_wait_selftest_kernel(int which, unsigned long long limit_ns, const uint32_t* never_written,
                                             int32_t* err) {
  __shared__ __align__(8) unsigned long long s_bar;
  __shared__ int s_flag;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&s_bar), 1);
    s_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  volatile int* abort_flag = &s_flag;
  bool ok;
  if (which == 0) ok = mbar_wait(smem_u32(&s_bar), 0, abort_flag, 91, true, limit_ns);
  else            ok = word_wait(never_written, 0xFFFFFFFFu, abort_flag, 92, lane, 256, limit_ns);
  __syncthreads();
  if (threadIdx.x == 0 && !ok && *abort_flag) atomicCAS(err, 0, *abort_flag);
}

// Device-side controller: the work list of the next launch without the runs of finished requests; hdr[0] = 0 where
// there are none (the launch then takes the plan's list).  One block.  The requests' flags are read once (a record may be
// changing under a statistic kernel of the previous layer that is still running: whatever is read here holds for the
// whole launch).  Runs stay whole, so that the sums of the requests still observed come out bit for bit as in a launch
// that skips nothing; groups that have shrunk are merged until they hold about `most` tiles, and a merged group's runs
// are dealt to the CTAs by where their middle lies among its tiles.
__device__ unsigned long long block_scan_1024(unsigned long long v, unsigned long long* warp_tot, unsigned long long& total) {   // exclusive
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned long long incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  __syncthreads();
  if (lane == 31) warp_tot[wid] = incl;
  __syncthreads();
  unsigned long long before = 0;
  total = 0;
  for (int w = 0; w < 32; ++w) { total += warp_tot[w]; if (w < wid) before += warp_tot[w]; }
  return before + incl - v;
}
__global__ void __launch_bounds__(1024) live_list_kernel(const TcRun* __restrict__ all, int n1, int n2, const TcFold* __restrict__ all_folds, int nseg,
                                                         int n_groups, int most, const asl_stat* __restrict__ latch, int cur, int batch, int grid,
                                                         int32_t* __restrict__ hdr, TcRun* __restrict__ runs, int32_t* __restrict__ first,
                                                         TcFold* __restrict__ folds, int32_t* __restrict__ scratch) {
  __shared__ uint32_t fin[ASL_SKIP_MAX_BATCH / 32];
  __shared__ unsigned long long warp_tot[32];
  const int tid = threadIdx.x, lane = tid & 31, n = n1 + n2;
  int any = 0;
  for (int b0 = 0; b0 < batch; b0 += 1024) {
    const int b = b0 + tid;
    const uint32_t word = __ballot_sync(0xffffffffu, b < batch && asl_finished(latch + b, cur));
    if (lane == 0) fin[b >> 5] = word;
    any |= word != 0u;
  }
  any = __syncthreads_or(any);
  if (tid == 0) hdr[0] = any;
  if (!any) return;
  auto live = [&](int b) { return ((fin[b >> 5] >> (b & 31)) & 1u) == 0u; };
  int32_t* pos = scratch;                        // [n] live tiles of the pass before the run
  int32_t* num = pos + n;                        // [n] the pass's live runs in order, and where they go: merged group * grid + CTA
  int32_t* key = num + n;
  int32_t* group_tiles = key + n;                // [groups]
  int32_t* merged = group_tiles + n_groups;      // [groups]
  int32_t* tiles = merged + n_groups;            // [2][groups] live tiles of a merged group, and before it
  int32_t* base = tiles + 2 * n_groups;
  int32_t* head = base + 2 * n_groups;           // [groups + 1 stages][2 passes][grid] first and last run (-1: none)
  const int n_lists = 2 * (n_groups + 1) * grid;
  int32_t* tail = head + n_lists;
  for (int i = tid; i < n_groups; i += 1024) group_tiles[i] = 0;
  for (int i = tid; i < 2 * n_groups; i += 1024) { tiles[i] = 0; base[i] = 0x7fffffff; }
  for (int i = tid; i < 2 * n_lists; i += 1024) head[i] = -1;
  for (int s = tid; s < nseg; s += 1024) {
    TcFold f = all_folds[s];
    if (!live(f.b)) f.nruns = 0;
    folds[s] = f;
  }
  __syncthreads();
  for (int i = n1 + tid; i < n; i += 1024)
    if (live(all[i].b)) atomicAdd(&group_tiles[all[i].group], all[i].ntiles);
  __syncthreads();
  if (tid == 0) {
    int held = 0, id = 0;
    for (int g = 0; g < n_groups; ++g) {
      if (held > 0 && held + group_tiles[g] > most) { ++id; held = 0; }
      held += group_tiles[g];
      merged[g] = id;
    }
  }
  __syncthreads();
  int n_live[2];
  for (int p = 0; p < 2; ++p) {
    const int at = p ? n1 : 0, np = p ? n2 : n1;
    unsigned long long sum = 0;                  // runs << 32 | tiles so far
    for (int i0 = 0; i0 < np; i0 += 1024) {
      const int i = i0 + tid;
      const bool mine = i < np && live(all[at + i].b);
      const int nt = mine ? all[at + i].ntiles : 0;
      unsigned long long total;
      const unsigned long long here = sum + block_scan_1024(mine ? (1ull << 32) + (unsigned)nt : 0ull, warp_tot, total);
      if (mine) {
        const int mg = merged[all[at + i].group];
        pos[at + i] = (int)(uint32_t)here;
        num[at + (int)(here >> 32)] = at + i;
        atomicAdd(&tiles[p * n_groups + mg], nt);
        atomicMin(&base[p * n_groups + mg], (int)(uint32_t)here);
      }
      sum += total;
    }
    n_live[p] = (int)(sum >> 32);
  }
  __syncthreads();
  for (int p = 0; p < 2; ++p)
    for (int r = tid; r < n_live[p]; r += 1024) {
      const int at = (p ? n1 : 0) + r, i = num[at], mg = merged[all[i].group];
      const int64_t middle = 2 * (pos[i] - base[p * n_groups + mg]) + all[i].ntiles;
      key[at] = mg * grid + (int)(middle * grid / (2 * tiles[p * n_groups + mg]));
    }
  __syncthreads();
  for (int p = 0; p < 2; ++p)
    for (int r = tid; r < n_live[p]; r += 1024) {
      const int at = (p ? n1 : 0) + r, i = num[at], k = key[at];
      TcRun run = all[i];
      const bool last = r + 1 == n_live[p] || key[at + 1] != k;
      run.next = last ? -1 : num[at + 1];
      runs[i] = run;
      const int list = ((k / grid + p) * 2 + p) * grid + k % grid;      // pass 2 of a group comes a stage after its pass 1
      if (r == 0 || key[at - 1] != k) head[list] = i;
      if (last) tail[list] = i;
    }
  __syncthreads();
  for (int i = tid; i < n_lists; i += 1024) {                  // chain a CTA's lists
    int j = i;
    if (i < grid) {
      while (j < n_lists && head[j] < 0) j += grid;
      first[i] = j < n_lists ? head[j] : -1;
    }
    if (tail[i] < 0) continue;
    for (j = i + grid; j < n_lists && head[j] < 0;) j += grid;
    if (j < n_lists) runs[tail[i]].next = head[j];
  }
}

// Row offsets (log2 of the softmax denominators) of the latest two-pass call as natural-log denominators [B][H_q][W]
__global__ void __launch_bounds__(256) offsets_to_lse_kernel(const float* __restrict__ offsets, float* __restrict__ lse, int n, int W, int G, int m,
                                                             int Wp, int pieces, int nchunk, int NC) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  const int t = i % W, hq = i / W, g = hq % G, bh = hq / G;                  // bh: request x kv head
  const int chunk = pieces > 1 ? g * pieces + t / MAX_ROWS : g / m;
  const int row = pieces > 1 ? t % MAX_ROWS : (g % m) * Wp + t;
  lse[i] = __ldcg(offsets + ((int64_t)bh * nchunk + chunk) * NC + row) * 0.6931471805599453f;
}

// FP8 keys: the bf16 window queries, scaled by Q8_SCALE, as two E4M3 terms hi + lo (hi = nearest code,
// lo = nearest code of the remainder; together exact whenever the remainder's bits fit the format, i.e.
// for 1/64 <= |q| <= 28): out[t][b][head][row][c], dense.
constexpr float Q8_SCALE = 16.0f;
__global__ void __launch_bounds__(256) split_queries_e4m3_kernel(const __nv_bfloat16* __restrict__ q, int64_t qs_b, int64_t qs_h,
                                                                 int64_t qs_r, int Hq, int W, int64_t total,
                                                                 uint8_t* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const int c = (int)(i & 127);
  const int64_t r = i >> 7;
  const int row = (int)(r % W), head = (int)((r / W) % Hq);
  const int64_t b = r / ((int64_t)W * Hq);
  const float x = __bfloat162float(q[b * qs_b + head * qs_h + row * qs_r + c]) * Q8_SCALE;
  const __nv_fp8_storage_t hi = __nv_cvt_float_to_fp8(x, __NV_SATFINITE, __NV_E4M3);
  const float xh = __half2float(__half(__nv_cvt_fp8_to_halfraw(hi, __NV_E4M3)));
  const __nv_fp8_storage_t lo = __nv_cvt_float_to_fp8(x - xh, __NV_SATFINITE, __NV_E4M3);
  out[i] = hi;
  out[total + i] = lo;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

bool make_map(CUtensorMap* tm, CUtensorMapDataType dtype, const void* base, int rank, const cuuint64_t* dims,
              const cuuint64_t* strides_bytes, const cuuint32_t* box) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  return fn(tm, dtype, rank, const_cast<void*>(base), dims, strides_bytes, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct ScoreKernel {
  void (*fn)(CUtensorMap, CUtensorMap, TcArgs);
  int smem;
};
template <int I>
constexpr ScoreKernel score_instance() { return {score_tc_kernel<(I & 8) != 0, (I & 4) != 0, (I & 2) != 0, (I & 1) != 0>, Smem<(I & 4) != 0, (I & 2) != 0>::BYTES}; }
const ScoreKernel& score_kernel(int i) {       // bits: max pooling, FP8 keys, wide, full halves
  static const ScoreKernel k[16] = {score_instance<0>(), score_instance<1>(), score_instance<2>(), score_instance<3>(),
                                    score_instance<4>(), score_instance<5>(), score_instance<6>(), score_instance<7>(),
                                    score_instance<8>(), score_instance<9>(), score_instance<10>(), score_instance<11>(),
                                    score_instance<12>(), score_instance<13>(), score_instance<14>(), score_instance<15>()};
  return k[i];
}
int score_kernel_of(const asl_params& p, const AslTcPlan& tp) {
  return (p.pool_mode == ASL_POOL_MAX ? 8 : 0) + (p.k_dtype == ASL_K_FP8_E4M3 ? 4 : 0) + (tp.wide ? 2 : 0) + (tp.HR == 128 ? 1 : 0);
}

}  // namespace

// ---------------------------------------------------------------- host side
namespace {

// The FP8 windows that asl.h names.  (plan_chunks cuts any window; the scorer before this one took chunks of whole heads
// in multiples of 64 rows only, and what it refused is refused still: no other window is tested with FP8 keys.)
bool fp8_shape(const asl_params& p) {
  const int W = p.window, R = p.n_q_heads / p.n_kv_heads * W;
  if (W % 32 || W > MAX_ROWS) return false;
  for (int m = MAX_ROWS / W; m >= 1; --m) {
    const int nc = m * W;
    if (p.pool_mode == ASL_POOL_MAX ? R % nc == 0 : nc % 64 == 0) return nc % 64 == 0;
  }
  return false;
}

// counters, launch number and ticket, offsets
size_t sync_bytes(const AslTcPlan& tp) {
  return (2 * (size_t)tp.nseg + 1) * SYNC_STRIDE * sizeof(uint32_t) + 2 * (size_t)tp.nseg * tp.NC * sizeof(unsigned long long);
}

int round_up(int x, int to) { return (x + to - 1) / to * to; }
int div_up(int x, int by) { return (x + by - 1) / by; }

// How the G*W rows of a kv head are cut into chunks of at most 256 buffer rows in halves of HR.  Average pooling adds
// all rows of a kv head, so heads follow one another without gaps; max pooling keeps column sums per query head, so
// heads start on 32-row blocks and no head straddles the halves (unless it needs both).  As few chunks as possible
// (each streams K again), heads spread evenly over them.
void plan_chunks(const asl_params& p, AslTcPlan& tp) {
  const int W = p.window, G = p.n_q_heads / p.n_kv_heads;
  const bool per_q = p.pool_mode == ASL_POOL_MAX;
  tp.pieces = 1;
  if (W > MAX_ROWS) {
    tp.pieces = div_up(W, MAX_ROWS);
    tp.Wp = MAX_ROWS; tp.m = 1; tp.nchunk = G * tp.pieces; tp.wide = true; tp.HR = 128;
  } else if (!per_q) {
    tp.Wp = W;
    tp.nchunk = div_up(G, MAX_ROWS / W);
    tp.m = div_up(G, tp.nchunk);
    tp.wide = tp.m * W > 128;
    tp.HR = round_up(tp.wide ? div_up(tp.m * W, 2) : tp.m * W, 32);
  } else if (W > 128) {
    tp.Wp = round_up(W, 64); tp.m = 1; tp.nchunk = G; tp.wide = true; tp.HR = tp.Wp / 2;
  } else {
    tp.Wp = round_up(W, 32);
    const int in_half = 128 / tp.Wp;
    tp.wide = G > in_half;
    tp.nchunk = div_up(G, tp.wide ? 2 * in_half : in_half);
    tp.m = div_up(G, tp.nchunk);
    if (tp.wide) tp.m = round_up(tp.m, 2);
    tp.HR = tp.m * tp.Wp / (tp.wide ? 2 : 1);
  }
  tp.NC = tp.HR * (tp.wide ? 2 : 1);
}

// Tiles [deal_lo(c), deal_lo(c + 1)) of a group's N belong to CTA c of G (G <= N).  The remainder r moves from group to
// group so that no CTA always has the odd tile.
int64_t deal_lo(int64_t c, int64_t N, int64_t G, int64_t r) { return (c * N + r) / G; }

// A work list: groups cut[0] .. cut[1] - 1 and so on of segments `segs`; pass 1 of a group (unless one_pass), then pass 2
// of the group before it.  Every pass of a group is dealt to the CTAs in contiguous runs.
struct HostList {
  std::vector<TcRun> runs[2];
  std::vector<int32_t> first;
  std::vector<TcStage> stages;
  std::vector<TcFold> folds;
  int32_t most = 0;                        // tiles of the largest group in pass 2
  int grid = 1;                            // CTAs
};
HostList deal(const std::vector<TcRun>& segs, const std::vector<int>& cut, const asl_ctx* c, int most_ctas, bool one_pass) {
  HostList l;
  const int ng = (int)cut.size() - 1;
  // no more CTAs than the largest group has tiles: what has no work leaves its SM to others from the start
  for (int g = 0; g < ng; ++g) {
    int64_t N = 0;
    for (int s = cut[g]; s < cut[g + 1]; ++s) N += (c->req[segs[s].b].n + KT - 1) / KT;
    if (N > l.grid) l.grid = N < most_ctas ? (int)N : most_ctas;
  }
  const int grid = l.grid;
  l.folds.resize(segs.size());
  std::vector<int> at[2];                  // first run of each group
  for (int p = one_pass ? 1 : 0; p < 2; ++p)
    for (int g = 0; g < ng; ++g) {
      std::vector<TcRun>& runs = l.runs[p];
      at[p].push_back((int)runs.size());
      int64_t N = 0, g0 = 0;
      auto tiles = [&](int s) { const AslReq& r = c->req[segs[s].b]; return ((p ? r.T : r.n) + KT - 1) / KT; };
      for (int s = cut[g]; s < cut[g + 1]; ++s) N += tiles(s);
      const int64_t G = N < grid ? N : grid, r = (int64_t)g * (N % G) % G;
      for (int s = cut[g]; s < cut[g + 1]; ++s) {
        const int slot0 = (int)runs.size();
        for (int64_t t = g0; t < g0 + tiles(s);) {
          int64_t cta = (t * G - r) / N;
          while (deal_lo(cta + 1, N, G, r) <= t) ++cta;
          int64_t end = deal_lo(cta + 1, N, G, r);
          if (end > g0 + tiles(s)) end = g0 + tiles(s);
          TcRun run = segs[s];
          run.tile0 = (int32_t)(t - g0); run.ntiles = (int32_t)(end - t); run.pass = p + 1; run.group = g;
          run.slot = (int32_t)runs.size(); run.cta = (int32_t)cta; run.next = -1;
          runs.push_back(run);
          t = end;
        }
        if (p == 0 || one_pass) l.folds[s] = TcFold{slot0, (int32_t)runs.size() - slot0, segs[s].rows, segs[s].b};
        g0 += tiles(s);
      }
      if (p && N > l.most) l.most = (int32_t)N;
    }
  for (int p = 0; p < 2; ++p) at[p].push_back((int)l.runs[p].size());
  l.first.assign(grid, -1);
  std::vector<int> last(grid, -1);
  const int n1 = (int)l.runs[0].size();
  auto chain = [&](int p, int g) {
    for (int i = at[p][g]; i < at[p][g + 1]; ++i) {
      const int cta = l.runs[p][i].cta, index = p * n1 + i, before = last[cta];
      if (before < 0) l.first[cta] = index;
      else (before < n1 ? l.runs[0][before] : l.runs[1][before - n1]).next = index;
      last[cta] = index;
    }
  };
  for (int g = 0; g <= ng; ++g) {
    if (g < ng && !one_pass) chain(0, g);
    if (g < ng) l.stages.push_back(TcStage{cut[g], cut[g + 1] - cut[g], 0, 0});
    if (g > 0) chain(1, g - 1);
  }
  return l;
}

}  // namespace

bool asl_tc_plan(asl_ctx* c) {
  const asl_params& p = c->p;
  AslTcPlan& tp = c->tc;
  tp = AslTcPlan();
  const int W = p.window, G = p.n_q_heads / p.n_kv_heads;
  if (p.k_dtype == ASL_K_FP8_E4M3 && !fp8_shape(p)) return false;
  plan_chunks(p, tp);

  // segments in (request, head, chunk) order
  std::vector<TcRun> segs;
  int64_t tiles = 0;
  for (int b = 0; b < p.batch; ++b)
    for (int h = 0; h < p.n_kv_heads; ++h)
      for (int ch = 0; ch < tp.nchunk; ++ch) {
        TcRun s{};
        s.seg = (int32_t)segs.size();
        s.b = b; s.h = h; s.chunk = ch;
        s.T = c->req[b].T; s.u_off = c->req[b].u_off; s.tok_off = c->req[b].tok_off;
        const int heads = G - ch * tp.m < tp.m ? G - ch * tp.m : tp.m;
        const int rest = W - ch % tp.pieces * MAX_ROWS;
        s.rows = tp.pieces > 1 ? (rest < MAX_ROWS ? rest : MAX_ROWS) : (heads - 1) * tp.Wp + W;
        s.kscale = p.k_dtype == ASL_K_FP8_E4M3 ? c->k_scale[h] / Q8_SCALE : 1.0f;
        segs.push_back(s);
        tiles += (c->req[b].n + KT - 1) / KT;
      }
  tp.nseg = (int)segs.size();
  if (tiles >= (int64_t)1 << 30) return false;

  // Groups of segments: pass 1 of a group, then pass 2 of the one before it, so that the fold of the row denominators is
  // hidden behind other tiles; at least two of them, of up to 140 MB of K each, 70 MB where a kv head has several chunks.  (One, where no CTA of
  // any call has more than one tile of a pass: there is then nothing to hide the fold behind, and it is waited for once
  // instead of twice.  In us with two groups and one: 1500 tokens of 8 kv heads 21.2, 15.8, 4096 of 2 heads 13.9, 11.6.  It
  // would pay up to 1.3 tiles a CTA, 3000 tokens 19.6, 16.7, but asl_score_layer and its halves then add in different
  // orders; at 2.5 tiles not, 6000 tokens 19.0, 21.4.)  Small groups leave more of K in L2 for pass 2
  // (above), large ones need fewer hand-offs, and the hand-offs count for more.  In us at 36, 50, 70, 100, 140 and 270 MB,
  // passes issued back to back: four layers of 128K tokens 835, 836, 827, 834, 819, 824; of 100K 667, 657, 636, 638, 630, 631;
  // of 64K 448, 447, 438, 441, 441, 439; two of eight ragged requests 587, 555, 579, 569, 562, 559; two with W = 128 and 64
  // query heads at 64K 769, 760, 774, 760, 769, 771; three with FP8 keys at 48K 238, 240, 239, 236, 238, 237.  Every chunk of a kv
  // head reads its K again, in either pass: with several, what does not stay in L2 counts for more.  At 70, 100, 140 MB, four
  // layers: 64 query heads, W = 128 (four chunks) 128K 2799, 2761, 2971, 96K 2092, 2090, 2213, eight ragged requests 6375,
  // 6418, 6665; W = 64 (two) 128K 1466, 1502, 1558; 32 query heads, W = 128 (two) 100K 1124, 1136, 1184.
  const int given = p.score_ctas > 0 && p.score_ctas < c->sm_count ? p.score_ctas : 0;
  std::vector<int> cut{0};
  {
    const double limit = tp.nchunk > 1 ? 70.0e6 : 140.0e6;
    auto seg_bytes = [&](int s) { return (double)c->req[segs[s].b].n * 128 * c->k_elem_bytes / tp.nchunk; };
    double total = 0, run = 0;
    int groups = 1;
    for (int s = 0; s < tp.nseg; ++s) {
      total += seg_bytes(s);
      if (run > 0 && run + seg_bytes(s) > limit) { ++groups; run = 0; }
      run += seg_bytes(s);
    }
    if (groups < 2 && tiles > (given ? given : c->sm_count - 32)) groups = 2;
    run = 0;
    for (int s = 0; s + 1 < tp.nseg; ++s) {                // evenly sized
      run += seg_bytes(s);
      if (run + 0.5 * seg_bytes(s + 1) > total / groups * cut.size()) cut.push_back(s + 1);
    }
    cut.push_back(tp.nseg);
  }
  // CTAs: as many as the caller says; else one per SM, and where the call is one half of a layer (asl_score_columns) 16
  // fewer, so that the rest of the layer before runs beside it, 32 fewer for the shorter one-pass call with one chunk
  // per kv head
  const int spare[2] = {16, tp.nchunk == 1 ? 32 : 16};
  const int n_lists = given || p.score_ctas > 0 ? 2 : 4;
  HostList lists[4];
  for (int i = 0; i < n_lists; ++i) {
    const int ctas = given ? given : (i < 2 || c->sm_count <= 2 * spare[i & 1] ? c->sm_count : c->sm_count - spare[i & 1]);
    lists[i] = (i & 1) ? deal(segs, {0, tp.nseg}, c, ctas, true) : deal(segs, cut, c, ctas, false);
  }

  // one allocation for everything the kernels read or count in
  size_t bytes = 0;
  std::vector<char> host;
  auto put = [&](const void* data, size_t n) {
    const size_t at = bytes;
    bytes = asl_align256(bytes + n);
    host.resize(bytes, 0);
    if (n) memcpy(host.data() + at, data, n);
    return at;
  };
  struct ListAt { size_t runs, first, stages, folds; } at[4];
  size_t n_runs = 0, groups = 0, ctas = 0;                    // of the longest lists
  for (int i = 0; i < n_lists; ++i) {
    const HostList& l = lists[i];
    TcList& out = tp.lists[i >> 1][i & 1];
    out.grid = l.grid;
    out.n1 = (int32_t)l.runs[0].size();
    out.n2 = (int32_t)l.runs[1].size();
    out.n_groups = (int32_t)l.stages.size();
    out.most = l.most;
    std::vector<TcRun> runs(l.runs[0]);
    runs.insert(runs.end(), l.runs[1].begin(), l.runs[1].end());
    at[i] = ListAt{put(runs.data(), runs.size() * sizeof(TcRun)), put(l.first.data(), l.first.size() * sizeof(int32_t)),
                   put(l.stages.data(), l.stages.size() * sizeof(TcStage)), put(l.folds.data(), l.folds.size() * sizeof(TcFold))};
    if (runs.size() > n_runs) n_runs = runs.size();
    if (l.stages.size() > groups) groups = l.stages.size();
    if ((size_t)l.grid > ctas) ctas = l.grid;
    if (out.n1 > tp.partial_slots) tp.partial_slots = out.n1;
  }
  const std::vector<char> zeros(sync_bytes(tp), 0);
  const size_t sync_at = put(zeros.data(), zeros.size());
  const size_t host_bytes = bytes;
  auto take = [&](size_t n) { const size_t t = bytes; bytes = asl_align256(bytes + n); return t; };
  const size_t live_at[5] = {take(n_runs * sizeof(TcRun)), take(ctas * sizeof(int32_t)), take((size_t)tp.nseg * sizeof(TcFold)),
                             take((3 * n_runs + 6 * groups + 4 * (groups + 1) * ctas) * sizeof(int32_t)),
                             take(sizeof(int32_t))};
  cudaError_t e = cudaMalloc(&tp.d_blob, bytes);
  if (e == cudaSuccess) e = cudaMemcpy(tp.d_blob, host.data(), host_bytes, cudaMemcpyHostToDevice);
  const ScoreKernel& kern = score_kernel(score_kernel_of(p, tp));
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kern.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kern.smem);
  if (e != cudaSuccess) { cudaGetLastError(); asl_tc_free(c); return false; }
  char* d = static_cast<char*>(tp.d_blob);
  for (int i = 0; i < n_lists; ++i) {
    TcList& out = tp.lists[i >> 1][i & 1];
    out.d_runs = reinterpret_cast<TcRun*>(d + at[i].runs);
    out.d_first = reinterpret_cast<int32_t*>(d + at[i].first);
    out.d_stages = reinterpret_cast<TcStage*>(d + at[i].stages);
    out.d_folds = reinterpret_cast<TcFold*>(d + at[i].folds);
  }
  if (n_lists == 2) { tp.lists[1][0] = tp.lists[0][0]; tp.lists[1][1] = tp.lists[0][1]; }
  tp.d_sync = reinterpret_cast<uint32_t*>(d + sync_at);
  tp.d_live_runs = reinterpret_cast<TcRun*>(d + live_at[0]);
  tp.d_live_first = reinterpret_cast<int32_t*>(d + live_at[1]);
  tp.d_live_folds = reinterpret_cast<TcFold*>(d + live_at[2]);
  tp.d_live_scratch = reinterpret_cast<int32_t*>(d + live_at[3]);
  tp.d_live_hdr = reinterpret_cast<int32_t*>(d + live_at[4]);
  return encode_fn() != nullptr;
}

size_t asl_tc_partial_bytes(const asl_ctx* c) { return (size_t)c->tc.partial_slots * (c->tc.wide ? GROUPS / 2 : GROUPS) * c->tc.NC * sizeof(float2); }

void asl_tc_free(asl_ctx* c) {
  AslTcPlan& tp = c->tc;
  if (tp.d_blob) cudaFree(tp.d_blob);
  tp = AslTcPlan();
}

asl_status asl_launch_wait_selftest(asl_ctx* c, int which, unsigned long long limit_ns, cudaStream_t st) {
  bounded_wait_selftest_kernel<<<1, 32, 0, st>>>(which, limit_ns, reinterpret_cast<const uint32_t*>(c->d_err), c->d_err);   // the error word is never all ones
  c->launches += 1;
  ASL_CUDA(cudaGetLastError());
  return ASL_OK;
}

asl_status asl_launch_window_lse(asl_ctx* c, const char* ws, float* lse_out, cudaStream_t st) {
  const AslTcPlan& tp = c->tc;
  const int n = c->p.batch * c->p.n_q_heads * c->p.window;
  offsets_to_lse_kernel<<<(n + 255) / 256, 256, 0, st>>>(reinterpret_cast<const float*>(ws + c->ws.score_offsets), lse_out, n, c->p.window,
                                                         c->p.n_q_heads / c->p.n_kv_heads, tp.m, tp.Wp, tp.pieces, tp.nchunk, tp.NC);
  c->launches += 1;
  ASL_CUDA(cudaGetLastError());
  return ASL_OK;
}

asl_status asl_launch_live_phases(asl_ctx* c, bool two_pass, bool beside, cudaStream_t st) {
  AslTcPlan& tp = c->tc;
  const TcList& l = tp.lists[beside][!two_pass];
  live_list_kernel<<<1, 1024, 0, st>>>(l.d_runs, l.n1, l.n2, l.d_folds, tp.nseg, l.n_groups, l.most + l.most / 4, c->latch_stat, c->cur_layer,
                                       c->p.batch, l.grid, tp.d_live_hdr, tp.d_live_runs, tp.d_live_first, tp.d_live_folds, tp.d_live_scratch);
  c->launches += 1;
  ASL_CUDA(cudaGetLastError());
  return ASL_OK;
}

// after a reported device error the counters may be inconsistent: start over
asl_status asl_tc_reset_sync(asl_ctx* c, cudaStream_t st) {
  AslTcPlan& tp = c->tc;
  if (!tp.d_sync) return ASL_OK;
  ASL_CUDA(cudaMemsetAsync(tp.d_sync, 0, sync_bytes(tp), st));
  return ASL_OK;
}

asl_status asl_launch_score_tc(asl_ctx* c, const void* q, const void* k, const float* lse, float* u, char* ws, bool beside,
                               cudaStream_t st) {
  const asl_params& p = c->p;
  AslTcPlan& tp = c->tc;
  const int W = p.window, G = p.n_q_heads / p.n_kv_heads;
  const bool fp8 = p.k_dtype == ASL_K_FP8_E4M3;
  CUtensorMap tm_q, tm_k;
  // one copy brings all heads of a chunk where they follow one another in the buffer as in the tensor
  const cuuint32_t box_t = (cuuint32_t)(W < MAX_ROWS ? W : MAX_ROWS), box_h = (cuuint32_t)(tp.pieces == 1 && tp.Wp == W ? tp.m : 1);
  if (fp8) {
    // the queries as two E4M3 terms in the workspace, then 8-bit maps: rows of 128 one-byte channels
    uint8_t* q8 = reinterpret_cast<uint8_t*>(ws + c->ws.score_q8);
    const int64_t total = (int64_t)p.batch * p.n_q_heads * W * 128;
    split_queries_e4m3_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(
        static_cast<const __nv_bfloat16*>(q), p.q_stride[0], p.q_stride[1], p.q_stride[2], p.n_q_heads, W, total, q8);
    c->launches += 1;
    const cuuint64_t qdims[5] = {128, (cuuint64_t)W, (cuuint64_t)p.n_q_heads, (cuuint64_t)p.batch, 2};
    const cuuint64_t qstr[4] = {128, (cuuint64_t)W * 128, (cuuint64_t)p.n_q_heads * W * 128, (cuuint64_t)total};
    const cuuint32_t qbox[5] = {128, box_t, box_h, 1, 1};
    if (!make_map(&tm_q, CU_TENSOR_MAP_DATA_TYPE_UINT8, q8, 5, qdims, qstr, qbox)) return ASL_ERR_CUDA;
    const cuuint64_t kdims[3] = {128, (cuuint64_t)p.n_kv_heads, (cuuint64_t)c->sum_tokens};
    const cuuint64_t kstr[2] = {(cuuint64_t)p.k_stride[1], (cuuint64_t)p.k_stride[0]};
    const cuuint32_t kbox[3] = {128, 1, (cuuint32_t)KT};
    if (!make_map(&tm_k, CU_TENSOR_MAP_DATA_TYPE_UINT8, k, 3, kdims, kstr, kbox)) return ASL_ERR_CUDA;
  } else {
    const cuuint64_t dims[4] = {128, (cuuint64_t)W, (cuuint64_t)p.n_q_heads, (cuuint64_t)p.batch};
    const cuuint64_t strides[3] = {(cuuint64_t)p.q_stride[2] * 2, (cuuint64_t)p.q_stride[1] * 2, (cuuint64_t)p.q_stride[0] * 2};
    const cuuint32_t box[4] = {64, box_t, box_h, 1};
    if (!make_map(&tm_q, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, q, 4, dims, strides, box)) return ASL_ERR_CUDA;
    const cuuint64_t kdims[3] = {128, (cuuint64_t)p.n_kv_heads, (cuuint64_t)c->sum_tokens};
    const cuuint64_t kstr[2] = {(cuuint64_t)p.k_stride[1] * 2, (cuuint64_t)p.k_stride[0] * 2};
    const cuuint32_t kbox[3] = {64, 1, (cuuint32_t)KT};
    if (!make_map(&tm_k, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, k, 3, kdims, kstr, kbox)) return ASL_ERR_CUDA;
  }
  TcArgs a{};
  const TcList& list = tp.lists[beside][lse != nullptr];
  a.list = {list.d_runs, list.d_first, list.d_folds};
  if (c->latch_stat && c->cur_layer >= 0 && p.batch <= ASL_SKIP_MAX_BATCH) {      // written by asl_launch_live_phases just before
    a.live = {tp.d_live_runs, tp.d_live_first, tp.d_live_folds};
    a.live_hdr = tp.d_live_hdr;
  }
  a.stages = list.d_stages;
  a.n_stages = lse ? 0 : list.n_groups;
  a.lse = lse;
  a.partials = reinterpret_cast<float2*>(ws + c->ws.score_partials);
  a.offsets = reinterpret_cast<float*>(ws + c->ws.score_offsets);
  a.u = u;
  a.counters = tp.d_sync;                                            // the one-pass launch touches neither these
  a.launch = tp.d_sync + 2 * (size_t)tp.nseg * SYNC_STRIDE;         // nor these
  a.ready = reinterpret_cast<unsigned long long*>(a.launch + SYNC_STRIDE);
  a.err = c->d_err;
  a.u_stride = c->u_stride;
  a.nseg = tp.nseg;
  a.NC = tp.NC; a.HR = tp.HR; a.W = W; a.Wp = tp.Wp; a.m = tp.m; a.pieces = tp.pieces; a.G = G; a.Hq = p.n_q_heads;
  a.u_rows_per_kv = c->u_rows_per_kv;
  a.u_parts = c->u_parts;
  a.scale_log2 = (float)(1.4426950408889634 / sqrt((double)p.head_dim));
  // every CTA must be resident at once (pass 2 waits for counters other CTAs advance): one CTA per SM at most
  const ScoreKernel& kern = score_kernel(score_kernel_of(p, tp));
  if (a.live_hdr) kern.fn<<<list.grid, THREADS, kern.smem, st>>>(tm_q, tm_k, a);     // (the kernel before writes the list, which is read as constant)
  else launch_after_smem(kern.fn, dim3(list.grid), dim3(THREADS), kern.smem, st, tm_q, tm_k, a);
  c->launches += 1;
  ASL_CUDA(cudaGetLastError());
  return ASL_OK;
}
