// Tensor-core attention over the packed cache (Eq. 1 with the dequantisation of
// Eq. 10) for sm_100a: tcgen05.mma with accumulators in tensor memory, operands
// staged by bulk asynchronous copies (TMA) and dequantised in shared memory.
//
// Work.  An item is (head, pair of 128-query tiles); it meets every 128-slot key
// tile of the cache.  Items x key tiles are laid out on one line of steps, and the
// line is cut into equal pieces, one per CTA (one CTA per SM).  A piece that does
// not cover an item completely leaves partial results (accumulator, running max
// and sum) in a scratch slot; a second kernel merges them.
//
// One CTA.  24 warps:
//   16 warps    softmax: a warp takes 16 whole rows of a query tile, half of a TMEM lane quarter; a quad of
//               lanes holds 128 scores each of two rows, loaded into registers at once, exchanges their
//               maxima by shuffles and writes P (16-bit) back to tensor memory.  O is rescaled only when
//               the running maximum grew by more than 2^14.  Registers move to these warps with setmaxnreg.
//   4 warps     operand producers (4 and 8 bits): packed codes (raw, as copied by TMA) -> fp16 K~ (per channel
//               and key group) and V~ (per token) in the 128-byte-swizzled layouts the MMA
//               descriptors expect.  One dequantised tile serves both query tiles.
//   2 warps     issue the MMAs of query tile 0 resp. 1 through an elected lane:
//               S_t = Q_t K~^T (M128 N128 K64) and O_t += P_t V~ (M128 N64 K128,
//               A = P from tensor memory).  The warps stay converged: a lone thread in a branch
//               gets one tcgen05.mma through every 48-62 clk at best (its operands are moved into
//               uniform registers each time), an elected lane every 30 clk for P V~.  Measured
//               (16384 cached tokens, 1374 queries): 4-bit 160.3 -> 158.6 us, keys quantised once
//               188.5 -> 181.9 us, 16-bit at 32768 tokens 287.1 -> 273.8 us.
//   1 thread    issues the bulk copies of the raw tiles, several steps ahead; its warp owns the
//               tensor-memory allocation (all 512 columns).
//   1 warp      with keys quantised once asks for the key constants a few tiles ahead of the producers,
//               else idle.
// 4-bit caches multiply in fp16 (the dequantised keys are not bf16-representable:
// rounding them to bf16 alone costs ~1e-2 relative L2 with outlier channels);
// 16-bit caches hold bf16 rows in the operands' order, which the copies bring to the operand tiles, and multiply in
// bf16.  Accumulation is fp32.
//
// Every mbarrier wait is bounded (one second of running time): when the bound is hit the CTA carries on
// without waiting and records XKV_E_TIMEOUT in the status words of the caches in its piece, so the
// kernel always terminates, drains its copies and frees its tensor memory.
#include <mutex>
#include <stdlib.h>

#include "xkv_internal.cuh"

namespace xkv {

namespace {

constexpr int kMaxDevices = 64;
// Warps: 0-15 softmax, 16-19 producers, 20 and 22 issue the MMAs of query tile 0 resp. 1, 21 issues the
// copies and owns the tensor memory; 23 asks for the key constants ahead of the producers (keys
// quantised once; else it only completes the warpgroup that setmaxnreg needs).
constexpr int kThreads = 768;
// registers per thread after the reallocation (setmaxnreg)
constexpr int kRegsSoftmax = 96;
// (24 layers, three streams in turn: tail at 16384 4225 us with 56 + 40, 4118 with 64 + 32, 4048 with 72 + 24, which is not
// taken up here; keys once at 16384 4515 with 48 + 48, 4329 with 56 + 40, 4326 with 64 + 32, 8-bit at 8192 2096, 1988 and
// 1973; 4-bit at 16384 3761, 3763, 3768 and 3757 with 40, 48, 56 and 64 for the producers, within the noise.  16-bit
// caches give the producers, who have nothing to do there, 48 as well.)
__host__ __device__ constexpr int regs_producers(bool once, bool tail) { return tail ? 64 : once ? 56 : 48; }
__host__ __device__ constexpr int regs_misc(bool once, bool tail) { return 96 - regs_producers(once, tail); }   // MMA issuers, copy thread
constexpr int kQRows = 128;
constexpr int kMaxGrid = 160;                 // CTAs the scratch is sized for (>= SM count of the part)
constexpr uint32_t kSpinLimit = 1u << 22;
// The reference maximum of a row moves only when the row maximum exceeds it by more than 2^kGrow
// (log2 units).  Until then exponentials reach at most 2^14 = 16384, inside the fp16 range.  Sums are
// rescaled row by row, but the accumulator as soon as one of a warp's 16 rows asks for it, so a low
// threshold would trip it at every few tiles (24 layers at 4096: 14, 8, 4 take 1018, 1034, 1058 us; at 16384
// 3764, 3793, 3827).
constexpr float kGrow = 14.f;

constexpr uint32_t kAhead = 4;        // tiles whose constants are asked for ahead of the producers (keys quantised once)

// ring depths: kNK, kNV operand tiles of K~ and V~, kNR raw stages
template <int BITS> struct Cfg;
template <> struct Cfg<4> {
  static constexpr int kNK = 3, kNV = 3;
  static constexpr int kNR = 4;               // raw stages
  static constexpr int kRawK = 4096, kRawV = 4096, kRawKP = 1024, kRawVP = 1024;
  static constexpr int kRawStage = kRawK + kRawV + kRawKP + kRawVP;
};
template <> struct Cfg<8> {                    // 8-bit codes, keys quantised once: K, V rows of 64 bytes,
  static constexpr int kNK = 3, kNV = 3;
  static constexpr int kNR = 4;               // 128 group references (in the K-parameter region), V parameters
  static constexpr int kRawK = 8192, kRawV = 8192, kRawKP = 1024, kRawVP = 1024;
  static constexpr int kRawStage = kRawK + kRawV + kRawKP + kRawVP;
};
// 16-bit caches: no raw stages and no work for the producers, whose copies within shared memory (64 KB a tile, read and
// written) cost time and, at the power cap, clock.  24 layers, 1374 tokens at 32768: 7783 -> 7641 us a step.
template <> struct Cfg<16> {                   // rows are stored as the MMA wants them (BufSet): the copies fill the
  static constexpr int kNK = 4, kNV = 4;      // operand tiles themselves
  static constexpr int kNR = 1;               // (no raw stages: two unused barriers)
  static constexpr int kRawK = 16384, kRawV = 16384, kRawKP = 0, kRawVP = 0;
  static constexpr int kRawStage = 0;
};

// shared memory map (offsets from a 1024-byte aligned base)
constexpr int kOffQ = 0;                          // 2 x 16 KB  Q tiles, K-major, SW128
constexpr int kOffK = 32768;                      // kNK x 16 KB  K~ tiles
constexpr int kTabBytes = 768 + 2048;             // K table 768 B + V table 2048 B of fp16 parameters
constexpr int kBarBytes = 512;                    // barriers, tmem base, abort flag
template <int BITS> struct Map {
  static constexpr int kOffV = kOffK + Cfg<BITS>::kNK * 16384;          // kNV x 16 KB  V~ tiles
  static constexpr int kOffTab = kOffV + Cfg<BITS>::kNV * 16384;        // two tables (512 bytes that keep the alignment in 16-bit caches)
  static constexpr int kOffBar = kOffTab + (BITS == 16 ? 512 : 2 * kTabBytes);
  static constexpr int kOffRaw = kOffBar + kBarBytes;                   // raw stages (16-byte aligned)
};
template <int BITS> constexpr int smem_bytes() {
  return Map<BITS>::kOffRaw + Cfg<BITS>::kNR * Cfg<BITS>::kRawStage + 1024;
}

// Tensor memory columns (all 512).  A query tile has three blocks of 64 columns, B0 B1 B2.  In even
// steps its scores take B0 B1 and P (16-bit pairs) goes over B0 once the scores are in registers; in
// odd steps the scores take B1 B2 and P goes over B2.  So the scores of a step are computed during the
// softmax of the step before, whose P they do not touch, and P never waits for the P V~ before.
constexpr int kColTile = 192;      // * t
constexpr int kColO = 384;         // + 64 t : 64 fp32 columns, the accumulator
constexpr int kTmemCols = 512;

// one partial slot: two query tiles x 128 rows x (64 accumulators + max + sum)
constexpr size_t kSlotFloats = 2 * 128 * 64;
constexpr size_t kSlotBytes = kSlotFloats * sizeof(float) + 2 * 128 * sizeof(float2);

// One cache (or a prefix of one) and the queries that attend to it.
struct Job {
  const __nv_bfloat16* q;
  __nv_bfloat16* out;
  const uint8_t* k;
  const float2* kpar;
  const uint8_t* v;
  const float2* vpar;
  int* status;
  // Newest frame unquantised (Eq. 1 read literally): when k_tail is set, the key slots
  // [tail_lo, t_phys) take K~, V~ from these bf16 tensors ([head][token][64] with the strides
  // of Args, token = slot - tail_lo) instead of the packed rows.
  const __nv_bfloat16* k_tail;
  const __nv_bfloat16* v_tail;
  // Quantise-once mode: every token refers to the parameter-table slot of its key group
  // (kslot [cap]); ktab16 [slot][n_heads][8][12] holds, per 8-channel word, the four fp16 pairs
  // of scales, offsets and constants that dequant_word_h takes.
  const int32_t* kslot;
  const uint32_t* ktab16;
  int n, cap, t_first, t_phys, tail_lo, n_heads;
  int n_tiles;          // key tiles of the cache
  int q_tiles;          // 128-row query tiles of the frame
  int n_pairs;          // ceil(q_tiles / 2)
  uint32_t step_lo, step_hi;   // its steps on the line: n_heads * n_pairs items of n_tiles steps
};

// Layers of a stack or frames of a chunk in one launch: fewer pieces are cut (an item that is cut
// costs its queries, first scores and epilogue once more, about 3.3 steps, and a merge), and the
// multiprocessors run out of work together once per launch.  The table travels in the kernel's
// parameters, whose classic limit of 4 KB it stays below.
constexpr int kMaxJobs = kMaxLayers;
struct Args {
  int64_t ts, hs;       // strides of q, out, k_tail and v_tail
  float scale_log2;
  int n_jobs;
  int grid;             // pieces that the line of all steps is cut into: the first `longer` of them have
  uint32_t piece, longer;      // piece + 1 steps, the others `piece`
  float* part_o;        // [2 * grid][2][128][64]
  float2* part_ml;      // [2 * grid][2][128]
  Job job[kMaxJobs];
};
static_assert(sizeof(Args) <= 4096, "the job table");

__device__ __forceinline__ uint32_t piece_start(const Args& a, int b) {
  return (uint32_t)b * a.piece + min((uint32_t)b, a.longer);
}

// A CTA's walk along the line: the parts of items that its piece covers, one after the other.
struct Walk {
  uint32_t pos, end;
  int job;
  // of the current segment
  int h, pair, tile_lo, nt;
  __device__ __forceinline__ Walk(const Args& a) {
    pos = piece_start(a, blockIdx.x);
    end = piece_start(a, blockIdx.x + 1);
    job = 0;
  }
  __device__ __forceinline__ bool next(const Args& a) {
    if (pos >= end) return false;
    while (pos >= a.job[job].step_hi) ++job;
    const uint32_t tiles = (uint32_t)a.job[job].n_tiles, pairs = (uint32_t)a.job[job].n_pairs;
    const uint32_t rel = pos - a.job[job].step_lo;
    const uint32_t item = rel / tiles, head = item / pairs;
    tile_lo = (int)(rel - item * tiles);
    nt = (int)min(tiles - (uint32_t)tile_lo, end - pos);
    h = (int)head;
    pair = (int)(item - head * pairs);
    pos += (uint32_t)nt;
    return true;
  }
};

// ---- PTX wrappers -----------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
constexpr uint32_t kSuspendNs = 2000;
// The same with a time the hardware may keep the thread suspended before it answers "not yet"
// (it answers at once when the phase completes).
__device__ __forceinline__ bool mbar_try_suspend(uint32_t bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(ns) : "memory");
  return ok != 0;
}
// Up to 64 suspended tries in a loop of three instructions (try, branch out, count and branch back).
__device__ __forceinline__ bool mbar_try_many(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .pred q;\n\t.reg .u32 n;\n\t"
      "mov.u32 n, 64;\n\t"
      "XKV_TRY_%=:\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "@p bra XKV_DONE_%=;\n\t"
      "sub.u32 n, n, 1;\n\t"
      "setp.ne.u32 q, n, 0;\n\t"
      "@q bra XKV_TRY_%=;\n\t"
      "XKV_DONE_%=:\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(kSuspendNs) : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait.  On exhaustion a per-CTA flag goes up, and every later wait of the CTA gives up at
// once; at its end the CTA records the failure in the status words of the caches that it worked on.
struct WaitCtx { uint32_t abort_flag; };      // address in shared memory
__device__ __forceinline__ uint32_t ld_shared_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_shared_u32(uint32_t addr, uint32_t v) {
  asm volatile("st.volatile.shared.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// Threads on the critical chain (softmax warps, MMA issuers: SLEEP_NS below 128) retry at once, each
// try suspended by the hardware for a short while: their wake-up latency is part of every step.
// Threads that wait long and have slack (operand producers, the copy thread) sleep SLEEP_NS between
// tries, so that their polls (shared-memory instructions) do not take issue slots and queue space
// from the softmax warps.  The wait gives up after one second AND kWaitMinRounds rounds of tries
// (32 or 64 each): the rounds only count while the thread runs, so that a kernel that was
// descheduled for a while (a GPU shared between processes) does not time out on the clock alone.
constexpr uint64_t kWaitLimitNs = 1000000000ull;      // one second ...
constexpr uint32_t kWaitMinRounds = 1u << 12;         // ... and this many rounds, then XKV_E_TIMEOUT
constexpr int kSlack = 1000;     // sleep of the producers and the copy thread (256: 16-bit at 32768 tokens 6440 instead of 6290 us)
template <int SLEEP_NS = 32>
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, const WaitCtx& wc) {
  if (mbar_try(bar, parity)) return;          // the common case costs one instruction
  if (ld_shared_u32(wc.abort_flag)) return;
  const uint64_t t0 = global_ns();
  uint32_t rounds = 0;
  do {
    if (SLEEP_NS >= 128) {
#pragma unroll 1
      for (int it = 0; it < 32; ++it) {
        if (mbar_try_suspend(bar, parity, kSuspendNs)) return;
        __nanosleep(SLEEP_NS);
      }
    } else if (mbar_try_many(bar, parity)) {
      return;
    }
  } while (++rounds < kWaitMinRounds || global_ns() - t0 < kWaitLimitNs);
  st_shared_u32(wc.abort_flag, 1u);
}
// A wait of the CTA ran out: the results of the caches with steps in its piece are void.
__device__ __forceinline__ void report_timeout(const Args& a) {
  const uint32_t lo = piece_start(a, blockIdx.x), hi = piece_start(a, blockIdx.x + 1);
  for (int j = 0; j < a.n_jobs; ++j)
    if (a.job[j].step_lo < hi && a.job[j].step_hi > lo) atomicExch(a.job[j].status, (int)XKV_E_TIMEOUT);
}
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// packed fp32 pairs (two floats in one 64-bit register)
__device__ __forceinline__ uint64_t pack_f2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float f2_lo(uint64_t v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float f2_hi(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }
__device__ __forceinline__ uint64_t fma_f2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add_f2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul_f2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// One lane of a converged warp.  The issuing warps run converged and let one elected lane issue, so
// that descriptors and addresses stay warp-uniform and live in uniform registers: inside a branch
// that only one lane takes, every tcgen05.mma is preceded by moves of its operands into them.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}
// D[tmem] (+)= A[smem] * B[smem]
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(acc) : "memory");
}

// Tensor memory <-> registers, 16 lanes (rows) of the calling warp's quarter.  Of every 8 columns lane l holds, as in
// the accumulators of a warp-level MMA, columns 2 (l mod 4) and the next of row l / 4 (registers 4g, 4g + 1) and of row
// l / 4 + 8 (4g + 2, 4g + 3).  A pair of neighbours makes one 32-bit word of 16-bit P, and of every 4 words lane l
// holds word l mod 4 of the same two rows (2g, 2g + 1).  LD_64, ST_64: 64 columns; ST_P32: 32 words.
#define XKV_TMEM_LD_64(taddr, r, o)                                                                 \
  asm volatile(                                                                                     \
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 {"                                                    \
      "%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"                                      \
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"                    \
      : "=r"(r[(o) + 0]), "=r"(r[(o) + 1]), "=r"(r[(o) + 2]), "=r"(r[(o) + 3]),                     \
        "=r"(r[(o) + 4]), "=r"(r[(o) + 5]), "=r"(r[(o) + 6]), "=r"(r[(o) + 7]),                     \
        "=r"(r[(o) + 8]), "=r"(r[(o) + 9]), "=r"(r[(o) + 10]), "=r"(r[(o) + 11]),                   \
        "=r"(r[(o) + 12]), "=r"(r[(o) + 13]), "=r"(r[(o) + 14]), "=r"(r[(o) + 15]),                 \
        "=r"(r[(o) + 16]), "=r"(r[(o) + 17]), "=r"(r[(o) + 18]), "=r"(r[(o) + 19]),                 \
        "=r"(r[(o) + 20]), "=r"(r[(o) + 21]), "=r"(r[(o) + 22]), "=r"(r[(o) + 23]),                 \
        "=r"(r[(o) + 24]), "=r"(r[(o) + 25]), "=r"(r[(o) + 26]), "=r"(r[(o) + 27]),                 \
        "=r"(r[(o) + 28]), "=r"(r[(o) + 29]), "=r"(r[(o) + 30]), "=r"(r[(o) + 31])                  \
      : "r"(taddr) : "memory")

#define XKV_TMEM_ST_64(taddr, r)                                                                    \
  asm volatile(                                                                                     \
      "tcgen05.st.sync.aligned.16x256b.x8.b32 [%0], {"                                              \
      "%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"                                     \
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"                           \
      ::"r"(taddr),                                                                                 \
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]),                                                 \
        "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),                                                 \
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]),                                               \
        "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),                                             \
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),                                             \
        "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),                                             \
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),                                             \
        "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]) : "memory")

#define XKV_TMEM_ST_P32(taddr, r)                                                                   \
  asm volatile(                                                                                     \
      "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], {"                                              \
      "%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"                                    \
      ::"r"(taddr),                                                                                 \
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]),                                                 \
        "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),                                                 \
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]),                                               \
        "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory")

// Shared-memory matrix descriptor, 128-byte swizzle, 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFF);        // start address
  d |= (uint64_t)1 << 16;                        // leading byte offset (unused with one swizzle span)
  d |= (uint64_t)(1024 >> 4) << 32;              // stride byte offset between 8-row groups
  d |= (uint64_t)1 << 46;                        // descriptor version of this architecture
  d |= (uint64_t)2 << 61;                        // SWIZZLE_128B
  return d;
}

// Instruction descriptor for kind::f16: fp32 accumulate, M = 128.
__device__ __forceinline__ uint32_t make_idesc(int n_dim, bool bf16, bool b_mn_major) {
  uint32_t d = 0;
  d |= 1u << 4;                                  // D format fp32
  d |= (bf16 ? 1u : 0u) << 7;                    // A format
  d |= (bf16 ? 1u : 0u) << 10;                   // B format
  d |= (b_mn_major ? 1u : 0u) << 16;             // B major
  d |= (uint32_t)(n_dim >> 3) << 17;
  d |= (uint32_t)(128 >> 4) << 24;
  return d;
}

__device__ __forceinline__ uint32_t swz_off(int row, int chunk) {
  return (uint32_t)((row >> 3) * 1024 + (row & 7) * 128 + ((chunk ^ (row & 7)) << 4));
}

__device__ __forceinline__ uint32_t pack_h2(float a, float b) {
  const __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t pack_bf2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t h2_sub(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}


__device__ __forceinline__ uint32_t h2_fma(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t r;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}

// Eight 4-bit codes of one packed word -> four fp16 pairs of s * (q - z)  (Eq. 10).
// (w & 0x000F000F) | 0x6400 is the fp16 number 1024 + q and (w & 0x00F000F0) | 0x5400 is 64 + q.
// Every pair is formed as  fma(biased - zo, s, c)  with the constants of dequant_consts.
// Pairs 0 and 2 of a word carry the bias 1024, pairs 1 and 3 the bias 64.
__device__ __forceinline__ uint4 dequant_word_h(uint32_t w, const uint32_t (&s2)[4], const uint32_t (&zo)[4],
                                                const uint32_t (&c2)[4]) {
  const uint32_t t = w >> 8;
  const uint32_t a0 = (w & 0x000F000Fu) | 0x64006400u;
  const uint32_t a1 = (w & 0x00F000F0u) | 0x54005400u;
  const uint32_t a2 = (t & 0x000F000Fu) | 0x64006400u;
  const uint32_t a3 = (t & 0x00F000F0u) | 0x54005400u;
  uint4 r;
  r.x = h2_fma(h2_sub(a0, zo[0]), s2[0], c2[0]);
  r.y = h2_fma(h2_sub(a1, zo[1]), s2[1], c2[1]);
  r.z = h2_fma(h2_sub(a2, zo[2]), s2[2], c2[2]);
  r.w = h2_fma(h2_sub(a3, zo[3]), s2[3], c2[3]);
  return r;
}

// The same for eight 8-bit codes (two words, channels 4i..4i+3 as c0 | c2<<8 | c1<<16 | c3<<24):
// (w & 0x00FF00FF) | 0x6400 is the fp16 pair (1024 + c0, 1024 + c1), the word shifted by 8 gives
// (1024 + c2, 1024 + c3); every pair carries the bias 1024.
__device__ __forceinline__ uint4 dequant_word_h(uint2 w, const uint32_t (&s2)[4], const uint32_t (&zo)[4],
                                                const uint32_t (&c2)[4]) {
  const uint32_t a0 = (w.x & 0x00FF00FFu) | 0x64006400u;
  const uint32_t a1 = ((w.x >> 8) & 0x00FF00FFu) | 0x64006400u;
  const uint32_t a2 = (w.y & 0x00FF00FFu) | 0x64006400u;
  const uint32_t a3 = ((w.y >> 8) & 0x00FF00FFu) | 0x64006400u;
  uint4 r;
  r.x = h2_fma(h2_sub(a0, zo[0]), s2[0], c2[0]);
  r.y = h2_fma(h2_sub(a1, zo[1]), s2[1], c2[1]);
  r.z = h2_fma(h2_sub(a2, zo[2]), s2[2], c2[2]);
  r.w = h2_fma(h2_sub(a3, zo[3]), s2[3], c2[3]);
  return r;
}

// fp16 can hold magnitudes up to 65504; anything beyond (or not a number) is reported.
__device__ __forceinline__ bool beyond_fp16(float x) { return !(fabsf(x) <= 65504.f); }
__device__ __noinline__ void report_range(int* status) { atomicCAS(status, 0, (int)XKV_E_RANGE); }

// true when one of the two fp16 numbers is an infinity or a NaN (all exponent bits set)
__device__ __forceinline__ bool h2_not_finite(uint32_t h) {
  return (h & 0x7C00u) == 0x7C00u || (h & 0x7C000000u) == 0x7C000000u;
}

// Eight bf16 values -> eight fp16 values (exact whenever the value is in fp16's range).
__device__ __forceinline__ uint4 bf16x8_to_h8(const uint4& u) {
  const uint32_t r[4] = {u.x, u.y, u.z, u.w};
  uint32_t h[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) h[i] = pack_h2(__uint_as_float(r[i] << 16), __uint_as_float(r[i] & 0xFFFF0000u));
  return make_uint4(h[0], h[1], h[2], h[3]);
}

// Rows of the unquantised newest frame over the dequantised rows of a K~ or V~ tile: keys
// row0 + STEP i of the tile (whose first slot is `base`) that lie in [tail_lo, t_phys) are replaced by
// the caller's bf16 rows (src already points at this thread's head and 8-channel chunk w).  The rows
// are those that the same thread has dequantised.  A real call, so that the producers' loop carries
// none of this code.
template <int STEP>
__device__ __noinline__ void tail_rows_over(uint8_t* tile, const __nv_bfloat16* src, int64_t ts, int base, int row0, int w,
                                            int tail_lo, int t_phys, int* status) {
  bool bad = false;       // something beyond fp16
#pragma unroll 1
  for (int i0 = 0; i0 < 8; i0 += 4) {
    uint4 u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int slot = base + row0 + STEP * (i0 + i);
      u[i] = make_uint4(0, 0, 0, 0);
      if (slot >= tail_lo && slot < t_phys) u[i] = *reinterpret_cast<const uint4*>(src + (int64_t)(slot - tail_lo) * ts);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int row = row0 + STEP * (i0 + i), slot = base + row;
      if (slot >= tail_lo && slot < t_phys) {
        const uint4 hv = bf16x8_to_h8(u[i]);
        *reinterpret_cast<uint4*>(tile + swz_off(row, w)) = hv;
        bad |= h2_not_finite(hv.x) || h2_not_finite(hv.y) || h2_not_finite(hv.z) || h2_not_finite(hv.w);
      }
    }
  }
  if (bad) report_range(status);
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Bulk asynchronous copy global -> this CTA's shared memory, completion counted on an mbarrier.
// Addresses 16-byte aligned, size a multiple of 16.  No multicast.
__device__ __forceinline__ void tma_load_1d(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
// Keys quantised once: the rows of one K~ tile.  Thread t = (8-channel word, eight consecutive keys);
// the constants of a key's group come from the table in global memory, and only where the group
// changes: neighbours mostly belong to the same one, so a thread fetches them once or twice instead
// of eight times (keys 16 apart, two at a time, took 4650 clk a tile in this kernel).
// WORD: the codes of eight channels (uint32_t: 4-bit, uint2: 8-bit).
template <typename WORD>
__device__ __forceinline__ void once_keys(const uint8_t* codes, const uint8_t* refs, uint8_t* tile, const uint32_t* ktab16,
                                          int n_heads, int h, int t, uint32_t b_free, uint32_t parity, const WaitCtx& wc) {
  const int w = t & 7, k0 = (t >> 3) * 8;
  const int4 ra = *reinterpret_cast<const int4*>(refs + 4 * k0), rb = *reinterpret_cast<const int4*>(refs + 4 * k0 + 16);
  const int ref[8] = {ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z, rb.w};
  const uint4* table = reinterpret_cast<const uint4*>(ktab16) + (h * 8 + w) * 3;
  uint4 sv, zv, cv;
  auto fetch = [&](int r) {
    const uint4* e = table + (size_t)r * n_heads * 24;
    sv = __ldg(e); zv = __ldg(e + 1); cv = __ldg(e + 2);
  };
  fetch(ref[0]);
  WORD wd[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) wd[i] = *reinterpret_cast<const WORD*>(codes + (k0 + i) * (8 * sizeof(WORD)) + w * sizeof(WORD));
  mbar_wait<kSlack>(b_free, parity, wc);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if (i > 0 && ref[i] != ref[i - 1]) fetch(ref[i]);
    const uint32_t s2[4] = {sv.x, sv.y, sv.z, sv.w}, zo[4] = {zv.x, zv.y, zv.z, zv.w}, c2[4] = {cv.x, cv.y, cv.z, cv.w};
    *reinterpret_cast<uint4*>(tile + (k0 + i) * 128 + ((w ^ i) << 4)) = dequant_word_h(wd[i], s2, zo, c2);
  }
}
// O *= alpha for the calling warp's 16 rows (two per thread); a real call, to keep its registers out of the
// softmax loop.  Warp-collective.
__device__ __noinline__ void rescale_rows(uint32_t col_o, float alpha0, float alpha1) {
  uint32_t ro[32];
  XKV_TMEM_LD_64(col_o, ro, 0);
  tc_wait_ld();
#pragma unroll
  for (int i = 0; i < 32; ++i) ro[i] = __float_as_uint(__uint_as_float(ro[i]) * ((i & 2) ? alpha1 : alpha0));
  XKV_TMEM_ST_64(col_o, ro);
  tc_wait_st();
}
__device__ __forceinline__ void producer_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }

}  // namespace

// TAIL: the newest frame's keys and values come unquantised from Args::k_tail, v_tail (a separate
// instantiation, so that the kernel without a tail carries none of its code).
// ONCE: the keys' dequantisation constants are looked up per token (quantise-once mode) instead of
// per 64-slot run.
template <int BITS, bool TAIL = false, bool ONCE = false>
__global__ void __launch_bounds__(kThreads, 1) attn_tc_kernel(const __grid_constant__ Args a) {
  using C = Cfg<BITS>;
  constexpr int kSW = 16;                    // softmax warps
  constexpr uint32_t kRowThreads = 256;      // threads that work on one query tile
  constexpr int kNK = C::kNK, kNV = C::kNV;
  constexpr int kOffV = Map<BITS>::kOffV, kOffTab = Map<BITS>::kOffTab, kOffBar = Map<BITS>::kOffBar, kOffRaw = Map<BITS>::kOffRaw;
  constexpr int kRegProd = regs_producers(ONCE, TAIL), kRegMisc = regs_misc(ONCE, TAIL);
  extern __shared__ uint8_t smem_raw[];
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* sgen = smem_raw + (sbase - smem_u32(smem_raw));
  const uint32_t sQ = sbase + kOffQ, sK = sbase + kOffK, sV = sbase + kOffV, sRaw = sbase + kOffRaw;
  const uint32_t bar0 = sbase + kOffBar;
  // barrier slots (8 bytes each)
  const uint32_t b_kfull = bar0, b_kfree = bar0 + 8 * kNK;
  const uint32_t b_vfull = b_kfree + 8 * kNK, b_vfree = b_vfull + 8 * kNV;
  const uint32_t b_rfull = b_vfree + 8 * kNV, b_rfree = b_rfull + 8 * C::kNR;
  const uint32_t b_qfull = b_rfree + 8 * C::kNR;      // [2]
  const uint32_t b_sfull = b_qfull + 16, b_sfree = b_sfull + 16;
  // [2 tiles][2], even and odd steps: P V~ done, P written.  A parity wait is only sound while the
  // waiter is at most one completion away from the barrier; and the warps of a tile may be almost a
  // step apart (the next scores are there early), so arrivals of a step and of the next one need
  // barriers of their own.
  const uint32_t b_pvdone = b_sfree + 16, b_pfull = b_pvdone + 32;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(sgen + kOffBar + kBarBytes - 16);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sgen + kOffBar + kBarBytes - 12);
  const WaitCtx wc{sbase + kOffBar + kBarBytes - 12};
  const uint32_t s_progress = sbase + kOffBar + kBarBytes - 8;      // tiles that the producers have begun

  const int tid = threadIdx.x;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);     // (known to be the same in all lanes)
  constexpr bool kBf16 = (BITS == 16);

  if (tid == 0) {
    *abort_flag = 0;           // (the status words are older launches' too: they say nothing about this one)
    st_shared_u32(s_progress, 0u);
    for (int i = 0; i < kNK; ++i) { mbar_init(b_kfull + 8 * i, BITS == 16 ? 1 : 128); mbar_init(b_kfree + 8 * i, 2); }
    for (int i = 0; i < kNV; ++i) { mbar_init(b_vfull + 8 * i, BITS == 16 ? 1 : 128); mbar_init(b_vfree + 8 * i, 2); }
    for (int i = 0; i < C::kNR; ++i) { mbar_init(b_rfull + 8 * i, 1); mbar_init(b_rfree + 8 * i, 128); }
    for (int t = 0; t < 2; ++t) {
      mbar_init(b_qfull + 8 * t, kRowThreads); mbar_init(b_sfull + 8 * t, 1);
      mbar_init(b_sfree + 8 * t, kRowThreads);
      mbar_init(b_pvdone + 16 * t, 1); mbar_init(b_pvdone + 16 * t + 8, 1);
      mbar_init(b_pfull + 16 * t, kRowThreads); mbar_init(b_pfull + 16 * t + 8, kRowThreads);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kSW + 5) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32((const void*)tmem_slot)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_dependency_wait();        // the cache and the queries (all of the above ran beside the kernel before)
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  {
    // Registers move from the warps that need few to the softmax warps, whose threads keep 64 scores
    // in registers.  The pool is what the CTA was launched with (per scheduler 6 warps x 80
    // registers per lane = 480); afterwards 4 x 96 + 48 + 48 (or 56 + 40, 64 + 32 where the producers hold more)
    // of them are in use: all 480.
    if (warp < 16) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
    else if (warp < 20) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegProd));
    else asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegMisc));
  }

  if (warp < 16) {
    // ============== softmax warps, 16 rows of a query tile each ==============
    // Warps w and w + 8 may access the same quarter of the TMEM lanes and take 16 of its 32 rows each, whole rows:
    // a quad of lanes holds 128 scores of a row and of the row 8 further, 32 of each per lane.  The scores are
    // read into registers at once and their columns released, so that the next S = Q K~^T runs while the
    // exponentials are computed.  What a row needs as a whole (its maximum, its sum) goes around the quad by
    // shuffles; no warp waits for another one.
    // (Before, warps w and w + 8 shared 32 rows, 64 columns each, and exchanged maxima through shared memory and
    // a barrier in every step, 360 of its 2900 clk, which also kept the two in step.  Separate, three streams in turn:
    // one layer of 261 tokens at 1024 39.8 -> 38.2 us, of 1374 at 8192, all four calls, 132.2 -> 122.1; 24 layers: chunks of four
    // frames 7024 -> 6381, at 4096 1038 -> 1026, at 16384 3862 -> 3791, with the tail 4206 -> 4142, 16-bit at 32768
    // 8011 -> 7922; keys once 4450 -> 4588 and 8-bit 2035 -> 2059, which storing P 64 columns at a time makes up.)
    const int t = (warp >> 2) & 1;           // query tile of the pair
    const int hf = warp >> 3;                // half of the quarter's rows
    const int lane = tid & 31;
    const int r = (warp & 3) * 32 + 16 * hf + (lane >> 2);        // rows r and r + 8 of the tile
    const bool odd = lane & 1, second = lane & 2;
    const int cq2 = 2 * (lane & 3);          // this thread's columns: cq2 and the next of every 8
    const uint32_t lane_addr = tmem + ((uint32_t)((warp & 3) * 32 + 16 * hf) << 16);
    const uint32_t col_t = lane_addr + kColTile * t;
    const uint32_t colO = lane_addr + kColO + 64 * t;
    const uint32_t sfull = b_sfull + 8 * t, pfull = b_pfull + 16 * t, pvdone = b_pvdone + 16 * t;
    const uint64_t sc2 = pack_f2(a.scale_log2, a.scale_log2);
    uint32_t cnt = 0;                        // steps this tile has been through (barrier phases)
    int seg_idx = 0;
    for (Walk walk(a); walk.next(a); ++seg_idx) {
      const Job& job = a.job[walk.job];
      const int h = walk.h, tile_lo = walk.tile_lo, nt = walk.nt;
      const int qt = 2 * walk.pair + t;
      // steps whose tile has masked columns: the pad slots after the first frame, the end
      const int jj_pad = (job.t_first & 127) ? (job.t_first >> 7) - tile_lo : -1, jj_last = job.n_tiles - 1 - tile_lo;
      if (qt >= job.q_tiles) continue;          // the pair has no second tile
      // ---- Q tile: half a row per thread, bf16 -> operand type, into the swizzled K-major layout ----
      {
        const int rq = (warp & 3) * 32 + lane, row = qt * kQRows + rq;
        uint4 u[4];
        if (row < job.n) {
          const __nv_bfloat16* qp = job.q + (int64_t)h * a.hs + (int64_t)row * a.ts + 32 * hf;
#pragma unroll
          for (int c = 0; c < 4; ++c) u[c] = *reinterpret_cast<const uint4*>(qp + 8 * c);
        } else {
#pragma unroll
          for (int c = 0; c < 4; ++c) u[c] = make_uint4(0, 0, 0, 0);
        }
        bool q_bad = false;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint4 o = u[c];
          if (!kBf16) {
            const uint32_t rr[4] = {u[c].x, u[c].y, u[c].z, u[c].w};
            uint32_t hh[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              hh[i] = pack_h2(__uint_as_float(rr[i] << 16), __uint_as_float(rr[i] & 0xFFFF0000u));
              q_bad |= h2_not_finite(hh[i]);
            }
            o = make_uint4(hh[0], hh[1], hh[2], hh[3]);
          }
          *reinterpret_cast<uint4*>(sgen + kOffQ + t * 16384 + swz_off(rq, 4 * hf + c)) = o;
        }
        if (q_bad) report_range(job.status);
        fence_proxy_async();
        mbar_arrive(b_qfull + 8 * t);
      }
      float m0 = -INFINITY, m1 = -INFINITY;     // reference maxima of the two rows (scaled, log2 units; the same in the quad)
      uint64_t l0 = 0ull, l1 = 0ull;            // partial sums of this thread's columns (packed fp32 pairs)
      for (int jj = 0; jj < nt; ++jj, ++cnt) {
        int lim = 128;           // columns [lim, 128) are masked
        if (jj == jj_pad) lim = job.t_first & 127;
        if (jj == jj_last) lim = min(lim, job.t_phys - (tile_lo + jj) * 128);
        mbar_wait(sfull, cnt & 1, wc);
        __syncwarp();            // the waits may leave the warp diverged; tcgen05.ld/st are warp-collective
        tc_fence_after();
        // ---- the scores into registers; after that their columns may take the next tile's scores ----
        uint32_t sc[64];
        XKV_TMEM_LD_64(col_t + 64 * (cnt & 1), sc, 0);
        XKV_TMEM_LD_64(col_t + 64 * (cnt & 1) + 64, sc, 32);
        tc_wait_ld();
        tc_fence_before();
        mbar_arrive(b_sfree + 8 * t);
        if (lim < 128) {
#pragma unroll
          for (int i = 0; i < 64; ++i)
            if (8 * (i >> 2) + cq2 + (i & 1) >= lim) sc[i] = 0xff800000u;           // -inf: exponential 0
        }
        float mx0 = -INFINITY, mx1 = -INFINITY, low0 = 0.f, low1 = 0.f;
#pragma unroll
        for (int g = 0; g < 16; ++g) {
          if (kBf16 && g == 8) {         // (16-bit caches: the two halves of the columns apart, see below)
            low0 = mx0; low1 = mx1;
            mx0 = mx1 = -INFINITY;
          }
          mx0 = max3(mx0, __uint_as_float(sc[4 * g]), __uint_as_float(sc[4 * g + 1]));
          mx1 = max3(mx1, __uint_as_float(sc[4 * g + 2]), __uint_as_float(sc[4 * g + 3]));
        }
        float half_max = 0.f;
        if (kBf16) {
          // the quad's four maxima of half a row: row r in lanes 0 (columns below 64) and 1, row r + 8 in lanes 2 and 3
          const float low = fmaxf(odd ? mx0 : low0, __shfl_xor_sync(0xffffffffu, odd ? low0 : mx0, 1));
          const float high = fmaxf(odd ? mx1 : low1, __shfl_xor_sync(0xffffffffu, odd ? low1 : mx1, 1));
          half_max = fmaxf(second ? high : low, __shfl_xor_sync(0xffffffffu, second ? low : high, 2));
          mx0 = fmaxf(mx0, low0);
          mx1 = fmaxf(mx1, low1);
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
          mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, o));
          mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, o));
        }
        mx0 *= a.scale_log2;
        mx1 *= a.scale_log2;
        // The reference maximum moves only when the row maximum grew by more than 2^kGrow over it;
        // then the sums and (at the end of the step, when the registers are free) the accumulator
        // are rescaled.  Every tile has a column that is not masked, so the maxima are finite.
        float alpha0 = 1.f, alpha1 = 1.f;
        const bool grow = mx0 > m0 + kGrow || mx1 > m1 + kGrow;
        if (grow) {
          if (mx0 > m0 + kGrow) {
            alpha0 = exp2f(m0 - mx0);      // 0 on the first tile (-inf)
            m0 = mx0;
            l0 = mul_f2(l0, pack_f2(alpha0, alpha0));
          }
          if (mx1 > m1 + kGrow) {
            alpha1 = exp2f(m1 - mx1);
            m1 = mx1;
            l1 = mul_f2(l1, pack_f2(alpha1, alpha1));
          }
        }
        const uint64_t nm0 = pack_f2(-m0, -m0), nm1 = pack_f2(-m1, -m1);
        if (kBf16) {
          // A weight rounded to bf16 and the sum that it is divided by: where one key dominates a row its
          // rounding error drops out if the sum holds the rounded weight as well.  The largest weight of
          // every 64 columns is enough (error against float64 at 32760 tokens 2.16e-3 -> 1.90e-3, of which the
          // rounding of the output is 1.66e-3; 24 layers at 32768 7636 -> 7905 us); all rounded weights were no
          // better and cost 6 % of the step, measured before the warps took whole rows.  Which columns go together
          // is part of the result: a thread's own 32 instead saved 0.7 % and moved outputs by 2e-4.
          const float top = fast_exp2(fmaf(half_max, a.scale_log2, second ? -m1 : -m0));
          const float off = __bfloat162float(__float2bfloat16_rn(top)) - top;
          l0 = add_f2(l0, pack_f2(second ? 0.f : off, 0.f));
          l1 = add_f2(l1, pack_f2(second ? off : 0.f, 0.f));
        }
        const uint32_t colP = col_t + 128 * (cnt & 1);       // (over scores of these rows only)
        // Exponentials against the reference; P (16-bit pairs) -> TMEM, 64 columns at a time (32 at a time, three streams
        // in turn: 24 layers at 4096 1019 -> 1075 us, at 16384 3762 -> 3983, keys once 4384 -> 4547, tail 4119 -> 4273,
        // 8-bit 1981 -> 2036).
        auto columns = [&](int g0, uint32_t* pk) {
#pragma unroll
          for (int g = 0; g < 8; ++g) {
            const uint32_t* x = sc + 4 * (g0 + g);
            const uint64_t x0 = fma_f2(pack_f2(__uint_as_float(x[0]), __uint_as_float(x[1])), sc2, nm0);
            const uint64_t x1 = fma_f2(pack_f2(__uint_as_float(x[2]), __uint_as_float(x[3])), sc2, nm1);
            const float e0 = fast_exp2(f2_lo(x0)), e1 = fast_exp2(f2_hi(x0)), e2 = fast_exp2(f2_lo(x1)), e3 = fast_exp2(f2_hi(x1));
            l0 = add_f2(l0, pack_f2(e0, e1));
            l1 = add_f2(l1, pack_f2(e2, e3));
            pk[2 * g] = kBf16 ? pack_bf2(e0, e1) : pack_h2(e0, e1);
            pk[2 * g + 1] = kBf16 ? pack_bf2(e2, e3) : pack_h2(e2, e3);
          }
        };
        {
          uint32_t pk[16];
          columns(0, pk); XKV_TMEM_ST_P32(colP, pk);
          columns(8, pk); XKV_TMEM_ST_P32(colP + 32, pk);
        }
        if (jj > 0 && __any_sync(0xffffffffu, grow)) {
          // the accumulator is quiescent once the previous step's PV has completed
          mbar_wait(pvdone + 8 * ((cnt - 1) & 1), ((cnt - 1) >> 1) & 1, wc);
          __syncwarp();
          tc_fence_after();
          rescale_rows(colO, alpha0, alpha1);
        }
        tc_wait_st();
        tc_fence_before();
        mbar_arrive(pfull + 8 * (cnt & 1));
      }
      // ---- epilogue of the segment ----
      mbar_wait(pvdone + 8 * ((cnt - 1) & 1), ((cnt - 1) >> 1) & 1, wc);    // the last PV (they complete in order)
      __syncwarp();
      tc_fence_after();
      float s0 = f2_lo(l0) + f2_hi(l0), s1 = f2_lo(l1) + f2_hi(l1);
#pragma unroll
      for (int o = 1; o < 4; o <<= 1) {
        s0 += __shfl_xor_sync(0xffffffffu, s0, o);
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      }
      const bool whole = (tile_lo == 0 && nt == job.n_tiles);
      uint32_t ro[32];
      XKV_TMEM_LD_64(colO, ro, 0);
      tc_wait_ld();
      if (whole) {
        const float inv0 = 1.f / s0, inv1 = 1.f / s1;
        const int row = qt * kQRows + r;
        __nv_bfloat16* op = job.out + (int64_t)h * a.hs + (int64_t)row * a.ts + cq2;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          if (row < job.n)
            *reinterpret_cast<uint32_t*>(op + 8 * g) = pack_bf2(__uint_as_float(ro[4 * g]) * inv0, __uint_as_float(ro[4 * g + 1]) * inv0);
          if (row + 8 < job.n)
            *reinterpret_cast<uint32_t*>(op + 8 * a.ts + 8 * g) = pack_bf2(__uint_as_float(ro[4 * g + 2]) * inv1, __uint_as_float(ro[4 * g + 3]) * inv1);
        }
      } else {
        const size_t slot = (size_t)2 * blockIdx.x + (seg_idx == 0 ? 0 : 1);
        const size_t prow = (slot * 2 + t) * 128 + r;
        float* dst = a.part_o + prow * 64 + cq2;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          *reinterpret_cast<float2*>(dst + 8 * g) = make_float2(__uint_as_float(ro[4 * g]), __uint_as_float(ro[4 * g + 1]));
          *reinterpret_cast<float2*>(dst + 512 + 8 * g) = make_float2(__uint_as_float(ro[4 * g + 2]), __uint_as_float(ro[4 * g + 3]));
        }
        if ((lane & 3) == 0) { a.part_ml[prow] = make_float2(m0, s0); a.part_ml[prow + 8] = make_float2(m1, s1); }
      }
      tc_fence_before();
    }
  } else if (warp < kSW + 4) {
    // =========================== operand producers ===========================
    const int t = tid - 32 * kSW;
    const int w = t & 7;          // 16-byte chunk = 8 channels
    const int kb = t >> 3;        // keys kb + 16 i
    const uint32_t row_off = (uint32_t)((kb >> 3) * 1024 + (kb & 7) * 128 + ((w ^ (kb & 7)) << 4));
    uint32_t g = 0;               // steps so far (ring positions)
    for (Walk walk(a); BITS != 16 && walk.next(a);) {
      const Job& job = a.job[walk.job];
      const int tile_lo = walk.tile_lo, nt = walk.nt;
      const int h = walk.h;
      for (int jj = 0; jj < nt; ++jj, ++g) {
        // keys of this tile that belong to the unquantised newest frame (none without a tail)
        const int slot0 = (tile_lo + jj) * 128 + kb;              // this thread's keys: slot0 + 16 i
        const bool tail_tile = TAIL && BITS == 4 && (tile_lo + jj) * 128 + 127 >= job.tail_lo;
        const int64_t tail_off = (int64_t)h * a.hs + 8 * w;
        const uint32_t rs = g % C::kNR, ru = g / C::kNR;
        const uint32_t kbuf = g % kNK, ku = g / kNK;
        const uint32_t vbuf = g % kNV, vu = g / kNV;
        const uint8_t* raw = sgen + kOffRaw + rs * C::kRawStage;
        if (ONCE && t == 0) st_shared_u32(s_progress, g + 1);
        mbar_wait<kSlack>(b_rfull + 8 * rs, ru & 1, wc);
        if (TAIL && BITS == 4 && (tile_lo + jj) * 128 >= job.tail_lo && (tile_lo + jj) * 128 + 127 < job.t_phys) {
          // ---- a tile that lies in the unquantised frame as a whole: K~ and V~ are the caller's
          // bf16 rows converted to fp16, the packed codes of the stage are not looked at ----
          // (The parameter tables take turns by step.  A table is filled again once all producers have
          // passed the step between, which must therefore make them meet although it fills no table.)
          producer_sync();
          bool bad = false;
#pragma unroll
          for (int kv = 0; kv < 2; ++kv) {
            const __nv_bfloat16* src = (kv ? job.v_tail : job.k_tail) + tail_off + (int64_t)(slot0 - job.tail_lo) * a.ts;
            uint4 u[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) u[i] = *reinterpret_cast<const uint4*>(src + (int64_t)(16 * i) * a.ts);
            if (kv == 0) mbar_wait<kSlack>(b_kfree + 8 * kbuf, (ku & 1) ^ 1, wc);
            else mbar_wait<kSlack>(b_vfree + 8 * vbuf, (vu & 1) ^ 1, wc);
            uint8_t* dst = sgen + (kv ? kOffV + vbuf * 16384 : kOffK + kbuf * 16384) + row_off;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const uint4 hv = bf16x8_to_h8(u[i]);
              bad |= h2_not_finite(hv.x) || h2_not_finite(hv.y) || h2_not_finite(hv.z) || h2_not_finite(hv.w);
              *reinterpret_cast<uint4*>(dst + i * 2048) = hv;
            }
            fence_proxy_async();
            mbar_arrive(kv ? b_vfull + 8 * vbuf : b_kfull + 8 * kbuf);
          }
          if (bad) report_range(job.status);
          mbar_arrive(b_rfree + 8 * rs);
          continue;
        }
        if (BITS == 4) {
          // ---- fp16 parameter tables of this tile (one (group, channel) and one key per thread) ----
          uint8_t* tab = sgen + kOffTab + (g & 1) * kTabBytes;
          {
            bool k_bad = false;
            if (!ONCE) {
              const float2 kp = *reinterpret_cast<const float2*>(raw + C::kRawK + C::kRawV + 8 * t);  // (group t>>6, channel t&63)
              float zl, zh, kc;
              dequant_consts(kp.x, kp.y, zl, zh, kc);
              __half* ks = reinterpret_cast<__half*>(tab);              // [2][64] scales, [2][64] offsets, [2][64] constants
              ks[t] = __float2half_rn(kp.x);
              ks[128 + t] = __float2half_rn((((t & 7) >> 1) & 1) ? zh : zl);
              ks[256 + t] = __float2half_rn(kc);
              k_bad = beyond_fp16(fabsf(kp.x) * (fabsf(kp.y) + 15.f));
            }
            const float2 vp = *reinterpret_cast<const float2*>(raw + C::kRawK + C::kRawV + C::kRawKP + 8 * t);   // key t
            float vl, vh, vc;
            dequant_consts(vp.x, vp.y, vl, vh, vc);
            *reinterpret_cast<uint4*>(tab + 768 + 16 * t) =
                make_uint4(pack_h2(vp.x, vp.x), pack_h2(vl, vl), pack_h2(vh, vh), pack_h2(vc, vc));
            // largest magnitude a code of this group / token can dequantise to
            if (k_bad || beyond_fp16(fabsf(vp.x) * (fabsf(vp.y) + 15.f))) report_range(job.status);
          }
          producer_sync();
          // ---- keys ----
          uint32_t wd[8];
          if (ONCE) {
            once_keys<uint32_t>(raw, raw + C::kRawK + C::kRawV, sgen + kOffK + kbuf * 16384, job.ktab16, job.n_heads, h, t,
                                b_kfree + 8 * kbuf, (ku & 1) ^ 1, wc);
          } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) wd[i] = *reinterpret_cast<const uint32_t*>(raw + (kb + 16 * i) * 32 + 4 * w);
            mbar_wait<kSlack>(b_kfree + 8 * kbuf, (ku & 1) ^ 1, wc);
#pragma unroll
            for (int grp = 0; grp < 2; ++grp) {
              const uint4 sv = *reinterpret_cast<const uint4*>(tab + grp * 128 + 16 * w);
              const uint4 zv = *reinterpret_cast<const uint4*>(tab + 256 + grp * 128 + 16 * w);
              const uint4 cv = *reinterpret_cast<const uint4*>(tab + 512 + grp * 128 + 16 * w);
              const uint32_t s2[4] = {sv.x, sv.y, sv.z, sv.w}, zo[4] = {zv.x, zv.y, zv.z, zv.w};
              const uint32_t c2[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const uint4 o = dequant_word_h(wd[4 * grp + i], s2, zo, c2);
                *reinterpret_cast<uint4*>(sgen + kOffK + kbuf * 16384 + row_off + (4 * grp + i) * 2048) = o;
              }
            }
          }
          if (TAIL && tail_tile)
            tail_rows_over<ONCE ? 1 : 16>(sgen + kOffK + kbuf * 16384, job.k_tail + tail_off, a.ts, slot0 - kb, ONCE ? (t >> 3) * 8 : kb, w, job.tail_lo,
                                          job.t_phys, job.status);
          fence_proxy_async();
          mbar_arrive(b_kfull + 8 * kbuf);
          // ---- values ----
#pragma unroll
          for (int i = 0; i < 8; ++i) wd[i] = *reinterpret_cast<const uint32_t*>(raw + C::kRawK + (kb + 16 * i) * 32 + 4 * w);
          mbar_wait<kSlack>(b_vfree + 8 * vbuf, (vu & 1) ^ 1, wc);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint4 pv = *reinterpret_cast<const uint4*>(tab + 768 + 16 * (kb + 16 * i));
            const uint32_t s2[4] = {pv.x, pv.x, pv.x, pv.x}, zo[4] = {pv.y, pv.z, pv.y, pv.z};
            const uint32_t c2[4] = {pv.w, pv.w, pv.w, pv.w};
            const uint4 o = dequant_word_h(wd[i], s2, zo, c2);
            *reinterpret_cast<uint4*>(sgen + kOffV + vbuf * 16384 + row_off + i * 2048) = o;
          }
          if (TAIL && tail_tile)
            tail_rows_over<16>(sgen + kOffV + vbuf * 16384, job.v_tail + tail_off, a.ts, slot0 - kb, kb, w, job.tail_lo, job.t_phys, job.status);
          fence_proxy_async();
          mbar_arrive(b_vfull + 8 * vbuf);
          // The raw stage is released only here, after the words read from it have been used and
          // the fence above: released right after the loads, the refill of the stage was observed
          // to reach some of those loads when the wait in between was long.
          mbar_arrive(b_rfree + 8 * rs);
        } else if (BITS == 8) {
          // ---- 8-bit codes (keys quantised once): the same steps with rows of 64 bytes ----
          uint8_t* tab = sgen + kOffTab + (g & 1) * kTabBytes;
          {
            const float2 vp = *reinterpret_cast<const float2*>(raw + C::kRawK + C::kRawV + C::kRawKP + 8 * t);   // key t
            float vl, vh, vc;
            dequant_consts(vp.x, vp.y, vl, vh, vc);
            *reinterpret_cast<uint4*>(tab + 768 + 16 * t) = make_uint4(pack_h2(vp.x, vp.x), pack_h2(vl, vl), 0u, pack_h2(vc, vc));
            if (beyond_fp16(fabsf(vp.x) * (fabsf(vp.y) + 255.f))) report_range(job.status);
          }
          producer_sync();
          uint2 wd8[8];
          once_keys<uint2>(raw, raw + C::kRawK + C::kRawV, sgen + kOffK + kbuf * 16384, job.ktab16, job.n_heads, h, t,
                           b_kfree + 8 * kbuf, (ku & 1) ^ 1, wc);
          fence_proxy_async();
          mbar_arrive(b_kfull + 8 * kbuf);
#pragma unroll
          for (int i = 0; i < 8; ++i) wd8[i] = *reinterpret_cast<const uint2*>(raw + C::kRawK + (kb + 16 * i) * 64 + 8 * w);
          mbar_wait<kSlack>(b_vfree + 8 * vbuf, (vu & 1) ^ 1, wc);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint4 pv = *reinterpret_cast<const uint4*>(tab + 768 + 16 * (kb + 16 * i));
            const uint32_t s2[4] = {pv.x, pv.x, pv.x, pv.x}, zo[4] = {pv.y, pv.y, pv.y, pv.y};
            const uint32_t c2[4] = {pv.w, pv.w, pv.w, pv.w};
            const uint4 o = dequant_word_h(wd8[i], s2, zo, c2);
            *reinterpret_cast<uint4*>(sgen + kOffV + vbuf * 16384 + row_off + i * 2048) = o;
          }
          fence_proxy_async();
          mbar_arrive(b_vfull + 8 * vbuf);
          mbar_arrive(b_rfree + 8 * rs);
        }
      }
    }
  } else if (warp == kSW + 4 || warp == kSW + 6) {
    // =========================== MMA issuers ==================================
    // One converged warp per query tile; an elected lane issues.  Step j: S = Q K~_j^T as soon as
    // the softmax warps hold the scores of step j - 1 in registers, then O += P V~_(j-1) as soon as
    // P is there: the scores are a whole step ahead of the softmax.  Both warps release the K~/V~
    // stages (two arrivals each), also for an item that has no second tile.
    const uint32_t t = (warp == kSW + 4) ? 0u : 1u;
    const uint32_t idesc_qk = make_idesc(128, kBf16, false);
    const uint32_t idesc_pv = make_idesc(64, kBf16, true);
    const uint64_t dq = make_desc(sQ + t * 16384), dk0 = make_desc(sK), dv0 = make_desc(sV);
    const uint32_t d_tile = tmem + kColTile * t, d_o = tmem + kColO + 64 * t;
    uint32_t kb = 0, kph = 0, vb = 0, vph = 0;      // ring positions and their parities
    uint32_t cs = 0, cq = 0;                        // scores and query tiles so far
    for (Walk walk(a); walk.next(a);) {
      const int nt = walk.nt;
      const bool active = 2 * walk.pair + (int)t < a.job[walk.job].q_tiles;
#pragma unroll 1
      for (int jj = 0; jj <= nt; ++jj) {
        if (jj < nt) {
          mbar_wait(b_kfull + 8 * kb, kph, wc);
          if (active) {
            // The scores of the step before are in registers, P of the one before that is consumed.  At
            // the start of a segment Q is written after the epilogue of the segment before, so
            // everything earlier has completed.  (Asking for an older phase would be wrong there: its
            // parity comes round again.)
            if (jj == 0) mbar_wait(b_qfull + 8 * t, cq & 1, wc); else mbar_wait(b_sfree + 8 * t, (cs - 1) & 1, wc);
            if (jj > 1) mbar_wait(b_pvdone + 16 * t + 8 * (cs & 1), ((cs >> 1) - 1) & 1, wc);
          }
          __syncwarp();
          tc_fence_after();
          if (elect_one()) {
            if (active) {
              const uint64_t dk = dk0 + (uint64_t)(kb * (16384 >> 4));
              const uint32_t d_s = d_tile + 64 * (cs & 1);
#pragma unroll
              for (int ks = 0; ks < 4; ++ks)   // 16 channels per step: 32 B inside the swizzle span
                mma_ss(d_s, dq + (uint64_t)(ks * 2), dk + (uint64_t)(ks * 2), idesc_qk, ks > 0 ? 1u : 0u);
              tc_commit(b_sfull + 8 * t);
            }
            tc_commit(b_kfree + 8 * kb);
          }
          __syncwarp();
          if (active) ++cs;
          if (++kb == (uint32_t)kNK) { kb = 0; kph ^= 1; }
        }
        if (jj > 0) {
          const uint32_t c = cs - ((jj < nt) ? 2u : 1u);       // the step whose P V~ this is
          mbar_wait(b_vfull + 8 * vb, vph, wc);
          if (active) mbar_wait(b_pfull + 16 * t + 8 * (c & 1), (c >> 1) & 1, wc);
          __syncwarp();
          tc_fence_after();
          if (elect_one()) {
            if (active) {
              const uint64_t dv = dv0 + (uint64_t)(vb * (16384 >> 4));
              const uint32_t d_p = d_tile + 128 * (c & 1);
#pragma unroll
              for (int ks = 0; ks < 8; ++ks)   // 16 keys per step: 2 swizzle atoms = 2048 B of V~, 8 columns of P
                mma_ts(d_o, d_p + 8 * ks, dv + (uint64_t)((ks * 2048) >> 4), idesc_pv, (jj > 1 || ks > 0) ? 1u : 0u);
              tc_commit(b_pvdone + 16 * t + 8 * (c & 1));
            }
            tc_commit(b_vfree + 8 * vb);
          }
          __syncwarp();
          if (++vb == (uint32_t)kNV) { vb = 0; vph ^= 1; }
        }
      }
      if (active) ++cq;
    }
    tc_fence_before();
  } else if (ONCE && warp == kSW + 7) {
    // =========================== constants, ahead of the producers =============
    // The constants of a tile's key groups lie anywhere in a table of hundreds of megabytes a layer: a
    // look-up can miss the L2 and the TLB, and the producers' look-ups depend on one another.  This
    // warp asks for the lines a few tiles before the producers need them.  (24 layers at 16384, three
    // streams taking turns: 5290 us a frame without it, 4440 with; 8-bit at 8192 2440 and 1970.  One
    // stream alone, whose constants the L2 holds better: 3920 and 3790, 1590 and 1550.)
    const int lane = tid & 31;
    uint32_t g = 0;
    for (Walk walk(a); walk.next(a);) {
      const Job& job = a.job[walk.job];
      for (int jj = 0; jj < walk.nt; ++jj, ++g) {
        for (int it = 0; it < (1 << 16); ++it) {           // (only a pace: nothing depends on it)
          if (g < ld_shared_u32(s_progress) + kAhead || ld_shared_u32(wc.abort_flag)) break;
          __nanosleep(500);
        }
        const int4 sl = *(reinterpret_cast<const int4*>(job.kslot + (size_t)(walk.tile_lo + jj) * 128) + lane);
        int before = __shfl_up_sync(0xffffffffu, sl.w, 1);
        if (lane == 0) before = -1;
        auto ask = [&](int slot, int prev) {
          if (slot == prev) return;
          const uint8_t* e = reinterpret_cast<const uint8_t*>(job.ktab16 + ((size_t)slot * job.n_heads + walk.h) * 96);
#pragma unroll
          for (int i = 0; i < 4; ++i) asm volatile("prefetch.global.L2 [%0];" ::"l"(e + min(128 * i, 383)));
        };
        ask(sl.x, before); ask(sl.y, sl.x); ask(sl.z, sl.y); ask(sl.w, sl.z);
        __syncwarp();
      }
    }
  } else if (tid == 32 * (kSW + 5)) {
    // =========================== TMA loader ===================================
    uint32_t g = 0;
    for (Walk walk(a); walk.next(a);) {
      const Job& job = a.job[walk.job];
      const int tile_lo = walk.tile_lo, nt = walk.nt;
      const int h = walk.h;
      const size_t head_slot = (size_t)h * job.cap;
      for (int jj = 0; jj < nt; ++jj, ++g) {
        const int tile = tile_lo + jj;
        const size_t slot0 = head_slot + (size_t)tile * 128;
        if (BITS == 16) {
          const uint32_t ks = g % kNK, vs = g % kNV;
          mbar_wait<kSlack>(b_kfree + 8 * ks, ((g / kNK) & 1) ^ 1, wc);
          mbar_expect_tx(b_kfull + 8 * ks, C::kRawK);
          tma_load_1d(sK + ks * 16384, job.k + slot0 * 128, C::kRawK, b_kfull + 8 * ks);
          mbar_wait<kSlack>(b_vfree + 8 * vs, ((g / kNV) & 1) ^ 1, wc);
          mbar_expect_tx(b_vfull + 8 * vs, C::kRawV);
          tma_load_1d(sV + vs * 16384, job.v + slot0 * 128, C::kRawV, b_vfull + 8 * vs);
          continue;
        }
        const uint32_t rs = g % C::kNR, ru = g / C::kNR;
        mbar_wait<kSlack>(b_rfree + 8 * rs, (ru & 1) ^ 1, wc);
        const uint32_t dst = sRaw + rs * C::kRawStage, bar = b_rfull + 8 * rs;
        const uint32_t kp_bytes = ONCE ? 512u : (uint32_t)C::kRawKP;    // 128 group references instead of 2 x 64 parameters
        mbar_expect_tx(bar, C::kRawStage - C::kRawKP + kp_bytes);
        if (BITS == 4) {
          tma_load_1d(dst, job.k + slot0 * 32, C::kRawK, bar);
          tma_load_1d(dst + C::kRawK, job.v + slot0 * 32, C::kRawV, bar);
          if (ONCE) tma_load_1d(dst + C::kRawK + C::kRawV, job.kslot + (size_t)tile * 128, kp_bytes, bar);
          else tma_load_1d(dst + C::kRawK + C::kRawV, job.kpar + ((size_t)h * (job.cap >> 6) + 2 * tile) * 64, C::kRawKP, bar);
          tma_load_1d(dst + C::kRawK + C::kRawV + C::kRawKP, job.vpar + slot0, C::kRawVP, bar);
        } else if (BITS == 8) {
          tma_load_1d(dst, job.k + slot0 * 64, C::kRawK, bar);
          tma_load_1d(dst + C::kRawK, job.v + slot0 * 64, C::kRawV, bar);
          tma_load_1d(dst + C::kRawK + C::kRawV, job.kslot + (size_t)tile * 128, kp_bytes, bar);
          tma_load_1d(dst + C::kRawK + C::kRawV + C::kRawKP, job.vpar + slot0, C::kRawVP, bar);
        }
      }
    }
    // Drain: every copy this thread started has landed once the last use of each stage completed
    // (bounded, and not cut short by the abort flag, so that nothing is in flight at exit).
    const uint32_t issued = g;
    auto drain = [&](uint32_t full, uint32_t stages) {
      for (uint32_t i = 0; i < stages && i < issued; ++i) {
        const uint32_t gi = issued - 1 - i;
        for (uint32_t it = 0; it < kSpinLimit; ++it)
          if (mbar_try(full + 8 * (gi % stages), (gi / stages) & 1)) break;
      }
    };
    if (BITS == 16) { drain(b_kfull, kNK); drain(b_vfull, kNV); }
    else drain(b_rfull, C::kNR);
  }
  __syncthreads();
  if (tid == 0 && *abort_flag) report_timeout(a);
  if (warp == kSW + 5) {
    __syncwarp();
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

// ---------------------------------------------------------------------------
// Merge of the partial results of the items that were cut between CTAs:
// out = sum_s 2^(m_s - M) O_s / sum_s 2^(m_s - M) l_s.  Eight blocks per cut of the line (the start
// of a piece); the first cut inside an item does the whole item, the others have nothing to do.
// Thread = (row, 8-channel chunk) of a query tile.  Items that one CTA covered alone were
// written by it.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
attn_combine_kernel(const __grid_constant__ Args a) {
  grid_dependency_wait();
  const int cut = (int)(blockIdx.x >> 3) + 1, t = (int)(blockIdx.x >> 2) & 1;
  const int r = (int)(blockIdx.x & 3) * 32 + (int)(threadIdx.x >> 3), ch = (int)(threadIdx.x & 7);
  const uint32_t at = piece_start(a, cut), before = piece_start(a, cut - 1);
  int jn = 0;
  while (at >= a.job[jn].step_hi) ++jn;
  const Job& job = a.job[jn];
  const uint32_t tiles = (uint32_t)job.n_tiles, pairs = (uint32_t)job.n_pairs;
  const uint32_t item = (at - job.step_lo) / tiles;
  const uint32_t lo = job.step_lo + item * tiles, hi = lo + tiles;
  if (at == lo || before > lo) return;           // between two items; not the item's first cut
  const int h = (int)(item / pairs), pair = (int)(item % pairs);
  const int qt = 2 * pair + t;
  const int row = qt * 128 + r;
  if (qt >= job.q_tiles || row >= job.n) return;
  const int b_first = cut - 1;
  // the piece before the cut holds the item in its second slot if it began with another item
  const bool first_is_second_slot = before < lo;
  // The partials are fetched four at a time, all loads before the first use (an item is cut into
  // two or three pieces unless the cache is very long); the running maximum and the weights are
  // those of the online softmax, in the fixed order of the pieces.
  float m = -INFINITY, l = 0.f;
  float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  for (int b0 = b_first; b0 < a.grid && (b0 == b_first || piece_start(a, b0) < hi); b0 += 4) {
    float2 ml[4];
    float4 x[4], y[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int b = b0 + j;
      ml[j] = make_float2(-INFINITY, 0.f);
      x[j] = y[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (b < a.grid && (b == b_first || piece_start(a, b) < hi)) {
        const size_t slot = (size_t)2 * b + ((b == b_first && first_is_second_slot) ? 1 : 0);
        const size_t prow = (slot * 2 + t) * 128 + r;
        ml[j] = a.part_ml[prow];
        const float4* po = reinterpret_cast<const float4*>(a.part_o + prow * 64 + 8 * ch);
        x[j] = po[0];
        y[j] = po[1];
      }
    }
    const float mc = fmaxf(fmaxf(m, fmaxf(ml[0].x, ml[1].x)), fmaxf(ml[2].x, ml[3].x));
    const float sc = exp2f(m - mc);                // 0 for the first group (m = -inf)
    m = mc;
    l *= sc;
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] *= sc;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float wgt = exp2f(ml[j].x - m);        // 0 for an absent piece
      l += wgt * ml[j].y;
      acc[0] += wgt * x[j].x; acc[1] += wgt * x[j].y; acc[2] += wgt * x[j].z; acc[3] += wgt * x[j].w;
      acc[4] += wgt * y[j].x; acc[5] += wgt * y[j].y; acc[6] += wgt * y[j].z; acc[7] += wgt * y[j].w;
    }
  }
  const float inv = 1.f / l;
  uint32_t o[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) o[i] = pack_bf2(acc[2 * i] * inv, acc[2 * i + 1] * inv);
  *reinterpret_cast<uint4*>(job.out + (int64_t)h * a.hs + (int64_t)row * a.ts + 8 * ch) = make_uint4(o[0], o[1], o[2], o[3]);
}

size_t attn_tc_scratch_bytes(const xkv_params*) { return (size_t)2 * kMaxGrid * kSlotBytes + 512; }

// Per device, on first use with that device current: the SM count, and the opt-in to more than
// 48 KB of dynamic shared memory for the attention kernels (a per-device function attribute).
static std::mutex g_setup_mutex;
static int g_sm_count[kMaxDevices] = {0};       // 0: not set up yet

// The kernel moves registers between its warps with setmaxnreg; the pool they move in is what the CTA
// was launched with.  If a compiler ever gave the kernel fewer registers at launch than the
// reallocation needs, setmaxnreg.inc would wait for ever: refuse to run instead.
template <int BITS, bool TAIL, bool ONCE>
static cudaError_t prepare_kernel() {
  const auto kernel = attn_tc_kernel<BITS, TAIL, ONCE>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes<BITS>());
  if (e != cudaSuccess) return e;
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess) return e;
  const int warps_per_scheduler = kThreads / 32 / 4;
  return (fa.numRegs * warps_per_scheduler >= 4 * kRegsSoftmax + regs_producers(ONCE, TAIL) + regs_misc(ONCE, TAIL))
             ? cudaSuccess : cudaErrorLaunchOutOfResources;
}

static cudaError_t attn_device_setup(int* sm_count) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (g_sm_count[dev] == 0) {
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    e = prepare_kernel<4, false, false>();
    if (e == cudaSuccess) e = prepare_kernel<4, true, false>();
    if (e == cudaSuccess) e = prepare_kernel<4, false, true>();
    if (e == cudaSuccess) e = prepare_kernel<4, true, true>();
    if (e == cudaSuccess) e = prepare_kernel<8, false, true>();
    if (e == cudaSuccess) e = prepare_kernel<16, false, false>();
    if (e != cudaSuccess) return e;
    g_sm_count[dev] = sms;
  }
  *sm_count = g_sm_count[dev];
  return cudaSuccess;
}

static void fill_job(Job* j, const AttnCall& call) {
  const xkv_cache* c = call.cache;
  const BufSet& b = c->buf[c->cur];
  j->q = reinterpret_cast<const __nv_bfloat16*>(call.q);
  j->out = reinterpret_cast<__nv_bfloat16*>(call.out);
  j->k = b.k; j->kpar = b.kpar; j->v = b.v; j->vpar = b.vpar;
  j->kslot = b.kslot; j->ktab16 = c->ktab16;
  j->status = c->status;
  j->n = call.n; j->cap = c->cap; j->n_heads = c->p.n_heads;
  j->t_first = c->T_first;
  j->t_phys = c->rest_base + (c->T - c->T_first);
  if (c->T == c->T_first) j->t_phys = c->T_first;         // only the first frame: no pad tile beyond it
  if (call.prefix > 0 && call.prefix < c->T) {
    // a prefix of the cache in logical order: inside the first frame it ends the first segment,
    // after it the rest segment
    if (call.prefix <= c->T_first) { j->t_first = call.prefix; j->t_phys = call.prefix; }
    else j->t_phys = c->rest_base + (call.prefix - c->T_first);
  }
  j->k_tail = j->v_tail = nullptr;
  j->tail_lo = j->t_phys;
  if (call.k_tail && c->p.kv_bits == 4) {      // a 16-bit cache holds the frame exactly as it arrived
    j->k_tail = reinterpret_cast<const __nv_bfloat16*>(call.k_tail);
    j->v_tail = reinterpret_cast<const __nv_bfloat16*>(call.v_tail);
    j->tail_lo = j->t_phys - call.n;           // the newest frame holds the last n slots
  }
  j->n_tiles = (j->t_phys + 127) / 128;
  j->q_tiles = (call.n + kQRows - 1) / kQRows;
  j->n_pairs = (j->q_tiles + 1) / 2;
}

// One launch (and its merge) for the jobs in `a`, which are those caches'.  `part` holds the partial slots: accumulators float
// [slots][2][128][64], then (max, sum) float2 [slots][2][128], slots = part_bytes / kSlotBytes.  The
// grid is the SM count, capped by the slots available (two per CTA) and by the number of steps.
static cudaError_t launch_jobs(xkv_cache* const* caches, int n_caches, Args& a, uint32_t total, bool tail, float* part,
                               size_t part_bytes, int sm_count, cudaStream_t st) {
  const xkv_cache* c = caches[0];
  const size_t slots = part_bytes / kSlotBytes;
  long long grid = sm_count;
  if (grid > (long long)(slots / 2)) grid = (long long)(slots / 2);
  if (c->attn_max_blocks > 0 && grid > c->attn_max_blocks) grid = c->attn_max_blocks;
  if (grid > (long long)total) grid = total;
  if (grid < 1) return cudaErrorMemoryAllocation;
  a.grid = (int)grid;
  a.piece = total / (uint32_t)grid;
  a.longer = total % (uint32_t)grid;
  a.part_o = part;
  a.part_ml = reinterpret_cast<float2*>(part + slots * kSlotFloats);
  {
    LaunchScope ls(caches, n_caches, XKV_PROF_ATTN, st);
    const bool once = c->p.key_mode == XKV_KEYS_ONCE;
    const void* fn;
    int smem = smem_bytes<4>();
    if (c->p.kv_bits == 16) { fn = (const void*)attn_tc_kernel<16>; smem = smem_bytes<16>(); }
    else if (c->p.kv_bits == 8) { fn = (const void*)attn_tc_kernel<8, false, true>; smem = smem_bytes<8>(); }
    else if (tail && once) fn = (const void*)attn_tc_kernel<4, true, true>;
    else if (tail) fn = (const void*)attn_tc_kernel<4, true>;
    else if (once) fn = (const void*)attn_tc_kernel<4, false, true>;
    else fn = (const void*)attn_tc_kernel<4>;
    void* params[1] = {(void*)&a};
    const cudaError_t e = launch_overlapped(fn, dim3((unsigned)grid), dim3(kThreads), params, (size_t)smem, st);
    if (e != cudaSuccess) return e;
  }
  if (grid > 1) {
    LaunchScope ls(caches, n_caches, XKV_PROF_COMBINE, st);
    void* params[1] = {(void*)&a};
    const cudaError_t e = launch_overlapped((const void*)attn_combine_kernel, dim3((unsigned)(grid - 1) * 8), dim3(256), params, 0, st);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

static cudaError_t launch_attn_tc_on(const AttnCall* calls, int count, int64_t ts, int64_t hs, float scale, float* part,
                                     size_t part_bytes, cudaStream_t st) {
  int sm_count = 0;
  {
    const cudaError_t e = attn_device_setup(&sm_count);
    if (e != cudaSuccess) return e;
  }
  xkv_cache* lead = calls[0].cache;
  const bool tail = calls[0].k_tail && lead->p.kv_bits == 4;
  if (calls[0].k_tail && lead->p.kv_bits == 8) return cudaErrorNotSupported;      // (the unquantised tail is built for 4-bit caches)
  Args a;
  a.ts = ts; a.hs = hs;
  a.scale_log2 = scale * 1.4426950408889634f;
  for (int i = 0; i < count;) {
    a.n_jobs = 0;
    uint32_t total = 0;
    xkv_cache* caches[kMaxJobs];
    int n_caches = 0;
    for (; i < count && a.n_jobs < kMaxJobs; ++i) {
      Job* j = &a.job[a.n_jobs];
      fill_job(j, calls[i]);
      const uint64_t steps = (uint64_t)j->n_heads * j->n_pairs * j->n_tiles;
      if (total + steps >= (1ull << 32)) {
        if (a.n_jobs > 0) break;
        return cudaErrorNotSupported;          // (no workspace of that size fits a GPU)
      }
      j->step_lo = total;
      total += (uint32_t)steps;
      j->step_hi = total;
      a.n_jobs++;
      // (the frames of a chunk are jobs of one cache)
      if (n_caches == 0 || caches[n_caches - 1] != calls[i].cache) caches[n_caches++] = calls[i].cache;
    }
    const cudaError_t e = launch_jobs(caches, n_caches, a, total, tail, part, part_bytes, sm_count, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_attn_tc(const AttnCall* calls, int count, int64_t ts, int64_t hs, float scale, cudaStream_t st) {
  return launch_attn_tc_on(calls, count, ts, hs, scale, calls[0].cache->attn_part, calls[0].cache->attn_part_bytes, st);
}

// ---------------------------------------------------------------------------
// attn_packed_causal_static: the same attention with its partial slots in a
// fixed array that is part of the loaded library image instead of the caller's
// workspace.  See xkv.h for who needs this and for the rules of use.
// ---------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_static_partials[XKV_STATIC_SCRATCH_BYTES];

// In host code `g_static_partials` only names the symbol; the device address has to be asked
// for, once per device, while that device is current.
static std::mutex g_static_mutex;
static void* g_static_addr[kMaxDevices] = {nullptr};

cudaError_t launch_attn_tc_static(const AttnCall& call, int64_t ts, int64_t hs, float scale, cudaStream_t st) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  void* addr = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_addr[dev]) {
      void* p = nullptr;
      e = cudaGetSymbolAddress((void**)&p, g_static_partials);
      if (e != cudaSuccess) return e;
      g_static_addr[dev] = p;
    }
    addr = g_static_addr[dev];
  }
  return launch_attn_tc_on(&call, 1, ts, hs, scale, reinterpret_cast<float*>(addr), (size_t)XKV_STATIC_SCRATCH_BYTES, st);
}

// ---------------------------------------------------------------------------
// Test hook: the bounded wait of the attention kernel on a barrier that nothing completes.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(32) timeout_probe_kernel(const __grid_constant__ Args a) {
  __shared__ __align__(8) unsigned long long bar;
  __shared__ volatile int abort_flag;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    mbar_init(smem_u32(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const WaitCtx wc{smem_u32((const void*)&abort_flag)};
  if (threadIdx.x == 0) mbar_wait(smem_u32(&bar), 0, wc);     // phase 0 never completes: runs into the limit
  __syncthreads();
  mbar_wait(smem_u32(&bar), 0, wc);                           // the flag is up: every later wait returns at once
  __syncthreads();
  if (threadIdx.x == 0 && abort_flag) report_timeout(a);
}

cudaError_t launch_timeout_probe(xkv_cache* c, cudaStream_t st) {
  Args a;
  a.n_jobs = 1;
  a.piece = 1;                       // one step, all of it this cache's
  a.longer = 0;
  a.job[0].step_lo = 0;
  a.job[0].step_hi = 1;
  a.job[0].status = c->status;
  timeout_probe_kernel<<<1, 32, 0, st>>>(a);
  c->launches++;
  return cudaGetLastError();
}

}  // namespace xkv
