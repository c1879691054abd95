// Cache maintenance: append (+ per-token value quantisation), pooled query,
// importance scores, top-k selection, key regroup / re-quantisation and the
// survivor gather.  All bandwidth- or latency-bound; fp32 arithmetic whose every
// operation and order is fixed, because it decides integers (kept indices, 4-bit
// codes) that must be reproducible bit for bit.
//
// One persistent kernel of up to two thread blocks per SM (fewer where the busiest phase has less work)
// runs the phases that a call needs.  A launch takes one layer or up to 28; every layer has blocks of
// its own, with barriers among them (the launch is cooperative where there is one):
//
//   APPEND  values quantised per token (Eq. 7-9) into their final slot; keys staged
//           (4-bit) or copied (16-bit)                                 [kv_append]
//   POOL    pooled query rows, Eq. 2-3                                 [kv_score_evict]
//   KBAR    head means of the cached keys after the first frame, Eq. 4, when the
//           stored ones are stale
//   ---- barrier ----
//   SCORE   row mean of the pooled query, scores S = w . K-bar (Eq. 5-6), histogram
//           of the top 12 bits of the score keys
//   ---- barrier ----
//   SEL1    every block finds the histogram bin that holds the k-th largest key;
//           keys in higher bins are kept, keys in that bin become candidates
//   ---- barrier ----
//   SEL2    every block finds the k-th largest (key, position) among the candidates
//           (a histogram of their next 8 key bits, then a ranking inside each warp) and
//           writes the kept positions of its own tokens in order
//   ---- barrier ----
//   PACK    16-bit caches and keys quantised once: the survivor gather  [kv_quant_pack]
//
// xkv_stream_step runs all of them in one launch; the per-call entry points launch
// the same kernel with the phases of that call.  The 4-bit kv_quant_pack (key regroup +
// re-quantisation, Eq. 7-9, fused with the survivor gather) is a kernel of its own,
// launched right behind.
#include <stdlib.h>

#include <mutex>

#include "xkv_internal.cuh"

namespace xkv {

namespace {

constexpr int kMT = 512;                 // threads per block
constexpr int kBlocksPerSM = 2;
constexpr uint32_t kBarSpin = 1u << 21;  // polls of a barrier before it gives up (each a sleep and an L2 round trip)

// ---------------------------------------------------------------------------
// Eq. 7-8, fixed-order fp32:  s = (max-min)/(2^b - 1) (1 if the range is 0),
// inv = 1/s, z = rint(-min*inv) + 0, q = clamp(rint(x*inv) + z, 0, 2^b - 1).  qmax = 2^b - 1.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void quant_params(float mn, float mx, float& s, float& inv, float& z, float qmax = 15.f) {
  const float r = __fsub_rn(mx, mn);
  s = (r == 0.f) ? 1.f : __fdiv_rn(r, qmax);
  inv = __fdiv_rn(1.f, s);
  z = __fadd_rn(rintf(__fmul_rn(-mn, inv)), 0.f);
}

__device__ __forceinline__ uint32_t quant_code(float x, float inv, float z, float qmax = 15.f) {
  float q = __fadd_rn(rintf(__fmul_rn(x, inv)), z);
  q = fminf(fmaxf(q, 0.f), qmax);
  return (uint32_t)q;
}

// 8-bit storage: the codes of channels 4i..4i+3 form the word c0 | c2<<8 | c1<<16 | c3<<24, so that
// the mask 0x00FF00FF yields the adjacent channels (0, 1) and, after a shift by 8, (2, 3).
__device__ __forceinline__ uint32_t pack4_bytes(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3) {
  return c0 | (c2 << 8) | (c1 << 16) | (c3 << 24);
}
__device__ __forceinline__ void unpack8_bytes(uint2 w, uint32_t (&c)[8]) {
  c[0] = w.x & 0xFFu; c[2] = (w.x >> 8) & 0xFFu; c[1] = (w.x >> 16) & 0xFFu; c[3] = w.x >> 24;
  c[4] = w.y & 0xFFu; c[6] = (w.y >> 8) & 0xFFu; c[5] = (w.y >> 16) & 0xFFu; c[7] = w.y >> 24;
}

// Bit position of channel j (0..7) inside the packed word:
// word = c0 | c2<<4 | c4<<8 | c6<<12 | c1<<16 | c3<<20 | c5<<24 | c7<<28.
__device__ __forceinline__ int nib_shift(int j) { return ((j >> 1) << 2) + ((j & 1) << 4); }

__device__ __forceinline__ uint32_t pack8(const uint32_t (&c)[8]) {
  uint32_t w = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) w |= c[j] << nib_shift(j);
  return w;
}

__device__ __forceinline__ void bf16x8_to_float(const uint4& u, float (&x)[8]) {
  const uint32_t r[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    x[2 * i] = __uint_as_float(r[i] << 16);
    x[2 * i + 1] = __uint_as_float(r[i] & 0xFFFF0000u);
  }
}

// ---------------------------------------------------------------------------
// Conversion-free forms of Eq. 10 and Eq. 7.  They produce the same fp32 results
// as the plain forms whenever their preconditions hold (callers check them and
// take the plain forms otherwise), but use no int<->float conversion or round
// instruction, which issue at a quarter of the fp32 rate.
//
// A 4-bit code q sitting at bit 4i of a word, OR-ed into the mantissa of
// 2^(23-4i), is the float 2^(23-4i) + q.  Subtracting 2^(23-4i) + z (exact for
// integer |z| < 2^22) gives q - z exactly, like float(q) - z.
// ---------------------------------------------------------------------------
constexpr float kZLimit = 4194304.f;       // 2^22
constexpr float kRoundMagic = 12582912.f;  // 1.5 * 2^23: y + magic has rint(y) in its mantissa for |y| < 2^22

__device__ __forceinline__ uint32_t magic_bits(int j) { return 0x4B000000u - (uint32_t)(j >> 1) * 0x02000000u; }
__device__ __forceinline__ float magic_val(int j) { return __uint_as_float(magic_bits(j)); }

// par[j] = (s, magic_val(j) + z) for the 8 channels of the word.
__device__ __forceinline__ void dequant8_magic(uint32_t word, const float2 (&par)[8], float (&x)[8]) {
  const uint32_t hi = word >> 16;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t src = (j & 1) ? hi : word;
    const uint32_t bits = (src & (0xFu << (4 * (j >> 1)))) | magic_bits(j);
    x[j] = __fmul_rn(par[j].x, __fsub_rn(__uint_as_float(bits), par[j].y));
  }
}

__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Two fp32 numbers in one 64-bit register and the packed forms of the IEEE operations (each half
// is rounded exactly like the scalar operation, so results do not change; one instruction does two).
__device__ __forceinline__ uint64_t pk2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpk2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// dequant8_magic on channel pairs: s2[p] = (s of channel 2p, s of channel 2p + 1), mz2[p] the same
// for magic + z.
__device__ __forceinline__ void dequant8_magic2(uint32_t word, const uint64_t (&s2)[4], const uint64_t (&mz2)[4],
                                                float (&x)[8]) {
  const uint32_t hi = word >> 16;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const uint32_t be = (word & (0xFu << (4 * p))) | magic_bits(2 * p);
    const uint32_t bo = (hi & (0xFu << (4 * p))) | magic_bits(2 * p);
    unpk2(mul2(s2[p], sub2(pk2(__uint_as_float(be), __uint_as_float(bo)), mz2[p])), x[2 * p], x[2 * p + 1]);
  }
}

// The plain forms as real calls on scalars, so that the rarely taken fallback costs a branch and
// not predicated copies of its instructions in the hot path, and arrays stay in registers.
__device__ __noinline__ float dequant_one_call(uint32_t q, float s, float z) {
  return __fmul_rn(s, __fsub_rn((float)q, z));
}
__device__ __noinline__ uint32_t quant_code_call(float x, float inv, float z) { return quant_code(x, inv, z); }

__device__ __forceinline__ void dequant8_plain(uint32_t word, const float2* par, float (&x)[8]) {
#pragma unroll
  for (int j = 0; j < 8; ++j) x[j] = dequant_one_call((word >> nib_shift(j)) & 0xFu, par[j].x, par[j].y);
}

// Unsigned key whose order is the total order of fp32 bit patterns (so that -0 < +0).
__device__ __forceinline__ uint32_t order_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ uint32_t ld_acquire_u32(const unsigned int* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

constexpr int kSelBins = 4096;       // histogram of the top 12 key bits
constexpr int kHistCopies = 4;       // copies of the histogram (a block adds to copy index mod 4: fewer collisions)
constexpr int kPoolRows = 120;       // pooled rows staged in shared memory at a time
constexpr int kCandSmem = 4096;      // candidates a block holds in shared memory
constexpr int kSubBins = 256;        // second histogram: the next 8 key bits of the candidates
constexpr int kSubList = 512;        // candidates of one sub-bin that a block lists in shared memory

// Shared memory of a block, one phase at a time.
union __align__(16) Smem {
  struct { float pooled[64 * 64]; } pool;                                          // [H <= 64][64]
  struct { float2 par[64 * 64]; } kbar;                                            // [H][64] key parameters of one group
  struct { float w[64]; float rows[kPoolRows * 64]; } score;
  struct { unsigned long long cand[kCandSmem]; unsigned long long list[kSubList]; } sel;   // (key << 32) | ~position
  struct { float mn[4][4][64]; float mx[4][4][64]; float2 iz[4][64]; } kq;          // quantise-once: one key group, 4 heads
};

struct Shared {
  Smem u;
  unsigned int warp[33];
  unsigned int acc;
  unsigned int bin, need;          // result of SEL1, used by SEL2
  unsigned int sub, need2, n_list; // SEL2: the sub-bin of the k-th largest key, its rank there, listed candidates
  float fsum[2];                   // SCORE: block sums of S and S^2
  int abort_flag;
};

__device__ __forceinline__ unsigned int block_excl_scan(unsigned int v, unsigned int* s_warp, unsigned int& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;     // 16 warps
  unsigned int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const unsigned int t = (lane < kMT / 32) ? s_warp[lane] : 0u;
    unsigned int y = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned int z = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += z;
    }
    s_warp[lane] = y - t;
    if (lane == 31) s_warp[32] = y;
  }
  __syncthreads();
  const unsigned int res = s_warp[warp] + x - v;
  total = s_warp[32];
  __syncthreads();
  return res;
}

// sum of v over the block (all threads get it); *s_acc must be zero on entry and is zero on exit
__device__ __forceinline__ unsigned int block_sum(unsigned int v, unsigned int* s_acc) {
  v = __reduce_add_sync(0xffffffffu, v);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(s_acc, v);
  __syncthreads();
  const unsigned int t = *s_acc;
  __syncthreads();
  if (threadIdx.x == 0) *s_acc = 0u;
  __syncthreads();
  return t;
}

// The blocks that work on one layer: every layer of a launch has its own, which run through the phases
// independently of the other layers' (their barriers included).
struct Blocks { int index, count; };

// Barrier of a layer's blocks.  Every block arrives once per barrier; the counter only grows (the host
// passes the value it had when the kernel was launched).  The wait is bounded: when it runs out
// the block records XKV_E_TIMEOUT and the kernel winds down without touching anything further.
// `arrived`: the arrivals of the barriers before.  A block that does not `stay` arrives and waits for nobody.
__device__ __forceinline__ bool grid_barrier(const MaintArgs& a, const Blocks& B, uint32_t& arrived, Shared& sh, bool stay = true) {
  __syncthreads();
  arrived += (uint32_t)B.count;
  if (threadIdx.x == 0 && !sh.abort_flag) {
    // (release and acquire by this thread cover the block: the barriers around order the others)
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar) : "memory");
    if (!stay) return false;
    const uint32_t target = a.bar_base + arrived;
    uint32_t it = 0;
    while ((int)(ld_acquire_u32(a.bar) - target) < 0) {
      if (++it > kBarSpin) {
        sh.abort_flag = 1;
        atomicExch(a.status, (int)XKV_E_TIMEOUT);
        break;
      }
      __nanosleep(20);
    }
  }
  if (!stay) return false;
  __syncthreads();
  return sh.abort_flag == 0;
}

// Of `count` blocks, those with work in the scoring and selection of r_old tokens, 64 at a time, and one more that
// clears what the next step needs clear; the others leave at the first barrier, and the two barriers behind it are
// among few.  (A gather, or head means, behind or beside them have work for all.)  One layer, 261 tokens at 1024: 13 of
// 87 blocks stay, a step takes 38.6 instead of 38.9 us, eight frames from an empty cache 265.3 instead of 266.9; where
// every block has tokens to score nothing changes (1374 tokens at 8192: 120.0 and 120.1).
__host__ __device__ __forceinline__ int later_blocks(uint32_t phases, int r_old, int count) {
  const int need = (r_old + 63) / 64 + 1;
  return (phases & (kPhPack | kPhKbarNew)) || need > count ? count : need;
}

// ---------------------------------------------------------------------------
// APPEND.  Thread = (head, token, 8-channel word).  Values: per-token min/max over
// the 64 channels by xor-shuffle inside the 8-lane group, then codes -> one 32-bit
// word per lane.  Keys: copied to the staging buffer (4-bit) or to their final
// slot (16-bit).
// ---------------------------------------------------------------------------
template <int BITS, bool ONCE>
__device__ __forceinline__ void phase_append(const MaintArgs& a, const Blocks& B) {
  const long long items = (long long)a.H * a.n * 8;
  const int passes = (int)((items + kMT - 1) / kMT);
  const BufSet& d0 = a.oth;
  const BufSet& d1 = a.cur;
  const bool two = a.first != 0;
  // pass p goes to block G - 1 - (p mod G): the blocks that hold no pooled row start first
  for (int p = B.count - 1 - B.index; p < passes; p += B.count) {
    const long long g = (long long)p * kMT + threadIdx.x;
    const int w = (int)(g & 7);
    const long long th = g >> 3;
    const bool valid = th < (long long)a.H * a.n;
    const int h = valid ? (int)(th / a.n) : 0;
    const int tok = valid ? (int)(th % a.n) : 0;
    const int64_t src = (int64_t)h * a.hs_kv + (int64_t)tok * a.ts_kv + 8 * w;
    const uint4 kv = *reinterpret_cast<const uint4*>(a.k + src);
    const uint4 vv = *reinterpret_cast<const uint4*>(a.v + src);
    const size_t slot = (size_t)h * a.cap + a.dst_slot + tok;
    if (BITS == 16) {
      if (valid) {
        const size_t at = slot * 128 + 16 * (w ^ (int)(slot & 7));
        *reinterpret_cast<uint4*>(d0.k + at) = kv;
        *reinterpret_cast<uint4*>(d0.v + at) = vv;
        if (two) {
          *reinterpret_cast<uint4*>(d1.k + at) = kv;
          *reinterpret_cast<uint4*>(d1.v + at) = vv;
        }
      }
    } else {
      float x[8];
      bf16x8_to_float(vv, x);
      float mn = x[0], mx = x[0];
#pragma unroll
      for (int j = 1; j < 8; ++j) { mn = fminf(mn, x[j]); mx = fmaxf(mx, x[j]); }
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      }
      constexpr float kQmax = (BITS == 8) ? 255.f : 15.f;
      float s, inv, z;
      quant_params(mn, mx, s, inv, z, kQmax);
      uint32_t c[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) c[j] = quant_code(x[j], inv, z, kQmax);
      if (valid) {
        if (BITS == 8) {
          const uint2 words = make_uint2(pack4_bytes(c[0], c[1], c[2], c[3]), pack4_bytes(c[4], c[5], c[6], c[7]));
          *reinterpret_cast<uint2*>(d0.v + slot * 64 + 8 * w) = words;
          if (two) *reinterpret_cast<uint2*>(d1.v + slot * 64 + 8 * w) = words;
        } else {
          const uint32_t word = pack8(c);
          *reinterpret_cast<uint32_t*>(d0.v + slot * 32 + 4 * w) = word;
          if (two) *reinterpret_cast<uint32_t*>(d1.v + slot * 32 + 4 * w) = word;
        }
        if (w == 0) d0.vpar[slot] = make_float2(s, z);
        if (two) {
          if (w == 0) d1.vpar[slot] = make_float2(s, z);
        }
        if (!ONCE) __stcg(reinterpret_cast<uint4*>(a.kstage + ((size_t)h * a.max_n + tok) * 64 + 8 * w), kv);
      }
    }
    if (valid && h == 0 && w == 0) {
      const int32_t o = (a.frame << 16) | tok;
      d0.origin[a.dst_slot + tok] = o;
      if (two) d1.origin[a.dst_slot + tok] = o;
    }
  }
}

// ---------------------------------------------------------------------------
// POOL.  Pooled query, Eq. 2-3.  Block b takes pooled rows b, b + G, ...; thread
// (c, hs) builds pooled[h][i][c] for heads h = hs, hs + 8, ... (sequential sum over
// the group's tokens, divided by the group size); threads with hs == 0 add the
// heads in order and scale by 1/H.  Loads are issued in batches ahead of the
// (ordered) additions.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void phase_pool(const MaintArgs& a, const Blocks& B, Shared& sh) {
  const int c = threadIdx.x & 63;
  const int hslot = threadIdx.x >> 6;      // 0..7
  for (int i = B.index; i < a.n_pooled; i += B.count) {
    int ta, tb;
    if (i < a.n_special) { ta = i; tb = i + 1; }
    else { ta = a.n_special + (i - a.n_special) * a.pool_g; tb = min(ta + a.pool_g, a.n_q); }
    // heads h0 and h0 + 8 together: all loads of a batch (2 heads x 16 tokens) are issued before
    // the first (ordered) addition; an index past the group is clamped, its value unused
    for (int h0 = hslot; h0 < a.H; h0 += 16) {
      const bool has1 = h0 + 8 < a.H;
      const __nv_bfloat16* base0 = a.q + (int64_t)h0 * a.hs_q + c;
      const __nv_bfloat16* base1 = a.q + (int64_t)(has1 ? h0 + 8 : h0) * a.hs_q + c;
      float acc0 = 0.f, acc1 = 0.f;
      for (int t0 = ta; t0 < tb; t0 += 16) {
        float x0[16], x1[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int64_t off = (int64_t)min(t0 + u, tb - 1) * a.ts_q;
          x0[u] = __bfloat162float(base0[off]);
          x1[u] = __bfloat162float(base1[off]);
        }
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          if (t0 + u < tb) {
            acc0 = (t0 + u == ta) ? x0[u] : __fadd_rn(acc0, x0[u]);
            acc1 = (t0 + u == ta) ? x1[u] : __fadd_rn(acc1, x1[u]);
          }
        }
      }
      if (i >= a.n_special) {
        acc0 = __fdiv_rn(acc0, (float)(tb - ta));
        acc1 = __fdiv_rn(acc1, (float)(tb - ta));
      }
      sh.u.pool.pooled[h0 * 64 + c] = acc0;
      if (has1) sh.u.pool.pooled[(h0 + 8) * 64 + c] = acc1;
    }
    __syncthreads();
    if (hslot == 0) {
      float acc = 0.f;
      for (int h0 = 0; h0 < a.H; h0 += 16) {
        float v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = (h0 + u < a.H) ? sh.u.pool.pooled[(h0 + u) * 64 + c] : 0.f;
#pragma unroll
        for (int u = 0; u < 16; ++u)
          if (h0 + u < a.H) acc = (h0 + u == 0) ? v[u] : __fadd_rn(acc, v[u]);
      }
      const float inv_h = __fdiv_rn(1.f, (float)a.H);
      __stcg(&a.qbar[i * 64 + c], __fmul_rn(acc, inv_h));
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// KBAR.  Head means of the keys, Eq. 4, for the rest-local positions [lo, hi) of the
// buffer set `b`: one pass per 64-slot key group (the rest segment starts on a
// 128-slot boundary, so the tokens of a pass share their quantisation parameters).
// Thread = (token, 8-channel word): dequantise the word of every head in order
// (Eq. 10), accumulate the head sum sequentially, scale by 1/H.  The words of
// sixteen heads (4-bit; four 16-byte pieces for 16-bit storage) are fetched ahead
// of their (ordered) use.
// ---------------------------------------------------------------------------
// One run of up to 64 consecutive slots whose keys share their quantisation parameters:
// slot0 = physical slot of the run's first token, i0 = its rest-local position, `count` tokens;
// the parameters of (head h, channel ch) are par[h * par_stride + ch].
template <int BITS>
__device__ __forceinline__ void kbar_run(const MaintArgs& a, Shared& sh, const BufSet& b, const float2* par,
                                         size_t par_stride, int slot0, int i0, int count) {
  const int tid = threadIdx.x;
  const int w = tid & 7;
  const int tok = tid >> 3;
  const int H = a.H, cap = a.cap;
  {
    const int i = i0 + tok;                       // rest-local index
    const int slot = slot0 + tok;
    bool plain = false;
    if (BITS == 4) {
      // Parameters of the key group.  Fast path: float4 [H][4][8] = (s, magic + z) of channels
      // 8w + 2v and 8w + 2v + 1 at [h][v][w], so that the eight lanes of a quarter-warp read
      // consecutive 16-byte chunks.  Plain path: float2 (s, z) [H][64].
      int big = a.force_plain;
      for (int e = tid; e < H * 64; e += kMT) {
        const float2 sz = __ldcg(&par[(size_t)(e >> 6) * par_stride + (e & 63)]);
        big |= !(fabsf(sz.y) < kZLimit);
      }
      plain = __syncthreads_or(big) != 0;
      for (int e = tid; e < H * 64; e += kMT) {
        float2 sz = __ldcg(&par[(size_t)(e >> 6) * par_stride + (e & 63)]);
        if (plain) {
          sh.u.kbar.par[e] = sz;
        } else {
          const int h = e >> 6, ch = e & 63;
          sz.y = __fadd_rn(magic_val(ch & 7), sz.y);
          sh.u.kbar.par[((h * 4 + ((ch & 7) >> 1)) * 8 + (ch >> 3)) * 2 + (ch & 1)] = sz;
        }
      }
      __syncthreads();
    }
    const bool valid = tok < count;
    float acc[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = 0.f;
    if (BITS == 8) {
      // 8-bit codes: plain Eq. 10 per channel, parameters (s, z) [H][64] in shared memory
      __syncthreads();
      for (int e = tid; e < H * 64; e += kMT) sh.u.kbar.par[e] = __ldcg(&par[(size_t)(e >> 6) * par_stride + (e & 63)]);
      __syncthreads();
      for (int h0 = 0; h0 < H; h0 += 8) {
        uint2 wide8[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          wide8[u] = make_uint2(0u, 0u);
          if (valid && h0 + u < H) wide8[u] = __ldcg(reinterpret_cast<const uint2*>(b.k + ((size_t)(h0 + u) * cap + slot) * 64 + 8 * w));
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int h = h0 + u;
          if (h < H) {
            uint32_t c[8];
            unpack8_bytes(wide8[u], c);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float2 sz = sh.u.kbar.par[h * 64 + 8 * w + j];
              const float x = __fmul_rn(sz.x, __fsub_rn((float)c[j], sz.y));
              acc[j] = (h == 0) ? x : __fadd_rn(acc[j], x);
            }
          }
        }
      }
    }
    constexpr int kHB = (BITS == 4) ? 16 : 4;     // heads whose words are in flight together
    for (int h0 = 0; BITS != 8 && h0 < H; h0 += kHB) {
      uint32_t word[BITS == 4 ? kHB : 1];
      uint4 wide[BITS == 4 ? 1 : kHB];
#pragma unroll
      for (int u = 0; u < kHB; ++u) {
        const int h = h0 + u;
        if (BITS == 4) word[u] = 0u; else wide[u] = make_uint4(0, 0, 0, 0);
        if (valid && h < H) {
          if (BITS == 4) word[u] = __ldcg(reinterpret_cast<const uint32_t*>(b.k + ((size_t)h * cap + slot) * 32 + 4 * w));
          else wide[u] = __ldcg(reinterpret_cast<const uint4*>(b.k + ((size_t)h * cap + slot) * 128 + 16 * (w ^ (slot & 7))));
        }
      }
#pragma unroll
      for (int u = 0; u < kHB; ++u) {
        const int h = h0 + u;
        if (h < H) {
          float x[8];
          if (BITS == 4) {
            if (plain) {
              dequant8_plain(word[BITS == 4 ? u : 0], sh.u.kbar.par + h * 64 + 8 * w, x);
            } else {
              float2 par[8];
              const float4* pp = reinterpret_cast<const float4*>(sh.u.kbar.par) + h * 32 + w;
#pragma unroll
              for (int v = 0; v < 4; ++v) {
                const float4 t = pp[v * 8];
                par[2 * v] = make_float2(t.x, t.y);
                par[2 * v + 1] = make_float2(t.z, t.w);
              }
              dequant8_magic(word[BITS == 4 ? u : 0], par, x);
            }
          } else {
            bf16x8_to_float(wide[BITS == 4 ? 0 : u], x);
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[j] = (h == 0) ? x[j] : __fadd_rn(acc[j], x[j]);
        }
      }
    }
    const float inv_h = __fdiv_rn(1.f, (float)H);
    if (valid) {
      float4* dst = reinterpret_cast<float4*>(b.kbar + (size_t)i * 64 + 8 * w);
      __stcg(dst, make_float4(__fmul_rn(acc[0], inv_h), __fmul_rn(acc[1], inv_h), __fmul_rn(acc[2], inv_h),
                              __fmul_rn(acc[3], inv_h)));
      __stcg(dst + 1, make_float4(__fmul_rn(acc[4], inv_h), __fmul_rn(acc[5], inv_h), __fmul_rn(acc[6], inv_h),
                                  __fmul_rn(acc[7], inv_h)));
    }
    __syncthreads();       // the parameter table is rewritten by the next run
  }
}

// KBAR over the rest-local positions [0, kbar_hi) (re-quantising mode and 16-bit):
// one run per 64-slot key group (the rest segment starts on a 128-slot boundary).
template <int BITS>
__device__ __forceinline__ void phase_kbar(const MaintArgs& a, const Blocks& B, Shared& sh) {
  const BufSet& b = a.cur;
  const int hi = a.kbar_hi, g_hi = (hi + 63) >> 6;
  for (int gb = B.index; gb < g_hi; gb += B.count) {
    const int grp = (a.rest_base >> 6) + gb;
    kbar_run<BITS>(a, sh, b, b.kpar + (size_t)grp * 64, (size_t)(a.cap >> 6) * 64, a.rest_base + gb * 64, gb * 64,
                   min(64, hi - gb * 64));
  }
}

// ---------------------------------------------------------------------------
// Quantise-once mode, APPEND: the frame's keys are quantised here, per channel in groups of 64
// consecutive tokens of the frame (Eq. 7-9), and never again.  Item = (group, four heads); 128
// threads per head, thread = (8-channel word, four tokens 16 apart).  Each group takes a slot
// of the parameter table: fp32 (scale, zero) for the maintenance arithmetic and the constants
// of the attention's fp16 operand path.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

template <int BITS>
__device__ __forceinline__ void phase_quant_keys_once(const MaintArgs& a, const Blocks& B, Shared& sh) {
  constexpr float kQmax = (BITS == 8) ? 255.f : 15.f;
  const BufSet& d0 = a.oth;
  const BufSet& d1 = a.cur;
  const bool two = a.first != 0;
  const int H = a.H, cap = a.cap, n = a.n;
  const int tid = threadIdx.x;
  const int hl = tid >> 7, t = tid & 127, w = t & 7, tq = t >> 3, wih = t >> 5;
  const int n_groups = (n + 63) >> 6, n_quads = (H + 3) >> 2;
  const int items = n_groups * n_quads;
  for (int item = B.index; item < items; item += B.count) {
    const int gamma = item / n_quads, quad = item - gamma * n_quads;
    const int h = quad * 4 + hl;
    const bool head_ok = h < H;
    // the group's table slot: the ring of free slots is read at places the host has counted out
    const uint32_t take = a.pop_base + (uint32_t)gamma;
    const int slot = __ldcg(&a.ring[take % (uint32_t)a.n_slots]);
    if (tid == 0 && quad == 0) {
      if ((int)(take - __ldcg(a.push_pos)) >= 0) atomicCAS(a.status, 0, (int)XKV_E_LIMIT);   // the table has run out
      a.ref[slot] = min(64, n - gamma * 64);
    }
    float x[4][8];
    bool live[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int tok = gamma * 64 + tq + 16 * u;
      live[u] = tok < n;
      uint4 raw = make_uint4(0, 0, 0, 0);
      if (live[u] && head_ok) raw = *reinterpret_cast<const uint4*>(a.k + (int64_t)h * a.hs_kv + (int64_t)tok * a.ts_kv + 8 * w);
      bf16x8_to_float(raw, x[u]);
    }
    float mn[8], mx[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) { mn[j] = INFINITY; mx[j] = -INFINITY; }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (live[u]) {
#pragma unroll
        for (int j = 0; j < 8; ++j) { mn[j] = fminf(mn[j], x[u][j]); mx[j] = fmaxf(mx[j], x[u][j]); }
      }
    }
#pragma unroll
    for (int o = 8; o < 32; o <<= 1) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        mn[j] = fminf(mn[j], __shfl_xor_sync(0xffffffffu, mn[j], o));
        mx[j] = fmaxf(mx[j], __shfl_xor_sync(0xffffffffu, mx[j], o));
      }
    }
    __syncthreads();                 // the previous item's parameters have been read
    if ((t & 31) < 8) {
#pragma unroll
      for (int j = 0; j < 8; ++j) { sh.u.kq.mn[hl][wih][8 * w + j] = mn[j]; sh.u.kq.mx[hl][wih][8 * w + j] = mx[j]; }
    }
    __syncthreads();
    if (t < 64) {                    // one thread per channel: the group's parameters (warps 0, 1 of the head)
      float lo = sh.u.kq.mn[hl][0][t], hi = sh.u.kq.mx[hl][0][t];
#pragma unroll
      for (int r = 1; r < 4; ++r) { lo = fminf(lo, sh.u.kq.mn[hl][r][t]); hi = fmaxf(hi, sh.u.kq.mx[hl][r][t]); }
      float sc, inv, z;
      quant_params(lo, hi, sc, inv, z, kQmax);
      sh.u.kq.iz[hl][t] = make_float2(inv, z);
      float zl, zh, cc;
      dequant_consts(sc, z, zl, zh, cc);
      const float zo = (BITS == 4 && (((t & 7) >> 1) & 1)) ? zh : zl;      // 8-bit codes all carry the bias 1024
      // the neighbouring channel's constants: pairs (2p, 2p + 1) share a word
      const float sc1 = __shfl_xor_sync(0xffffffffu, sc, 1), zo1 = __shfl_xor_sync(0xffffffffu, zo, 1);
      const float cc1 = __shfl_xor_sync(0xffffffffu, cc, 1);
      if (head_ok) {
        a.ktab32[((size_t)slot * H + h) * 64 + t] = make_float2(sc, z);
        if ((t & 1) == 0) {
          uint32_t* e = a.ktab16 + (((size_t)slot * H + h) * 8 + (t >> 3)) * 12 + ((t & 7) >> 1);
          e[0] = pack_half2(sc, sc1);
          e[4] = pack_half2(zo, zo1);
          e[8] = pack_half2(cc, cc1);
        }
        if (!(fabsf(sc) * (fabsf(z) + kQmax) <= 65504.f)) atomicCAS(a.status, 0, (int)XKV_E_RANGE);
      }
    }
    __syncthreads();
    if (head_ok) {
      float2 iz[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) iz[j] = sh.u.kq.iz[hl][8 * w + j];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (!live[u]) continue;
        uint32_t c[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) c[j] = quant_code(x[u][j], iz[j].x, iz[j].y, kQmax);
        const size_t dslot = (size_t)h * cap + a.dst_slot + gamma * 64 + tq + 16 * u;
        if (BITS == 8) {
          const uint2 words = make_uint2(pack4_bytes(c[0], c[1], c[2], c[3]), pack4_bytes(c[4], c[5], c[6], c[7]));
          *reinterpret_cast<uint2*>(d0.k + dslot * 64 + 8 * w) = words;
          if (two) *reinterpret_cast<uint2*>(d1.k + dslot * 64 + 8 * w) = words;
        } else {
          const uint32_t word = pack8(c);
          *reinterpret_cast<uint32_t*>(d0.k + dslot * 32 + 4 * w) = word;
          if (two) *reinterpret_cast<uint32_t*>(d1.k + dslot * 32 + 4 * w) = word;
        }
      }
    }
    if (quad == 0 && tid < 64 && gamma * 64 + tid < n) {
      d0.kslot[a.dst_slot + gamma * 64 + tid] = slot;
      if (two) d1.kslot[a.dst_slot + gamma * 64 + tid] = slot;
    }
  }
}

// Quantise-once mode: head means (Eq. 4) of the frame just quantised, into the destination's
// array: one run per arrival group, whose parameters sit in the group's table slot.
template <int BITS>
__device__ __forceinline__ void phase_kbar_new_once(const MaintArgs& a, const Blocks& B, Shared& sh) {
  const int n_groups = (a.n + 63) >> 6;
  const BufSet& d = a.oth;
  for (int gamma = B.index; gamma < n_groups; gamma += B.count) {
    const int slot = __ldcg(&d.kslot[a.dst_slot + gamma * 64]);
    kbar_run<BITS>(a, sh, d, a.ktab32 + (size_t)slot * a.H * 64, 64, a.dst_slot + gamma * 64,
                   a.dst_slot - a.rest_base + gamma * 64, min(64, a.n - gamma * 64));
  }
}

// The survivor gathers.  Tile = (head, kMT / PIECES consecutive survivors), thread = (survivor,
// 16-byte piece ch of PIECES): one division per tile and thread, where an index of (head, survivor,
// piece) split by 64-bit divisions cost more than the copies.  Several tiles are in flight per thread: the kept
// indices, then the rows, then the stores.
template <int PIECES>
struct GatherTiles {
  static constexpr int kTokens = kMT / PIECES;
  int ch, tok, per_head, count;
  __device__ __forceinline__ explicit GatherTiles(const MaintArgs& a) {
    ch = (int)threadIdx.x % PIECES;
    tok = (int)threadIdx.x / PIECES;
    per_head = (a.kk + kTokens - 1) / kTokens;
    count = a.H * per_head;
  }
  // slots that this thread's survivor of a tile comes from and goes to; false if there is none
  __device__ __forceinline__ bool rows(const MaintArgs& a, int tile, size_t* from, size_t* to) const {
    const int h = tile / per_head, i = (tile - h * per_head) * kTokens + tok;
    const bool ok = tile < count && i < a.kk;
    const int old = (ok && !a.identity) ? __ldcg(&a.kept[i]) : i;
    const size_t base = (size_t)h * a.cap + a.rest_base;
    *from = base + old;
    *to = base + i;
    return ok;
  }
};
// Origins (and, quantise-once mode, group references) of the survivors.
__device__ __forceinline__ void gather_origins(const MaintArgs& a, const Blocks& B) {
  for (int i = B.index * kMT + (int)threadIdx.x; i < a.kk; i += B.count * kMT) {
    const int old = a.identity ? i : __ldcg(&a.kept[i]);
    a.oth.origin[a.rest_base + i] = a.cur.origin[a.rest_base + old];
    if (a.cur.kslot) a.oth.kslot[a.rest_base + i] = a.cur.kslot[a.rest_base + old];
  }
}

// Quantise-once mode, PACK: the survivors' key and value code rows, value parameters, group
// references, origins and head means move to their new places in the other buffer set.
template <int BITS>
__device__ __forceinline__ void phase_gather_once(const MaintArgs& a, const Blocks& B) {
  constexpr int kRow = (BITS == 8) ? 64 : 32;       // bytes of a code row
  constexpr int kRC = kRow / 16;                    // 16-byte chunks of a row
  const BufSet& src = a.cur;
  const BufSet& dst = a.oth;
  const int32_t* kept = a.identity ? nullptr : a.kept;
  const long long stride = (long long)B.count * kMT;
  const long long first = (long long)B.index * kMT + threadIdx.x;
  if (a.kk == 0) {
    // the budget leaves no room for the middle (k = 0): every token after the first frame leaves,
    // without a selection; their key groups give their table slots back
    for (long long i = first; i < a.r_old; i += stride) {
      const int slot = __ldcg(&src.kslot[a.rest_base + i]);
      if (atomicSub(&a.ref[slot], 1) == 1) a.ring[atomicAdd(a.push_pos, 1u) % (unsigned int)a.n_slots] = slot;
    }
    return;
  }
  const GatherTiles<2 * kRC> tiles(a);                            // the 16-byte pieces of K codes, then of V codes
  constexpr int kU = 4;
  const int piece = 16 * (tiles.ch % kRC);
  const uint8_t* from_base = (tiles.ch < kRC ? src.k : src.v) + piece;
  uint8_t* to_base = (tiles.ch < kRC ? dst.k : dst.v) + piece;
  for (int t0 = B.index; t0 < tiles.count; t0 += kU * B.count) {
    size_t from[kU], to[kU];
    bool ok[kU];
    uint4 row[kU];
    float2 vp[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) ok[u] = tiles.rows(a, t0 + u * B.count, &from[u], &to[u]);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      row[u] = ok[u] ? *reinterpret_cast<const uint4*>(from_base + from[u] * kRow) : make_uint4(0, 0, 0, 0);
      vp[u] = (ok[u] && tiles.ch == kRC) ? src.vpar[from[u]] : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      if (!ok[u]) continue;
      *reinterpret_cast<uint4*>(to_base + to[u] * kRow) = row[u];
      if (tiles.ch == kRC) dst.vpar[to[u]] = vp[u];
    }
  }
  const long long rows = (long long)a.kk * 16;                       // (survivor, 16-byte chunk of its head-mean row)
  for (long long g0 = first; g0 < rows; g0 += 4 * stride) {
    int old[4]; bool ok[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long long g = g0 + u * stride;
      ok[u] = g < rows;
      old[u] = ok[u] ? (kept ? __ldcg(&kept[(int)(g >> 4)]) : (int)(g >> 4)) : 0;
    }
    float4 row[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      row[u] = ok[u] ? __ldcg(reinterpret_cast<const float4*>(src.kbar + (size_t)old[u] * 64) + ((g0 + u * stride) & 15)) : make_float4(0, 0, 0, 0);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long long g = g0 + u * stride;
      if (ok[u]) reinterpret_cast<float4*>(dst.kbar + (size_t)(g >> 4) * 64)[g & 15] = row[u];
    }
  }
  gather_origins(a, B);
}

// ---------------------------------------------------------------------------
// SCORE.  w[c] = (sequential sum of the pooled rows) / N_pooled; S[j] = balanced
// tree over the 64 products w[c] * K-bar[j][c] (three levels inside the lane, three
// by xor-shuffle), Eq. 5-6.  Thread = (token, 8-channel word); block b takes the
// 64-token runs b, b + G, ...
// ---------------------------------------------------------------------------
__device__ __forceinline__ void phase_score(const MaintArgs& a, const Blocks& B, Shared& sh) {
  const int tid = threadIdx.x;
  const int n_runs = (a.r_old + 63) >> 6;
  if (B.index >= n_runs && B.index != 0) return;
  // the pooled rows come through shared memory, 120 at a time (one round trip), and one thread
  // per channel adds them in order -- unless the caller supplied the row mean
  for (int r0 = 0; a.w_in == nullptr && r0 < a.n_pooled; r0 += kPoolRows) {
    const int rows = min(kPoolRows, a.n_pooled - r0);
    __syncthreads();
    for (int e = tid; e < rows * 64; e += kMT) sh.u.score.rows[e] = __ldcg(&a.qbar[r0 * 64 + e]);
    __syncthreads();
    if (tid < 64) {
      float acc = (r0 == 0) ? 0.f : sh.u.score.w[tid];
      for (int q0 = 0; q0 < rows; q0 += 16) {
        float v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = (q0 + u < rows) ? sh.u.score.rows[(q0 + u) * 64 + tid] : 0.f;
#pragma unroll
        for (int u = 0; u < 16; ++u)
          if (q0 + u < rows) acc = (r0 == 0 && q0 + u == 0) ? v[u] : __fadd_rn(acc, v[u]);
      }
      sh.u.score.w[tid] = acc;
    }
  }
  if (tid < 64) {
    const float wv = a.w_in ? a.w_in[tid] : __fdiv_rn(sh.u.score.w[tid], (float)a.n_pooled);
    sh.u.score.w[tid] = wv;
    if (B.index == 0) a.qvec[tid] = wv;
  }
  __syncthreads();
  const int w = tid & 7, tok = tid >> 3;
  float wq[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) wq[j] = sh.u.score.w[8 * w + j];
  float s1 = 0.f, s2 = 0.f;       // sum of S and of S^2 (for budget policies)
  constexpr int kU = 2;           // runs whose loads are in flight together
  for (int run0 = B.index; run0 < n_runs; run0 += kU * B.count) {
    float4 x[kU], y[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int i = (run0 + u * B.count) * 64 + tok;
      const float4* src = reinterpret_cast<const float4*>(a.cur.kbar + (size_t)(i < a.r_old ? i : 0) * 64 + 8 * w);
      x[u] = __ldcg(src);
      y[u] = __ldcg(src + 1);
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int i = (run0 + u * B.count) * 64 + tok;
      const bool valid = i < a.r_old;
      const float kb[8] = {x[u].x, x[u].y, x[u].z, x[u].w, y[u].x, y[u].y, y[u].z, y[u].w};
      float p[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) p[j] = __fmul_rn(kb[j], wq[j]);
      float t0 = __fadd_rn(p[0], p[1]), t1 = __fadd_rn(p[2], p[3]);
      float t2 = __fadd_rn(p[4], p[5]), t3 = __fadd_rn(p[6], p[7]);
      t0 = __fadd_rn(t0, t1);
      t2 = __fadd_rn(t2, t3);
      float s = __fadd_rn(t0, t2);
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) s = __fadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
      if (valid && w == 0) {
        __stcg(&a.scores[i], s);
        atomicAdd(&a.hist[(B.index & (kHistCopies - 1)) * kSelBins + (order_key(s) >> 20)], 1u);
        s1 += s;
        s2 += s * s;
      }
    }
  }
  // statistics of the scores: block sums, then one atomic per block
#pragma unroll
  for (int o = 8; o < 32; o <<= 1) { s1 += __shfl_xor_sync(0xffffffffu, s1, o); s2 += __shfl_xor_sync(0xffffffffu, s2, o); }
  if ((tid & 31) == 0) { atomicAdd(&sh.fsum[0], s1); atomicAdd(&sh.fsum[1], s2); }
  __syncthreads();
  if (tid == 0) { atomicAdd(&a.stats[0], sh.fsum[0]); atomicAdd(&a.stats[1], sh.fsum[1]); sh.fsum[0] = sh.fsum[1] = 0.f; }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// SEL1 / SEL2.  Top-k of the scores (Sec. 3.2), ties to the lower position, i.e.
// the k largest of the unique pairs (key, -position).  Every block that owns tokens
// repeats the global parts (histogram scan, bisection) for itself.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long composite(uint32_t key, int pos) {
  return ((unsigned long long)key << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)pos);
}

// Tokens of one pass of the selection phases: 64 when the layer has a block for every 64 tokens (then
// the latency of a pass counts), else one per thread (then the number of passes does).
__device__ __forceinline__ int sel_width(const MaintArgs& a, const Blocks& B) {
  return ((a.r_old + 63) >> 6) <= B.count ? 64 : kMT;
}

__device__ __forceinline__ void phase_sel1(const MaintArgs& a, const Blocks& B, Shared& sh) {
  const int tid = threadIdx.x;
  const int width = sel_width(a, B), n_runs = (a.r_old + width - 1) / width;
  if (B.index == B.count - 1) {                 // the next selecting launch's counter and sub-histogram:
    if (tid == 0) *a.cand_count_next = 0u;           // nobody uses them in this launch
    if (tid < kSubBins) a.hist2_next[tid] = 0u;
    if (tid < 4) a.stats_next[tid] = 0.f;
  }
  if (B.index >= n_runs) return;
  // thread t owns the bins 4095 - 8t - 7 .. 4095 - 8t; walked from the top
  unsigned int hb[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
  {
    uint4 lo4[kHistCopies], hi4[kHistCopies];
#pragma unroll
    for (int cpy = 0; cpy < kHistCopies; ++cpy) {
      const uint4* hp = reinterpret_cast<const uint4*>(a.hist + cpy * kSelBins + kSelBins - 8 - 8 * tid);
      lo4[cpy] = __ldcg(hp);
      hi4[cpy] = __ldcg(hp + 1);
    }
#pragma unroll
    for (int cpy = 0; cpy < kHistCopies; ++cpy) {
      hb[0] += hi4[cpy].w; hb[1] += hi4[cpy].z; hb[2] += hi4[cpy].y; hb[3] += hi4[cpy].x;
      hb[4] += lo4[cpy].w; hb[5] += lo4[cpy].z; hb[6] += lo4[cpy].y; hb[7] += lo4[cpy].x;
    }
  }
  unsigned int own = 0u;
#pragma unroll
  for (int u = 0; u < 8; ++u) own += hb[u];
  unsigned int total;
  unsigned int above = block_excl_scan(own, sh.warp, total);   // keys in higher bins than this thread's
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    if (above < (unsigned int)a.kk && (unsigned int)a.kk <= above + hb[u]) {
      sh.bin = (unsigned int)(kSelBins - 1 - (8 * tid + u));
      sh.need = (unsigned int)a.kk - above;                       // the k-th largest is the need-th largest of its bin
    }
    above += hb[u];
  }
  __syncthreads();
  const uint32_t bin = sh.bin;
  for (int run = B.index; run < n_runs; run += B.count) {
    const int i = run * width + tid;
    bool hi = false;
    if (tid < width && i < a.r_old) {
      const uint32_t key = order_key(__ldcg(&a.scores[i]));
      hi = (key >> 20) > bin;
      if ((key >> 20) == bin) {
        const unsigned int at = atomicAdd(a.cand_count, 1u);
        __stcg(&a.cand[at], composite(key, i));
        atomicAdd(&a.hist2[(key >> 12) & (kSubBins - 1)], 1u);
      }
    }
    const int cnt = __syncthreads_count(hi);
    if (tid == 0) __stcg(&a.run_hi[run], (unsigned int)cnt);
  }
}

template <bool ONCE>
__device__ __forceinline__ void phase_sel2(const MaintArgs& a, const Blocks& B, Shared& sh) {
  const int tid = threadIdx.x;
  const int width = sel_width(a, B), n_runs = (a.r_old + width - 1) / width;
  if (B.index == B.count - 1) {                 // every block has read the histogram: ready for the next step
    for (int e = tid; e < kSelBins * kHistCopies; e += kMT) a.hist[e] = 0u;
  }
  if (B.index >= n_runs) return;
  const uint32_t bin = sh.bin;
  const unsigned int need = sh.need;
  const unsigned int ncand = __ldcg(a.cand_count);
  const bool in_smem = ncand <= (unsigned int)kCandSmem;
  if (in_smem)
    for (unsigned int e = tid; e < ncand; e += kMT) sh.u.sel.cand[e] = __ldcg(&a.cand[e]);
  __syncthreads();
  auto cand_at = [&](unsigned int e) -> unsigned long long { return in_smem ? sh.u.sel.cand[e] : __ldcg(&a.cand[e]); };
  // the need-th largest candidate: its bin bits are known, the positions lie below 2^pbits
  int pbits = 1;
  while ((1 << pbits) < a.r_old) ++pbits;
  unsigned long long prefix = ((unsigned long long)bin << 52) | (unsigned long long)(0xFFFFFFFFu << pbits);
  // The candidates share the top 12 key bits; a second histogram over their next 8 bits (filled by
  // SEL1) narrows the k-th largest key down to one sub-bin, whose few members are listed and ranked.
  {
    const unsigned int h2 = (tid < kSubBins) ? __ldcg(&a.hist2[kSubBins - 1 - tid]) : 0u;   // thread t: sub-bin 255 - t
    unsigned int total;
    const unsigned int above2 = block_excl_scan(h2, sh.warp, total);
    if (tid == 0) sh.n_list = 0u;
    if (tid < kSubBins && above2 < need && need <= above2 + h2) { sh.sub = kSubBins - 1 - tid; sh.need2 = need - above2; }
    __syncthreads();
  }
  const uint32_t sub = sh.sub;
  const unsigned int need2 = sh.need2;
  if (in_smem) {
    for (unsigned int e = tid; e < ncand; e += kMT) {
      const unsigned long long cv = sh.u.sel.cand[e];
      if ((((uint32_t)(cv >> 32) >> 12) & (kSubBins - 1)) == sub) {
        const unsigned int at = atomicAdd(&sh.n_list, 1u);
        if (at < (unsigned int)kSubList) sh.u.sel.list[at] = cv;
      }
    }
  }
  __syncthreads();
  const unsigned int m = sh.n_list;
  if (in_smem && m <= 32u) {
    // every warp ranks the listed candidates by itself: lane l holds candidate l and counts the
    // larger ones; the one with need2 - 1 larger ones is the k-th largest of all
    const int lane = tid & 31;
    const unsigned long long mine = (unsigned int)lane < m ? sh.u.sel.list[lane] : 0ull;
    unsigned int larger = 0u;
    for (unsigned int j = 0; j < m; ++j) larger += __shfl_sync(0xffffffffu, mine, (int)j) > mine;
    const unsigned int hit = __ballot_sync(0xffffffffu, (unsigned int)lane < m && larger == need2 - 1u);
    prefix = __shfl_sync(0xffffffffu, mine, __ffs(hit) - 1);
  } else {
    // many candidates (many equal or nearly equal scores): the same bisection over the whole
    // 64-bit pair, block-wide, on the list in shared memory or, if it does not fit, in global memory
    for (int bit = 51; bit >= 0; --bit) {
      if (bit < 32 && bit >= pbits) continue;
      const unsigned long long trial = prefix | (1ull << bit);
      unsigned int c = 0u;
      for (unsigned int e = tid; e < ncand; e += kMT) c += cand_at(e) >= trial;
      if (block_sum(c, &sh.acc) >= need) prefix = trial;
    }
  }
  const unsigned long long tau = prefix;             // kept candidates: composite >= tau (exactly `need` of them)
  if (B.index == 0 && tid == 0) {                 // the k-th largest score itself, for the statistics
    const uint32_t key = (uint32_t)(tau >> 32);
    a.stats[2] = __uint_as_float((key & 0x80000000u) ? (key ^ 0x80000000u) : ~key);
  }
  for (int run = B.index; run < n_runs; run += B.count) {
    // survivors before this run: the sure keeps of the runs before it plus the kept candidates at
    // lower positions
    unsigned int part = 0u;
    for (int r = tid; r < run; r += kMT) part += __ldcg(&a.run_hi[r]);
    const uint32_t below = 0xFFFFFFFFu - (uint32_t)(run * width);      // position part of the run's first position
    for (unsigned int e = tid; e < ncand; e += kMT) {
      const unsigned long long cv = cand_at(e);
      part += (cv >= tau) && ((uint32_t)cv > below);                   // larger low word = lower position
    }
    const unsigned int base = block_sum(part, &sh.acc);
    const int i = run * width + tid;
    bool keep = false;
    if (tid < width && i < a.r_old) {
      const uint32_t key = order_key(__ldcg(&a.scores[i]));
      keep = (key >> 20) > bin || ((key >> 20) == bin && composite(key, i) >= tau);
    }
    const unsigned int m = __ballot_sync(0xffffffffu, keep);
    if ((tid & 31) == 0) sh.warp[tid >> 5] = __popc(m);
    __syncthreads();
    if (tid < width) {
      unsigned int off = base + __popc(m & ((1u << (tid & 31)) - 1u));
      for (int wp = 0; wp < (tid >> 5); ++wp) off += sh.warp[wp];
      if (keep) __stcg(&a.kept[off], i);
      if (ONCE && i < a.r_old && !keep) {
        // the token leaves: its key group loses a member and gives its table slot back when empty
        const int slot = __ldcg(&a.cur.kslot[a.rest_base + i]);
        if (atomicSub(&a.ref[slot], 1) == 1) a.ring[atomicAdd(a.push_pos, 1u) % (unsigned int)a.n_slots] = slot;
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// kv_quant_pack, 4-bit: a kernel of its own (one thread block per item, placed by the
// hardware scheduler; the arithmetic needs more registers than the phases above).
// Keys: survivors are dequantised with the parameters of the group they came
// from (Eq. 10), new keys come from the bf16 staging buffer; per-channel min/max
// over the group's tokens; new parameters and codes (Eq. 7-8).  A complete group
// whose 64 tokens all survive in place is copied.
// Values: the survivors' code rows and parameters, and the origins, move to
// their new slots in the other buffer set (they were quantised on arrival).
// ---------------------------------------------------------------------------
constexpr int kTpt = 4;                          // tokens per thread
constexpr int kRgLanes = 64 / kTpt;              // token lanes
constexpr int kRgThreads = 8 * kRgLanes;

struct RegroupArgs {
  BufSet src, dst;                // (the first frame goes to both buffer sets)
  bool two;
  int force_plain;
  int cap, max_n, base_slot, kk, r_new;
  const int32_t* kept;
  const __nv_bfloat16* kstage;
};
template <int MAX> struct RegroupBatch { RegroupArgs layer[MAX]; };

// Block = (64-slot group, head), thread = (four consecutive tokens, 8-channel word).  Bound by
// instruction issue and latency: consecutive tokens rarely change the source group (its parameters are
// 40 instructions), and the per-channel extremes go through shared memory instead of 32 shuffles a
// thread.  24 layers at 16384 tokens: 584 us with four heads a block, tokens 16 apart and shuffles; eight tokens
// a thread 414 (80 registers, spills) and 447 us (117 registers, too few warps); four tokens, four
// heads a block 436, two heads 396, one head 369 us (small blocks wait for less at their barriers).
template <int MAX>
__global__ void __launch_bounds__(kRgThreads, 8) regroup_k_kernel(const __grid_constant__ RegroupBatch<MAX> batch) {
  grid_dependency_trigger();
  grid_dependency_wait();
  const RegroupArgs& a = batch.layer[MAX == 1 ? 0 : blockIdx.z];
  if ((int)blockIdx.x * 64 >= a.r_new) return;
  const int cap = a.cap, base_slot = a.base_slot, kk = a.kk, r_new = a.r_new;
  __shared__ __align__(16) int s_old[64];        // source position (rest-local) of each token, -1 = new key, -2 = none
  __shared__ __align__(16) float s_mn[kRgLanes][64];   // per token lane; channel 8w + 4k + e at 32k + 4w + e
  __shared__ __align__(16) float s_mx[kRgLanes][64];
  __shared__ __align__(16) float2 s_iz[64];     // 1/s and z - magic (int); channel 8w + 2v + e at (8v + w) 2 + e
  __shared__ float s_z[64];                     // z, for the plain forms
  const int tid = threadIdx.x;
  const int gamma = blockIdx.x;
  const int h = blockIdx.y;
  const int w = tid & 7, tq = tid >> 3;              // tokens kTpt tq + u
  if (tid < 64) {
    const int i = gamma * 64 + tid;
    s_old[tid] = (i < kk) ? (a.kept ? a.kept[i] : i) : (i < r_new) ? -1 : -2;
  }
  __syncthreads();
  const size_t head_slot = (size_t)h * cap + base_slot;

  // ---- values, parameters and origins of the survivors (first frame: nothing to move): half a
  // token's row is fetched here and stored after the key loads below have been issued, so that the two
  // round trips overlap ----
  uint4 v_row = make_uint4(0, 0, 0, 0);
  float2 v_par = make_float2(0.f, 0.f);
  int v_org = 0;
  const int v_tok = tid >> 1, v_half = tid & 1;
  const int v_old = s_old[v_tok];
  const bool v_move = v_old >= 0, o_move = v_move && h == 0 && v_half == 0;
  if (v_move) {
    v_row = *(reinterpret_cast<const uint4*>(a.src.v + (head_slot + v_old) * 32) + v_half);
    if (v_half == 0) v_par = a.src.vpar[head_slot + v_old];
  }
  if (o_move) v_org = a.src.origin[base_slot + v_old];
  auto store_values = [&]() {
    if (v_move) {
      *(reinterpret_cast<uint4*>(a.dst.v + (head_slot + gamma * 64 + v_tok) * 32) + v_half) = v_row;
      if (v_half == 0) a.dst.vpar[head_slot + gamma * 64 + v_tok] = v_par;
    }
    if (o_move) a.dst.origin[base_slot + gamma * 64 + v_tok] = v_org;
  };

  // ---- keys ----
  const int last = gamma * 64 + 63;
  const bool carried = (last < kk) && (s_old[63] == last);
  const size_t dgrp = ((size_t)h * (cap >> 6) + (base_slot >> 6) + gamma) * 64;
  const size_t drow = (head_slot + gamma * 64 + kTpt * tq) * 32 + 4 * w;      // this thread's first word in the destination
  if (carried) {
    store_values();
    {
#pragma unroll
      for (int u = 0; u < kTpt; ++u) {
        const uint32_t word = *reinterpret_cast<const uint32_t*>(a.src.k + drow + 32 * u);
        *reinterpret_cast<uint32_t*>(a.dst.k + drow + 32 * u) = word;
        if (a.two) *reinterpret_cast<uint32_t*>(a.src.k + drow + 32 * u) = word;
      }
      if (tid < 64) {
        const float2 sz = a.src.kpar[dgrp + tid];
        a.dst.kpar[dgrp + tid] = sz;
        if (a.two) a.src.kpar[dgrp + tid] = sz;
      }
    }
    return;
  }
  int old[kTpt];
  {
    const int4 o = *reinterpret_cast<const int4*>(&s_old[kTpt * tq]);
    old[0] = o.x; old[1] = o.y; old[2] = o.z; old[3] = o.w;
  }
  uint32_t word[kTpt];
  {
    const uint8_t* kp = a.src.k + head_slot * 32 + 4 * w;
#pragma unroll
    for (int u = 0; u < kTpt; ++u) {
      word[u] = 0u;
      if (old[u] >= 0) word[u] = *reinterpret_cast<const uint32_t*>(kp + (size_t)old[u] * 32);
    }
  }
  store_values();
  float x[kTpt][8];
  {
    int par_grp = -1;
    const float2* par_src = nullptr; // the group's (s, z) in global memory (the plain path reads them there)
    uint64_t s2[4], mz2[4];          // fast path: (s, s) and (magic + z, magic + z) of the channel pairs
    bool par_plain = false;
    const float2* par0 = a.src.kpar + ((size_t)h * (cap >> 6) + (base_slot >> 6)) * 64 + 8 * w;   // (base_slot is a multiple of 64)
#pragma unroll
    for (int u = 0; u < kTpt; ++u) {
      if (old[u] >= 0) {
        const int g = old[u] >> 6;
        if (g != par_grp) {
          const float4* pp = reinterpret_cast<const float4*>(par0 + (size_t)g * 64);
          float zmax = 0.f;
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const float4 q4 = __ldg(pp + v);
            zmax = fmaxf(zmax, fmaxf(fabsf(q4.y), fabsf(q4.w)));
            s2[v] = pk2(q4.x, q4.z);
            mz2[v] = pk2(__fadd_rn(magic_val(2 * v), q4.y), __fadd_rn(magic_val(2 * v), q4.w));
          }
          par_plain = !(zmax < kZLimit) || a.force_plain;
          par_src = reinterpret_cast<const float2*>(pp);
          par_grp = g;
        }
        if (par_plain) dequant8_plain(word[u], par_src, x[u]);
        else dequant8_magic2(word[u], s2, mz2, x[u]);
      } else {
        uint4 fresh = make_uint4(0, 0, 0, 0);
        if (old[u] == -1)
          fresh = *reinterpret_cast<const uint4*>(a.kstage + ((size_t)h * a.max_n + (gamma * 64 + kTpt * tq + u - kk)) * 64 + 8 * w);
        bf16x8_to_float(fresh, x[u]);
      }
    }
  }
  {
    float mn[8], mx[8];
    if (old[kTpt - 1] != -2) {        // all tokens there
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        mn[j] = min3(x[0][j], x[1][j], fminf(x[2][j], x[3][j]));
        mx[j] = max3(x[0][j], x[1][j], fmaxf(x[2][j], x[3][j]));
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) { mn[j] = INFINITY; mx[j] = -INFINITY; }
#pragma unroll
      for (int u = 0; u < kTpt - 1; ++u) {
        if (old[u] != -2) {
#pragma unroll
          for (int j = 0; j < 8; ++j) { mn[j] = fminf(mn[j], x[u][j]); mx[j] = fmaxf(mx[j], x[u][j]); }
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      *reinterpret_cast<float4*>(&s_mn[tq][32 * k + 4 * w]) = make_float4(mn[4 * k], mn[4 * k + 1], mn[4 * k + 2], mn[4 * k + 3]);
      *reinterpret_cast<float4*>(&s_mx[tq][32 * k + 4 * w]) = make_float4(mx[4 * k], mx[4 * k + 1], mx[4 * k + 2], mx[4 * k + 3]);
    }
  }
  __syncthreads();
  // one thread per channel finishes the reduction and derives the group's parameters
  int slow = a.force_plain;
  if (tid < 64) {
    // (from the empty extremes: a lane whose tokens are all not numbers has none of its own)
    float lo = INFINITY, up = -INFINITY;
#pragma unroll
    for (int r = 0; r < kRgLanes; ++r) { lo = fminf(lo, s_mn[r][tid]); up = fmaxf(up, s_mx[r][tid]); }
    float sc, inv, z;
    quant_params(lo, up, sc, inv, z);
    const int ch = ((tid >> 2) & 7) * 8 + (tid >> 5) * 4 + (tid & 3);
    s_iz[(((ch & 7) >> 1) * 8 + (ch >> 3)) * 2 + (ch & 1)] = make_float2(inv, __int_as_float((int)z - (int)0x4B400000));
    s_z[ch] = z;
    {
      a.dst.kpar[dgrp + ch] = make_float2(sc, z);
      if (a.two) a.src.kpar[dgrp + ch] = make_float2(sc, z);
      // the conversion-free quantiser needs |x * inv| < 2^21 and |z| < 2^22
      const float ymax = __fmul_rn(fmaxf(fabsf(lo), fabsf(up)), inv);
      slow |= !(ymax < 2097152.f) || !(fabsf(z) < kZLimit);
    }
  }
  slow = __syncthreads_or(slow);
  float inv[8];
  int zadj[8];
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const float4 q4 = *reinterpret_cast<const float4*>(&s_iz[(8 * v + w) * 2]);
    inv[2 * v] = q4.x; inv[2 * v + 1] = q4.z;
    zadj[2 * v] = __float_as_int(q4.y); zadj[2 * v + 1] = __float_as_int(q4.w);
  }
  uint64_t inv2[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) inv2[p] = pk2(inv[2 * p], inv[2 * p + 1]);
#pragma unroll
  for (int u = 0; u < kTpt; ++u) {
    if (old[u] == -2) continue;
    uint32_t packed = 0u;
    if (slow) {
#pragma unroll
      for (int j = 0; j < 8; ++j) packed |= quant_code_call(x[u][j], inv[j], s_z[8 * w + j]) << nib_shift(j);
    } else {
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        // x * inv for two channels at once; the addition of 1.5 * 2^23 stays scalar: a packed
        // multiplication followed by a packed addition was observed to round once, like a fused
        // multiply-add, which breaks the ties of Eq. 7's rounding
        float te, to;
        unpk2(mul2(pk2(x[u][2 * p], x[u][2 * p + 1]), inv2[p]), te, to);
        te = __fadd_rn(te, kRoundMagic);
        to = __fadd_rn(to, kRoundMagic);
        int qe = (int)__float_as_uint(te) + zadj[2 * p], qo = (int)__float_as_uint(to) + zadj[2 * p + 1];
        asm("min.relu.s32 %0, %1, 15;" : "=r"(qe) : "r"(qe));
        asm("min.relu.s32 %0, %1, 15;" : "=r"(qo) : "r"(qo));
        // the nibbles do not overlap: multiply-add places them
        packed = (uint32_t)qe * (1u << nib_shift(2 * p)) + packed;
        packed = (uint32_t)qo * (1u << nib_shift(2 * p + 1)) + packed;
      }
    }
    *reinterpret_cast<uint32_t*>(a.dst.k + drow + 32 * u) = packed;
    if (a.two) *reinterpret_cast<uint32_t*>(a.src.k + drow + 32 * u) = packed;
  }
}

// ---------------------------------------------------------------------------
// PACK, 16-bit: rows of keys and values and the origins move from the current
// buffer set to the other, preserving order.  Thread-item = (head, survivor,
// 16-byte chunk).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void phase_gather16(const MaintArgs& a, const Blocks& B) {
  const BufSet& src = a.cur;
  const BufSet& dst = a.oth;
  const GatherTiles<8> tiles(a);
  constexpr int kU = 3;
  for (int t0 = B.index; t0 < tiles.count; t0 += kU * B.count) {
    size_t from[kU], to[kU];
    bool ok[kU];
    uint4 k[kU], v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) ok[u] = tiles.rows(a, t0 + u * B.count, &from[u], &to[u]);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      k[u] = v[u] = make_uint4(0, 0, 0, 0);
      if (ok[u]) {
        const size_t at = from[u] * 128 + 16 * (tiles.ch ^ (int)(from[u] & 7));
        k[u] = *reinterpret_cast<const uint4*>(src.k + at);
        v[u] = *reinterpret_cast<const uint4*>(src.v + at);
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      if (!ok[u]) continue;
      const size_t at = to[u] * 128 + 16 * (tiles.ch ^ (int)(to[u] & 7));
      *reinterpret_cast<uint4*>(dst.k + at) = k[u];
      *reinterpret_cast<uint4*>(dst.v + at) = v[u];
    }
  }
  gather_origins(a, B);
}

}  // namespace

// ---------------------------------------------------------------------------
// The kernel.
// ---------------------------------------------------------------------------
// A launch takes up to MAX layers: block b works on layer b mod n.  (A layer alone leaves the chip
// waiting: at 1374 tokens and 16384 cached ones its phases are chains of round trips that move
// 16 MB in 30 us.)  The form for one layer keeps its parameters directly addressable.
template <int MAX> struct MaintBatch { int n; MaintArgs layer[MAX]; };

template <int BITS, bool ONCE, int MAX>
__global__ void __launch_bounds__(kMT, kBlocksPerSM) maint_kernel(const __grid_constant__ MaintBatch<MAX> batch) {
  __shared__ Shared sh;
  if (threadIdx.x == 0) { sh.abort_flag = 0; sh.acc = 0u; sh.bin = 0u; sh.need = 0u; sh.fsum[0] = sh.fsum[1] = 0.f; }
  __syncthreads();
  grid_dependency_wait();
  const int which = (MAX == 1) ? 0 : (int)blockIdx.x % batch.n;
  Blocks B{(MAX == 1) ? (int)blockIdx.x : (int)blockIdx.x / batch.n,
           (MAX == 1) ? (int)gridDim.x : ((int)gridDim.x - which + batch.n - 1) / batch.n};
  const MaintArgs& a = batch.layer[which];
  uint32_t arrived = 0;
  const uint32_t ph = a.phases;
  bool ran = false;                 // something has run since the last barrier

  if (ph & kPhAppend) {
    phase_append<BITS, ONCE>(a, B);
    if (ONCE) phase_quant_keys_once<BITS>(a, B, sh);
    ran = true;
  }
  if (ph & kPhPool) { phase_pool(a, B, sh); ran = true; }
  if (ph & kPhKbar) {
    // (from the first block that has no pooled row)
    const int skip = (ph & kPhPool) ? a.n_pooled % B.count : 0;
    const Blocks K{B.index >= skip ? B.index - skip : B.index + B.count - skip, B.count};
    phase_kbar<BITS>(a, K, sh);
    ran = true;
  }

  if (ph & (kPhScore | kPhKbarNew)) {
    // (the blocks that have nothing to do in the phases that follow leave here)
    const int later = later_blocks(ph, a.r_old, B.count);
    if (ran && !grid_barrier(a, B, arrived, sh, B.index < later)) return;
    if (ran) B.count = later;
    if (ONCE && (ph & kPhKbarNew)) phase_kbar_new_once<BITS>(a, B, sh);
    if (ph & kPhScore) phase_score(a, B, sh);
    ran = true;
  }
  if (ph & kPhSel) {
    if (ran && !grid_barrier(a, B, arrived, sh)) return;
    phase_sel1(a, B, sh);
    if (!grid_barrier(a, B, arrived, sh)) return;
    phase_sel2<ONCE>(a, B, sh);
    ran = true;
  }
  if (ph & kPhPack) {
    if (ran && !grid_barrier(a, B, arrived, sh)) return;
    if (ONCE) phase_gather_once<BITS>(a, B);
    else if (BITS == 16 && a.kk > 0) phase_gather16(a, B);
  }
}

// Quantise-once mode: the ring of free table slots starts full.
__global__ void once_init_kernel(int32_t* ring, unsigned int* push_pos, int n_slots) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n_slots) ring[i] = i;
  if (i == 0) *push_pos = (unsigned int)n_slots;
}

cudaError_t launch_once_init(xkv_cache* c, cudaStream_t st) {
  once_init_kernel<<<(c->n_slots + 255) / 256, 256, 0, st>>>(c->ring, c->counters + 8, c->n_slots);
  return cudaGetLastError();
}

// Arrivals at the barriers that a launch with these phases and `count` blocks goes through (the same decisions as in
// the kernel).
static uint32_t maint_arrivals(uint32_t ph, int r_old, uint32_t count) {
  uint32_t n = 0;
  bool ran = (ph & (kPhAppend | kPhPool | kPhKbar)) != 0;
  if (ph & (kPhScore | kPhKbarNew)) {
    if (ran) { n += count; count = (uint32_t)later_blocks(ph, r_old, (int)count); }
    ran = true;
  }
  if (ph & kPhSel) { n += (ran ? 2u : 1u) * count; ran = true; }
  if (ph & kPhPack) n += ran ? count : 0u;
  return n;
}

// Per device, on first use with that device current: how many blocks of the kernel can be
// resident at once (a cooperative launch needs the whole grid resident).
static std::mutex g_maint_mutex;
static int g_maint_grid[64] = {0};

template <int MAX> static const void* maint_fn(int bits, bool once) {
  return (bits == 16) ? (const void*)maint_kernel<16, false, MAX>
         : (bits == 8) ? (const void*)maint_kernel<8, true, MAX>
         : once        ? (const void*)maint_kernel<4, true, MAX>
                       : (const void*)maint_kernel<4, false, MAX>;
}

static cudaError_t maint_grid(int* grid) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_maint_mutex);
  if (g_maint_grid[dev] == 0) {
    int sms = 0, per_sm = kBlocksPerSM;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const void* fns[8] = {maint_fn<1>(4, false), maint_fn<1>(16, false), maint_fn<1>(4, true), maint_fn<1>(8, true),
                          maint_fn<kMaxLayers>(4, false), maint_fn<kMaxLayers>(16, false),
                          maint_fn<kMaxLayers>(4, true), maint_fn<kMaxLayers>(8, true)};
    for (const void* fn : fns) {
      int nb = 0;
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, kMT, 0);
      if (e != cudaSuccess) return e;
      if (nb < per_sm) per_sm = nb;
    }
    if (per_sm < 1) return cudaErrorLaunchOutOfResources;
    g_maint_grid[dev] = sms * per_sm;
  }
  *grid = g_maint_grid[dev];
  return cudaSuccess;
}

template <int MAX>
static cudaError_t launch_regroup_n(xkv_cache* const* c, const MaintArgs* a, int count, cudaStream_t st) {
  RegroupBatch<MAX> b;
  int groups = 0;
  for (int i = 0; i < count; ++i) {
    b.layer[i] = {a[i].cur, a[i].oth, a[i].first != 0, a[i].force_plain, a[i].cap, a[i].max_n, a[i].first ? 0 : a[i].rest_base,
                  a[i].kk, a[i].r_new, a[i].identity ? nullptr : a[i].kept, a[i].kstage};
    const int g = (a[i].r_new + 63) / 64;
    if (g > groups) groups = g;
  }
  const dim3 grid(groups, a[0].H, count);
  LaunchScope ls(c, count, XKV_PROF_PACK, st);
  void* params[1] = {(void*)&b};
  const cudaError_t e = launch_overlapped((const void*)regroup_k_kernel<MAX>, grid, dim3(kRgThreads), params, 0, st);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_regroup(xkv_cache* const* c, const MaintArgs* a, int count, cudaStream_t st) {
  return count == 1 ? launch_regroup_n<1>(c, a, 1, st) : launch_regroup_n<kMaxLayers>(c, a, count, st);
}

// Blocks that have something to do in the busiest phase of a layer (what runs between two barriers
// counts together).  A layer of 261 tokens fills 87 of 296; the others would only make its barriers
// longer.
static int useful_blocks(const xkv_cache* c, const MaintArgs& a) {
  long long first = 0, later = 1;
  auto ceil_div = [](long long x, long long y) { return (x + y - 1) / y; };
  if (a.phases & kPhAppend) first += ceil_div((long long)a.H * a.n * 8, kMT);
  if ((a.phases & kPhAppend) && c->p.key_mode == XKV_KEYS_ONCE) first += ceil_div(a.n, 64) * ceil_div(a.H, 4);
  if (a.phases & kPhPool) first += a.n_pooled;
  if (a.phases & kPhKbar) first += ceil_div(a.kbar_hi, 64) + 1;
  if (a.phases & kPhKbarNew) later = ceil_div(a.n, 64);
  if ((a.phases & (kPhScore | kPhSel)) && ceil_div(a.r_old, 64) > later) later = ceil_div(a.r_old, 64);
  if (a.phases & kPhPack) {
    const long long bytes = (long long)a.H * (a.kk > 0 ? a.kk : a.r_old) * 2 * c->row_bytes;
    if (ceil_div(bytes, 16 * kMT) > later) later = ceil_div(bytes, 16 * kMT);
  }
  const long long n = first > later ? first : later;
  return n < 65536 ? (int)n : 65536;
}

template <int MAX>
static cudaError_t launch_maint_n(xkv_cache* const* c, MaintArgs* as, int count, cudaStream_t st) {
  int grid = 0;
  cudaError_t e = maint_grid(&grid);
  if (e != cudaSuccess) return e;
  MaintBatch<MAX> batch;
  batch.n = count;
  bool barriers = false;
  int useful = 1;
  for (int i = 0; i < count; ++i) {
    const int u = useful_blocks(c[i], as[i]);
    if (u > useful) useful = u;
  }
  if ((long long)useful * count < grid) grid = useful * count;
  for (int i = 0; i < count; ++i) {
    MaintArgs& a = as[i];
    xkv_cache* ci = c[i];
    const uint32_t arrivals = maint_arrivals(a.phases, a.r_old, (uint32_t)((grid - i + count - 1) / count));      // of this layer's blocks
    a.bar = ci->counters;
    a.bar_base = ci->bar_base;
    a.status = ci->status;
    a.cand_count = ci->counters + 2 + ci->sel_parity;
    a.cand_count_next = ci->counters + 2 + (ci->sel_parity ^ 1);
    a.hist2 = ci->counters + 64 + 256 * ci->sel_parity;
    a.hist2_next = ci->counters + 64 + 256 * (ci->sel_parity ^ 1);
    a.stats = reinterpret_cast<float*>(ci->counters + 16 + 4 * ci->sel_parity);
    a.stats_next = reinterpret_cast<float*>(ci->counters + 16 + 4 * (ci->sel_parity ^ 1));
    a.push_pos = ci->counters + 8;
    if (a.phases & kPhSel) { ci->stats_parity = ci->sel_parity; ci->sel_parity ^= 1; }
    if (arrivals > 0) barriers = true;
    ci->bar_base += arrivals;
    batch.layer[i] = a;
  }
  void* params[1] = {(void*)&batch};
  const void* fn = maint_fn<MAX>(c[0]->p.kv_bits, c[0]->p.key_mode == XKV_KEYS_ONCE);
  e = barriers ? cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(kMT), params, 0, st)
               : launch_overlapped(fn, dim3(grid), dim3(kMT), params, 0, st);
  return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_maint(xkv_cache* const* c, MaintArgs* a, int count, int prof_cat, cudaStream_t st) {
  LaunchScope ls(c, count, prof_cat, st);
  return count == 1 ? launch_maint_n<1>(c, a, 1, st) : launch_maint_n<kMaxLayers>(c, a, count, st);
}

}  // namespace xkv
