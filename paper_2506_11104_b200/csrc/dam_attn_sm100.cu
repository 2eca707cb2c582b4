// Sparse flash attention on the 5th-generation tensor cores (sm_100a): bf16 inputs, head_dim 128 or 64.
//
// One persistent CTA per SM walks the work list of the mask blob.  A work item is a pair of adjacent
// 128-row query blocks (2p, 2p+1) of one (sequence, head), two query tiles ("streams" A and B).  Step t multiplies the
// t-th tile of either block's list; where that is the same tile (gathered columns, dense rows) it is loaded once, otherwise
// the step has a K and a V tile for each.  The items follow one another without a gap: the steps of the next one are in
// flight while this one's output is written.
// Warp roles:
//   warp 0      TMA producer: K and V of every step into a ring of shared-memory slots (128-byte swizzle); for every step it
//               leaves a descriptor word in shared memory (which streams have a tile in it, whether it is a stream's first or
//               last of the item, whether the streams' tiles differ);
//   warp 1      MMA issuer (one elected thread), driven by those descriptors alone (it reads no global memory):
//               O_X += P_X V with P_X read from TMEM, then S_X = Q_X K^T of the next step into the same TMEM columns; the two
//               streams take turns, so that one stream's softmax runs under the other stream's MMAs;
//   warp 2      scheduler: claims the next item when this one is nearly loaded, leaves a record of it (item, first tile
//               entries, the head's bit-set pointers) for the other roles, and loads Q_X when the last S_X has been made;
//   warp 3      idle;
//   warps 4-7   softmax of stream A, warps 8-11 of stream B: one thread per query row reads its S row from
//               TMEM (twice: running max, then probabilities), applies the tile's mask bits where the tile
//               is not fully active, writes P (bf16) back to TMEM and rescales O in TMEM when the running max
//               moved by more than 2^8; after a block's last tile it leaves the row's reference and sum;
//   warps 12-15 output of both streams: O / sum and the log-sum-exp, 32 bytes per thread and store.
// What bounds it: a stream's chain from P to the next S to the next P (P V and S about 1400 cycles, softmax 1700 to 1950),
// two of which share the tensor pipe.  In the form before this one the softmax warps also wrote the output, the steps were those of
// the merged lists (in a quarter of them one stream had no tile) and the item's record and Q came when everything before was
// done: an item of 12.5 tiles took 30300 cycles at 32768 tokens, 10500 of them between a stream's last P of an item
// and its first of the next.  Attention alone, that form -> this one, timed in turn: 1237 tokens 26.5 -> 24.7 us, 8192 tokens 97.1 ->
// 90.1, 32768 tokens 413 -> 380, 131072 tokens 1995 -> 1872, mixed lengths 1645 -> 1515, 16001 tokens at head_dim 64 124 -> 110, 2048 rows
// of 26624 43.0 -> 38.4; all-ones 8192 tokens 524 -> 525.
// The kernel's code is kept small: all of it is executed for every item, the instruction cache holds about 64 KB, and the
// same roles in 78 KB were a fifth slower than in 66.  So what waits or issues is written once and looped over
// streams, operands and chunks where it is not hot, and mask words are made at one place.
// A head's lone diagonal (dam_internal.cuh) is served by one tile per query block that starts at the block's first key on
// it, multiplied last, in place of the two listed tiles it lies across; the softmax of that tile is one entry per row.
// Only the tiles the mask lists are ever loaded or multiplied (paper Sec. 4.3: masked logits are -inf).
// Every wait is bounded; an expired wait sets the status word in the scratch buffer and the CTA drains
// and exits.
#include <cuda_bf16.h>
#include <math_constants.h>

#include <type_traits>

#include "dam_internal.cuh"
#include "sm100_ptx.cuh"

using namespace sm100;

namespace {

constexpr int kThreads = 512;   // four warpgroups: {producer, MMA issuer, scheduler, an idle warp}, softmax of stream A, of stream B, output
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kColS = 0;      // S_A at 0, S_B at 128 (P_X overwrites columns [0, 64) of S_X)
constexpr uint32_t kColO = 256;    // O_A at 256, O_B at 384
constexpr float kRescaleThreshold = 8.0f;
// Step descriptor bits of stream A (those of stream B lie one higher): the stream has a tile in the step; it is the stream's
// first / last tile of its item.  kStepDual: the streams' tiles are different ones (K of A, K of B, V of A, V of B).
// kStepEnd: no step, the work list is done.
constexpr uint32_t kStepTile = 1u, kStepFirst = 4u, kStepLast = 16u, kStepDual = 64u, kStepEnd = 128u;
constexpr int kPolyPer8 = 2;   // of every 8 exponentials, how many use the FMA-pipe polynomial (0, 2 or 4)

// Work lists whose items inside the row ranges are marked: up to 3840 or 16384 items (a word for 32).
constexpr int kRowBitWords = 120, kRowBitWordsLong = 512;

// RANGED: 0 no row ranges, 1 row ranges, 2 row ranges and a list of more than 3840 items (head_dim 128).
template <int RANGED, int D>
struct SmemLayout {
  static constexpr int kSlotBytes = 256 * D;            // a Q, K or V tile
  // A step with two tiles per operand holds four slots; a fifth lets the next K tile come early (32768 tokens 388 us with four
  // and K waited for before P V, 359 with four and after, 353 with five; 256 rows of 30000, 8 heads, 31.9 with four and 30.7 with
  // five, 2048 rows of 8192, 32 heads, 40.6 and 38.4).  Beside the row bits of a long list there is room for four.
  static constexpr int kSlots = D == 64 ? 10 : RANGED == 2 ? 4 : 5;
  static constexpr int kBitWords = RANGED == 0 ? 0 : RANGED == 1 && D == 128 ? kRowBitWords : kRowBitWordsLong;
  static constexpr int q = 0;                           // Q_A, Q_B
  static constexpr int slots = 2 * kSlotBytes;
  static constexpr int bars = kSlotBytes * (2 + kSlots);
  // slot_full[kSlots], slot_empty[kSlots], claim, and pairs: q_full, q_empty, s_full, p_full, o_final, o_free, row_full (one
  // per stream), rec_full, rec_empty (one per record)
  static constexpr int n_bars = 2 * kSlots + 1 + 18;
  static constexpr int step_desc = (bars + 8 * n_bars + 15) & ~15;   // u32[16]: what the producer found at each step (kStep*)
  static constexpr int item_rec = step_desc + 64;                    // ItemRec[2]: what the other roles need to start an item
  static constexpr int stat = item_rec + 2 * 112;                    // float2 [stream][128]: reference and sum of every row
  static constexpr int tmem_slot = stat + 2 * DAM_TILE * 8;
  static constexpr int abort_flag = tmem_slot + 4;
  static constexpr int row_bits = abort_flag + 4;           // u32[kBitWords]: the work list's items inside the row ranges
  static constexpr int total = row_bits + 4 * kBitWords;
  static_assert(item_rec % 16 == 0 && bars % 8 == 0 && stat % 8 == 0, "shared-memory records must be aligned");
  static_assert(total <= 232448, "227 KB of shared memory");
};

// What the scheduler hands to the other roles with every work-list position: the item record, the first tile entry of each
// stream and the head's bit-set pointers, so that their set-up reads shared memory instead of walking item -> sequence
// record -> tile list in global memory.
struct alignas(16) ItemRec {
  uint4 u, v;               // the two words of the DamItem (u.x < 0: the work list is done)
  int2 lone;                // the head's lone diagonal and the entries in front of it
  uint32_t e[2][2];         // the first two entries of each stream's list (entries left out are not counted)
  DamHeadBits hb;
  int lone_from;            // the first query block it is served on
  int gath_row;             // first row of the (sequence, head)'s gathered-column tiles in the scratch buffer
};
static_assert(sizeof(ItemRec) == 112, "ItemRec must be 112 bytes");

__device__ __forceinline__ void st_global_v8(void* p, const uint32_t* v) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
               "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}

struct AttnParams {
  const unsigned char* blob;
  __nv_bfloat16* O;
  float* lse;
  uint32_t* status;         // scratch status word
  uint32_t* work_counter;   // scratch word 2, zero at launch
  unsigned long long scratch_bytes;
  int group, total_tokens, causal;
  int64_t o_stride_tok, o_stride_head;
  int o_vec8;               // every row of O starts on a 32-byte boundary
  float scale_log2;         // softmax scale * log2(e)
  const int32_t* ranges;    // row ranges [begin, end) per sequence (chunked prefill), or NULL
};

__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// One work item: a pair of query blocks of one (sequence, head) and the tile-list ranges of both.
struct Item {
  int head, tok0, qb0, S, hasB, seq;
  uint32_t a0, a1, b0, b1;      // tile list [a0, a1) of block 2p, [b0, b1) of block 2p+1
};

__device__ __forceinline__ Item item_from_words(const uint4& u, const uint4& v) {
  Item it;
  it.head = (int)u.x; it.tok0 = (int)u.y; it.qb0 = (int)u.z; it.S = (int)u.w;
  it.a0 = v.x; it.a1 = v.y; it.b0 = v.y; it.b1 = v.z;
  it.hasB = (int)(v.w >> 31); it.seq = (int)(v.w & 0x7FFFFFFFu);
  return it;
}

// The lone diagonal of a head on one query block: the `n` entries from `at` on list tiles that hold its cells and nothing
// else; they are left out, and one tile of keys from `key` on takes their place behind the list.  n = 0: nothing of the
// kind on this block.
struct Lone {
  uint32_t at, n;
  int key;
  __device__ __forceinline__ Lone(int2 lone, int from, uint32_t t0, int qb, int S) : at(0u), n(0u), key(0) {
    const int i0 = qb * DAM_TILE, r = lone.x;
    if (qb >= from && i0 < S) {
      key = i0 - r;
      n = (uint32_t)(min(i0 + DAM_TILE, S) - 1 - r) / DAM_TILE - (uint32_t)key / DAM_TILE + 1u;
      at = t0 + (uint32_t)lone.y;
    }
  }
};

// The tiles of one query block in the order they are multiplied: its list, without the entries the lone diagonal makes
// superfluous, then the lone diagonal's tile.
struct TileWalk {
  const uint32_t* tiles;
  uint32_t i, end, cur, at, n;
  int row;                      // first key row of the lone diagonal's tile, -1: none (left)
  // first: the first entry that is not left out (where there is any); tok0: first row of the sequence
  __device__ __forceinline__ TileWalk(const uint32_t* t, uint32_t t0, uint32_t t1, const Lone& ln, uint32_t first, int tok0)
      : tiles(t), i(t0), end(t1), at(ln.at), n(ln.n), row(ln.n ? tok0 + ln.key : -1) {
    if (n && i == at) i += n;
    cur = first;
  }
  // (from the positions: an entry that has just been asked for is not waited for)
  __device__ __forceinline__ bool more() const { return i < end || row >= 0; }
  __device__ __forceinline__ uint32_t left() const { return end - i + (row >= 0 ? 1u : 0u); }    // (an upper bound)
  // where the next tile's K rows are: bit 31 set: row of the gathered columns
  __device__ __forceinline__ uint32_t next(int tok0, int gath_row) {
    if (i >= end) { const uint32_t r = (uint32_t)row; row = -1; return r; }
    const uint32_t e = cur;
    ++i;
    if (n && i == at) i += n;
    if (i < end) cur = __ldg(tiles + i);
    return (e >> 28) == DAM_KIND_GATHERED ? 0x80000000u | (uint32_t)(gath_row + (int)(e & 0xFFFFu) * 2 * DAM_TILE)
                                          : (uint32_t)(tok0 + (int)(e & 0x0FFFFFFFu) * DAM_TILE);
  }
};

// ---- packed fp32x2 arithmetic (one instruction for two lanes of a register pair) -----------------------
__device__ __forceinline__ void fma2(float& d0, float& d1, float a0, float a1, float b0, float b1, float c0, float c1) {
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\t"
      "mov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d0), "=f"(d1) : "f"(a0), "f"(a1), "f"(b0), "f"(b1), "f"(c0), "f"(c1));
}
__device__ __forceinline__ void add2(float& d0, float& d1, float a0, float a1, float b0, float b1) {
  asm("{\n\t.reg .b64 ra, rb, rd;\n\t"
      "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\t"
      "mov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d0), "=f"(d1) : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// 2^y for a pair of values on the FMA / ALU pipes instead of the special-function unit: split y into its
// nearest integer (added to the exponent field) and a remainder in [-0.5, 0.5] (degree-3 minimax polynomial,
// relative error 7.6e-5, far below the bf16 rounding of P).  y is the fp32 argument the special-function unit gets, rounded
// once, however large the logits are.  It is clamped at -125 so that the exponent stays in range; that turns an underflowing
// probability into 2^-125 instead of 0.
__device__ __forceinline__ void ex2_poly2(float y0, float y1, float& p0, float& p1) {
  const float kMagic = 12582912.f;    // 1.5 * 2^23: adding it leaves round(y) in the low mantissa bits
  y0 = fmaxf(y0, -125.f); y1 = fmaxf(y1, -125.f);
  float r0, r1, i0, i1, f0, f1, q0, q1;
  add2(r0, r1, y0, y1, kMagic, kMagic);
  add2(i0, i1, r0, r1, -kMagic, -kMagic);
  add2(f0, f1, y0, y1, -i0, -i1);
  fma2(q0, q1, f0, f1, 0.05520550534129143f, 0.05520550534129143f, 0.24261397123336792f, 0.24261397123336792f);
  fma2(q0, q1, q0, q1, f0, f1, 0.6932547688484192f, 0.6932547688484192f);
  fma2(q0, q1, q0, q1, f0, f1, 0.9999276995658875f, 0.9999276995658875f);
  // (a multiply-add for shift and add; of the magic number nothing is left in the upper bits)
  int b0, b1;
  asm("mad.lo.s32 %0, %1, 8388608, %2;" : "=r"(b0) : "r"(__float_as_int(r0)), "r"(__float_as_int(q0)));
  asm("mad.lo.s32 %0, %1, 8388608, %2;" : "=r"(b1) : "r"(__float_as_int(r1)), "r"(__float_as_int(q1)));
  p0 = __int_as_float(b0);
  p1 = __int_as_float(b1);
}

// Sweep 1 over one S row held in TMEM (4 chunks of 32 columns, next chunk in flight while one is reduced).
__device__ __forceinline__ float sweep_max(uint32_t tS) {
  uint32_t ra[32], rb[32];
  float mx0 = -CUDART_INF_F, mx1 = -CUDART_INF_F;
  tmem_ld32(tS, ra);
  tc_wait_ld();
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    uint32_t* cur = (c & 1) ? rb : ra;
    uint32_t* nxt = (c & 1) ? ra : rb;
    if (c < 3) tmem_ld32(tS + (c + 1) * 32, nxt);
#pragma unroll
    for (int q = 0; q < 32; q += 4) {
      mx0 = max3(mx0, __uint_as_float(cur[q]), __uint_as_float(cur[q + 1]));
      mx1 = max3(mx1, __uint_as_float(cur[q + 2]), __uint_as_float(cur[q + 3]));
    }
    if (c < 3) tc_wait_ld();
  }
  return fmaxf(mx0, mx1);
}

// The maximum over the active entries, as small code: it runs on the first tile of a list and where the bound was exceeded.
__device__ __forceinline__ float sweep_max_masked(uint32_t tS, uint4 bits) {
  float mx0 = -CUDART_INF_F, mx1 = -CUDART_INF_F;
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    const uint32_t word = bits.x;
    bits.x = bits.y; bits.y = bits.z; bits.z = bits.w;
    if (!__any_sync(0xFFFFFFFFu, word != 0u)) continue;
    uint32_t cur[32];
    tmem_ld32(tS + c * 32, cur);
    tc_wait_ld();
#pragma unroll
    for (int q = 0; q < 32; q += 4) {
      const float v0 = ((word >> q) & 1u) ? __uint_as_float(cur[q]) : -CUDART_INF_F;
      const float v1 = ((word >> (q + 1)) & 1u) ? __uint_as_float(cur[q + 1]) : -CUDART_INF_F;
      const float v2 = ((word >> (q + 2)) & 1u) ? __uint_as_float(cur[q + 2]) : -CUDART_INF_F;
      const float v3 = ((word >> (q + 3)) & 1u) ? __uint_as_float(cur[q + 3]) : -CUDART_INF_F;
      mx0 = max3(mx0, v0, v1); mx1 = max3(mx1, v2, v3);
    }
  }
  return fmaxf(mx0, mx1);
}

// 32 probabilities p = 2^(s * scale + neg_m), zero where the mask bit is clear, packed to bf16; their sums are taken in fp32,
// before the bf16 rounding.  Of every 8, 6 go through the special-function unit and 2 through the polynomial.
template <bool MASKED>
__device__ __forceinline__ void exp_chunk(const uint32_t* cur, uint32_t word, float scale, float neg_m, uint32_t* pk,
                                          float& s0, float& s1, float& s2, float& s3) {
#pragma unroll
  for (int q = 0; q < 32; q += 8) {
    float y[8], p[8];
    constexpr int kEx2 = 8 - kPolyPer8;
#pragma unroll
    for (int u = 0; u < 8; u += 2)
      fma2(y[u], y[u + 1], __uint_as_float(cur[q + u]), __uint_as_float(cur[q + u + 1]), scale, scale, neg_m, neg_m);
#pragma unroll
    for (int u = 0; u < kEx2; ++u) p[u] = ex2(y[u]);
#pragma unroll
    for (int u = kEx2; u < 8; u += 2) ex2_poly2(y[u], y[u + 1], p[u], p[u + 1]);
    if (MASKED) {
#pragma unroll
      for (int u = 0; u < 8; ++u) p[u] = ((word >> (q + u)) & 1u) ? p[u] : 0.f;
    }
    add2(s0, s1, s0, s1, p[0], p[1]);
    add2(s2, s3, s2, s3, p[2], p[3]);
    add2(s0, s1, s0, s1, p[4], p[5]);
    add2(s2, s3, s2, s3, p[6], p[7]);
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      __nv_bfloat162 h = __floats2bfloat162_rn(p[u], p[u + 1]);
      pk[(q + u) >> 1] = *reinterpret_cast<uint32_t*>(&h);
    }
  }
}

// Sweep 2: the probabilities of the halves [lo, hi) of a row, stored over the first 64 columns of the row's S (those of the
// first half over columns of the first half, which is in registers by then); a half that is inactive for every row of the
// warp is zero.  Bound by the latency of its chains: a half is one block of straight code without votes or branches, so that
// the arithmetic of one chunk runs under the exponentials of the other.  With a vote per chunk of 32 columns, to skip
// the inactive ones, a masked tile took 1584 cycles in a warp alone on its scheduler and 2334 beside another, now 1230 and
// 1988; an unmasked one takes 1190 and 1940.  So the tiles of a mask that are active throughout go the same way: a copy without
// the selects is 4 KB of code that the other roles' has to share the instruction cache with (8192 tokens 87.2 -> 83.8 us, 32768 tokens
// 347 -> 340, 131072 tokens 1670 -> 1637, head_dim 64 117 -> 112).  MASKED = false is for lists of active tiles alone.
template <bool MASKED>
__device__ __forceinline__ float sweep_exp(uint32_t tS, const uint4& bits, int lo, int hi, float scale, float neg_m) {
  float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 1
  for (int h = lo; h < hi; ++h) {
    uint32_t ra[32], rb[32], pk[32];
    tmem_ld32(tS + 64 * h, ra);
    tmem_ld32(tS + 64 * h + 32, rb);
    tc_wait_ld();
    exp_chunk<MASKED>(ra, h ? bits.z : bits.x, scale, neg_m, pk, s0, s1, s2, s3);
    exp_chunk<MASKED>(rb, h ? bits.w : bits.y, scale, neg_m, pk + 16, s0, s1, s2, s3);
    tmem_st32(tS + 32 * h, pk);
  }
  if (MASKED && hi - lo < 2) {
    uint32_t z[32];
#pragma unroll
    for (int q = 0; q < 32; ++q) z[q] = 0u;
    if (hi < 2) tmem_st32(tS + 32, z);
    if (lo > 0) tmem_st32(tS, z);
  }
  return (s0 + s1) + (s2 + s3);
}

// RANGED: only the work items whose first row lies in the row range of their sequence are processed.
// D: head_dim, 128 or 64.  With 64 a Q / K / V tile is one 16 KB box of the tensor maps, S = Q K^T takes four MMAs instead of
// eight and O has 64 columns.
template <int RANGED, int D>
__global__ void __launch_bounds__(kThreads, 1)
attn_sm100_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                  const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmG, const AttnParams prm,
                  const __grid_constant__ DamRowRanges rows) {
  using Smem = SmemLayout<RANGED, D>;
  constexpr uint32_t kSlots = Smem::kSlots, kSlotBytes = Smem::kSlotBytes;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = smem_raw;
  const uint32_t sbase = smem_u32(smem);
  const uint32_t sQ = sbase + Smem::q;
  const uint32_t sSlots = sbase + Smem::slots;
  const uint32_t bar0 = sbase + Smem::bars;
  const uint32_t bSlotFull = bar0, bSlotEmpty = bSlotFull + 8 * kSlots, bClaim = bSlotEmpty + 8 * kSlots;
  const uint32_t bQFull = bClaim + 8, bQEmpty = bQFull + 16, bSFull = bQEmpty + 16, bPFull = bSFull + 16, bOFinal = bPFull + 16;
  const uint32_t bOFree = bOFinal + 16, bRow = bOFree + 16, bRecFull = bRow + 16, bRecEmpty = bRecFull + 16;
  volatile uint32_t* step_desc = reinterpret_cast<volatile uint32_t*>(smem + Smem::step_desc);
  ItemRec* item_rec = reinterpret_cast<ItemRec*>(smem + Smem::item_rec);
  float2* stat = reinterpret_cast<float2*>(smem + Smem::stat);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + Smem::tmem_slot);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + Smem::abort_flag);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const unsigned char* blob = prm.blob;
  const DamHeader* H = reinterpret_cast<const DamHeader*>(blob);
  const int nitems = H->prows;
  const uint32_t* tiles = reinterpret_cast<const uint32_t*>(blob + H->off_tiles);
  // a blob with gathered-column tiles needs the larger scratch: nothing is computed without it, and the status
  // word says why (the gather kernel is not even launched when the scratch holds no tile at all).  The kernel in front
  // clears that word: the error is written, and the CTA ends, only after it.  (The blob itself may be read before: the
  // kernel in front lets this one begin after its own wait for the kernels that wrote the blob.)
  if ((H->flags & DAM_FLAG_GATHER) && H->attn_scratch_bytes > prm.scratch_bytes) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (blockIdx.x == 0 && tid == 0) atomicMax(prm.status, (uint32_t)DAM_ERR_BUFFER_TOO_SMALL);
    return;
  }
  // Dynamic scheduling: the work list is sorted longest first; the scheduler takes positions from a global counter (the
  // first one is the CTA index) and hands a record of each to the other roles through a two-entry ring in shared memory.
  const bool row_list = RANGED && nitems <= 32 * Smem::kBitWords;
  uint32_t* row_bits = reinterpret_cast<uint32_t*>(smem + Smem::row_bits);

  if (tid == 0) {
    for (int s = 0; s < kSlots; ++s) { mbar_init(bSlotFull + 8 * s, 1); mbar_init(bSlotEmpty + 8 * s, 1); }
    mbar_init(bClaim, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(bQFull + 8 * s, 1); mbar_init(bQEmpty + 8 * s, 1); mbar_init(bSFull + 8 * s, 1); mbar_init(bPFull + 8 * s, 4);
      mbar_init(bOFinal + 8 * s, 1); mbar_init(bOFree + 8 * s, 4); mbar_init(bRow + 8 * s, 4);
      mbar_init(bRecFull + 8 * s, 1); mbar_init(bRecEmpty + 8 * s, 13);       // producer, 8 softmax warps, 4 output warps
    }
    *abort_flag = 0u;
    mbar_fence_init();
    tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV); tma_prefetch_desc(&tmG);
  }
  if (warp == 0) { tmem_alloc(smem_u32(tmem_slot), kTmemCols); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // launched as a programmatic dependent of the kernel that gathers the matched columns: everything above ran
  // under that kernel's tail; its tiles (and the cleared work counter) are visible from here on
  asm volatile("griddepcontrol.wait;" ::: "memory");

  // Row ranges: every CTA marks the items of the work list that lie inside them, and the schedulers claim the k-th marked
  // one.  With every position claimed and the others skipped, a position cost the producer three dependent reads and the
  // nine consumers a hand-over (2048 of 26624 rows, 256 of 3328 items: 65.1 us a pass, now 52.9).
  if (row_list) {
    const uint4* list = reinterpret_cast<const uint4*>(blob + H->off_work);
    const int nwords = (nitems + 31) >> 5;
    for (int x0 = warp; x0 < nwords; x0 += 4 * (kThreads / 32)) {
      int qb0[4], seq[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int w = (x0 + k * (kThreads / 32)) * 32 + lane;
        qb0[k] = 0; seq[k] = -1;
        if (w < nitems) {
          qb0[k] = (int)__ldg(&list[2 * (size_t)w].z);
          seq[k] = (int)(__ldg(&list[2 * (size_t)w + 1].w) & 0x7FFFFFFFu);
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int x = x0 + k * (kThreads / 32);
        const uint32_t bits = __ballot_sync(0xFFFFFFFFu, seq[k] >= 0 && rows.holds(prm.ranges, seq[k], qb0[k]));
        if (lane == 0 && x < nwords) row_bits[x] = bits;
      }
    }
    __syncthreads();
  }

  // Registers are handed out per warpgroup: 72 a thread for the single-thread roles, 184 for the softmax and 72 for the
  // output warps (72 * 128 + 2 * 184 * 128 + 72 * 128 = the 128 * 512 the CTA starts with).
  if (warp < 4) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (elect_one()) {
      uint32_t sc = 0, step = 0;                             // K / V tiles loaded; steps
      bool ok = true;
      for (uint32_t n = 0;; ++n) {
        const uint32_t slot = n & 1u;
        if (!(ok = mbar_wait(bRecFull + 8 * slot, (n >> 1) & 1u, abort_flag))) break;
        const ItemRec& rec = item_rec[slot];
        const Item it = item_from_words(rec.u, rec.v);
        const int2 lone = rec.lone;
        const int lone_from = rec.lone_from, gath_row = rec.gath_row;
        const uint32_t eA = rec.e[0][0], eB = rec.e[1][0];
        mbar_arrive(bRecEmpty + 8 * slot);
        if (it.head < 0) break;
        const int kvh = it.head / prm.group;
        const Lone lA(lone, lone_from, it.a0, it.qb0, it.S), lB(lone, lone_from, it.b0, it.qb0 + 1, it.S);
        TileWalk A(tiles, it.a0, it.a1, lA, eA, it.tok0), B(tiles, it.b0, it.b1, lB, eB, it.tok0);
        uint32_t first = 3u;                                 // streams (bit 0: A, bit 1: B) that have had no tile yet
        bool claim = true;
        // the steps: the next tile of either block, loaded once where it is the same one
#pragma unroll 1
        while (ok) {
          uint32_t d = 0u, ra = 0u, rb = 0u;
          if (A.more()) { ra = A.next(it.tok0, gath_row); d |= kStepTile | (A.more() ? 0u : kStepLast); }
          if (B.more()) { rb = B.next(it.tok0, gath_row); d |= 2u * (kStepTile | (B.more() ? 0u : kStepLast)); }
          if (!d) break;
          const bool dual = (d & 3u) == 3u && ra != rb;
          if (!(d & 1u)) ra = rb;
          // the next item is claimed when a step or two are still to come
          if (claim && A.left() <= 1u && B.left() <= 1u) { mbar_arrive(bClaim); claim = false; }
          // (visible to the issuer once the step's K tile has landed)
          step_desc[step++ & 15u] = d | (d & first) * kStepFirst | (dual ? kStepDual : 0u);
          first &= ~d;
          const int nload = dual ? 4 : 2;
#pragma unroll 1
          for (int v = 0; v < nload; ++v) {                  // K, V
            const bool isV = 2 * v >= nload;
            const uint32_t s = sc % kSlots, bar = bSlotFull + 8 * s, dst = sSlots + s * kSlotBytes;
            if (!(ok = mbar_wait(bSlotEmpty + 8 * s, ((sc / kSlots) & 1u) ^ 1u, abort_flag))) break;
            ++sc;
            mbar_arrive_expect_tx(bar, DAM_TILE * D * 2);
            const uint32_t r = dual && (v & 1) ? rb : ra;
            const bool gathered = r >> 31;
            const CUtensorMap* tm = gathered ? &tmG : isV ? &tmV : &tmK;
            const int head = gathered ? 0 : kvh, r0 = (int)(r & 0x7FFFFFFFu) + (gathered && isV ? DAM_TILE : 0);
            tma_load_3d(dst, tm, bar, 0, head, r0);
            if (D == 128) tma_load_3d(dst + 16384, tm, bar, 64, head, r0);
          }
        }
        if (!ok) break;
        if (claim) mbar_arrive(bClaim);                      // an item without steps
      }
      if (ok && mbar_wait(bSlotEmpty + 8 * (sc % kSlots), ((sc / kSlots) & 1u) ^ 1u, abort_flag)) {
        step_desc[step & 15u] = kStepEnd;
        mbar_arrive(bSlotFull + 8 * (sc % kSlots));
      } else {
        // drain: copies already issued still write into shared memory; wait for them (bounded)
        uint32_t dummy = 0;
#pragma unroll 1
        for (uint32_t k = sc < kSlots ? 0u : sc - kSlots; k < sc; ++k)
          mbar_wait(bSlotFull + 8 * (k % kSlots), (k / kSlots) & 1u, &dummy, kDrainPolls);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    // (the lane is elected, not `lane == 0`: see elect_one.  32k-token layer 558 -> 491 us, mixed-length batch
    // 1827 -> 1506 us, dense list 2150 -> 1960 us)
    if (elect_one()) {
      const uint32_t idesc_qk = idesc_bf16_f32(128, 128, 0);
      const uint32_t idesc_pv = idesc_bf16_f32(128, D, 1);
      uint32_t sc = 0, step = 0;
      uint32_t p_ph = 0, q_ph = 0;         // bit X: parity of the P tiles of stream X, of its items
      bool ok = true;
      // descriptors: the high words are invariant, the low words step by (byte offset >> 4)
      const uint64_t dQ = smem_desc_sw128(sQ, 16, 1024);
      const uint64_t dK = smem_desc_sw128(sSlots, 16, 1024);
      const uint64_t dV = smem_desc_sw128(sSlots, 16384, 1024);
      const uint32_t dQ_lo = (uint32_t)dQ, dQ_hi = (uint32_t)(dQ >> 32);
      const uint32_t dK_lo = (uint32_t)dK, dK_hi = (uint32_t)(dK >> 32);
      const uint32_t dV_lo = (uint32_t)dV, dV_hi = (uint32_t)(dV >> 32);
      // One trip: P V of step d, S of step dn, the streams in turn (the code of both is there once: it is fetched again for
      // every trip, between the softmax warps' code).
      uint32_t d = 0, dn = 0, sv = 0, sk = 0;                // sv, sk: positions in the ring of the V tile(s) of d, the K tile(s) of dn
      auto slot_wait = [&](uint32_t at) -> bool { return mbar_wait(bSlotFull + 8 * (at % kSlots), (at / kSlots) & 1u, abort_flag); };
      auto slot_free = [&](uint32_t at) { tc_commit(bSlotEmpty + 8 * (at % kSlots)); };
      for (;;) {
        // K of the next step, then V of this one: they are there long before P, and between P V and S nothing is waited for.
        // A step's descriptor is readable once its K tile (or the end mark in its place) is there.
        if (d) {
          sv = sc;
          sc += (d & kStepDual) ? 2u : 1u;
        }
        sk = sc;
        // K that is late is waited for between the P V of A and of B, but not behind B's last tile: the next K may then come
        // from a record that the output warps free, and they wait for that P V.  Such a step is a trip of its own (dn = 0),
        // S of the next one another (d = 0).  Never waiting there costs 8192 tokens 84.3 -> 86.6 us.
        bool have = mbar_try_wait(bSlotFull + 8 * (sk % kSlots), (sk / kSlots) & 1u);
        if (d ? !(ok = slot_wait(sv)) : !have && !(ok = have = slot_wait(sk))) break;
        dn = have ? step_desc[step & 15u] : 0u;
#pragma unroll
        for (int X = 0; X < 2; ++X) {
          const uint32_t dx = d >> X, bX = 8 * X;
          const uint32_t v = X && (d & kStepDual) ? sv + 1u : sv;
          if (dx & kStepTile) {
            if (X && (d & kStepDual) && !(ok = slot_wait(v))) break;
            const uint32_t fresh = (dx & kStepFirst) ? 1u : 0u;
            // the output warps have read the O of the stream's last item
            if (fresh && !(ok = mbar_wait(bOFree + bX, (q_ph >> X) & 1u, abort_flag))) break;
            if (!(ok = mbar_wait(bPFull + bX, (p_ph >> X) & 1u, abort_flag))) break;
            p_ph ^= 1u << X;
            tc_fence_after();
            const uint32_t b0 = dV_lo + (v % kSlots) * (kSlotBytes >> 4), o = tmem + kColO + X * 128, a = tmem + kColS + X * 128;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
              // V is MN-major: 16 keys per step = 2048 bytes; 64-column halves 16384 bytes apart
              mma_ts_lh(o, a + ks * 8, b0 + ks * (2048 >> 4), dV_hi, idesc_pv, ks > 0 ? 1u : fresh ^ 1u);
            // a stream's output is final right after the P V of its last tile
            if (dx & kStepLast) tc_commit(bOFinal + bX);
          }
          if (X == 0) {
            if (!have && !(d & 2u * kStepLast)) {
              if (!(ok = have = slot_wait(sk))) break;
              dn = step_desc[step & 15u];
            }
            if (have) {
              ++step;
              sc += (dn & kStepDual) ? 2u : 1u;
            }
          }
          const uint32_t nx = dn >> X, k = X && (dn & kStepDual) ? sk + 1u : sk;
          if (X && (dn & kStepDual) && !(ok = slot_wait(k))) break;
          if (nx & kStepTile) {
            if (nx & kStepFirst) {
              if (!(ok = mbar_wait(bQFull + bX, (q_ph >> X) & 1u, abort_flag))) break;
              q_ph ^= 1u << X;
            }
            tc_fence_after();
            const uint32_t a0 = dQ_lo + X * (kSlotBytes >> 4), b0 = dK_lo + (k % kSlots) * (kSlotBytes >> 4), o = tmem + kColS + X * 128;
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
              const uint32_t off = ((ks >> 2) * 16384 + (ks & 3) * 32) >> 4;
              mma_ss_lh(o, a0 + off, dQ_hi, b0 + off, dK_hi, idesc_qk, ks > 0 ? 1u : 0u);
            }
            tc_commit(bSFull + bX);
            if (nx & kStepLast) tc_commit(bQEmpty + bX);
          }
          if (X ? d != 0u : (d & kStepDual) != 0u) slot_free(v);
          if (X ? have && !(dn & kStepEnd) : (dn & kStepDual) != 0u) slot_free(k);
        }
        if (!ok || (dn & kStepEnd)) break;
        d = dn;
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ scheduler
    // Claims the next position of the work list when the producer is near the end of the current one, reads what the other
    // roles need of it (three dependent reads that none of them waits for), and loads the query tiles as soon as the last S
    // of a stream is there.
    if (elect_one()) {
      int row_word = 0, row_seen = 0;
      uint32_t q_ph = 0;                                     // bit X: parity of the Q tiles of stream X
      uint32_t claims = 0;
      for (uint32_t n = 0;; ++n) {
        const uint32_t slot = n & 1u;
        if (n > 0 && !mbar_wait(bClaim, (n - 1u) & 1u, abort_flag)) break;
        if (!mbar_wait(bRecEmpty + 8 * slot, ((n >> 1) & 1u) ^ 1u, abort_flag)) break;
        ItemRec& rec = item_rec[slot];
        uint4 u, v;
        int w;
        do {
          w = claims++ == 0 ? (int)blockIdx.x : (int)(gridDim.x + atomicAdd(prm.work_counter, 1u));
          if (row_list) {
            const int nwords = (nitems + 31) >> 5;              // (claims grow: the words before row_word hold row_seen marks)
            while (row_word < nwords && row_seen + __popc(row_bits[row_word]) <= w) row_seen += __popc(row_bits[row_word++]);
            if (row_word < nwords) {
              uint32_t left = row_bits[row_word];
              for (int k = row_seen; k < w; ++k) left &= left - 1u;
              w = 32 * row_word + __ffs(left) - 1;
            } else {
              w = nitems;
            }
          }
          if (w >= nitems) break;
          const uint4* src = reinterpret_cast<const uint4*>(blob + H->off_work) + 2 * (size_t)w;
          u = __ldg(src); v = __ldg(src + 1);
        } while (RANGED && !row_list && !rows.holds(prm.ranges, (int)(v.w & 0x7FFFFFFFu), (int)u.z));
        if (w >= nitems) {
          rec.u.x = 0xFFFFFFFFu;
          mbar_arrive(bRecFull + 8 * slot);
          break;
        }
        const Item it = item_from_words(u, v);
        rec.u = u; rec.v = v;
        const DamSeq sq = reinterpret_cast<const DamSeq*>(blob + H->off_seq)[it.seq];
        int4 lone = make_int4(-1, 0, 0x7FFFFFFF, 0);
        if (H->off_lone) lone = __ldg(reinterpret_cast<const int4*>(blob + H->off_lone) + it.seq * H->num_q_heads + it.head);
#pragma unroll
        for (int X = 0; X < 2; ++X) {
          const uint32_t t0 = X ? it.b0 : it.a0, t1 = X ? it.b1 : it.a1;
          const Lone ln(make_int2(lone.x, lone.y), lone.z, t0, it.qb0 + X, it.S);
#pragma unroll
          for (uint32_t k = 0; k < 2; ++k) {
            const uint32_t t = t0 + k >= ln.at ? t0 + k + ln.n : t0 + k;
            rec.e[X][k] = t < t1 ? __ldg(tiles + t) : 0u;
          }
        }
        rec.lone = make_int2(lone.x, lone.y);
        rec.lone_from = lone.z;
        rec.hb = dam_head_bits(blob, H, sq, it.head);
        // gathered-column tiles of this (sequence, head): K tile at rows (2T) * 128, V tile at (2T + 1) * 128
        rec.gath_row = (int)(((long long)sq.gath_off + (long long)it.head * sq.nL) * 2 * DAM_TILE);
        mbar_arrive(bRecFull + 8 * slot);
        bool ok = true;
#pragma unroll 1
        for (int X = 0; X < 2 && ok; ++X) {
          if (X ? it.b0 == it.b1 : it.a0 == it.a1) continue;
          const uint32_t bar = bQFull + 8 * X, dst = sQ + X * kSlotBytes;
          const int row = it.tok0 + (it.qb0 + X) * DAM_TILE;
          if (!(ok = mbar_wait(bQEmpty + 8 * X, ((q_ph >> X) & 1u) ^ 1u, abort_flag))) break;
          q_ph ^= 1u << X;
          mbar_arrive_expect_tx(bar, DAM_TILE * D * 2);
          tma_load_3d(dst, &tmQ, bar, 0, it.head, row);
          if (D == 128) tma_load_3d(dst + 16384, &tmQ, bar, 64, it.head, row);
        }
        if (!ok) break;
      }
      if (*abort_flag) {
        // drain: copies already issued still write into shared memory; wait for them (bounded)
        uint32_t dummy = 0;
#pragma unroll 1
        for (int X = 0; X < 2; ++X) mbar_wait(bQFull + 8 * X, ((q_ph >> X) & 1u) ^ 1u, &dummy, kDrainPolls);
      }
    }
  }
  } else if (warp < 12) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 184;");
    // ------------------------------------------------------------------ softmax warps
    const int X = (warp - 4) >> 2;                           // stream: 0 = block 2p, 1 = block 2p+1
    const int r = (warp & 3) * 32 + lane;                    // row of the tile = TMEM lane
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t tS = tmem + lane_addr + kColS + X * 128;
    const uint32_t tO = tmem + lane_addr + kColO + X * 128;
    const uint32_t bS = bSFull + 8 * X, bP = bPFull + 8 * X;
    // An all-ones blob has a copy of this role to itself, in which a tile without a mask goes without selects: 8192 tokens 531 ->
    // 518 us, 32768 tokens 8.30 -> 8.08 ms.  (As a branch for each tile the copy costs the other lists 1-2 %, beside the role 0.2 %.)
    auto softmax = [&](auto all_ones_c) {
    constexpr bool all_ones = decltype(all_ones_c)::value;
    uint32_t cS = 0, cO = 0;
    bool ok = true;
    for (uint32_t n = 0; ok; ++n) {
      const uint32_t slot = n & 1u;
      if (!(ok = mbar_wait(bRecFull + 8 * slot, (n >> 1) & 1u, abort_flag))) break;
      const ItemRec& rec = item_rec[slot];
      const Item it = item_from_words(rec.u, rec.v);
      const DamHeadBits hb = rec.hb;
      uint32_t e = rec.e[X][0], e_nx = rec.e[X][1];          // entries of the next tile and of the one behind it
      const int2 lone = rec.lone;
      const int lone_from = rec.lone_from;
      __syncwarp();
      if (lane == 0) mbar_arrive(bRecEmpty + 8 * slot);               // the whole warp has read the record
      if (it.head < 0) break;
      const int qb = it.qb0 + X;
      const uint32_t t0 = X ? it.b0 : it.a0;
      uint32_t t1 = X ? it.b1 : it.a1;
      const int i = qb * DAM_TILE + r;
      const bool row_valid = i < it.S;
      if (t0 == t1) continue;
      float m_ref = -CUDART_INF_F;   // reference max (scaled, log2 domain) that P and O are expressed against
      float l = 0.f;
      // The mask words of a tile come from global memory: they are fetched one tile ahead, without branches, from what is
      // the same for all tiles of the row (dam_tile_row_bits says what they are): four words of the true mask or of the
      // matched columns, and a window of the reversed diagonals that moves by four words from tile to tile.
      const uint32_t* wide = i < hb.L ? hb.M + (size_t)i * hb.W : hb.V;
      const int wide_end = row_valid && (i < hb.L || i < hb.gather_from) ? hb.L : 0;      // keys below this one
      const int dx = hb.L - 1 - i, dw = row_valid && i >= hb.L ? dx >> 5 : 0x40000000;
      auto tile_bits = [&](uint32_t e, bool& need) -> uint4 {
        const uint32_t kind = e >> 28;
        const int kb = (int)(e & 0x0FFFFFFFu);
        if (kind == DAM_KIND_PARTIAL) {
          need = true;
          uint4 b = make_uint4(0u, 0u, 0u, 0u);
          if (kb * DAM_TILE < wide_end) b = __ldg(reinterpret_cast<const uint4*>(wide) + kb);
          const int w = dw + 4 * kb;
          uint32_t v[5];
#pragma unroll
          for (int k = 0; k < 5; ++k) v[k] = (uint32_t)(w + k) < (uint32_t)hb.W ? __ldg(hb.Drev + w + k) : 0u;
          b.x |= __funnelshift_r(v[0], v[1], dx);
          b.y |= __funnelshift_r(v[1], v[2], dx);
          b.z |= __funnelshift_r(v[2], v[3], dx);
          b.w |= __funnelshift_r(v[3], v[4], dx);
          return b;
        }
        // the first n: of a gathered tile, the columns it holds; of a full one, the keys that exist (and not beyond the row)
        int n = kind == DAM_KIND_GATHERED ? (int)((e >> 16) & 0xFFu) + 1 : it.S - kb * DAM_TILE;
        if (kind == DAM_KIND_FULL && prm.causal) n = min(n, i - kb * DAM_TILE + 1);
        need = __any_sync(0xFFFFFFFFu, n < DAM_TILE);
        // rows beyond the sequence keep nothing, but do not make a tile a masked one for their warp: without a reference they would
        // have it take the masked maximum, too, in every tile (all-ones: 1000 tokens 26.6 -> 22.4 us, 3000 tokens 116.9 -> 97.5)
        if (!row_valid) n = 0;
        return dam_low_ones128(n);
      };
      // entries left out: entry t of what remains is entry t + ln.n of the list from ln.at on
      const Lone ln(lone, lone_from, t0, qb, it.S);
      t1 -= ln.n;
      auto entry = [&](uint32_t t) -> uint32_t { return __ldg(tiles + (t >= ln.at ? t + ln.n : t)); };
      // (a trip fetches the mask words of tile t and then does tile t - 1: the code for the words is there once)
      bool need_mask = false, need_nx = false;
      uint4 bits, bits_nx = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
      for (uint32_t tn = t0; tn <= t1; ++tn) {
        need_mask = need_nx;
        bits = bits_nx;
        if (tn < t1) {
          bits_nx = tile_bits(e, need_nx);
          e = e_nx;
          if (tn + 2 < t1) e_nx = entry(tn + 2);
        }
        if (tn == t0) continue;
        const uint32_t t = tn - 1;
        // the halves of the row with an active entry in some row of the warp
        const int lo = __any_sync(0xFFFFFFFFu, (bits.x | bits.y) != 0u) ? 0 : 1, hi = __any_sync(0xFFFFFFFFu, (bits.z | bits.w) != 0u) ? 2 : 1;
        if (!(ok = mbar_wait(bS, cS & 1u, abort_flag))) break;
        ++cS;
        tc_fence_after();
        // ---- sweep 1: row maximum of the raw dot products.  On a masked tile the maximum over all entries is
        //      tried first: it bounds the masked one from above, so when it does not exceed the reference by more
        //      than the threshold for any row of the warp, the reference stays where it is and the masked
        //      maximum (two more instructions per element) is never needed.  The result is the same either way.
        bool masked_max = need_mask && (t == t0);            // the first tile sets the reference
        float mx = -CUDART_INF_F;
        if (!masked_max) {
          const float mu = sweep_max(tS);
          if (!need_mask) mx = mu;
          else masked_max = __any_sync(0xFFFFFFFFu, mu * prm.scale_log2 - m_ref > kRescaleThreshold);   // -inf reference: true
        }
        if (masked_max) mx = sweep_max_masked(tS, bits);
        const float m_new = fmaxf(m_ref, mx * prm.scale_log2);
        // move the reference only on the first tile or when the max grew by more than the threshold
        bool move = (t == t0) || (m_new - m_ref > kRescaleThreshold);   // -inf reference: inf > 8 is true
        if (m_new == -CUDART_INF_F) move = false;
        float alpha = 1.f;
        if (move) {
          alpha = (m_ref == -CUDART_INF_F) ? 0.f : ex2(m_ref - m_new);
          m_ref = m_new;
        }
        const float mm = (m_ref == -CUDART_INF_F) ? 0.f : m_ref;
        // ---- sweep 2: probabilities against the reference max, packed to bf16 into the first half of S
        const float tsum = all_ones && !need_mask ? sweep_exp<false>(tS, bits, 0, 2, prm.scale_log2, -mm)
                                                  : sweep_exp<true>(tS, bits, lo, hi, prm.scale_log2, -mm);
        l = l * alpha + tsum;
        // ---- O is complete up to the previous tile of this stream (its MMAs precede S of this tile)
        if (t > t0) {
          const bool resc = alpha != 1.f;
          if (__any_sync(0xFFFFFFFFu, resc)) {
#pragma unroll 1
            for (int c = 0; c < D / 32; ++c) {
              uint32_t rr[32];
              tmem_ld32(tO + c * 32, rr);
              tc_wait_ld();
#pragma unroll
              for (int q = 0; q < 32; ++q) rr[q] = __float_as_uint(__uint_as_float(rr[q]) * alpha);
              tmem_st32(tO + c * 32, rr);
            }
          }
        }
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bP);
      }
      if (!ok) break;
      if (ln.n) {
        // ---- the lone diagonal's tile: row r needs its entry r alone, which lies in the warp's own 32-column chunk
        if (!(ok = mbar_wait(bS, cS & 1u, abort_flag))) break;
        ++cS;
        tc_fence_after();
        uint32_t v[32];
        tmem_ld32(tS + (warp & 3) * 32, v);
        tc_wait_ld();
#pragma unroll
        for (int w = 16; w >= 1; w >>= 1)
#pragma unroll
          for (int q = 0; q < w; ++q) v[q] = (lane & w) ? v[q + w] : v[q];
        const float y = row_valid ? __uint_as_float(v[0]) * prm.scale_log2 : -CUDART_INF_F;
        float alpha = 1.f;
        if (y - m_ref > kRescaleThreshold) {                 // (-inf reference: inf > 8; NaN when y is -inf too)
          alpha = (m_ref == -CUDART_INF_F) ? 0.f : ex2(m_ref - y);
          m_ref = y;
        }
        // (as in the sweeps: an infinite reference counts as zero, so that a logit of -inf gives zero and not a NaN)
        const float p = row_valid ? ex2(y - (m_ref == -CUDART_INF_F ? 0.f : m_ref)) : 0.f;
        l = l * alpha + p;
        const __nv_bfloat16 pb = __float2bfloat16_rn(p);
        const uint32_t pw = (uint32_t)*reinterpret_cast<const unsigned short*>(&pb) << (16 * (lane & 1));
        // P: zeros but for that entry
#pragma unroll
        for (int q = 0; q < 32; ++q) v[q] = 0u;
        tmem_st32(tS, v);
        tmem_st32(tS + 32, v);
        tc_wait_st();
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = q == (lane >> 1) ? pw : 0u;
        tmem_st16(tS + (warp & 3) * 16, v);
        if (t0 < t1 && __any_sync(0xFFFFFFFFu, alpha != 1.f)) {
#pragma unroll 1
          for (int c = 0; c < D / 32; ++c) {
            tmem_ld32(tO + c * 32, v);
            tc_wait_ld();
#pragma unroll
            for (int q = 0; q < 32; ++q) v[q] = __float_as_uint(__uint_as_float(v[q]) * alpha);
            tmem_st32(tO + c * 32, v);
          }
        }
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bP);
      }
      // ---- the output warps take it from here (once they have read what the item before left here)
      if (!(ok = mbar_wait(bOFree + 8 * X, (cO & 1u) ^ 1u, abort_flag))) break;
      stat[X * DAM_TILE + r] = make_float2(m_ref, l);
      ++cO;
      __syncwarp();
      if (lane == 0) mbar_arrive(bRow + 8 * X);
    }
    };
    if (H->flags & DAM_FLAG_ALL_ONES) softmax(std::true_type());
    else softmax(std::false_type());
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    // ------------------------------------------------------------------ output warps: O / l and the log-sum-exp
    // (of both streams; the next item's first tiles are in the softmax warps meanwhile)
    const int r = (warp & 3) * 32 + lane;
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    uint32_t o_ph = 0;                                       // bit X: parity of the items of stream X
    bool ok = true;
    for (uint32_t n = 0; ok; ++n) {
      const uint32_t slot = n & 1u;
      if (!(ok = mbar_wait(bRecFull + 8 * slot, (n >> 1) & 1u, abort_flag))) break;
      const Item it = item_from_words(item_rec[slot].u, item_rec[slot].v);
      __syncwarp();
      if (lane == 0) mbar_arrive(bRecEmpty + 8 * slot);
      if (it.head < 0) break;
#pragma unroll 1
      for (int X = 0; X < 2; ++X) {
        if (X == 1 && !it.hasB) break;
        const int i = (it.qb0 + X) * DAM_TILE + r;
        const bool row_valid = i < it.S;
        __nv_bfloat16* orow = prm.O + (int64_t)(it.tok0 + i) * prm.o_stride_tok + (int64_t)it.head * prm.o_stride_head;
        float* lse_p = prm.lse + (int64_t)it.head * prm.total_tokens + it.tok0 + i;
        if (X ? it.b0 == it.b1 : it.a0 == it.a1) {
          if (row_valid) {
            const uint4 z = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
            for (int c = 0; c < D / 8; ++c) reinterpret_cast<uint4*>(orow)[c] = z;
            *lse_p = -CUDART_INF_F;
          }
          continue;
        }
        if (!(ok = mbar_wait(bRow + 8 * X, (o_ph >> X) & 1u, abort_flag))) break;
        const float2 ml = stat[X * DAM_TILE + r];
        if (!(ok = mbar_wait(bOFinal + 8 * X, (o_ph >> X) & 1u, abort_flag))) break;
        o_ph ^= 1u << X;
        tc_fence_after();
        const float inv = ml.y > 0.f ? 1.0f / ml.y : 0.f;
        const uint32_t tO = tmem + lane_addr + kColO + X * 128;
#pragma unroll 1
        for (int c = 0; c < D / 32; ++c) {
          uint32_t rr[32], o[16];
          tmem_ld32(tO + c * 32, rr);
          tc_wait_ld();
          if (c + 1 == D / 32) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bOFree + 8 * X);
          }
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            __nv_bfloat162 hpair = __floats2bfloat162_rn(__uint_as_float(rr[2 * q]) * inv, __uint_as_float(rr[2 * q + 1]) * inv);
            o[q] = *reinterpret_cast<uint32_t*>(&hpair);
          }
          if (row_valid) {
            if (prm.o_vec8) {
              st_global_v8(orow + c * 32, o);
              st_global_v8(orow + c * 32 + 16, o + 8);
            } else {
#pragma unroll
              for (int q = 0; q < 4; ++q)
                reinterpret_cast<uint4*>(orow)[c * 4 + q] = make_uint4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
            }
          }
        }
        if (row_valid) *lse_p = ml.y > 0.f ? (ml.x + log2f(ml.y)) * 0.6931471805599453f : -CUDART_INF_F;
      }
    }
  }

  if (blockIdx.x == 0 && tid == 64) prm.status[3] = 1u;      // word 4 of the scratch block: which kernel served the call
  tc_fence_before();
  report_expired_wait(abort_flag, prm.status, DAM_ERR_DEVICE_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

// The n-th matched column of a head, counted off its pattern words (0xFFFF: it has no more), for the blobs of an earlier
// build, which have no list.  Out of line: the hot path is a short chain of loads.
__device__ __noinline__ int nth_column(const unsigned char* dv, const DamSeq& sq, int h, int n) {
  const uint32_t* Vw = reinterpret_cast<const uint32_t*>(dv) + sq.dv_off + (uint64_t)h * 3 * sq.W + 2 * sq.W;
  for (int w = 0; w < sq.W; ++w) {
    const uint32_t word = __ldg(Vw + w);
    const int c = __popc(word);
    if (n < c) return 32 * w + (int)__fns(word, 0, n + 1);
    n -= c;
  }
  return 0xFFFF;
}

// Copies the K and V rows of the matched columns of every (sequence, head) into dense tiles of 128 keys in
// the scratch buffer (K tile at rows (2T) * 128, V tile at rows (2T + 1) * 128 of a [rows][head_dim] bf16 array;
// T = gath_off + head * nL + g).  Rows past the last matched column are zero.  One block per tile, grid-stride.
// Bound by latency: a chain of header, column index, row.  The indices are read from the list that the classification
// leaves; found here instead, from the V words by prefix counts and a search per place, they took
// another 1-1.5 us of every call (a 2048-row chunk against a 2048-token window 66.4 us, now 64.9; 1237 tokens with a
// 512-token window 59.3, now 58.6; 8192 tokens 151.2, now 149.7).
constexpr int kGatherThreads = 256;
__global__ void __launch_bounds__(kGatherThreads)
gather_columns_kernel(const unsigned char* __restrict__ blob, const __nv_bfloat16* __restrict__ K,
                      const __nv_bfloat16* __restrict__ V, int Hq, int group, int d, int64_t kst, int64_t ksh, int64_t vst,
                      int64_t vsh, unsigned char* scratch, unsigned long long scratch_bytes) {
  asm volatile("griddepcontrol.wait;" ::: "memory");     // (launched under the tail of the kernel before it)
  asm volatile("griddepcontrol.launch_dependents;");     // the attention kernel behind this one may start its prologue
  // the attention kernel's status block starts at zero
  if (blockIdx.x == 0) {
    if (threadIdx.x < 64) reinterpret_cast<uint32_t*>(scratch)[threadIdx.x] = 0u;
    __syncthreads();
  }
  const DamHeader* H = reinterpret_cast<const DamHeader*>(blob);
  if (!(H->flags & DAM_FLAG_GATHER)) return;
  if (H->attn_scratch_bytes > scratch_bytes) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicMax(reinterpret_cast<uint32_t*>(scratch) + 1, (uint32_t)DAM_ERR_BUFFER_TOO_SMALL);
    return;
  }
  __shared__ int col[DAM_TILE];
  uint4* out = reinterpret_cast<uint4*>(scratch + 256);
  const bool cols_missing = H->off_cols == 0;
  // (without a list: words of the tiles' own memory, twice 128 rows of head_dim per tile, which are not used)
  const unsigned short* cols = reinterpret_cast<const unsigned short*>(cols_missing ? scratch + 256 : blob + H->off_cols);
  const DamSeq* seqs = reinterpret_cast<const DamSeq*>(blob + H->off_seq);
  const int tid = threadIdx.x;
  for (long long T = blockIdx.x; T < (long long)H->gath_tiles; T += gridDim.x) {
    int c_mine = tid < DAM_TILE ? __ldg(cols + T * DAM_TILE + tid) : 0;
    int b = 0;
    while (b + 1 < H->num_seqs && (long long)seqs[b + 1].gath_off <= T) ++b;
    const DamSeq sq = seqs[b];
    if (sq.nL == 0) continue;
    const int h = (int)((T - (long long)sq.gath_off) / sq.nL), g = (int)((T - (long long)sq.gath_off) % sq.nL);
    if (h >= Hq) continue;
    if (cols_missing) c_mine = nth_column(blob + H->off_dv, sq, h, g * DAM_TILE + tid);
    __syncthreads();
    if (tid < DAM_TILE) col[tid] = c_mine == 0xFFFF ? -1 : c_mine;
    __syncthreads();
    if (col[0] < 0) continue;                                 // capacity tile that no row list refers to
    const __nv_bfloat16* Kh = K + (int64_t)sq.tok_start * kst + (int64_t)(h / group) * ksh;
    const __nv_bfloat16* Vh = V + (int64_t)sq.tok_start * vst + (int64_t)(h / group) * vsh;
    const int ppr = d >> 3;                                      // 16-byte pieces per row (16 at head_dim 128, 8 at 64)
    const int part = tid % ppr, r0 = tid / ppr, step = kGatherThreads / ppr;
    // eight rows of K and of V per thread are requested before the first is stored (the block is one dependent
    // chain of loads as it is; one round trip per row would be most of its time), so 256 threads request the whole tile
    // at once (128 threads, two round trips: the call at 8192 tokens 105.4 us, now 104.0)
    for (int rb = r0; rb < DAM_TILE; rb += 8 * step) {
      uint4 kv[8], vv[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = rb + u * step;
        const int c = r < DAM_TILE ? col[r] : -1;
        kv[u] = make_uint4(0u, 0u, 0u, 0u); vv[u] = kv[u];
        if (c >= 0) {
          kv[u] = __ldg(reinterpret_cast<const uint4*>(Kh + (int64_t)c * kst) + part);
          vv[u] = __ldg(reinterpret_cast<const uint4*>(Vh + (int64_t)c * vst) + part);
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = rb + u * step;
        if (r < DAM_TILE) {
          out[((size_t)(2 * T) * DAM_TILE + r) * ppr + part] = kv[u];
          out[((size_t)(2 * T + 1) * DAM_TILE + r) * ppr + part] = vv[u];
        }
      }
    }
  }
}

// The status block of a call without a gather kernel in front: a kernel, so that the chain of launches is not broken.
__global__ void clear_status_kernel(uint32_t* scratch, int keep) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");     // (late, as in the gather kernel)
  if ((int)threadIdx.x >= keep) scratch[threadIdx.x] = 0u;
}

// Self-test of the bounded waits, on mbarriers that nothing ever arrives on, a waiting thread in a warp of its own for each:
// the attention kernel's by a count of polls (a fixed number of them, timed), the scoring kernel's by the wall clock (the
// given limit), and another of those that the expired one has to release long before its own limit.  The status word is written the
// way those kernels write it, by a thread that has nothing else to do.
// words: nanoseconds of the wait by the wall clock, of the count of polls as kWaitPolls of them would take, of the released wait;
// how many of the three gave up.
__global__ void bounded_wait_selftest_kernel(uint32_t* status, unsigned long long limit_ns, unsigned long long* words) {
  constexpr uint32_t kPolls = kWaitPolls / 800;
  __shared__ uint64_t bar;
  __shared__ uint32_t flag_polls, flag_clock, gave_up;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    flag_polls = flag_clock = gave_up = 0u;
    mbar_fence_init();
  }
  __syncthreads();
  const uint64_t t0 = globaltimer_ns();
  if (threadIdx.x == 32) {
    if (!mbar_wait_slow(smem_u32(&bar), 0u, &flag_clock, limit_ns)) atomicAdd(&gave_up, 1u);
    words[0] = globaltimer_ns() - t0;
  } else if (threadIdx.x == 64) {
    if (!mbar_wait(smem_u32(&bar), 0u, &flag_polls, kPolls)) atomicAdd(&gave_up, 1u);
    words[1] = (globaltimer_ns() - t0) * (kWaitPolls / kPolls);
  } else if (threadIdx.x == 96) {
    if (!mbar_wait_slow(smem_u32(&bar), 0u, &flag_clock, 2 * limit_ns + 1000000000ull)) atomicAdd(&gave_up, 1u);
    words[2] = globaltimer_ns() - t0;
  }
  report_expired_wait(&flag_clock, status, DAM_ERR_DEVICE_TIMEOUT);
  if (threadIdx.x == 0) words[3] = flag_polls ? gave_up : 0u;
}

template <int RANGED, int D>
cudaError_t allow_smem() {
  return cudaFuncSetAttribute(attn_sm100_kernel<RANGED, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, SmemLayout<RANGED, D>::total);
}

}  // namespace

cudaError_t dam_launch_bounded_wait_selftest(void* scratch, unsigned long long limit_ns, cudaStream_t st) {
  bounded_wait_selftest_kernel<<<1, 128, 0, st>>>(reinterpret_cast<uint32_t*>(scratch) + 1, limit_ns,
                                                  reinterpret_cast<unsigned long long*>(scratch) + 1);
  return cudaGetLastError();
}

cudaError_t dam_launch_attn_sm100(const void* Q, const void* K, const void* V, const void* blob,
                                  const dam_shape_t* s, int causal, float scale, void* O, float* lse, void* scratch,
                                  size_t scratch_bytes, const int32_t* ranges, const int32_t* ranges_host, bool run_gather,
                                  cudaStream_t st) {
  const int d = s->head_dim;
  if (s->dtype != DAM_BF16 || (d != 128 && d != 64)) return cudaErrorNotSupported;
  if (s->total_tokens == 0)                              // nothing to compute: the status block starts at zero all the same
    return dam_launch_chained(clear_status_kernel, dim3(1), dim3(64), 0, st, reinterpret_cast<uint32_t*>(scratch), run_gather ? 0 : 2);
  int dev = 0;
  DamDeviceInfo di;
  cudaError_t e;
  if ((e = dam_current_device(&dev, &di)) != cudaSuccess) return e;
  if (di.cc_major != 10 || di.smem_optin < 232448) return cudaErrorNotSupported;
  if ((e = dam_device_table().once(dev, DAM_SETUP_ATTN_SMEM, [](void) -> cudaError_t {
         cudaError_t r;
         if ((r = allow_smem<0, 128>()) != cudaSuccess || (r = allow_smem<1, 128>()) != cudaSuccess || (r = allow_smem<2, 128>()) != cudaSuccess) return r;
         return (r = allow_smem<0, 64>()) != cudaSuccess ? r : allow_smem<1, 64>();
       })) != cudaSuccess)
    return e;
  const int sm_count = di.sm_count;
  // gathered-column tiles (if the blob has any) live after the 256-byte status block of the scratch buffer
  const size_t grows = scratch_bytes > 256 ? (scratch_bytes - 256) / (size_t)(d * 2) : 0;      // rows of head_dim bf16
  CUtensorMap tq, tk, tv, tg;
  const bool has_g = grows >= 2 * DAM_TILE;
  if (!dam_make_tmap_bf16(&tg, has_g ? reinterpret_cast<const unsigned char*>(scratch) + 256 : Q, d, 1,
                          has_g ? (int64_t)grows : DAM_TILE, d, d))
    return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  if (has_g && run_gather) {
    // clears the status block too
    cfg.gridDim = dim3(sm_count * 4); cfg.blockDim = dim3(kGatherThreads);
    if ((e = cudaLaunchKernelEx(&cfg, gather_columns_kernel, reinterpret_cast<const unsigned char*>(blob),
                                reinterpret_cast<const __nv_bfloat16*>(K), reinterpret_cast<const __nv_bfloat16*>(V),
                                (int)s->num_q_heads, (int)(s->num_q_heads / s->num_kv_heads), d, s->k_stride_tok, s->k_stride_head,
                                s->v_stride_tok, s->v_stride_head, reinterpret_cast<unsigned char*>(scratch),
                                (unsigned long long)scratch_bytes)) != cudaSuccess)
      return e;
  } else {
    // status word and work counter start at zero (a further row range clears the work counter only)
    if ((e = dam_launch_chained(clear_status_kernel, dim3(1), dim3(64), 0, st, reinterpret_cast<uint32_t*>(scratch),
                                run_gather ? 0 : 2)) != cudaSuccess)
      return e;
  }
  if (!dam_make_tmap_bf16(&tq, Q, d, s->num_q_heads, s->total_tokens, s->q_stride_tok, s->q_stride_head) ||
      !dam_make_tmap_bf16(&tk, K, d, s->num_kv_heads, s->total_tokens, s->k_stride_tok, s->k_stride_head) ||
      !dam_make_tmap_bf16(&tv, V, d, s->num_kv_heads, s->total_tokens, s->v_stride_tok, s->v_stride_head))
    return cudaErrorInvalidValue;
  const DamRowRanges rows(ranges ? ranges_host : nullptr, s->num_seqs);
  int pairs = 0, all = 0;                                // (of the row ranges: whole pairs, as the caller has checked)
  for (int b = 0; b < s->num_seqs; ++b) {
    const int S = s->cu_seqlens_host[b + 1] - s->cu_seqlens_host[b];
    const int r0 = ranges ? ranges_host[2 * b] : 0, r1 = ranges ? ranges_host[2 * b + 1] : S;
    pairs += (r1 - r0 + 2 * DAM_TILE - 1) / (2 * DAM_TILE);
    all += (S + 2 * DAM_TILE - 1) / (2 * DAM_TILE);
  }
  pairs *= s->num_q_heads; all *= s->num_q_heads;
  if (pairs == 0) return cudaSuccess;
  // a CTA for every pair to compute, but where the list is too long to be marked the CTAs walk all of it, and the walk is
  // what takes the time: 256 rows of 204800 tokens, 32 pairs of 25600, 32 CTAs 565 us, 148 CTAs 134
  if (all > 32 * kRowBitWordsLong) pairs = all;
  if (s->o_stride_tok >= (int64_t)1 << 39 || s->o_stride_head >= (int64_t)1 << 39) return cudaErrorInvalidValue;   // (no such memory)
  AttnParams p;
  p.blob = reinterpret_cast<const unsigned char*>(blob);
  p.O = reinterpret_cast<__nv_bfloat16*>(O);
  p.lse = lse;
  p.status = reinterpret_cast<uint32_t*>(scratch) + 1;
  p.work_counter = reinterpret_cast<uint32_t*>(scratch) + 2;
  p.scratch_bytes = scratch_bytes;
  p.ranges = ranges;
  p.group = s->num_q_heads / s->num_kv_heads; p.total_tokens = s->total_tokens;
  p.causal = causal;
  p.o_vec8 = reinterpret_cast<uintptr_t>(O) % 32 == 0 && s->o_stride_tok % 16 == 0 && s->o_stride_head % 16 == 0;
  p.o_stride_tok = s->o_stride_tok; p.o_stride_head = s->o_stride_head;
  p.scale_log2 = scale * 1.4426950408889634f;
  const int grid = pairs < sm_count ? pairs : sm_count;
  cfg.gridDim = dim3(grid); cfg.blockDim = dim3(kThreads);
  auto launch = [&](auto* kernel, int smem) -> cudaError_t {
    cfg.dynamicSmemBytes = smem;
    return cudaLaunchKernelEx(&cfg, kernel, tq, tk, tv, tg, p, rows);
  };
  if (d == 128) {
    if (!ranges) return launch(attn_sm100_kernel<0, 128>, SmemLayout<0, 128>::total);
    return all <= 32 * kRowBitWords ? launch(attn_sm100_kernel<1, 128>, SmemLayout<1, 128>::total)
                                    : launch(attn_sm100_kernel<2, 128>, SmemLayout<2, 128>::total);
  }
  return ranges ? launch(attn_sm100_kernel<1, 64>, SmemLayout<1, 64>::total) : launch(attn_sm100_kernel<0, 64>, SmemLayout<0, 64>::total);
}
