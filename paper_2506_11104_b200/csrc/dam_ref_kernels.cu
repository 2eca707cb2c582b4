// Plain CUDA-core kernels (fp32 arithmetic, any head_dim that is a multiple of 8 up to 256, bf16
// or fp32 inputs).  They serve the fp32 configuration and every shape the tensor-core kernels do
// not cover, and are the on-device cross-check for those kernels.
#include <cuda_bf16.h>
#include <math_constants.h>

#include "dam_internal.cuh"

namespace {

constexpr int kRefWarps = 8;          // warps of a block
constexpr int kFewRows = 8, kFewKeys = 8;      // attn_ref_few_kernel: rows of a block, keys of a warp in a stage

template <typename T> struct Ld8;
template <> struct Ld8<float> {
  static __device__ __forceinline__ void load(const float* p, float* o) {
    float4 a = __ldg(reinterpret_cast<const float4*>(p));
    float4 b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w; o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
  }
  static __device__ __forceinline__ float one(const float* p) { return __ldg(p); }
  static __device__ __forceinline__ void store(float* p, float v) { *p = v; }
};
template <> struct Ld8<__nv_bfloat16> {
  static __device__ __forceinline__ void load(const __nv_bfloat16* p, float* o) {
    uint4 a = __ldg(reinterpret_cast<const uint4*>(p));
    const uint32_t w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      o[2 * q] = __uint_as_float(w[q] << 16);
      o[2 * q + 1] = __uint_as_float(w[q] & 0xFFFF0000u);
    }
  }
  static __device__ __forceinline__ float one(const __nv_bfloat16* p) { return __bfloat162float(*p); }
  static __device__ __forceinline__ void store(__nv_bfloat16* p, float v) { *p = __float2bfloat16_rn(v); }
};

// The keys a block works on at a time sit in shared memory as fp32 rows.  A K row is padded by four floats: the lanes of
// a warp read four consecutive floats of 32 different rows, and since d is a multiple of 8 the row pitch in 16-byte units
// is odd, so the eight rows of a quarter warp fall into eight different bank groups.
constexpr int kStageKeys = 64;
__host__ __device__ inline int k_pitch(int d) { return d + 4; }

// rows [j0, j0 + kStageKeys) of a [tokens][d] matrix (row stride `st` elements) into fp32 rows of `pitch` floats; rows
// from `n` on are zero
template <typename T>
__device__ __forceinline__ void load_stage(float* dst, int pitch, const T* __restrict__ src, int64_t st, int j0, int n, int d) {
  const int ppr = d >> 3;                                       // pieces of 8 elements per row
  for (int x = threadIdx.x; x < kStageKeys * ppr; x += blockDim.x) {
    const int r = x / ppr, piece = x % ppr;
    float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (j0 + r < n) Ld8<T>::load(src + (int64_t)(j0 + r) * st + piece * 8, v);
    float4* o = reinterpret_cast<float4*>(dst + r * pitch + piece * 8);
    o[0] = make_float4(v[0], v[1], v[2], v[3]);
    o[1] = make_float4(v[4], v[5], v[6], v[7]);
  }
}

// The same for fp32 rows with asynchronous copies: the caller commits and waits.
__device__ __forceinline__ void load_stage_async(float* dst, int pitch, const float* __restrict__ src, int64_t st, int j0, int n, int d) {
  const int ppr = d >> 2;                                       // 16-byte pieces per row
  for (int x = threadIdx.x; x < kStageKeys * ppr; x += blockDim.x) {
    const int r = x / ppr, piece = x % ppr;
    const uint32_t to = static_cast<uint32_t>(__cvta_generic_to_shared(dst + r * pitch + piece * 4));
    const bool in = j0 + r < n;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(src + (int64_t)(in ? j0 + r : 0) * st + piece * 4),
                 "r"(in ? 16 : 0) : "memory");                  // (0 source bytes: zeros)
  }
}

// Dot products of R query rows (fp32, shared memory, d floats apart) with the keys of rows k0 and k1: one fused
// multiply-add per dimension in ascending order.
template <int R>
__device__ __forceinline__ void dot_rows(const float* q_s, const float* k0, const float* k1, int d, float (&s)[R][2]) {
#pragma unroll
  for (int r = 0; r < R; ++r) s[r][0] = s[r][1] = 0.f;
#pragma unroll 4
  for (int t = 0; t < d; t += 4) {
    const float4 a = *reinterpret_cast<const float4*>(k0 + t), b = *reinterpret_cast<const float4*>(k1 + t);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float4 q = *reinterpret_cast<const float4*>(q_s + r * d + t);
      s[r][0] = fmaf(q.x, a.x, s[r][0]); s[r][1] = fmaf(q.x, b.x, s[r][1]);
      s[r][0] = fmaf(q.y, a.y, s[r][0]); s[r][1] = fmaf(q.y, b.y, s[r][1]);
      s[r][0] = fmaf(q.z, a.z, s[r][0]); s[r][1] = fmaf(q.z, b.z, s[r][1]);
      s[r][0] = fmaf(q.w, a.w, s[r][0]); s[r][1] = fmaf(q.w, b.w, s[r][1]);
    }
  }
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

// ---------------------------------------------------------------------------------------------
// Window scores: causal softmax over the first L tokens, then the single-compare threshold.
// Two sweeps over the keys of a row (max / sum, then probabilities); the fp32 probability that is
// compared with p* is the very value written to the dump.
// ---------------------------------------------------------------------------------------------
// `nbuf` stages of K fit in shared memory: a block that needs no more loads them all at once, before the first sweep, and
// neither sweep waits again (512 tokens, PCL 128: 12.4 -> 11.3 us).  Otherwise a stage is loaded when it is due.
// Bound by latency at the sizes this path serves.  A block takes 8 R adjacent rows (R per warp) of one map and walks
// the keys in stages of 64 held in shared memory, so that a key row is read from memory once per block and not once per
// row.  R = 1 while that leaves SMs idle, 4 otherwise (a stage then feeds four times the multiply-adds).
template <typename T, int R>
__global__ void __launch_bounds__(256)
scores_ref_kernel(unsigned char* blob, const T* __restrict__ Q, const T* __restrict__ K,
                  int Hq, int group, int d, int64_t qst, int64_t qsh, int64_t kst, int64_t ksh,
                  float scale, float pstar, float* __restrict__ dump, int nbuf) {
  dam_chain_prologue();
  extern __shared__ __align__(16) float smem[];
  const DamHeader* H = reinterpret_cast<const DamHeader*>(blob);
  const int sh = blockIdx.y;
  const int b = sh / Hq, h = sh % Hq;
  const DamSeq sq = reinterpret_cast<const DamSeq*>(blob + H->off_seq)[b];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int i_block = blockIdx.x * nw * R;
  if (i_block >= sq.L) return;
  const int i_end = min(i_block + nw * R, sq.L);                // keys 0 .. i_end - 1 matter to the block
  const int i0 = i_block + warp * R;
  const int stage = kStageKeys * k_pitch(d);
  float* k_s = smem;
  float* q_s = smem + nbuf * stage + warp * R * d;
  const int nstage = (i_end + kStageKeys - 1) / kStageKeys;
  const bool resident = nstage <= nbuf;
  const T* Kh = K + (int64_t)sq.tok_start * kst + (int64_t)(h / group) * ksh;
  if (resident) for (int t = 0; t < nstage; ++t) load_stage<T>(k_s + t * stage, k_pitch(d), Kh, kst, t * kStageKeys, sq.L, d);
  for (int x = lane; x < R * d; x += 32) {
    const int i = i0 + x / d;
    q_s[x] = i < sq.L ? Ld8<T>::one(Q + (int64_t)(sq.tok_start + i) * qst + (int64_t)h * qsh + x % d) : 0.f;
  }
  if (resident) __syncthreads();
  uint32_t* M = reinterpret_cast<uint32_t*>(blob + H->off_true) + sq.true_off + (uint64_t)h * sq.L * sq.W;
  float* Ph = dump ? dump + sq.p_off + (uint64_t)h * sq.L * sq.L : nullptr;
  float m[R], l[R], mw[R];
#pragma unroll
  for (int r = 0; r < R; ++r) { m[r] = -CUDART_INF_F; l[r] = 0.f; mw[r] = 0.f; }
  const float* k0 = k_s + lane * k_pitch(d);
  const float* k1 = k0 + 32 * k_pitch(d);
  for (int sweep = 0; sweep < 2; ++sweep) {
    for (int t = 0; t < nstage; ++t) {
      const int j0 = t * kStageKeys;
      if (!resident) {
        __syncthreads();
        load_stage<T>(k_s, k_pitch(d), Kh, kst, j0, sq.L, d);
        __syncthreads();
      }
      float s[R][2];
      const int at = resident ? t * stage : 0;
      dot_rows<R>(q_s, k0 + at, k1 + at, d, s);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int j = j0 + c * 32 + lane;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int i = i0 + r;
          const float x = s[r][c] * scale;
          if (sweep == 0) {
            if (j <= i) {
              const float mn = fmaxf(m[r], x);
              l[r] = l[r] * expf(m[r] - mn) + expf(x - mn);
              m[r] = mn;
            }
          } else {
            const float p = j <= i ? expf(x - mw[r]) / l[r] : 0.f;
            if (Ph && i < sq.L && j < sq.L) Ph[(uint64_t)i * sq.L + j] = p;
            const uint32_t word = __ballot_sync(0xFFFFFFFFu, p >= pstar);
            if (lane == 0 && i < sq.L && (j0 >> 5) + c < sq.W) M[(size_t)i * sq.W + (j0 >> 5) + c] = word;
          }
        }
      }
    }
    if (sweep == 0) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        mw[r] = warp_max(m[r]);
        l[r] = warp_sum((m[r] == -CUDART_INF_F) ? 0.f : l[r] * expf(m[r] - mw[r]));
      }
    }
  }
  // words (and map cells) to the right of the stages the block visited lie above the diagonal
  for (int r = 0; r < R; ++r) {
    const int i = i0 + r;
    if (i >= sq.L) break;
    for (int w = nstage * (kStageKeys / 32) + lane; w < sq.W; w += 32) M[(size_t)i * sq.W + w] = 0u;
    if (Ph) for (int j = nstage * kStageKeys + lane; j < sq.L; j += 32) Ph[(uint64_t)i * sq.L + j] = 0.f;
  }
}

// ---------------------------------------------------------------------------------------------
// Masked attention over the listed tiles, online softmax in fp32.  A block takes 8 R adjacent rows (R per warp) of one
// (head, q-block) row of the tile list and walks its tiles in stages of 64 keys whose K and V rows sit in shared memory;
// a stage without an active cell in the block's rows is not loaded.  The lanes of a warp are keys for the scores and
// dimensions for the output.  For many rows (R = 4; attn_ref_few_kernel serves few).
// PIPE (fp32, two stages fit in shared memory): the next stage with an active cell is looked for and its copies are
// started before this one is worked on (512 tokens, 2 heads, a row per warp: 28.5 -> 21.7 us; leaving out the keys no row keeps inside a stage: no change).
// ---------------------------------------------------------------------------------------------
template <typename T, int R, int ND, bool PIPE>
__global__ void __launch_bounds__(256)
attn_ref_kernel(const unsigned char* blob, const T* __restrict__ Q, const T* __restrict__ K,
                const T* __restrict__ V, int Hq, int group, int d, int64_t qst, int64_t qsh,
                int64_t kst, int64_t ksh, int64_t vst, int64_t vsh, int64_t ost, int64_t osh,
                int causal, float scale, T* __restrict__ O, float* __restrict__ lse, int total_tokens,
                const int32_t* __restrict__ ranges, const __grid_constant__ DamRowRanges rr, uint32_t* scratch, int keep) {
  // the status block starts at zero (its first `keep` words stay: a further row range of the same layer)
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x >= keep && threadIdx.x < 64) scratch[threadIdx.x] = 0u;
  extern __shared__ __align__(16) float smem[];
  const DamHeader* H = reinterpret_cast<const DamHeader*>(blob);
  const int row = blockIdx.x;
  const int h = row / H->total_qblocks, gqb = row % H->total_qblocks;
  const int b = reinterpret_cast<const int32_t*>(blob + H->off_qbseq)[gqb];
  const DamSeq sq = reinterpret_cast<const DamSeq*>(blob + H->off_seq)[b];
  const int qb = gqb - sq.first_qblock;
  if (ranges && !rr.holds(ranges, b, qb & ~1)) return;         // row ranges: whole pairs of query blocks
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int i_block = qb * DAM_TILE + blockIdx.y * nw * R;
  if (i_block >= sq.S) return;
  const int i0 = i_block + warp * R;
  const uint32_t* tile_ptr = reinterpret_cast<const uint32_t*>(blob + H->off_tile_ptr);
  const uint32_t* tiles = reinterpret_cast<const uint32_t*>(blob + H->off_tiles);
  const uint32_t t0 = tile_ptr[row], t1 = tile_ptr[row + 1];
  const DamHeadBits hb = dam_head_bits(blob, H, sq, h);
  const int pitch = k_pitch(d);
  const int stage = kStageKeys * (pitch + d);
  float* k_s = smem;
  float* v_s = k_s + kStageKeys * pitch;
  float* q_s = smem + (PIPE ? 2 : 1) * stage + warp * R * d;
  float* p_s = smem + (PIPE ? 2 : 1) * stage + nw * R * d + warp * R * kStageKeys;       // the warp's probabilities of a stage
  for (int x = lane; x < R * d; x += 32) {
    const int i = i0 + x / d;
    q_s[x] = i < sq.S ? Ld8<T>::one(Q + (int64_t)(sq.tok_start + i) * qst + (int64_t)h * qsh + x % d) : 0.f;
  }
  const T* Kh = K + (int64_t)sq.tok_start * kst + (int64_t)(h / group) * ksh;
  const T* Vh = V + (int64_t)sq.tok_start * vst + (int64_t)(h / group) * vsh;
  float acc[R][ND], m[R], l[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    m[r] = -CUDART_INF_F; l[r] = 0.f;
#pragma unroll
    for (int u = 0; u < ND; ++u) acc[r][u] = 0.f;
  }
  // the stages of the row's tiles that hold an active cell of the block's rows, in order
  struct Stage { uint32_t w0[R], w1[R], any; int j0; bool valid; };
  uint32_t t = t0;
  int half = 2, kb = 0;
  uint4 bits[R];
  auto find = [&](Stage& g) {
    while (true) {
      if (half == 2) {
        uint32_t e = 0u;
        while (t < t1 && ((e = __ldg(tiles + t)) >> 28) == 0u) ++t;     // padding behind the row's entries
        if (t >= t1) { g.valid = false; return; }
        ++t;
        kb = (int)(e & 0x0FFFFFFFu);
#pragma unroll
        for (int r = 0; r < R; ++r) bits[r] = dam_apply_bits(hb, e >> 28, i0 + r, kb, causal);
        half = 0;
      }
      g.any = 0u;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        g.w0[r] = half ? bits[r].z : bits[r].x;
        g.w1[r] = half ? bits[r].w : bits[r].y;
        g.any |= g.w0[r] | g.w1[r];
      }
      g.j0 = kb * DAM_TILE + half * kStageKeys;
      ++half;
      if (__syncthreads_or(g.any != 0u)) { g.valid = true; return; }    // (a barrier: the stage before the last is no longer read)
    }
  };
  auto work = [&](const Stage& g, const float* k_b, const float* v_b) {
    if (!g.any) return;                                 // (the same in all lanes: the words are the row's)
    float s[R][2];
    dot_rows<R>(q_s, k_b + lane * pitch, k_b + (32 + lane) * pitch, d, s);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const bool a0 = (g.w0[r] >> lane) & 1u, a1 = (g.w1[r] >> lane) & 1u;
      const float x0 = a0 ? s[r][0] * scale : -CUDART_INF_F, x1 = a1 ? s[r][1] * scale : -CUDART_INF_F;
      const float mn = fmaxf(m[r], warp_max(fmaxf(x0, x1)));
      // (an infinite maximum counts as zero: a row without a key so far, or whose logits are all -inf)
      const float at = mn == -CUDART_INF_F ? 0.f : mn, corr = expf(m[r] - at);
      const float p0 = a0 ? expf(x0 - at) : 0.f, p1 = a1 ? expf(x1 - at) : 0.f;
      l[r] = l[r] * corr + warp_sum(p0 + p1);
      m[r] = mn;
#pragma unroll
      for (int u = 0; u < ND; ++u) acc[r][u] *= corr;
      p_s[r * kStageKeys + lane] = p0;
      p_s[r * kStageKeys + 32 + lane] = p1;
    }
    __syncwarp();
#pragma unroll 2
    for (int k = 0; k < kStageKeys; k += 4) {
      float4 p[R];
#pragma unroll
      for (int r = 0; r < R; ++r) p[r] = *reinterpret_cast<const float4*>(p_s + r * kStageKeys + k);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int u = 0; u < ND; ++u) {
          const int t_ = lane + 32 * u;
          const float v = t_ < d ? v_b[(k + q) * d + t_] : 0.f;
#pragma unroll
          for (int r = 0; r < R; ++r) {
            // (a key the row does not keep is left out, whatever its V row holds)
            const float pk = q == 0 ? p[r].x : q == 1 ? p[r].y : q == 2 ? p[r].z : p[r].w;
            if (pk != 0.f) acc[r][u] = fmaf(pk, v, acc[r][u]);
          }
        }
      }
    }
    __syncwarp();
  };
  if constexpr (PIPE) {
    auto start = [&](const Stage& g, int buf) {
      if (g.valid) {
        load_stage_async(k_s + buf * stage, pitch, reinterpret_cast<const float*>(Kh), kst, g.j0, sq.S, d);
        load_stage_async(v_s + buf * stage, d, reinterpret_cast<const float*>(Vh), vst, g.j0, sq.S, d);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    Stage cur, nxt;
    find(cur);
    start(cur, 0);
    for (int buf = 0; cur.valid; buf ^= 1) {
      find(nxt);
      start(nxt, buf ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncthreads();
      work(cur, k_s + buf * stage, v_s + buf * stage);
      cur = nxt;
    }
  } else {
    Stage cur;
    for (find(cur); cur.valid; find(cur)) {
      load_stage<T>(k_s, pitch, Kh, kst, cur.j0, sq.S, d);
      load_stage<T>(v_s, d, Vh, vst, cur.j0, sq.S, d);
      __syncthreads();
      work(cur, k_s, v_s);
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = i0 + r;
    if (i >= sq.S) break;
    T* orow = O + (int64_t)(sq.tok_start + i) * ost + (int64_t)h * osh;
    const float inv = l[r] > 0.f ? 1.0f / l[r] : 0.f;
#pragma unroll
    for (int u = 0; u < ND; ++u) {
      const int t_ = lane + 32 * u;
      if (t_ < d) Ld8<T>::store(orow + t_, acc[r][u] * inv);
    }
    if (lane == 0) lse[(int64_t)h * total_tokens + sq.tok_start + i] = l[r] > 0.f ? m[r] + logf(l[r]) : -CUDART_INF_F;
  }
}

// The same for few rows: a block of eight warps takes eight adjacent rows, and a warp takes eight of the 64 keys of every stage
// for all of them.  Lane 4 r + c scores row r against keys c and c + 4; for the output a lane holds 2 dimensions (of every 64) of all
// eight rows.  Every warp has a running softmax of its own over its keys, merged at the end.  A warp per row reads all 64
// keys of a stage from shared memory for each row, 2300 cycles of its bandwidth; here a key is read once per block.
// What is left is latency: a stage's two barriers and chains, and what the first one waits for (header, records, list, mask
// words, rows).  fp32, 2 heads of 64: 512 tokens 21.6 -> 17.2 us (19.2 without the mask words asked for a tile ahead), 1100 tokens
// 27.6 -> 21.3, 4 heads, 700 tokens 45.3 -> 33.5.  Three blocks to an SM (1500 tokens 29.3 -> 25.4).
template <typename T, int ND, bool PIPE>
__global__ void __launch_bounds__(256, ND == 1 ? 3 : 1)
attn_ref_few_kernel(const unsigned char* blob, const T* __restrict__ Q, const T* __restrict__ K,
                    const T* __restrict__ V, int Hq, int group, int d, int64_t qst, int64_t qsh,
                    int64_t kst, int64_t ksh, int64_t vst, int64_t vsh, int64_t ost, int64_t osh,
                    int causal, float scale, T* __restrict__ O, float* __restrict__ lse, int total_tokens,
                    const int32_t* __restrict__ ranges, const __grid_constant__ DamRowRanges rr, uint32_t* scratch, int keep) {
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x >= keep && threadIdx.x < 64) scratch[threadIdx.x] = 0u;
  extern __shared__ __align__(16) float smem[];
  const DamHeader* H = reinterpret_cast<const DamHeader*>(blob);
  const int row = blockIdx.x;
  const int h = row / H->total_qblocks, gqb = row % H->total_qblocks;
  const int b = reinterpret_cast<const int32_t*>(blob + H->off_qbseq)[gqb];
  const DamSeq sq = reinterpret_cast<const DamSeq*>(blob + H->off_seq)[b];
  const int qb = gqb - sq.first_qblock;
  if (ranges && !rr.holds(ranges, b, qb & ~1)) return;         // row ranges: whole pairs of query blocks
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i0 = qb * DAM_TILE + blockIdx.y * kFewRows;
  if (i0 >= sq.S) return;
  const uint32_t* tile_ptr = reinterpret_cast<const uint32_t*>(blob + H->off_tile_ptr);
  const uint32_t* tiles = reinterpret_cast<const uint32_t*>(blob + H->off_tiles);
  const uint32_t t0 = tile_ptr[row], t1 = tile_ptr[row + 1];
  const DamHeadBits hb = dam_head_bits(blob, H, sq, h);
  const int pitch = k_pitch(d);
  const int stage = kStageKeys * (pitch + d);
  float* k_s = smem;
  float* v_s = k_s + kStageKeys * pitch;
  float* q_s = smem + (PIPE ? 2 : 1) * stage;                                  // kFewRows rows, `pitch` apart
  float* p_s = q_s + kFewRows * pitch + warp * (kFewKeys + 1) * kFewRows;      // the warp's probabilities, a row per key; corrections
  for (int x = threadIdx.x; x < kFewRows * d; x += blockDim.x) {
    const int r = x / d, c = x % d;
    q_s[r * pitch + c] = i0 + r < sq.S ? Ld8<T>::one(Q + (int64_t)(sq.tok_start + i0 + r) * qst + (int64_t)h * qsh + c) : 0.f;
  }
  const T* Kh = K + (int64_t)sq.tok_start * kst + (int64_t)(h / group) * ksh;
  const T* Vh = V + (int64_t)sq.tok_start * vst + (int64_t)(h / group) * vsh;
  const int my_row = lane >> 2, my_key = warp * kFewKeys + (lane & 3);          // and my_key + 4
  float acc[kFewRows][2 * ND], m = -CUDART_INF_F, l = 0.f;
#pragma unroll
  for (int r = 0; r < kFewRows; ++r)
#pragma unroll
    for (int u = 0; u < 2 * ND; ++u) acc[r][u] = 0.f;
  // the stages of the tiles that hold an active cell of the block's rows, in order
  struct Stage { uint32_t mine; int j0; bool valid; };                         // mine: bits 0 and 4: the lane's two cells
  // (the mask words of a tile are asked for one tile ahead, its entry two: a stage would wait for both in turn)
  uint32_t t = t0, e_next = t < t1 ? __ldg(tiles + t) : 0u;
  int half = 2, kb = 0, kb_next = 0;
  uint4 bits = make_uint4(0u, 0u, 0u, 0u), bits_next = bits;
  bool more = false;
  auto ask = [&]() {
    more = (e_next >> 28) != 0u;                                // (zero entries are padding behind the row's)
    if (!more) return;
    kb_next = (int)(e_next & 0x0FFFFFFFu);
    bits_next = dam_apply_bits(hb, e_next >> 28, i0 + my_row, kb_next, causal);
    ++t;
    e_next = t < t1 ? __ldg(tiles + t) : 0u;
  };
  ask();
  auto find = [&](Stage& g) {
    while (true) {
      if (half == 2) {
        if (!more) { g.valid = false; return; }
        kb = kb_next;
        bits = bits_next;
        ask();
        half = 0;
      }
      const uint32_t w0 = half ? bits.z : bits.x, w1 = half ? bits.w : bits.y;
      g.mine = ((my_key & 32) ? w1 : w0) >> (my_key & 31);
      g.j0 = kb * DAM_TILE + half * kStageKeys;
      ++half;
      if (__syncthreads_or((w0 | w1) != 0u)) { g.valid = true; return; }     // (a barrier: the stage before the last is no longer read)
    }
  };
  auto work = [&](const Stage& g, const float* k_b, const float* v_b) {
    const bool a0 = g.mine & 1u, a1 = (g.mine >> 4) & 1u;
    if (!__any_sync(0xFFFFFFFFu, a0 || a1)) return;
    float s0 = 0.f, s1 = 0.f;
    const float *k0 = k_b + my_key * pitch, *k1 = k0 + 4 * pitch, *q = q_s + my_row * pitch;
#pragma unroll 4
    for (int c = 0; c < d; c += 4) {
      const float4 x = *reinterpret_cast<const float4*>(q + c), y = *reinterpret_cast<const float4*>(k0 + c),
                   z = *reinterpret_cast<const float4*>(k1 + c);
      s0 = fmaf(x.x, y.x, s0); s1 = fmaf(x.x, z.x, s1);
      s0 = fmaf(x.y, y.y, s0); s1 = fmaf(x.y, z.y, s1);
      s0 = fmaf(x.z, y.z, s0); s1 = fmaf(x.z, z.z, s1);
      s0 = fmaf(x.w, y.w, s0); s1 = fmaf(x.w, z.w, s1);
    }
    const float x0 = a0 ? s0 * scale : -CUDART_INF_F, x1 = a1 ? s1 * scale : -CUDART_INF_F;
    float mn = fmaxf(x0, x1);
    mn = fmaxf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, 1));
    mn = fmaxf(mn, __shfl_xor_sync(0xFFFFFFFFu, mn, 2));
    mn = fmaxf(m, mn);
    // (an infinite maximum counts as zero: a row without a key so far, or whose logits are all -inf)
    const float at = mn == -CUDART_INF_F ? 0.f : mn, corr = expf(m - at);
    const float p0 = a0 ? expf(x0 - at) : 0.f, p1 = a1 ? expf(x1 - at) : 0.f;
    l = l * corr + (p0 + p1);
    m = mn;
    p_s[(lane & 3) * kFewRows + my_row] = p0;
    p_s[((lane & 3) + 4) * kFewRows + my_row] = p1;
    p_s[kFewKeys * kFewRows + my_row] = corr;
    __syncwarp();
    if (__any_sync(0xFFFFFFFFu, corr != 1.f)) {
#pragma unroll
      for (int r = 0; r < kFewRows; ++r) {
        const float f = p_s[kFewKeys * kFewRows + r];
#pragma unroll
        for (int u = 0; u < 2 * ND; ++u) acc[r][u] *= f;
      }
    }
#pragma unroll 4
    for (int k = 0; k < kFewKeys; ++k) {
      const float4 pa = *reinterpret_cast<const float4*>(p_s + k * kFewRows), pb = *reinterpret_cast<const float4*>(p_s + k * kFewRows + 4);
      const float pk[kFewRows] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
#pragma unroll
      for (int u = 0; u < ND; ++u) {
        const int c = 2 * lane + 64 * u;
        const float2 v = c < d ? *reinterpret_cast<const float2*>(v_b + (warp * kFewKeys + k) * d + c) : make_float2(0.f, 0.f);
#pragma unroll
        for (int r = 0; r < kFewRows; ++r)
          if (pk[r] != 0.f) {                          // (a key the row does not keep is left out, whatever its V row holds)
            acc[r][2 * u] = fmaf(pk[r], v.x, acc[r][2 * u]);
            acc[r][2 * u + 1] = fmaf(pk[r], v.y, acc[r][2 * u + 1]);
          }
      }
    }
    __syncwarp();
  };
  if constexpr (PIPE) {
    auto start = [&](const Stage& g, int buf) {
      if (g.valid) {
        load_stage_async(k_s + buf * stage, pitch, reinterpret_cast<const float*>(Kh), kst, g.j0, sq.S, d);
        load_stage_async(v_s + buf * stage, d, reinterpret_cast<const float*>(Vh), vst, g.j0, sq.S, d);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    Stage cur, nxt;
    find(cur);
    start(cur, 0);
    for (int buf = 0; cur.valid; buf ^= 1) {
      find(nxt);
      start(nxt, buf ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncthreads();
      work(cur, k_s + buf * stage, v_s + buf * stage);
      cur = nxt;
    }
  } else {
    Stage cur;
    for (find(cur); cur.valid; find(cur)) {
      load_stage<T>(k_s, pitch, Kh, kst, cur.j0, sq.S, d);
      load_stage<T>(v_s, d, Vh, vst, cur.j0, sq.S, d);
      __syncthreads();
      work(cur, k_s, v_s);
    }
  }
  // merge of the eight warps: their references and sums, then their outputs, in the memory of the stages
  l += __shfl_xor_sync(0xFFFFFFFFu, l, 1);
  l += __shfl_xor_sync(0xFFFFFFFFu, l, 2);
  __syncthreads();
  float2* ml = reinterpret_cast<float2*>(q_s);                                 // [warp][row]
  if ((lane & 3) == 0) ml[warp * kFewRows + my_row] = make_float2(m, l);
#pragma unroll
  for (int r = 0; r < kFewRows; ++r)
#pragma unroll
    for (int u = 0; u < ND; ++u) {
      const int c = 2 * lane + 64 * u;
      if (c < d) *reinterpret_cast<float2*>(smem + (warp * kFewRows + r) * d + c) = make_float2(acc[r][2 * u], acc[r][2 * u + 1]);
    }
  __syncthreads();
  const int r = warp, i = i0 + r;                                              // a row per warp
  if (i >= sq.S) return;
  float M = -CUDART_INF_F, f[kRefWarps], sum = 0.f;
#pragma unroll
  for (int w = 0; w < kRefWarps; ++w) M = fmaxf(M, ml[w * kFewRows + r].x);
#pragma unroll
  for (int w = 0; w < kRefWarps; ++w) {
    const float2 x = ml[w * kFewRows + r];
    f[w] = x.x == -CUDART_INF_F ? 0.f : expf(x.x - M);
    sum += x.y * f[w];
  }
  // (zero without a key.  A NaN stays one: a warp whose only key has a NaN logit has no reference, its output is left out below, but
  // its sum is NaN)
  const float inv = sum > 0.f ? 1.0f / sum : sum;
  T* orow = O + (int64_t)(sq.tok_start + i) * ost + (int64_t)h * osh;
  for (int c = lane; c < d; c += 32) {
    float o = 0.f;
#pragma unroll
    for (int w = 0; w < kRefWarps; ++w)
      if (f[w] != 0.f) o = fmaf(f[w], smem[(w * kFewRows + r) * d + c], o);
    Ld8<T>::store(orow + c, o * inv);
  }
  if (lane == 0) lse[(int64_t)h * total_tokens + sq.tok_start + i] = sum > 0.f ? M + logf(sum) : -CUDART_INF_F;
}

// Whether a call has many rows: `halves` / 2 for every warp of a block of eight on every SM.  Scoring takes four rows per warp
// from there on and one below, so that a short prompt's rows are spread over the whole chip (four for every warp).
inline bool many_rows(long long rows, int sm_count, int halves) { return 2 * rows >= (long long)sm_count * kRefWarps * halves; }
// Attention takes four rows per warp from five rows for every warp on, attn_ref_few_kernel below (fp32, head_dim 64, a warp per
// row, four rows per warp and it: 1400 rows 45.3, -, 33.5 us; 4000 54, -, 40; 4800 -, 62, 50; 6000 -, 62.4, 60.8; 8000 -, 62.5,
// 74.5; bf16, head_dim 40, 5800 -, 55.6, 37.3).  With a head_dim above 64 there is a block of the latter to an SM instead of
// three, and the line is at two and a half (2 heads, windows of 128, four rows per warp and it: 2560 rows fp32 head_dim 96 45.3 and
// 42.5, 128 51.5 and 49.4, 192 78.1 and 67.9, 256 92.4 and 102.6, bf16 96 47.0 and 47.4, 256 92.5 and 103; 3072 rows 45.3 and 48.5,
// 51.5 and 55.9, 78.1 and 78.1, 92.4 and 119, 46.2 and 54.3, 93.9 and 121; 4608 rows fp32 128 51.5 and 75.9, bf16 96 47.4 and 71.9;
// 5888 rows fp32 192 148 and 129, 256 174 and 197, bf16 96 62.7 and 88.5).
inline int attn_halves(int head_dim) { return head_dim <= 64 ? 10 : 5; }

size_t score_smem(int d, int R, int nbuf) { return ((size_t)nbuf * kStageKeys * k_pitch(d) + (size_t)kRefWarps * R * d) * sizeof(float); }
size_t attn_smem(int d, int R, int nbuf) {
  if (R == 1)
    return ((size_t)nbuf * kStageKeys * (k_pitch(d) + d) + (size_t)kFewRows * k_pitch(d) + kRefWarps * (kFewKeys + 1) * kFewRows) * sizeof(float);
  return ((size_t)nbuf * kStageKeys * (k_pitch(d) + d) + (size_t)kRefWarps * R * (d + kStageKeys)) * sizeof(float);
}

// Opt-in of one kernel instance to all the shared memory a block may have, once per device: the limit belongs to the
// instance, and its calls differ in what they use (head_dim, stages), so a limit set to the need of each call could be
// lowered by one thread between another's setting and launch.  (48 KB need no opt-in.)
template <typename K>
cudaError_t allow_all_smem(K* kernel) {
  int dev = 0, bytes = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&bytes, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return e == cudaSuccess ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) : e;
}
template <typename T, int R>
cudaError_t opt_in_scores(int dev, size_t bytes) {
  constexpr int key = DAM_SETUP_REF_SMEM + 2 * (sizeof(T) == 4) + (R == 4);
  return bytes <= 48 * 1024 ? cudaSuccess
                            : dam_device_table().once(dev, key, []() -> cudaError_t { return allow_all_smem(scores_ref_kernel<T, R>); });
}
template <typename T, int R, int ND, bool PIPE>
constexpr auto attn_kernel() {
  if constexpr (R == 1) return attn_ref_few_kernel<T, ND, PIPE>;
  else return attn_ref_kernel<T, R, 2 * ND, PIPE>;
}
template <typename T, int R, int ND, bool PIPE>
cudaError_t opt_in_attn(int dev, size_t bytes) {
  constexpr int dims = ND == 1 ? 0 : ND == 2 ? 1 : 2, type = PIPE ? 2 : sizeof(T) == 4;
  constexpr int key = DAM_SETUP_REF_SMEM + 4 + (3 * type + dims) * 2 + (R == 4);
  static_assert(key < DamDeviceTable::kMaxSetups, "a set-up step per instance");
  return bytes <= 48 * 1024
             ? cudaSuccess
             : dam_device_table().once(dev, key, []() -> cudaError_t { return allow_all_smem(attn_kernel<T, R, ND, PIPE>()); });
}

template <typename T, int R>
cudaError_t launch_scores(const void* Q, const void* K, const dam_shape_t* s, const DamBuildCtx& c, float* dump, int dev,
                          const DamDeviceInfo& di, cudaStream_t st) {
  const dim3 grid((c.max_L + kRefWarps * R - 1) / (kRefWarps * R), c.num_seqs * c.Hq);
  // all stages at once while every block has an SM of its own anyway (a block's shared memory then costs no occupancy)
  const int nstage = (c.max_L + kStageKeys - 1) / kStageKeys;
  const int nbuf = (long long)grid.x * grid.y <= di.sm_count && score_smem(c.d, R, nstage) <= (size_t)di.smem_optin ? nstage : 1;
  const size_t sm = score_smem(c.d, R, nbuf);
  cudaError_t e = opt_in_scores<T, R>(dev, sm);
  if (e != cudaSuccess) return e;
  return dam_launch_chained(scores_ref_kernel<T, R>, grid, dim3(kRefWarps * 32), sm, st, c.blob, (const T*)Q, (const T*)K, c.Hq,
                            c.Hq / c.Hkv, c.d, s->q_stride_tok, s->q_stride_head, s->k_stride_tok, s->k_stride_head, c.scale,
                            c.pstar, dump, nbuf);
}

template <typename T, int R, int ND>
cudaError_t launch_attn(const void* Q, const void* K, const void* V, const void* blob, const dam_shape_t* s, int causal,
                        float scale, void* O, float* lse, const int32_t* ranges, const DamRowRanges& rr, uint32_t* scratch, int keep, int rows, int dev, int smem_max, cudaStream_t st) {
  const bool pipe = sizeof(T) == 4 && attn_smem(s->head_dim, R, 2) <= (size_t)smem_max;
  const size_t sm = attn_smem(s->head_dim, R, pipe ? 2 : 1);
  auto kernel = attn_kernel<T, R, ND, false>();
  cudaError_t e;
  if (sizeof(T) == 4 && pipe) {
    if constexpr (sizeof(T) == 4) { kernel = attn_kernel<T, R, ND, true>(); e = opt_in_attn<T, R, ND, true>(dev, sm); }
  } else {
    e = opt_in_attn<T, R, ND, false>(dev, sm);
  }
  if (e != cudaSuccess) return e;
  const dim3 grid(rows, DAM_TILE / (kRefWarps * R));
  // (an ordinary launch: as a link of the chain its blocks are placed while the ordering kernel still holds SMs, several to
  // an SM where every one of them could have its own: fp32, 512 tokens, a pass 46.7 us against 44.9)
  kernel<<<grid, kRefWarps * 32, sm, st>>>(
      (const unsigned char*)blob, (const T*)Q, (const T*)K, (const T*)V, s->num_q_heads, s->num_q_heads / s->num_kv_heads, s->head_dim,
      s->q_stride_tok, s->q_stride_head, s->k_stride_tok, s->k_stride_head, s->v_stride_tok, s->v_stride_head, s->o_stride_tok,
      s->o_stride_head, causal, scale, (T*)O, lse, s->total_tokens, ranges, rr, scratch, keep);
  return cudaGetLastError();
}

template <typename T, int R>
cudaError_t launch_attn_dims(const void* Q, const void* K, const void* V, const void* blob, const dam_shape_t* s, int causal,
                             float scale, void* O, float* lse, const int32_t* ranges, const DamRowRanges& rr, uint32_t* scratch, int keep, int rows, int dev, int smem_max, cudaStream_t st) {
  const int nd = (s->head_dim + 63) / 64;
  if (nd <= 1) return launch_attn<T, R, 1>(Q, K, V, blob, s, causal, scale, O, lse, ranges, rr, scratch, keep, rows, dev, smem_max, st);
  if (nd <= 2) return launch_attn<T, R, 2>(Q, K, V, blob, s, causal, scale, O, lse, ranges, rr, scratch, keep, rows, dev, smem_max, st);
  return launch_attn<T, R, 4>(Q, K, V, blob, s, causal, scale, O, lse, ranges, rr, scratch, keep, rows, dev, smem_max, st);
}

}  // namespace

cudaError_t dam_launch_scores_ref(const void* Q, const void* K, const dam_shape_t* s, const DamBuildCtx& c,
                                  float* dump, cudaStream_t st) {
  if (c.max_L == 0) return cudaSuccess;
  int dev = 0;
  DamDeviceInfo di;
  cudaError_t e = dam_current_device(&dev, &di);
  if (e != cudaSuccess) return e;
  const bool four = many_rows((long long)c.max_L * c.num_seqs * c.Hq, di.sm_count, 8);
  if (c.dtype == DAM_F32)
    return four ? launch_scores<float, 4>(Q, K, s, c, dump, dev, di, st) : launch_scores<float, 1>(Q, K, s, c, dump, dev, di, st);
  return four ? launch_scores<__nv_bfloat16, 4>(Q, K, s, c, dump, dev, di, st) : launch_scores<__nv_bfloat16, 1>(Q, K, s, c, dump, dev, di, st);
}

cudaError_t dam_launch_attn_ref(const void* Q, const void* K, const void* V, const void* blob, const dam_shape_t* s,
                                int causal, float scale, void* O, float* lse, void* scratch, bool keep_status,
                                const int32_t* ranges, const int32_t* ranges_host, cudaStream_t st) {
  int rows = 0;
  for (int b = 0; b < s->num_seqs; ++b)
    rows += (s->cu_seqlens_host[b + 1] - s->cu_seqlens_host[b] + DAM_TILE - 1) / DAM_TILE;
  rows *= s->num_q_heads;
  uint32_t* scr = reinterpret_cast<uint32_t*>(scratch);
  const DamRowRanges rr(ranges ? ranges_host : nullptr, s->num_seqs);
  const int keep = keep_status ? 2 : 0;
  if (rows == 0) return cudaMemsetAsync(scr + keep, 0, 256 - 4 * keep, st);
  int dev = 0;
  DamDeviceInfo di;
  cudaError_t e = dam_current_device(&dev, &di);
  if (e != cudaSuccess) return e;
  const bool four = many_rows((long long)rows * DAM_TILE, di.sm_count, attn_halves(s->head_dim));
  if (s->dtype == DAM_F32)
    return four ? launch_attn_dims<float, 4>(Q, K, V, blob, s, causal, scale, O, lse, ranges, rr, scr, keep, rows, dev, di.smem_optin, st)
                : launch_attn_dims<float, 1>(Q, K, V, blob, s, causal, scale, O, lse, ranges, rr, scr, keep, rows, dev, di.smem_optin, st);
  return four ? launch_attn_dims<__nv_bfloat16, 4>(Q, K, V, blob, s, causal, scale, O, lse, ranges, rr, scr, keep, rows, dev, di.smem_optin, st)
              : launch_attn_dims<__nv_bfloat16, 1>(Q, K, V, blob, s, causal, scale, O, lse, ranges, rr, scr, keep, rows, dev, di.smem_optin, st);
}
