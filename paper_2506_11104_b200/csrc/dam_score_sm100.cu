// Window scoring on the 5th-generation tensor cores (sm_100a): bf16 inputs, head_dim 128 or 64 (template parameter:
// with 64 a Q / K tile is one 16 KB box of the tensor maps and S = Q K^T takes four MMAs instead of eight).
//
// For every (sequence, query head) the causal softmax map over the first L tokens is computed tile by
// tile and thresholded straight into the bit-packed true mask (paper Sec. 4.2.1 - 4.2.3); the map itself
// is never stored unless the caller asks for the fp32 dump.  An S buffer per softmax group in TMEM lets the MMA warp run ahead
// of them.  A work item is one 128-row query block of
// one (sequence, head).  Two sweeps over its kv tiles kb = 0 .. qb:
//   sweep A  S = Q K^T (tcgen05, accumulator in TMEM) -> per-row running max and sum;
//   sweep B  S again -> p = exp2(x - max) / sum in fp32 -> bit = [p >= p*] -> one 16-byte store of the
//            row's 128 bits per tile (and the optional dump of p).
// Warp roles: warp 0 TMA producer, warp 1 MMA issuer, then two or four groups of one thread per query row;
// group G owns TMEM buffer G, i.e. every second or fourth kv tile, and the groups merge their row statistics through
// shared memory between the sweeps.  Every wait is bounded.
#include <cuda_bf16.h>
#include <math_constants.h>

#include "dam_internal.cuh"
#include "sm100_ptx.cuh"

using namespace sm100;

namespace {

constexpr int kSlotBytes = 32768;

// kGroups: softmax groups of four warps, each with an S buffer (tile g uses buffer g % kGroups).
template <int kGroups>
struct SmemLayout {
  static constexpr int kSlots = kGroups == 4 ? 5 : 2;
  static constexpr int kThreads = 64 + 128 * kGroups;      // producer warp, MMA warp, softmax warps
  static constexpr int q = 0;
  static constexpr int slots = kSlotBytes;
  static constexpr int bars = kSlotBytes * (1 + kSlots);
  // q_full, q_empty, slot_full[kSlots], slot_empty[kSlots], s_full[kGroups], s_empty[kGroups], stat_ready,
  // sched_full[2], sched_empty[2]
  static constexpr int n_bars = 2 + 2 * kSlots + 2 * kGroups + 5;
  static constexpr int sched_items = bars + 8 * n_bars;     // int[2]
  static constexpr int stat = sched_items + 8;              // float2 [2][kGroups][128]
  static constexpr int tmem_slot = stat + 2 * kGroups * 128 * 8;
  static constexpr int abort_flag = tmem_slot + 4;
  static constexpr int total = abort_flag + 4 + 1024;
};

struct ScoreParams {
  unsigned char* blob;
  float* dump;
  uint32_t* status;
  uint32_t* work_counter;     // zero at launch
  int num_seqs, Hq, group, max_nL;
  int dump_vec8;              // every row of the dumped maps starts on a 32-byte boundary and is a multiple of 32 bytes
  float scale_log2, pstar;
  DamPlan plan;
};

__device__ __forceinline__ void st_global_v8(float* p, const float* v) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
               "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ void fma2(float& d0, float& d1, float a0, float a1, float b0, float b1, float c0, float c1) {
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d0), "=f"(d1) : "f"(a0), "f"(a1), "f"(b0), "f"(b1), "f"(c0), "f"(c1));
}
__device__ __forceinline__ void add2(float& d0, float& d1, float a0, float a1, float b0, float b1) {
  asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d0), "=f"(d1) : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

struct Item { int b, h, qb, valid; DamSeq sq; };

__device__ __forceinline__ Item decode_item(const unsigned char* blob, const ScoreParams& p, int w) {
  Item it;
  const int per = p.num_seqs * p.Hq;
  it.qb = p.max_nL - 1 - w / per;           // heaviest query blocks first
  const int sh = w % per;
  it.b = sh / p.Hq; it.h = sh % p.Hq;
  it.sq = dam_plan_seq(p.plan, blob, it.b);
  it.valid = it.qb < it.sq.nL;
  return it;
}

template <int D, int kGroups>
__global__ void __launch_bounds__(SmemLayout<kGroups>::kThreads, 4 / kGroups)
score_sm100_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ ScoreParams prm) {
  using Smem = SmemLayout<kGroups>;
  constexpr uint32_t kSlots = Smem::kSlots, kTmemCols = 128 * kGroups;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  const uint32_t sQ = sbase + Smem::q;
  const uint32_t sSlots = sbase + Smem::slots;
  const uint32_t bar0 = sbase + Smem::bars;
  const uint32_t bQFull = bar0, bQEmpty = bar0 + 8;
  const uint32_t bSlotFull = bar0 + 16, bSlotEmpty = bSlotFull + 8 * kSlots;
  const uint32_t bSFull = bSlotEmpty + 8 * kSlots, bSEmpty = bSFull + 8 * kGroups, bStat = bSEmpty + 8 * kGroups;
  const uint32_t bSchedFull = bStat + 8, bSchedEmpty = bSchedFull + 16;
  volatile int* sched_items = reinterpret_cast<volatile int*>(smem + Smem::sched_items);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + Smem::tmem_slot);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(smem + Smem::abort_flag);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* blob = prm.blob;
  const DamHeader* H = &prm.plan.h;
  const int nitems = prm.max_nL * prm.num_seqs * prm.Hq;
  // Items (heaviest query blocks first) are claimed from a global counter by the producer thread and handed
  // to the MMA thread and the softmax warps through a two-entry ring; a negative entry ends the loop.
  auto next_item_consumer = [&](uint32_t n) -> int {
    const uint32_t slot = n & 1u;
    if (!mbar_wait_slow(bSchedFull + 8 * slot, (n >> 1) & 1u, abort_flag)) return -2;
    return sched_items[slot];
  };

  if (tid == 0) {
    mbar_init(bQFull, 1); mbar_init(bQEmpty, 1);
    for (int s = 0; s < kSlots; ++s) { mbar_init(bSlotFull + 8 * s, 1); mbar_init(bSlotEmpty + 8 * s, 1); }
    for (int s = 0; s < kGroups; ++s) { mbar_init(bSFull + 8 * s, 1); mbar_init(bSEmpty + 8 * s, 4); }
    mbar_init(bStat, 4 * kGroups);
    for (int s = 0; s < 2; ++s) { mbar_init(bSchedFull + 8 * s, 1); mbar_init(bSchedEmpty + 8 * s, 1 + 4 * kGroups); }   // MMA thread + softmax warps
    *abort_flag = 0u;
    mbar_fence_init();
    tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmK);
  }
  if (warp == 0) { tmem_alloc(smem_u32(tmem_slot), kTmemCols); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // everything above is independent of the kernel before this one; the blob it initialises is read from here on
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (blockIdx.x == 0 && tid == 0) {
    reinterpret_cast<DamHeader*>(blob)->reserved[0] = 1ull;          // the map of this blob was scored on the tensor cores
    reinterpret_cast<DamHeader*>(blob)->reserved[1] = kGroups;
  }

  if (warp == 0) {
    if (elect_one()) {              // (elected, not lane 0: PCL 4096 292 -> 274 us for stage 1, PCL 2048 97.6 -> 95.8 us)
      uint32_t sc = 0, ic = 0;
      uint32_t armed[kSlots];
#pragma unroll
      for (int s = 0; s < kSlots; ++s) armed[s] = 2u;
      bool ok = true;
      for (uint32_t n = 0; ok; ++n) {
        const uint32_t sl = n & 1u;
        if (!(ok = mbar_wait_slow(bSchedEmpty + 8 * sl, ((n >> 1) & 1u) ^ 1u, abort_flag))) break;
        int w = n == 0 ? (int)blockIdx.x : (int)(gridDim.x + atomicAdd(prm.work_counter, 1u));
        if (w >= nitems) w = -1;
        sched_items[sl] = w;
        mbar_arrive(bSchedFull + 8 * sl);
        if (w < 0) break;
        const Item it = decode_item(blob, prm, w);
        if (!it.valid) continue;
        if (!(ok = mbar_wait_slow(bQEmpty, (ic & 1u) ^ 1u, abort_flag))) break;
        mbar_arrive_expect_tx(bQFull, DAM_TILE * D * 2);
        const int tokq = it.sq.tok_start + it.qb * DAM_TILE;
        tma_load_3d(sQ, &tmQ, bQFull, 0, it.h, tokq);
        if (D == 128) tma_load_3d(sQ + 16384, &tmQ, bQFull, 64, it.h, tokq);
        ++ic;
        const int kvh = it.h / prm.group;
        const int ntile = 2 * (it.qb + 1);
        for (int t = 0; t < ntile && ok; ++t) {
          const int kb = t % (it.qb + 1);
          const uint32_t s = sc % kSlots, ph = (sc / kSlots) & 1u;
          if (!(ok = mbar_wait_slow(bSlotEmpty + 8 * s, ph ^ 1u, abort_flag))) break;
          const uint32_t dst = sSlots + s * kSlotBytes, bar = bSlotFull + 8 * s;
          mbar_arrive_expect_tx(bar, DAM_TILE * D * 2);
          tma_load_3d(dst, &tmK, bar, 0, kvh, it.sq.tok_start + kb * DAM_TILE);
          if (D == 128) tma_load_3d(dst + 16384, &tmK, bar, 64, kvh, it.sq.tok_start + kb * DAM_TILE);
          armed[s] = ph;
          ++sc;
        }
      }
      if (!ok) {
        uint32_t dummy = 0;
        for (int s = 0; s < kSlots; ++s)
          if (armed[s] != 2u) mbar_wait_slow(bSlotFull + 8 * s, armed[s], &dummy, 20000000ull);
        mbar_wait_slow(bQFull, (ic + 1u) & 1u, &dummy, 20000000ull);
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      const uint32_t idesc = idesc_bf16_f32(128, 128, 0);
      const uint64_t dQ = smem_desc_sw128(sQ, 16, 1024), dK = smem_desc_sw128(sSlots, 16, 1024);
      const uint32_t dQ_lo = (uint32_t)dQ, dQ_hi = (uint32_t)(dQ >> 32), dK_lo = (uint32_t)dK, dK_hi = (uint32_t)(dK >> 32);
      uint32_t sc = 0, ic = 0, g = 0;
      bool ok = true;
      for (uint32_t n = 0; ok; ++n) {
        const int w = next_item_consumer(n);
        if (w != -2) mbar_arrive(bSchedEmpty + 8 * (n & 1u));
        if (w < 0) { ok = (w == -1); break; }
        const Item it = decode_item(blob, prm, w);
        if (!it.valid) continue;
        if (!(ok = mbar_wait_slow(bQFull, ic & 1u, abort_flag))) break;
        ++ic;
        const int ntile = 2 * (it.qb + 1);
        for (int t = 0; t < ntile && ok; ++t, ++g, ++sc) {
          const uint32_t buf = g % kGroups, s = sc % kSlots;
          if (!(ok = mbar_wait_slow(bSEmpty + 8 * buf, ((g / kGroups) & 1u) ^ 1u, abort_flag))) break;
          if (!(ok = mbar_wait_slow(bSlotFull + 8 * s, (sc / kSlots) & 1u, abort_flag))) break;
          tc_fence_after();
          const uint32_t b0 = dK_lo + s * (kSlotBytes >> 4);
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) {
            const uint32_t off = ((ks >> 2) * 16384 + (ks & 3) * 32) >> 4;
            mma_ss_lh(tmem + buf * 128, dQ_lo + off, dQ_hi, b0 + off, dK_hi, idesc, ks > 0 ? 1u : 0u);
          }
          tc_commit(bSlotEmpty + 8 * s);
          tc_commit(bSFull + 8 * buf);
          if (t + 1 == ntile) tc_commit(bQEmpty);
        }
      }
    }
  } else {
    // ---------------------------------------------------------------- row statistics and thresholding
    // Groups of four warps; group G owns the S buffer G, i.e. every kGroups-th kv tile of the item.
    const int G = (warp - 2) >> 2;
    const int r = (warp & 3) * 32 + lane;
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t tS0 = tmem + lane_addr;
    float2* stat = reinterpret_cast<float2*>(smem + Smem::stat);      // [2 item parities][kGroups][128 rows]
    uint32_t g = 0, cG = 0, nitem = 0;      // g: tiles issued so far (all groups); cG: tiles this group consumed
    bool ok = true;
    for (uint32_t n = 0; ok; ++n) {
      const int w = next_item_consumer(n);
      __syncwarp();
      if (lane == 0 && w != -2) mbar_arrive(bSchedEmpty + 8 * (n & 1u));
      if (w < 0) { ok = (w == -1); break; }
      const Item it = decode_item(blob, prm, w);
      if (!it.valid) continue;
      const int L = it.sq.L, W = it.sq.W;
      const int i = it.qb * DAM_TILE + r;
      const bool row_valid = i < L;
      uint32_t* Mrow = reinterpret_cast<uint32_t*>(blob + H->off_true) + it.sq.true_off + (uint64_t)it.h * L * W + (size_t)i * W;
      float* Prow = prm.dump ? prm.dump + it.sq.p_off + (uint64_t)it.h * L * L + (size_t)i * L : nullptr;
      const int nk = it.qb + 1;
      float m = -CUDART_INF_F, l = 0.f, inv_l = 0.f, thr_raw = 0.f, margin = 0.f;
      for (int t = 0; t < 2 * nk; ++t, ++g) {
        if (t == nk) {
          // all groups have finished sweep A: merge their (max, sum) per row through shared memory
          float2* base = stat + (nitem & 1u) * kGroups * DAM_TILE;
          base[G * DAM_TILE + r] = make_float2(m, l);
          __syncwarp();
          if (lane == 0) mbar_arrive(bStat);                       // release: the warp's 32 rows are written
          if (!(ok = mbar_wait_slow(bStat, nitem & 1u, abort_flag))) break;
          float mn = m;
#pragma unroll
          for (int q = 0; q < kGroups; ++q) mn = fmaxf(mn, base[q * DAM_TILE + r].x);
          float ls = 0.f;
#pragma unroll
          for (int q = 0; q < kGroups; ++q) {
            const float2 o = base[q * DAM_TILE + r];
            ls += (o.x == -CUDART_INF_F) ? 0.f : o.y * ex2(o.x - mn);
          }
          m = mn; l = ls;
          inv_l = l > 0.f ? 1.0f / l : 0.f;
          // the raw dot product at which p = p* (below 2^-126 the exponential is zero, and so is p)
          thr_raw = (fmaxf(log2f(prm.pstar * l), -126.f) + m) / prm.scale_log2;
          margin = (0.000244140625f + fabsf(m) * 7.62939453125e-6f) / prm.scale_log2;      // 2^-12 + |m| 2^-17
        }
        if (g % kGroups != (uint32_t)G) continue;
        const int kb = t % nk;
        const bool sweepB = t >= nk;
        const uint32_t buf = (uint32_t)G;
        const uint32_t tS = tS0 + buf * 128;
        if (!(ok = mbar_wait_slow(bSFull + 8 * buf, cG & 1u, abort_flag))) break;
        ++cG;
        tc_fence_after();
        // keys beyond the causal limit (and beyond the window, which the limit implies) do not exist
        const int nvalid = kb == it.qb ? r + 1 : DAM_TILE;
        const bool diag = kb == it.qb;
        uint4 words = make_uint4(0u, 0u, 0u, 0u);
        float tmax = -CUDART_INF_F, tsum = 0.f;
        uint32_t cur[32];
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
          tmem_ld32(tS + c * 32, cur);
          tc_wait_ld();
          // raw dot products; the softmax scale (in log2 units) is applied inside the exponent's multiply-add
          float x[32];
#pragma unroll
          for (int q = 0; q < 32; ++q) x[q] = __uint_as_float(cur[q]);
          if (diag) {
#pragma unroll
            for (int q = 0; q < 32; ++q) x[q] = (c * 32 + q < nvalid) ? x[q] : -CUDART_INF_F;
          }
          if (!sweepB) {
            float c0 = -CUDART_INF_F, c1 = -CUDART_INF_F;
#pragma unroll
            for (int q = 0; q < 32; q += 4) { c0 = max3(c0, x[q], x[q + 1]); c1 = max3(c1, x[q + 2], x[q + 3]); }
            const float mn = fmaxf(tmax, fmaxf(c0, c1));          // maximum of the raw values (the scale is positive)
            if (mn > -CUDART_INF_F) {
              const float nm = -(mn * prm.scale_log2);
              float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
              for (int q = 0; q < 32; q += 4) {
                float y0, y1, y2, y3;
                fma2(y0, y1, x[q], x[q + 1], prm.scale_log2, prm.scale_log2, nm, nm);
                fma2(y2, y3, x[q + 2], x[q + 3], prm.scale_log2, prm.scale_log2, nm, nm);
                add2(a0, a1, a0, a1, ex2(y0), ex2(y1));
                add2(a2, a3, a2, a3, ex2(y2), ex2(y3));
              }
              tsum = tsum * ex2((tmax - mn) * prm.scale_log2) + ((a0 + a1) + (a2 + a3));     // tmax = -inf gives a factor 0
              tmax = mn;
            }
          } else if (Prow) {
            // the caller wants the map itself: every probability is computed and stored
            uint32_t word = 0u;
#pragma unroll
            for (int q = 0; q < 32; ++q) {
              const float p = ex2(fmaf(x[q], prm.scale_log2, -m)) * inv_l;    // -inf beyond the causal limit gives 0
              x[q] = p;
              word |= (p >= prm.pstar ? 1u : 0u) << q;
            }
            if (c == 0) words.x = word; else if (c == 1) words.y = word; else if (c == 2) words.z = word; else words.w = word;
            // a thread's 32 columns go out 32 bytes at a time where the rows of the map allow it (whole sectors; 8 samples of
            // 512 tokens x 32 heads, 268 MB of maps: 460 -> 88 us for the kernel), element by element otherwise
            if (row_valid) {
              const int j0 = kb * DAM_TILE + c * 32;
              if (prm.dump_vec8) {
#pragma unroll
                for (int q = 0; q < 32; q += 8)
                  if (j0 + q < L) st_global_v8(Prow + j0 + q, x + q);
              } else {
#pragma unroll
                for (int q = 0; q < 32; ++q)
                  if (j0 + q < L) Prow[j0 + q] = x[q];
              }
            }
          } else {
            // only the decision p >= p* is needed, p = 2^(x scale - m) / l.  It is the sign of x - thr, thr being the raw
            // product at which p reaches p*, except where x lies within `margin` of it: a chunk with such an entry is
            // evaluated exactly as in the branch above.  (Rounding of thr and of p is below 2^-17 + |m| 2^-22 in log2
            // units, the margin is 32 times that.)  The special-function unit is not needed otherwise: with a candidate
            // test and the exact form for every candidate, rows of noise were candidates throughout.
            uint32_t word = 0u;
            float near = CUDART_INF_F;
#pragma unroll
            for (int q = 31; q >= 0; --q) {
              const float dlt = thr_raw - x[q];                            // negative: p > p*
              near = fminf(near, fabsf(dlt));
              word = __funnelshift_l(__float_as_uint(dlt), word, 1);       // its sign bit becomes the lowest bit
            }
            if (__any_sync(0xFFFFFFFFu, near <= margin)) {
              word = 0u;
#pragma unroll
              for (int q = 0; q < 32; ++q) {
                const float p = ex2(fmaf(x[q], prm.scale_log2, -m)) * inv_l;
                word |= (p >= prm.pstar ? 1u : 0u) << q;
              }
            }
            if (c == 0) words.x = word; else if (c == 1) words.y = word; else if (c == 2) words.z = word; else words.w = word;
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bSEmpty + 8 * buf);
        if (!sweepB) {
          if (tmax > -CUDART_INF_F) {
            const float tm = tmax * prm.scale_log2;               // the tile's maximum in the scaled domain
            const float mn = fmaxf(m, tm);
            l = l * ex2(m - mn) + tsum * ex2(tm - mn);
            m = mn;
          }
        } else if (row_valid) {
          *reinterpret_cast<uint4*>(Mrow + kb * 4) = words;
        }
      }
      if (!ok) break;
      ++nitem;
      // zeros above the diagonal for the tiles this item does not visit: the true-mask words, and the map itself
      // when it is dumped
      if (row_valid && G == 0) {
        for (int kb = it.qb + 1; kb * 4 < W; ++kb) *reinterpret_cast<uint4*>(Mrow + kb * 4) = make_uint4(0u, 0u, 0u, 0u);
      }
      if (prm.dump) {
        // the warp's rows one after the other, a row's zeros by all lanes; the groups share them out
        float* P0 = prm.dump + it.sq.p_off + (uint64_t)it.h * L * L;
        for (int rr = 32 / kGroups * G; rr < 32 / kGroups * (G + 1); ++rr) {
          const int ir = it.qb * DAM_TILE + (warp & 3) * 32 + rr;
          if (ir >= L) break;
          float* Pr = P0 + (size_t)ir * L;
          if (prm.dump_vec8) {
            for (int j = nk * DAM_TILE + 4 * lane; j < L; j += 128) *reinterpret_cast<float4*>(Pr + j) = make_float4(0.f, 0.f, 0.f, 0.f);
          } else {
            for (int j = nk * DAM_TILE + lane; j < L; j += 32) Pr[j] = 0.f;
          }
        }
      }
    }
  }

  tc_fence_before();
  report_expired_wait(abort_flag, prm.status, DAM_ERR_DEVICE_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

// Two CTAs per SM with two softmax groups each, or one with four.  The four groups of
// a CTA are in the same sweep of the same item: first they all want the special-function unit, then the integer pipe, then
// all wait at the merge or for the next query tile; two items side by side fill each other's gaps, but an item takes
// longer.  So two from three items per SM on, four for windows of more than 16 tiles.  Stage 1, one and two CTAs per SM: 256 items of up to 8 tiles (8192 tokens) 40.5 and 47.8 us, 256 of 16 tiles 53.9
// and 70.5, 384 67.8 and 70.5, 512 (32768 tokens) 79.8 and 76.9, 1024 of up to 32 (131072 tokens) 232 and 217, 1536 (mixed
// lengths) 140 and 126, 1024 of 4 with the map written 112 and 106; 512 of up to 32 tiles 125.6 and 129.2, 768 169 and 156.
// In a batch of several lengths the items are counted by their tiles, in units of what an item of the longest window has on
// average: one window of 2048 tokens and 15 prompts of 100 (8 heads, 248 items, but 142 such units) 68.0 and 86.2 us, with 9 of 1000 (704
// items, 433 units) 85.5 and 80.4.  A place of the list without an item costs a CTA a claim, which two share: a twelfth of a
// unit (one window of 2048 and 20 of 500: 316 units, 1920 empty places 92.6 and 88.3; 2 of 2048 and 15 of 100: 271, 1800 87.1 and
// 91.2; 2 and 30: 284, 3600 120.4 and 114.5).
inline bool two_ctas(const dam_shape_t* s, const DamBuildCtx& c, int sm_count) {
  int64_t tiles = 0, items = 0;
  for (int b = 0; b < s->num_seqs; ++b) {
    const int64_t S = s->cu_seqlens_host[b + 1] - s->cu_seqlens_host[b], nL = ((S < c.pcl_max ? S : c.pcl_max) + DAM_TILE - 1) / DAM_TILE;
    items += nL;
    tiles += nL * (nL + 1) / 2;
  }
  const int64_t empty = ((int64_t)c.max_nL * c.num_seqs - items) * c.Hq;
  return 24 * tiles * c.Hq / (c.max_nL + 1) + empty >= 12 * (c.max_nL <= 16 ? 3 : 4) * (int64_t)sm_count;
}

}  // namespace

cudaError_t dam_launch_scores_sm100(const void* Q, const void* K, const dam_shape_t* s, const DamBuildCtx& c,
                                    float* dump, cudaStream_t st) {
  const int d = s->head_dim;
  if (s->dtype != DAM_BF16 || (d != 128 && d != 64)) return cudaErrorNotSupported;
  if (c.max_nL == 0) return cudaSuccess;
  int dev = 0;
  DamDeviceInfo di;
  cudaError_t e;
  if ((e = dam_current_device(&dev, &di)) != cudaSuccess) return e;
  if (di.cc_major != 10 || di.smem_optin < SmemLayout<4>::total) return cudaErrorNotSupported;
  if ((e = dam_device_table().once(dev, DAM_SETUP_SCORE_SMEM, [](void) -> cudaError_t {
         cudaError_t r;
         if ((r = cudaFuncSetAttribute(score_sm100_kernel<128, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, SmemLayout<4>::total)) != cudaSuccess) return r;
         if ((r = cudaFuncSetAttribute(score_sm100_kernel<128, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, SmemLayout<2>::total)) != cudaSuccess) return r;
         if ((r = cudaFuncSetAttribute(score_sm100_kernel<64, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, SmemLayout<4>::total)) != cudaSuccess) return r;
         return cudaFuncSetAttribute(score_sm100_kernel<64, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, SmemLayout<2>::total);
       })) != cudaSuccess)
    return e;
  const int sm_count = di.sm_count;
  CUtensorMap tq, tk;
  if (!dam_make_tmap_bf16(&tq, Q, d, s->num_q_heads, s->total_tokens, s->q_stride_tok, s->q_stride_head) ||
      !dam_make_tmap_bf16(&tk, K, d, s->num_kv_heads, s->total_tokens, s->k_stride_tok, s->k_stride_head))
    return cudaErrorInvalidValue;
  ScoreParams p;
  p.blob = c.blob; p.dump = dump;
  p.status = reinterpret_cast<uint32_t*>(c.blob) + 1;
  p.work_counter = reinterpret_cast<uint32_t*>(c.scratch) + 2;
  // (the status block and the work counter at the start of the scratch buffer were cleared together with the
  // rule counters, before the blob was initialised: this kernel follows that one directly)
  p.num_seqs = c.num_seqs; p.Hq = c.Hq; p.group = c.Hq / c.Hkv; p.max_nL = c.max_nL;
  p.scale_log2 = c.scale * 1.4426950408889634f;
  p.pstar = c.pstar;
  p.plan = c.plan;
  bool vec8 = dump && reinterpret_cast<uintptr_t>(dump) % 32 == 0;
  for (int b = 0; b < s->num_seqs && vec8; ++b) {
    const int S = s->cu_seqlens_host[b + 1] - s->cu_seqlens_host[b];
    vec8 = (S < c.pcl_max ? S : c.pcl_max) % 8 == 0;
  }
  p.dump_vec8 = vec8 ? 1 : 0;
  const int items = c.max_nL * c.num_seqs * c.Hq;
  const bool two = two_ctas(s, c, sm_count);
  const int ctas = two ? 2 * sm_count : sm_count, grid = items < ctas ? items : ctas;
  // launched as a programmatic dependent of the kernel that initialises the blob: its launch latency and its
  // prologue (barriers, TMEM, descriptors) hide under that kernel; it waits before it reads the blob
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid); cfg.blockDim = dim3(two ? SmemLayout<2>::kThreads : SmemLayout<4>::kThreads);
  cfg.dynamicSmemBytes = two ? SmemLayout<2>::total : SmemLayout<4>::total; cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  if (d == 128) return two ? cudaLaunchKernelEx(&cfg, score_sm100_kernel<128, 2>, tq, tk, p) : cudaLaunchKernelEx(&cfg, score_sm100_kernel<128, 4>, tq, tk, p);
  return two ? cudaLaunchKernelEx(&cfg, score_sm100_kernel<64, 2>, tq, tk, p) : cudaLaunchKernelEx(&cfg, score_sm100_kernel<64, 4>, tq, tk, p);
}
