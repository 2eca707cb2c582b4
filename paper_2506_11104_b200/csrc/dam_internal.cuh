// Internal layout of the mask blob and device helpers shared by the DAM kernels.
//
// The blob is one flat, relocatable buffer (byte offsets from its start, little endian):
//
//   DamHeader (256 B)            magic, status word, counts, section offsets
//   DamSeq[num_seqs]             per sequence: token start, S, L = min(S, pcl_max), q-block range,
//                                word offsets of its bit sections
//   qb_seq[total_qblocks]        sequence index of every global 128-row query block
//   per (seq, head) pattern bits 3 * W words: D (matched diagonal offsets r), Drev (D reversed:
//                                bit x = D[L-1-x]), V (matched columns c); W = ceil(L/32) rounded
//                                up to a multiple of 4 words
//   per (seq, head) true mask    L rows x W words, bit (j % 32) of word (j / 32) = M[i][j]
//   pair_tab[total_pairs]        first global q-block of every pair of adjacent q-blocks (2p, 2p+1) of a
//                                sequence; bit 31 set when the second block exists
//   lone[num_seqs * num_q_heads] int4 per (seq, head): its lone diagonal (see dam_lone_first_qblock) or -1, how many
//                                entries the list of a query block it is served on has in front of the diagonal's own,
//                                and the first such block
//   cols (gathered columns only) u16 per place of every gathered-column tile of every (seq, head): the head's matched
//                                columns in ascending order, 0xFFFF behind the last one
//   tile_ptr[rows + 1]           start of every row's entries in tiles[], rows = head * total_qblocks + global
//                                q-block.  Every pair of adjacent q-blocks owns a fixed range of tiles[] (the sum
//                                of the two rows' upper bounds, known from the shapes alone): the first row's
//                                entries, directly followed by the second row's, then zero entries (kind 0) up to
//                                the next pair.  [tile_ptr[r], tile_ptr[r + 1]) therefore holds row r's entries
//                                and possibly zero entries behind them, which every reader skips.
//   items[prows]                 work list of the attention kernel (DamItem, 32 B): one entry per
//                                (head, pair), the pair with the most listed tiles (both blocks
//                                together) first, with everything a CTA needs to start on it
//   tiles[...]                   one u32 per listed tile: kv tile index | kind << 28
//
// A PARTIAL tile stores no bits of its own: inside the window they are the true-mask words of the
// row, below it they follow from V and Drev (Sec. 4.3, Case 2), see dam_tile_row_bits.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/dam.h"

#define DAM_TILE 128
#define DAM_MAGIC 0x4B4D4144u      /* "DAMK" */
#define DAM_KIND_FULL 1u
#define DAM_KIND_PARTIAL 2u
#define DAM_KIND_GATHERED 3u    /* entry = gathered tile index | (columns in it - 1) << 16 | kind << 28 */
#define DAM_FLAG_ALL_ONES 1u
#define DAM_FLAG_CAUSAL_LIST 2u    /* tile lists hold only kb <= qb */
#define DAM_FLAG_GATHER 4u         /* rows from 2L-1 on list gathered-column tiles instead of vertical tiles */
#define DAM_HIST 4096

struct DamHeader {
  uint32_t magic;
  uint32_t status;          // device-side dam_status_t, 0 = ok
  uint32_t version;
  uint32_t flags;
  int32_t num_seqs;
  int32_t num_q_heads;
  int32_t total_qblocks;
  int32_t rows;             // num_q_heads * total_qblocks
  uint32_t tile_capacity;   // entries that fit in tiles[]
  uint32_t total_tiles;     // entries in use
  uint32_t full_tiles;
  uint32_t pcl_max;
  uint64_t off_seq, off_qbseq, off_dv, off_true, off_tile_ptr, off_work, off_tiles;
  uint64_t bytes_used;
  uint64_t causal_tiles;    // sum over heads and sequences of nq (nq + 1) / 2
  uint64_t off_pairtab;
  int32_t total_pairs;      // sum over sequences of ceil(nq / 2)
  int32_t prows;            // num_q_heads * total_pairs
  uint64_t gath_tiles;      // gathered-column tiles over all (seq, head): sum Hq * nL (capacity, 128 keys each)
  uint64_t attn_scratch_bytes;   // scratch dam_sparse_attention needs for this blob
  uint64_t mask_tiles;      // 128 x 128 tiles of the masks that hold an active cell (= total_tiles unless gathered)
  uint64_t head_tile_cap;   // entries of tiles[] every head owns (sum of the row bounds of all sequences)
  uint64_t reserved[7];     // [0]: 1 when the window map was scored by the tensor-core kernel, [1]: the softmax groups of its CTAs (test hooks)
  uint64_t off_lone;        // 0: no section (all-ones blob)
  uint64_t off_cols;        // 0: no section (all-ones blob, or no gathered columns)
  uint64_t off_lone2;       // (0; blobs of an earlier build have 8-byte records of the lone diagonals here, which are not read)
  uint64_t exec_tiles;      // tiles the tensor-core attention kernel multiplies (total_tiles, or fewer: lone diagonals)
};
static_assert(sizeof(DamHeader) == 256, "DamHeader must be 256 bytes");

struct DamItem {            // one unit of attention work: query blocks (2p, 2p+1) of one (sequence, head)
  int32_t head, tok0, qb0, S;      // tok0 = first token of the sequence, qb0 = 2p, S = sequence length
  uint32_t a0, a1, b1;             // tile list [a0, a1) of block 2p and [a1, b1) of block 2p+1
  uint32_t seq_hasB;               // sequence index | (second block exists) << 31
};
static_assert(sizeof(DamItem) == 32, "DamItem must be 32 bytes");

struct DamSeq {
  int32_t tok_start, S, L, nq;
  int32_t first_qblock, W, nL, first_pair;
  uint64_t dv_off;     // u32 words from off_dv: head h at dv_off + h * 3 * W
  uint64_t true_off;   // u32 words from off_true: head h at true_off + h * L * W
  uint64_t p_off;      // fp32 elements into a score tensor: head h at p_off + h * L * L
  uint64_t cnt_off;    // int32 elements into the build scratch count area: head h at cnt_off + h * cnt_stride
  uint64_t gath_off;   // gathered-column tiles: head h owns tiles [gath_off + h * nL, +nL)
  uint64_t tile_base;  // first entry of the sequence's rows inside a head's range of tiles[]
};
static_assert(sizeof(DamSeq) == 80, "DamSeq must be 80 bytes");

// The layout a build call works on, handed to its kernels by value: the header as the host computed it and, for batches
// of up to 32 sequences, their records too.  The rule kernels are short and follow one another; every dependent read of the
// header and of the sequence table in the blob costs each of them most of a microsecond.  32 records are what 4 KB of launch
// parameters hold beside the tensor maps (rounded down to a power of two); unused ones cost nothing (one sequence of 8192
// tokens, room for 6 / 16 / 32: 40.2 / 40.2 / 40.2 us of stage 1), used ones save up to a microsecond or two (8 x 8000
// tokens, 6 or 16: 171.2 / 170.3 us; 32 x 1000, 16 or 32: 219.7 / 218.1).
constexpr int kDamTabSeqs = 32;
struct DamPlan {
  DamHeader h;
  int32_t nseq;            // sequences in seq[], 0: more than fit (the records are read from the blob)
  int32_t nkeys;           // work items have fewer than this many listed tiles (or DAM_HIST - 1 of them and more)
  DamSeq seq[kDamTabSeqs];
};
static_assert(sizeof(DamPlan) <= 4096 - 1024, "the plan travels in the launch parameters");
__device__ __forceinline__ DamSeq dam_plan_seq(const DamPlan& p, const unsigned char* blob, int b) {
  return p.nseq ? p.seq[b] : reinterpret_cast<const DamSeq*>(blob + p.h.off_seq)[b];
}

// Per-(seq, head) words in the build scratch count area:
//   cntD[L], cntV[L], prefD[W + 1], prefV[W + 1], tile_pop[nL * nL], padded to a multiple of 4.
__host__ __device__ inline uint64_t dam_cnt_stride(int L, int W, int nL) {
  uint64_t n = 2ull * L + 2ull * (W + 1) + (uint64_t)nL * nL;
  return (n + 3) & ~3ull;
}
__host__ __device__ inline int dam_words(int L) { return (((L + 31) >> 5) + 3) & ~3; }
__host__ __device__ inline uint64_t dam_align(uint64_t x, uint64_t a) { return (x + a - 1) / a * a; }

// Upper bound on listed tiles of one q-block row of a DAM mask (see dam_mask_sizes): the window's column
// tiles plus the diagonal band, never more than the causal tiles of the row.  A row served by gathered-column
// tiles lists at most nL gathered tiles plus the band tiles [qb - nL, qb].
__host__ __device__ inline int dam_row_tile_bound(int qb, int nL, int L, int gather) {
  const int gather_first = (2 * L - 1 + DAM_TILE - 1) / DAM_TILE;
  if (gather && L > 0 && qb >= gather_first) {
    const int band = qb + 1 < nL + 1 ? qb + 1 : nL + 1;
    return nL + band;
  }
  int a = qb + 1, b = 2 * nL + 1;
  return a < b ? a : b;
}

// Sum of dam_row_tile_bound over the query blocks 0 .. qb-1 of a sequence: where block qb's entries start inside
// the sequence's range of a head.  (From the first gathered block on every bound is 2 nL + 1: nL gathered tiles
// and the nL + 1 band tiles; before it, min(q + 1, 2 nL + 1).)
__host__ __device__ inline uint64_t dam_row_tile_prefix(int qb, int nL, int L, int gather) {
  const int gather_first = (2 * L - 1 + DAM_TILE - 1) / DAM_TILE;
  const uint64_t m = 2ull * nL + 1;
  const uint64_t k = (gather && L > 0 && qb > gather_first) ? (uint64_t)gather_first : (uint64_t)qb;   // blocks on the plain rule
  const uint64_t j = k < m ? k : m;
  return j * (j + 1) / 2 + (k - j) * m + ((uint64_t)qb - k) * m;
}

// Running offsets of the per-sequence sections: next() gives the record of one sequence after another.
// all_ones_causal: -1 for a DAM mask, otherwise the all-ones blob's flag (cnt_off is then a tile offset per head).
struct DamSeqCursor {
  uint64_t dv, tr, po, co, go, tb;
  int fq, fp;
  __host__ __device__ inline DamSeq next(int tok0, int S, int pcl_max, int Hq, int gather, int all_ones_causal) {
    int L = S < pcl_max ? S : pcl_max;
    if (L < 0) L = 0;
    const int W = L > 0 ? dam_words(L) : 0;
    const int nL = (L + DAM_TILE - 1) / DAM_TILE, nq = (S + DAM_TILE - 1) / DAM_TILE;
    DamSeq s;
    s.tok_start = tok0; s.S = S; s.L = L; s.nq = nq;
    s.first_qblock = fq; s.W = W; s.nL = nL; s.first_pair = fp;
    s.dv_off = dv; s.true_off = tr; s.p_off = po; s.cnt_off = co; s.gath_off = go; s.tile_base = tb;
    dv += (uint64_t)Hq * 3 * W;
    tr += (uint64_t)Hq * L * W;
    po += (uint64_t)Hq * L * L;
    if (all_ones_causal < 0) co += (uint64_t)Hq * dam_cnt_stride(L, W, nL);
    else co += all_ones_causal ? (uint64_t)nq * (nq + 1) / 2 : (uint64_t)nq * nq;
    go += (uint64_t)Hq * nL;
    if (all_ones_causal < 0) tb += dam_row_tile_prefix(nq, nL, L, gather);
    fq += nq;
    fp += (nq + 1) / 2;
    return s;
  }
};

// Gathered-column tiles serve the query blocks that start at or after row 2L - 1 (first multiple of 128).
__host__ __device__ inline int dam_gather_first_qblock(int L) { return (2 * L - 1 + DAM_TILE - 1) / DAM_TILE; }
__host__ __device__ inline int dam_gather_first_row(int L) { return dam_gather_first_qblock(L) * DAM_TILE; }

// A lone diagonal: the largest matched diagonal r of a head, when it is at least 255 and no other is within 254 of it, so
// that a 128 x 128 tile with a cell of it has cells of it alone (on the query blocks below).  The usual one is r = L - 1,
// which has a single cell in the window and so matches whenever the window's last row keeps the first key: every head
// with a sink.  Its 128 keys of a query block lie across two tiles of the grid that hold nothing else; the tensor-core
// attention kernel multiplies one tile that starts at the block's first such key instead, of which a row needs one entry
// (the two listed tiles were 18 % of the attention time at 8k and 32k tokens).  Query blocks from this one on: all their
// keys on the diagonal lie beyond the tiles of the window, so no matched column meets them, and their lists have the same
// number of entries in front of the diagonal's.  With gathered columns that holds from the first block that lists them:
// the blocks before it list window tiles instead, one per tile with a matched column (L = 1024, columns 10, 200 and 900:
// three entries, where the blocks after it have one).
constexpr int kLoneMin = 255;
__host__ __device__ inline int dam_lone_first_qblock(int r, int L, bool gather) {
  const int beyond = (L + DAM_TILE - 1) / DAM_TILE + (r + DAM_TILE - 1) / DAM_TILE, gathered = gather ? dam_gather_first_qblock(L) : 0;
  return beyond > gathered ? beyond : gathered;
}

struct DamHeadBits {
  const uint32_t* D;
  const uint32_t* Drev;
  const uint32_t* V;
  const uint32_t* M;
  int L, W, S;
  int gather_from;     // first row whose matched columns are served by gathered tiles (INT_MAX: none)
};

__device__ __forceinline__ DamHeadBits dam_head_bits(const unsigned char* blob, const DamHeader* hdr,
                                                     const DamSeq& sq, int head) {
  DamHeadBits hb;
  const uint32_t* dv = reinterpret_cast<const uint32_t*>(blob + hdr->off_dv) + sq.dv_off + (uint64_t)head * 3 * sq.W;
  hb.D = dv;
  hb.Drev = dv + sq.W;
  hb.V = dv + 2 * sq.W;
  hb.M = reinterpret_cast<const uint32_t*>(blob + hdr->off_true) + sq.true_off + (uint64_t)head * sq.L * sq.W;
  hb.L = sq.L;
  hb.W = sq.W;
  hb.S = sq.S;
  hb.gather_from = (hdr->flags & DAM_FLAG_GATHER) ? dam_gather_first_row(sq.L) : 0x7FFFFFFF;
  return hb;
}

// bits [x, x + 32) of a bit array of nwords words; zero outside the array. x may be negative.
__device__ __forceinline__ uint32_t dam_window32(const uint32_t* __restrict__ bits, int nwords, int x) {
  int w = x >> 5;  // arithmetic shift: floor
  int sh = x & 31;
  uint32_t lo = (w >= 0 && w < nwords) ? __ldg(bits + w) : 0u;
  uint32_t hi = (w + 1 >= 0 && w + 1 < nwords) ? __ldg(bits + w + 1) : 0u;
  return __funnelshift_r(lo, hi, sh);
}

// The 128 mask bits of row i (index inside the sequence) against kv tile kb of a PARTIAL tile.
// Inside the window (i < L): the true-mask words.  Below it: matched columns of this tile OR the
// matched diagonals, key j active iff D[i - j]; with Drev[x] = D[L-1-x] the keys j0 .. j0+127 read
// Drev bits x0 .. x0+127, x0 = L - 1 - i + j0 (ascending in j), which also excludes j > i.
// (The CUDA-core attention and dam_mask_expand_rows.  The tensor-core attention's tile_bits says the same for the rows of a warp
// without branches: the two have to agree.)
__device__ __forceinline__ uint4 dam_tile_row_bits(const DamHeadBits& hb, int i, int kb) {
  uint4 r = make_uint4(0u, 0u, 0u, 0u);
  const int j0 = kb * DAM_TILE;
  if (i >= hb.S) return r;
  if (i < hb.L) {
    if (j0 < hb.L) r = __ldg(reinterpret_cast<const uint4*>(hb.M + (size_t)i * hb.W + kb * 4));
  } else {
    if (j0 < hb.L && i < hb.gather_from) r = __ldg(reinterpret_cast<const uint4*>(hb.V + kb * 4));
    // (five words cover the four windows)
    const int x0 = hb.L - 1 - i + j0;
    if (x0 + DAM_TILE > 0 && x0 < hb.L) {
      const int w = x0 >> 5, sh = x0 & 31;
      uint32_t d[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) d[k] = (uint32_t)(w + k) < (uint32_t)hb.W ? __ldg(hb.Drev + w + k) : 0u;
      r.x |= __funnelshift_r(d[0], d[1], sh);
      r.y |= __funnelshift_r(d[1], d[2], sh);
      r.z |= __funnelshift_r(d[2], d[3], sh);
      r.w |= __funnelshift_r(d[3], d[4], sh);
    }
  }
  return r;
}

// ones for t in [0, n), n clipped to [0, 128]
__device__ __forceinline__ uint4 dam_low_ones128(int n) {
  // (the PTX shift gives zero for a count of 32 and more, and zero minus one is all ones)
  auto w = [](int k) -> uint32_t {
    uint32_t r;
    asm("shl.b32 %0, 1, %1;" : "=r"(r) : "r"(max(k, 0)));
    return r - 1u;
  };
  return make_uint4(w(n), w(n - 32), w(n - 64), w(n - 96));
}

// Final 128 bits the attention kernels apply for row i against tile kb.  The bits of a PARTIAL tile have no key beyond
// the row already; a FULL tile is clipped to the keys that exist (and, with `causal`, to the row's own position).
__device__ __forceinline__ uint4 dam_apply_bits(const DamHeadBits& hb, uint32_t kind, int i, int kb, int causal) {
  if (kind != DAM_KIND_FULL) return dam_tile_row_bits(hb, i, kb);
  if (i >= hb.S) return make_uint4(0u, 0u, 0u, 0u);
  const int j0 = kb * DAM_TILE;
  int n = hb.S - j0;                       // keys beyond the sequence end do not exist
  if (causal) { int c = i - j0 + 1; n = c < n ? c : n; }
  return dam_low_ones128(n);
}

// Row ranges of a chunked call, handed to the kernel by value for batches of a few sequences (n = 0: read from memory).
constexpr int kRangeSeqs = DAM_ROW_RANGES_BY_VALUE;
struct DamRowRanges {
  int n;
  int2 r[kRangeSeqs];
  DamRowRanges(const int32_t* host, int num_seqs) : n(host && num_seqs <= kRangeSeqs ? num_seqs : 0) {
    for (int b = 0; b < kRangeSeqs; ++b) r[b] = b < n ? make_int2(host[2 * b], host[2 * b + 1]) : make_int2(0, 0);
  }
  // whether the pair of query blocks that starts with block qb0 of sequence `seq` is inside
  __device__ __forceinline__ bool holds(const int32_t* __restrict__ ranges, int seq, int qb0) const {
    const int r0 = qb0 * DAM_TILE;
    if (n) return r0 >= r[seq].x && r0 < r[seq].y;
    return r0 >= __ldg(ranges + 2 * seq) && r0 < __ldg(ranges + 2 * seq + 1);
  }
};

// ---- launches that follow one another ----------------------------------------------------------
// Most kernels here form a chain of short, dependent launches.  Each lets the next launch begin as soon as all
// of its own blocks are running (programmatic dependent launch) and then waits for the kernel before it to
// have completed with its memory visible: the launch latency of every link is hidden under its predecessor.
// The first kernel of a call is a link too, and a call whose blob has no gathered columns clears its status block in a
// kernel instead of a fill, which would break the chain (a pass at 1237 tokens 57.6 -> 56.1 us, 8192 tokens 150.7 -> 147.1,
// 16001 tokens at head_dim 64 163.5 -> 158.4; generation, one sequence 11.0 -> 9.5, 64 sequences 42.0 -> 40.7).
// Both instructions do nothing in a kernel that was launched the ordinary way.
__device__ __forceinline__ void dam_chain_prologue() {
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... KArgs, typename... Args>
cudaError_t dam_launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// ---- per-device state ---------------------------------------------------------------------------
// What a launch needs to know about the device it runs on, and the one-off set-up steps that CUDA wants per
// device (cudaFuncSetAttribute for the large dynamic shared memory of the tensor-core kernels).  Records are kept
// per device ordinal and filled on first use under a mutex, so that one process may drive several GPUs from
// several threads.
struct DamDeviceInfo { int cc_major, sm_count, smem_optin; };
typedef cudaError_t (*dam_device_query_fn)(int device, DamDeviceInfo* out);
typedef cudaError_t (*dam_device_setup_fn)(void);

class DamDeviceTable {
 public:
  static constexpr int kMaxDevices = 64;
  static constexpr int kMaxSetups = 32;
  // The record of `device`, filled by `query` the first time the ordinal is seen.
  cudaError_t info(int device, dam_device_query_fn query, DamDeviceInfo* out);
  // Runs `fn` (with `device` current) unless set-up step `key` already succeeded on that device.
  cudaError_t once(int device, int key, dam_device_setup_fn fn);
 private:
  struct Slot { bool filled; DamDeviceInfo info; bool done[kMaxSetups]; };
  Slot slots_[kMaxDevices] = {};
};
// (from DAM_SETUP_REF_SMEM on: one step per instance of the CUDA-core kernels)
enum { DAM_SETUP_ATTN_SMEM = 0, DAM_SETUP_SCORE_SMEM = 1, DAM_SETUP_DECODE_SMEM = 2, DAM_SETUP_REF_SMEM = 3 };

DamDeviceTable& dam_device_table();                                       // the library's own table
cudaError_t dam_current_device(int* device, DamDeviceInfo* info);         // ordinal and record of the current device

// ---- host-side launch entry points of the kernel files -----------------------------------------
struct DamBuildCtx {
  unsigned char* blob;
  unsigned char* scratch;
  int num_seqs, Hq, Hkv, d, dtype;
  int total_qblocks, rows, prows;
  int max_L, max_W, max_nL, max_nq, pcl_max;
  float pstar;       // single-compare threshold on p equivalent to the Box-Cox chain
  int per_map;       // 0, or the dam_transform_t whose threshold depends on each map's own statistics
  float tau, eps;    // for the per-map thresholds
  float mu;
  int min_support;
  float scale;
  int gather;        // list gathered-column tiles
  uint64_t off_cnt, off_cnt_end, off_keys, off_items;   // scratch sections
  DamPlan plan;
};

// `clear` (clear_bytes bytes, may be NULL) is filled with zeros by the same launch
cudaError_t dam_launch_init_blob(const dam_shape_t* shape, int pcl_max, uint32_t flags, void* blob,
                                 const DamHeader& host_hdr, void* clear, size_t clear_bytes, cudaStream_t st);
cudaError_t dam_launch_scores_ref(const void* Q, const void* K, const dam_shape_t* shape, const DamBuildCtx& c,
                                  float* scores_dump, cudaStream_t st);
cudaError_t dam_launch_bits_from_scores(const float* P, const DamBuildCtx& c, cudaStream_t st);
cudaError_t dam_launch_rule(const DamBuildCtx& c, cudaStream_t st);
cudaError_t dam_launch_all_ones(const dam_shape_t* shape, int causal, void* blob, cudaStream_t st);
cudaError_t dam_launch_expand_rows(const void* blob, int seq, int head, int row_begin, int nrows, int words,
                                   int causal, uint32_t* out, cudaStream_t st);
cudaError_t dam_launch_active_elems(const void* blob, int num_seqs, int Hq, unsigned long long* out, cudaStream_t st);
// `ranges` (device, int32[2 * num_seqs], or NULL; `ranges_host`: the same values): only the pairs of query blocks whose first row lies in
// [ranges[2b], ranges[2b+1]) of sequence b are computed
cudaError_t dam_launch_attn_ref(const void* Q, const void* K, const void* V, const void* blob,
                                const dam_shape_t* shape, int causal, float scale, void* O, float* lse,
                                void* scratch, bool keep_status, const int32_t* ranges, const int32_t* ranges_host, cudaStream_t st);
// tensor-core paths (bf16, d = 128); return cudaErrorNotSupported when the shape does not qualify
cudaError_t dam_launch_attn_sm100(const void* Q, const void* K, const void* V, const void* blob,
                                  const dam_shape_t* shape, int causal, float scale, void* O, float* lse,
                                  void* scratch, size_t scratch_bytes, const int32_t* ranges, const int32_t* ranges_host,
                                  bool run_gather, cudaStream_t st);
cudaError_t dam_launch_scores_sm100(const void* Q, const void* K, const dam_shape_t* shape, const DamBuildCtx& c,
                                    float* scores_dump, cudaStream_t st);

cudaError_t dam_launch_capture_accumulate(const float* P, const dam_shape_t* shape, int Lmax, float* A, int32_t* C,
                                          cudaStream_t st);
cudaError_t dam_launch_capture_average(const float* A, const int32_t* C, int Lmax, float eps, const dam_shape_t* shape,
                                       float* P_out, cudaStream_t st);
cudaError_t dam_launch_decode_group(const void* q, const void* K, const void* V, const void* blob, const dam_shape_t* shape,
                                    const int32_t* pos_dev, float scale, void* O, float* lse, void* scratch, cudaStream_t st);
cudaError_t dam_launch_decode(const void* q, const void* K, const void* V, const void* blob, const dam_shape_t* shape,
                              const int32_t* pos_dev, float scale, void* O, float* lse, void* scratch, cudaStream_t st);

cudaError_t dam_launch_bounded_wait_selftest(void* scratch, unsigned long long limit_ns, cudaStream_t st);
