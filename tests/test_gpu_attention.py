"""Stage-2 parity on the GPU, through the C ABI: with an identical mask, O and LSE must match the
float64 oracle within max-abs 2e-2 / mean-abs 2e-3 (bf16 in, fp32 accumulate) and 1e-3 for LSE."""
import numpy as np
import pytest
import torch

from paper_2506_11104_b200 import binding as B
from paper_2506_11104_b200 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
TOL = {torch.bfloat16: (2e-2, 2e-3, 1e-3), torch.float32: (1e-4, 1e-5, 1e-5)}


def _shape(w):
    return B.make_shape(w.cu_seqlens, w.num_q_heads, w.num_kv_heads, w.head_dim, w.Q.dtype, DEV)


def _run(w, blob, shape, causal=True, sentinel=False):
    Q, K, V = w.Q.to(DEV), w.K.to(DEV), w.V.to(DEV)
    O = lse = None
    if sentinel:
        # every row of every head must be written: a work item that was dropped would leave the NaN fill behind
        O = torch.full_like(Q, float("nan"))
        lse = torch.full((w.num_q_heads, Q.shape[0]), float("nan"), dtype=torch.float32, device=DEV)
    O, lse, scratch = B.dam_sparse_attention(Q, K, V, blob, shape, causal=causal, O=O, lse=lse)
    assert B.dam_poll_status(scratch) == 0
    # bf16 with head_dim 128 or 64 is served by the tcgen05 kernel, everything else by the CUDA-core kernel
    assert B.attention_ran_on_tensor_cores(scratch) == (w.Q.dtype == torch.bfloat16 and w.head_dim in (64, 128))
    if sentinel:
        _assert_every_row_written(O, lse)
    return O, lse


def _assert_every_row_written(O, lse):
    """No fill value left: O finite everywhere, LSE finite or -inf, and O = 0 exactly on the rows whose LSE is -inf."""
    assert torch.isfinite(O).all(), "rows of O were not written"
    assert not torch.isnan(lse).any() and not torch.isposinf(lse).any(), "rows of LSE were not written"
    empty = torch.isneginf(lse).transpose(0, 1)                       # [T, Hq]
    assert (O[empty] == 0).all()


def _check(w, O, lse, masks, rows_for, heads=None, causal=True, all_ones=False):
    mx, mn, le = TOL[w.Q.dtype]
    worst = [0.0, 0.0, 0.0]
    for b in range(len(w.cu_seqlens) - 1):
        S = w.cu_seqlens[b + 1] - w.cu_seqlens[b]
        if S == 0:
            continue
        for h in (heads if heads is not None else range(w.num_q_heads)):
            e = H.attention_errors(O, lse, w, masks, b, h, rows_for(S), causal=causal, all_ones=all_ones)
            worst = [max(a, c) for a, c in zip(worst, e)]
    assert worst[0] <= mx and worst[1] <= mn and worst[2] <= le, worst
    return worst


def _all_rows(S):
    return list(range(S))


def _sample_rows(L, n_random=256, n_blocks=8):
    """The rows around the window edges and the first row without overlap of columns and diagonals, both edge rows
    of `n_blocks` random 128-row query blocks, and `n_random` random rows."""
    def f(S, L=L):
        rng = np.random.default_rng(S)
        fixed = [0, L - 1, L, L + 1, 2 * L - 2, 2 * L - 1, S - 1, 127, 128, S - 129]
        nq = (S + 127) // 128
        for qb in rng.choice(nq, size=min(nq, n_blocks), replace=False):
            fixed += [int(qb) * 128, min(S - 1, int(qb) * 128 + 127)]
        rows = set(r for r in fixed if 0 <= r < S) | set(int(x) for x in rng.choice(S, size=min(S, n_random), replace=False))
        return sorted(rows)
    return f


HEADS8 = [0, 5, 9, 13, 18, 22, 27, 31]


@pytest.mark.parametrize("lengths,Hq,Hkv,d,dtype,causal", [
    ([512], 2, 2, 64, torch.float32, True),
    ([300, 77, 129], 4, 2, 64, torch.bfloat16, True),
    ([200], 2, 1, 32, torch.float32, False),
    ([640], 4, 1, 128, torch.bfloat16, True),
    ([257, 1, 500], 8, 2, 128, torch.bfloat16, True),
    ([384], 2, 2, 128, torch.bfloat16, False),
])
def test_all_ones_mask_is_dense_attention(lengths, Hq, Hkv, d, dtype, causal):
    w = synth.small_case(0, Hq, Hkv, d, 64, seed=7, dtype=dtype, lengths=lengths, amp=3.0)
    shape = _shape(w)
    blob = B.dam_mask_all_ones(shape, causal, DEV)
    O, lse = _run(w, blob, shape, causal=causal)
    _check(w, O, lse, None, _all_rows, causal=causal, all_ones=True)


def _masked_case(w, rows_for, heads=None, gather=False, sentinel=False):
    shape = _shape(w)
    rule = B.make_rule(w.pcl_max, w.tau, w.mu, w.lam, w.eps, gather_columns=gather)
    n = sum(w.num_q_heads * min(S, w.pcl_max) ** 2 for S in shape.lengths)
    dump = torch.zeros(n, dtype=torch.float32, device=DEV)
    blob, _ = B.dam_build_masks(w.Q.to(DEV), w.K.to(DEV), shape, rule, scores_dump=dump)
    assert B.dam_poll_status(blob) == 0
    masks = H.oracle_masks_from_dump(w, dump.cpu().numpy(), heads=heads)      # identical mask on both sides
    O, lse = _run(w, blob, shape, sentinel=sentinel)
    worst = _check(w, O, lse, masks, rows_for, heads=heads)
    return blob, shape, masks, O, lse, worst


@pytest.mark.parametrize("d", [64, 128])
def test_every_column_has_the_same_scale_at_large_logits(d):
    """Eight adjacent keys share a logit, V sets one of the eight against the others: O is zero unless some columns of a tile
    get other probabilities than their neighbours.  Logits reach 11700 in log2 units, where an argument that is not rounded
    once, in fp32, is off by a share of that.  Bound: 7 / 8 of the polynomial's 7.6e-5, and 8192 roundings of P to bf16 (rms
    1.1e-3 each), averaged: 2.7 * 1.1e-3 / sqrt(8192) = 3.3e-5."""
    n = 8192
    rng = np.random.default_rng(3)
    Q = torch.zeros(n, 1, d)
    Q[:, 0, 0] = torch.arange(n) % 255
    Q[:, 0, 1:3] = 1.0
    K = torch.zeros(n, 1, d)
    K[:, 0, 0] = 256.0                                                  # every product and sum of a logit is exact
    K[:, 0, 1] = -torch.from_numpy(np.repeat(rng.integers(0, 128, n // 8), 8)) / 8.0
    K[:, 0, 2] = -torch.from_numpy(np.repeat(rng.integers(0, 16, n // 8), 8)) / 128.0
    V = torch.zeros(n, 1, d)
    V[:, 0, :8] = -1.0
    V[torch.arange(n), 0, torch.arange(n) % 8] = 7.0
    Q, K, V = (x.to(torch.bfloat16).to(DEV) for x in (Q, K, V))
    shape = B.make_shape([0, n], 1, 1, d, torch.bfloat16, DEV)
    O, lse, scr = B.dam_sparse_attention(Q, K, V, B.dam_mask_all_ones(shape, False, DEV), shape, causal=False, softmax_scale=0.125)
    assert B.dam_poll_status(scr) == 0 and B.attention_ran_on_tensor_cores(scr)
    assert O.float().abs().max() <= 1e-4


def test_config0_every_row():
    w = synth.config0()
    blob, shape, masks, O, lse, worst = _masked_case(w, _all_rows)
    # rows below the window with no matched pattern are empty: O = 0, LSE = -inf (checked inside)
    assert torch.isfinite(O).all()


@pytest.mark.parametrize("lengths,pcl,Hq,Hkv,d,dtype", [
    ([700], 256, 4, 2, 128, torch.bfloat16),
    ([333, 1000, 64], 200, 4, 1, 64, torch.bfloat16),
    ([1500, 130], 256, 8, 2, 128, torch.bfloat16),
    ([513], 300, 2, 2, 32, torch.float32),
    ([2100, 700], 384, 8, 2, 64, torch.bfloat16),            # head_dim 64 on the tensor cores, several tiles and a ragged tail
])
@pytest.mark.parametrize("gather", [False, True])
def test_masked_small_cases_every_row(lengths, pcl, Hq, Hkv, d, dtype, gather):
    w = synth.small_case(0, Hq, Hkv, d, pcl, seed=11, dtype=dtype, lengths=lengths)
    _masked_case(w, _all_rows, gather=gather)


@pytest.mark.parametrize("S,pcl,d,dtype", [
    (300, 150, 8, torch.float32), (300, 150, 160, torch.float32),        # one and two staged buffers' largest head_dim range
    (260, 130, 256, torch.float32), (260, 130, 256, torch.bfloat16),      # two buffers do not fit with four rows per warp
    (1300, 700, 64, torch.float32), (5000, 130, 40, torch.float32),       # four rows per warp; a window of more stages than fit
])
def test_cuda_core_kernels_every_row(S, pcl, d, dtype):
    w = synth.small_case(S, 2, 1, d, pcl, seed=14, dtype=dtype) if d >= 16 else None
    if w is None:                                                        # too narrow for planted structure: noise alone
        w = synth.small_case(S, 2, 1, 16, pcl, seed=14, dtype=dtype)
        w.Q, w.K, w.V = (x[..., -d:].contiguous() for x in (w.Q, w.K, w.V))
    _masked_case(w, _sample_rows(pcl) if S > 2000 else _all_rows)


@pytest.mark.parametrize("lengths,pcl,d,dtype", [
    ([9], 9, 64, torch.float32), ([77, 1, 130], 40, 72, torch.bfloat16), ([200, 500], 64, 200, torch.float32),
    ([2900], 100, 24, torch.float32), ([3000], 100, 24, torch.float32),   # 5888 and 6144 rows: on either side of the line
    ([1400], 100, 96, torch.bfloat16), ([1500], 100, 96, torch.bfloat16),   # 2816 and 3072: the line of wider heads
    ([1400], 100, 136, torch.float32), ([1500], 100, 136, torch.float32),
])
def test_cuda_core_attention_of_few_rows(lengths, pcl, d, dtype):
    """Eight rows per block, the keys of a stage dealt over its warps: remainders of rows, keys and dimensions, keys that no
    row of a warp keeps, and the sizes around the change to four rows per warp."""
    w = synth.small_case(0, 2, 1, d, pcl, seed=15, dtype=dtype, lengths=lengths)
    _masked_case(w, _sample_rows(pcl) if max(lengths) > 2000 else _all_rows)


def _one_odd_key(n, key, value):
    """fp32 attention of n rows (two heads, lower-triangular) with one logit of every row replaced: Q, K, V on the device, O, LSE
    and the float64 outputs without that key."""
    g = torch.Generator().manual_seed(31)
    Q, K, V = (torch.randn(n, 2, 64, generator=g) for _ in range(3))
    Q[:, :, 0] = 1.0
    K[key, :, 0] = value
    Q, K, V = (x.to(DEV) for x in (Q, K, V))
    shape = B.make_shape([0, n], 2, 2, 64, torch.float32, DEV)
    O, lse, scr = B.dam_sparse_attention(Q, K, V, B.dam_mask_all_ones(shape, True, DEV), shape)
    assert B.dam_poll_status(scr) == 0
    logits = torch.einsum("ihd,jhd->hij", Q.double(), K.double()) / 8.0
    keep = torch.ones(n, n, dtype=torch.bool, device=DEV).tril()
    keep[:, key] = False
    P = torch.where(keep, logits, float("-inf")).softmax(-1).nan_to_num(0.0)       # (a row without any other key)
    return O.double(), lse, torch.einsum("hij,jhd->ihd", P, V.double())


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("key", [8, 65])
@pytest.mark.parametrize("n", [200, 3000])        # eight rows to a block, four rows to a warp
def test_cuda_core_attention_keeps_a_nan(n, key, value):
    """A NaN logit, or one of +inf, makes its rows NaN, also where a warp has no other key in the row; the rows in front of it
    are not touched."""
    O, lse, ref = _one_odd_key(n, key, value)
    assert torch.isnan(O[key:]).all()
    assert (O[:key] - ref[:key]).abs().max() <= 1e-4 and torch.isfinite(lse[:, :key]).all()


@pytest.mark.parametrize("key", [0, 8, 65])
@pytest.mark.parametrize("n", [200, 3000])
def test_cuda_core_attention_leaves_out_a_logit_of_minus_infinity(n, key):
    """A logit of -inf has no weight, also where it is the first of its row or the row's only one (O = 0, LSE = -inf)."""
    O, lse, ref = _one_odd_key(n, key, float("-inf"))
    assert (O - ref).abs().max() <= 1e-4
    assert torch.equal(torch.isneginf(lse), (torch.arange(n, device=DEV) == 0).expand(2, n) & (key == 0))


@pytest.mark.parametrize("gather", [False, True])
@pytest.mark.parametrize("lengths,pcl,Hq,Hkv,d", [
    ([1700], 384, 4, 2, 128),                # the lone diagonal crosses two tiles of every block
    ([1283, 1153, 900], 500, 4, 1, 64),      # window not a multiple of the tile; last blocks of 3 and 1 rows; one without such blocks
    ([1664], 385, 2, 2, 128),                # r = 384: whole tiles of the grid
])
def test_lone_diagonal_every_row(lengths, pcl, Hq, Hkv, d, gather):
    """Heads whose window keeps the first key in its last row: the diagonal r = L - 1 stands alone and is served by a
    tile that starts at its first key.  Head 0 attends to the first key only (a block whose list has nothing else)."""
    w = synth.small_case(0, Hq, Hkv, d, pcl, seed=23, dtype=torch.bfloat16, lengths=lengths)
    plans = [[synth.HeadPlan(sink=True, band_m=0 if h == 0 else (8, 16, 24)[h % 3], stripes=[] if h == 0 else [5, pcl // 2])
              for h in range(Hq)] for _ in lengths]
    parts = [synth.make_sequence(S, Hq, Hkv, d, min(S, pcl), plans[b], 8.0, [23, b], "cpu") for b, S in enumerate(lengths)]
    w.Q, w.K, w.V = (torch.cat([p[k] for p in parts]).to(torch.bfloat16) for k in range(3))
    blob, shape, masks, _, _, _ = _masked_case(w, _all_rows, gather=gather, sentinel=True)
    st = B.dam_mask_stats(blob, shape)
    assert st["executed_tiles"] < st["tiles"] if pcl != 385 else st["executed_tiles"] == st["tiles"]


@pytest.mark.parametrize("gather", [False, True])
@pytest.mark.parametrize("L,d", [(512, 128), (1000, 64)])
def test_lone_diagonal_at_any_distance(L, d, gather):
    """A lone diagonal far below L - 1 (a head that attends at a fixed lag), one head per distance, with matched columns
    that lie in more window tiles than they would fill as gathered columns.  The blocks between the first one beyond the
    diagonal's reach into the window and the first one with gathered columns list the window's tiles."""
    distances = [255, 300, L - 129, L - 128, L - 1]
    Hq = len(distances)
    w = synth.small_case(0, Hq, 1, d, L, seed=29, dtype=torch.bfloat16, lengths=[3 * L + 77])
    # a row keeps a handful of keys, so O reaches the largest |V|, about 5: half a bf16 step there is 2^-6, and P's rounding
    # adds 2^-9 of |V|: 0.026, over the tolerance.  With V halved (exactly) both are halved: 0.013.
    w.V = w.V * 0.5
    i = np.arange(L)
    maps = np.zeros((Hq, L, L), np.float32)
    for h, r in enumerate(distances):
        for lag in (0, r):
            maps[h, i[lag:], i[:L - lag]] = 0.5
        for c in (5, L // 3, L - 100):
            maps[h, c:, c] = 0.5
    shape = _shape(w)
    rule = B.make_rule(L, w.tau, w.mu, w.lam, w.eps, gather_columns=gather)
    blob, _ = B.dam_build_masks_from_scores(torch.from_numpy(maps).to(DEV), shape, rule)
    masks = H.oracle_masks_from_dump(w, maps.reshape(-1))
    assert [int(np.flatnonzero(m.D)[-1]) for m in masks[0]] == distances
    O, lse = _run(w, blob, shape, sentinel=True)
    _check(w, O, lse, masks, _all_rows)
    # tiles the kernel leaves out: on every block served that way, all but one of those with a cell of the diagonal
    st, S, left_out = B.dam_mask_stats(blob, shape), shape.lengths[0], 0
    for r in distances:
        first = max((L + 127) // 128 + (r + 127) // 128, (2 * L - 1 + 127) // 128 if gather else 0)
        left_out += sum((min(i0 + 128, S) - 1 - r) // 128 - (i0 - r) // 128 for i0 in range(128 * first, S, 128))
    assert left_out > 0 and st["executed_tiles"] == st["tiles"] - left_out


@pytest.mark.parametrize("d", [128, 64])
def test_gathered_blob_of_an_earlier_build(d):
    """A blob whose header has neither the list of matched columns nor the records of lone diagonals (both offsets zero, as
    in a blob that was saved before these sections existed), and one with the older records where they used to be."""
    w = synth.small_case(0, 4, 2, d, 300, seed=8, dtype=torch.bfloat16, lengths=[1500, 900])
    shape = _shape(w)
    dump = torch.zeros(2 * 4 * 300 * 300, device=DEV)
    blob, _ = B.dam_build_masks(w.Q.to(DEV), w.K.to(DEV), shape, B.make_rule(w.pcl_max, w.tau, w.mu, gather_columns=True), scores_dump=dump)
    masks = H.oracle_masks_from_dump(w, dump.cpu().numpy())
    assert any(m.V.sum() > 0 for seq in masks for m in seq)
    O, lse = _run(w, blob, shape)

    def word(name, value=None):
        at = B._HDR.fields[name][1]
        if value is not None:
            blob[at:at + 8] = torch.from_numpy(np.array([value], np.uint64).view(np.uint8)).to(DEV)
        return int(blob[at:at + 8].cpu().numpy().view(np.uint64)[0])

    lone = word("off_lone")
    word("off_lone", 0)
    word("off_lone2", lone)
    _check(w, *_run(w, blob, shape, sentinel=True), masks, _all_rows)
    word("off_lone2", 0)
    word("off_cols", 0)
    O_old, lse_old = _run(w, blob, shape, sentinel=True)
    _check(w, O_old, lse_old, masks, _all_rows)


@pytest.mark.parametrize("gather", [False, True])
def test_lone_diagonal_with_logits_of_minus_infinity(gather):
    """Rows whose key on the lone diagonal has a logit that overflows to -inf, alone (head 0: O = 0 and LSE = -inf) and
    beside a key of a column (head 1): as without the record of the lone diagonal, and the rows beside them as ever."""
    L, S, r = 512, 1500, 300
    i = np.arange(L)
    maps = np.zeros((2, L, L), np.float32)
    maps[:, i[r:], i[:L - r]] = 0.5
    maps[1, :, 0] = 0.5
    torch.manual_seed(37)
    Q, K, V = (torch.randn(S, h, 64, device=DEV).to(torch.bfloat16) for h in (2, 1, 1))
    Q[:, :, 0] = 1e30
    K[:, 0, 0] = 0.0
    K[3::3, 0, 0] = -1e30                                                   # product below the smallest float
    shape = B.make_shape([0, S], 2, 1, 64, torch.bfloat16, DEV)
    blob, _ = B.dam_build_masks_from_scores(torch.from_numpy(maps).to(DEV), shape, B.make_rule(L, 0.1, 0.8, gather_columns=gather))
    O, lse, _ = B.dam_sparse_attention(Q, K, V, blob, shape)
    at = B._HDR.fields["off_lone"][1]
    blob[at:at + 8] = 0
    O_plain, lse_plain, _ = B.dam_sparse_attention(Q, K, V, blob, shape)
    first = 1024 if gather else 896                                         # the blocks the diagonal is served on
    rows = torch.arange(first, S, device=DEV)
    overflown = (rows - r) % 3 == 0
    assert not torch.isnan(O).any() and not torch.isnan(lse).any()
    assert torch.equal(torch.isneginf(lse[0, first:]), overflown) and torch.equal(torch.isneginf(lse_plain[0, first:]), overflown)
    assert (O[first:, 0][overflown] == 0).all()
    # (one key: O is its V row either way, and LSE the logit)
    fin = rows[~overflown]
    assert torch.equal(O[fin, 0], O_plain[fin, 0]) and (lse[0, fin] - lse_plain[0, fin]).abs().max() <= TOL[torch.bfloat16][2]
    assert (O[:, 1].float() - O_plain[:, 1].float()).abs().max() <= 2e-2 and (lse[1] - lse_plain[1]).abs().max() <= 1e-3


def test_empty_rows_and_no_patterns():
    """mu > 1: nothing matches, every row below the window is empty."""
    w = synth.small_case(0, 4, 2, 128, 128, seed=5, lengths=[600])
    w.mu = 1.5
    blob, shape, masks, O, lse, _ = _masked_case(w, _all_rows)
    assert torch.isneginf(lse[:, 128:]).all() and (O[128:] == 0).all()


@pytest.mark.parametrize("gather", [False, True])
def test_config1_sampled_rows(gather):
    w = synth.config1()
    _masked_case(w, _sample_rows(1024), heads=HEADS8, gather=gather, sentinel=True)


def test_config1_dense_causal_sampled_rows():
    w = synth.config1()
    shape = _shape(w)
    blob = B.dam_mask_all_ones(shape, True, DEV)
    O, lse = _run(w, blob, shape)
    _check(w, O, lse, None, lambda S: [0, 1, 127, 128, 4095, 8191], heads=[3, 30], all_ones=True)


@pytest.mark.parametrize("gather", [False, True])
def test_config4_varlen_sampled_rows(gather):
    w = synth.config4()
    _masked_case(w, _sample_rows(1024), heads=HEADS8, gather=gather, sentinel=True)


def test_config2_layer_sampled_rows():
    """One layer of the 32-layer stack (32768 tokens, PCL 2048), in the launch configuration the benchmark times."""
    w = synth.config2_layer(5, DEV)
    blob, shape, masks, O, lse, worst = _masked_case(w, _sample_rows(2048), heads=HEADS8, gather=True, sentinel=True)
    st = B.dam_mask_stats(blob, shape)
    assert 0.01 <= st["tiles"] / st["causal_tiles"] <= 0.30


def test_config3_sampled_rows():
    """131072 tokens, PCL 4096: sampled rows of a few heads against the oracle over all 131072 keys."""
    w = synth.config3(DEV)
    _masked_case(w, _sample_rows(4096), heads=HEADS8, gather=True, sentinel=True)


def test_gathered_blob_with_small_scratch_reports_error():
    """A blob with gathered-column tiles needs the larger scratch; a scratch that holds some tiles but not all, and
    the 256-byte scratch that is enough for every other blob, are both refused on the device: O and LSE stay as
    they were and the status word says BUFFER_TOO_SMALL."""
    w = synth.small_case(0, 4, 2, 128, 128, seed=4, lengths=[900])
    shape = _shape(w)
    rule = B.make_rule(w.pcl_max, w.tau, w.mu, gather_columns=True)
    blob, _ = B.dam_build_masks(w.Q.to(DEV), w.K.to(DEV), shape, rule)
    assert B.dam_mask_sizes(shape, rule)[2] > 256
    for nbytes in (256 + 65536, 256):
        small = torch.zeros(256 + 70000, dtype=torch.uint8, device=DEV)[:nbytes]
        O = torch.full_like(w.Q.to(DEV), 7.0)
        O, lse, scr = B.dam_sparse_attention(w.Q.to(DEV), w.K.to(DEV), w.V.to(DEV), blob, shape, scratch=small, O=O)
        torch.cuda.synchronize()
        assert B.dam_poll_status(scr) == 3
        assert (O == 7.0).all()


@pytest.mark.parametrize("d", [128, 64])
def test_small_scratch_is_reported_by_every_chunk(d):
    """The kernel that clears the status word runs right before the one that writes the error: the error stays, call
    after call, and no row is written."""
    w = synth.small_case(0, 4, 2, d, 128, seed=4, lengths=[900])
    shape = _shape(w)
    Q, K, V = w.Q.to(DEV), w.K.to(DEV), w.V.to(DEV)
    blob, _ = B.dam_build_masks(Q, K, shape, B.make_rule(w.pcl_max, w.tau, w.mu, gather_columns=True))
    O, lse = torch.full_like(Q, 7.0), torch.full((4, 900), 7.0, device=DEV)
    for nbytes in (256, 256 + 65536):
        small = torch.zeros(256 + 70000, dtype=torch.uint8, device=DEV)[:nbytes]
        for k in range(20):
            B.dam_sparse_attention_rows(Q, K, V, blob, shape, [(256 * (k % 3), 256 * (k % 3) + 256)], O, lse, scratch=small)
            assert B.dam_poll_status(small) == 3
    assert (O == 7.0).all() and (lse == 7.0).all()


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("ranges", [None, [(0, 0), (0, 0)]])
def test_empty_batch_clears_the_status_block(dtype, ranges):
    """A call with no tokens leaves a clean status block, whatever the buffer held."""
    shape = B.make_shape([0, 0, 0], 2, 1, 128, dtype, DEV)
    x, lse = torch.zeros(8, 2, 128, dtype=dtype, device=DEV), torch.zeros(2, 8, device=DEV)
    blob = torch.zeros(4096, dtype=torch.uint8, device=DEV)
    scratch = torch.full((256,), 3, dtype=torch.uint8, device=DEV)
    if ranges is None:
        B.dam_sparse_attention(x, x, x, blob, shape, O=x, lse=lse, scratch=scratch)
    else:
        B.dam_sparse_attention_rows(x, x, x, blob, shape, ranges, x, lse, scratch=scratch)
    assert B.dam_poll_status(scratch) == 0 and not scratch.any()


def test_threads_with_different_shared_memory_sizes():
    """Threads on streams of their own whose calls share a kernel instance but not the amount of shared memory it is
    launched with (fp32: head_dim 136 and 160 for the attention, windows of one and six stages for the scores)."""
    import threading
    failures = []

    def work(d, S):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            w = synth.small_case(S, 2, 1, d, S, seed=6, dtype=torch.float32)
            shape = _shape(w)
            rule = B.make_rule(S, 0.1, 0.8)
            Q, K, V = w.Q.to(DEV), w.K.to(DEV), w.V.to(DEV)
            blob, build = B.dam_build_masks(Q, K, shape, rule)
            O, lse, scratch = B.dam_sparse_attention(Q, K, V, blob, shape)
            first = O.clone()
            try:
                for _ in range(1500):
                    B.dam_build_masks(Q, K, shape, rule, blob, build)
                    B.dam_sparse_attention(Q, K, V, blob, shape, O=O, lse=lse, scratch=scratch)
                stream.synchronize()
                assert torch.equal(O, first)
            except Exception as e:                           # (an assertion in a thread would be lost)
                failures.append((d, S, repr(e)))

    threads = [threading.Thread(target=work, args=a) for a in ((160, 64), (136, 64), (160, 384), (136, 384))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures


def test_bounded_wait_times_out_cleanly():
    """Waits of both kinds that nothing satisfies give up, the one by the clock after its limit, the one by polls after a
    number of them that takes some seconds, and the expired one releases the other; the status word says so although the
    thread that writes it has long been done, and the device keeps working (the next kernel runs and is correct)."""
    status, (waited_ns, polls_ns, released_ns, gave_up) = B.bounded_wait_words(DEV, limit_us=20000)
    assert status == 5 and gave_up == 3                  # DAM_ERR_DEVICE_TIMEOUT
    assert 15e6 <= waited_ns <= 500e6 and released_ns <= waited_ns + 100e6
    assert 0.3e9 <= polls_ns <= 10e9
    w = synth.small_case(0, 4, 2, 128, 128, seed=9, lengths=[300])
    shape = _shape(w)
    blob = B.dam_mask_all_ones(shape, True, DEV)
    O, lse = _run(w, blob, shape)
    _check(w, O, lse, None, _all_rows, all_ones=True)


def test_strided_qkv_views():
    """Q, K, V as views of one fused [T, Hq + 2 Hkv, d] tensor: the strides of dam_shape_t are honoured by the
    TMA descriptors and by the plain kernels."""
    for dtype, d in ((torch.bfloat16, 128), (torch.float32, 64)):
        Hq, Hkv = 4, 2
        w = synth.small_case(0, Hq, Hkv, d, 128, seed=13, dtype=dtype, lengths=[400, 131])
        T = w.Q.shape[0]
        fused = torch.zeros(T, Hq + 2 * Hkv, d, dtype=dtype, device=DEV)
        fused[:, :Hq] = w.Q.to(DEV); fused[:, Hq:Hq + Hkv] = w.K.to(DEV); fused[:, Hq + Hkv:] = w.V.to(DEV)
        Qv, Kv, Vv = fused[:, :Hq], fused[:, Hq:Hq + Hkv], fused[:, Hq + Hkv:]
        st = ((Hq + 2 * Hkv) * d, d)
        shape = B.make_shape(w.cu_seqlens, Hq, Hkv, d, dtype, DEV, q_strides=st, k_strides=st, v_strides=st)
        rule = B.make_rule(w.pcl_max, w.tau, w.mu, gather_columns=True)
        n = sum(Hq * min(S, w.pcl_max) ** 2 for S in shape.lengths)
        dump = torch.zeros(n, dtype=torch.float32, device=DEV)
        blob, _ = B.dam_build_masks(Qv, Kv, shape, rule, scores_dump=dump)
        masks = H.oracle_masks_from_dump(w, dump.cpu().numpy())
        O = torch.empty(T, Hq, d, dtype=dtype, device=DEV)
        O, lse, scr = B.dam_sparse_attention(Qv, Kv, Vv, blob, shape, O=O)
        assert B.dam_poll_status(scr) == 0 and B.dam_poll_status(blob) == 0
        _check(w, O, lse, masks, _all_rows)


@pytest.mark.parametrize("offset,row_pad,head_pad", [(0, 8, 0), (8, 0, 0), (0, 0, 8), (16, 32, 16)])
@pytest.mark.parametrize("d", [64, 128])
def test_output_rows_of_any_alignment(d, offset, row_pad, head_pad):
    """O is written 32 bytes at a time where its rows start on 32-byte boundaries, 16 bytes otherwise: the same values
    either way, and nothing between the rows."""
    Hq, Hkv = 4, 2
    w = synth.small_case(0, Hq, Hkv, d, 128, seed=13, lengths=[700, 131])
    Q, K, V = w.Q.to(DEV), w.K.to(DEV), w.V.to(DEV)
    rule = B.make_rule(w.pcl_max, w.tau, w.mu, gather_columns=True)
    shape = _shape(w)
    blob, _ = B.dam_build_masks(Q, K, shape, rule)
    O_ref, lse_ref = _run(w, blob, shape, sentinel=True)
    T, hs = Q.shape[0], d + head_pad
    ts = Hq * hs + row_pad
    buf = torch.full((offset + T * ts,), 7.0, dtype=torch.bfloat16, device=DEV)
    O = buf[offset:].as_strided((T, Hq, d), (ts, hs, 1))
    padded = B.make_shape(w.cu_seqlens, Hq, Hkv, d, torch.bfloat16, DEV, o_strides=(ts, hs))
    _, lse, scr = B.dam_sparse_attention(Q, K, V, blob, padded, O=O)
    assert B.dam_poll_status(scr) == 0 and B.attention_ran_on_tensor_cores(scr)
    assert torch.equal(O, O_ref) and torch.equal(lse, lse_ref)
    O.fill_(7.0)
    assert (buf == 7.0).all()


@pytest.mark.parametrize("gather", [False, True])
@pytest.mark.parametrize("d", [64, 128])
def test_empty_items_behind_an_item_with_tiles(d, gather):
    """No pattern matches: 16 items with tiles in both blocks, then more than eight empty ones per multiprocessor, so the next
    key tile (or the end of the list) comes three records or more behind a last step.  Every row is written, over the whole
    batch and over row ranges."""
    S = 20000
    w = synth.small_case(0, 16, 4, d, 256, seed=23, lengths=[S], mu=1.5)
    blob, shape, masks, O, lse, _ = _masked_case(w, _sample_rows(256, 64, 2), heads=[0, 7, 15], gather=gather, sentinel=True)
    assert torch.isneginf(lse[:, 256:]).all() and torch.isfinite(lse[:, 0]).all()
    Q, K, V = w.Q.to(DEV), w.K.to(DEV), w.V.to(DEV)
    Or, lr = torch.full_like(O, float("nan")), torch.full_like(lse, float("nan"))
    for r in [(0, 9984), (9984, S)]:
        assert B.dam_poll_status(B.dam_sparse_attention_rows(Q, K, V, blob, shape, [r], Or, lr)) == 0
    assert torch.equal(Or, O) and torch.equal(lr, lse)


@pytest.mark.parametrize("gather", [False, True])
def test_degenerate_lengths(gather):
    """Empty and one-token sequences inside a packed batch, a sequence shorter than a tile, MHA (group 1)."""
    w = synth.small_case(0, 4, 4, 128, 64, seed=17, lengths=[0, 1, 5, 0, 257, 128])
    _masked_case(w, _all_rows, gather=gather)
    shape = _shape(w)
    blob = B.dam_mask_all_ones(shape, True, DEV)
    O, lse = _run(w, blob, shape)
    _check(w, O, lse, None, _all_rows, all_ones=True)


@pytest.mark.parametrize("lengths,Hq,Hkv,d,dtype,gather", [
    ([1024, 300, 700], 8, 2, 128, torch.bfloat16, False),
    ([1536], 4, 1, 128, torch.bfloat16, True),
    ([900, 512], 2, 2, 64, torch.float32, False),
])
def test_chunked_prefill_equals_one_call(lengths, Hq, Hkv, d, dtype, gather):
    """Row ranges: chunks of 256 / 512 rows, with the cache beyond each chunk's end poisoned, give the oracle's
    O and LSE on every row (Sec. 4.3, Case 2, applied to rows that arrive in chunks) and, bit for bit, the output of
    the single call (the arithmetic per row is the same and no row reads a key beyond itself)."""
    w = synth.small_case(0, Hq, Hkv, d, 128, seed=21, dtype=dtype, lengths=lengths)
    shape = _shape(w)
    rule = B.make_rule(w.pcl_max, w.tau, w.mu, w.lam, w.eps, gather_columns=gather)
    Q, K, V = w.Q.to(DEV), w.K.to(DEV), w.V.to(DEV)
    dump = torch.zeros(sum(Hq * min(S, w.pcl_max) ** 2 for S in lengths), dtype=torch.float32, device=DEV)
    blob, _ = B.dam_build_masks(Q, K, shape, rule, scores_dump=dump)
    masks = H.oracle_masks_from_dump(w, dump.cpu().numpy())
    O_ref, lse_ref, _ = B.dam_sparse_attention(Q, K, V, blob, shape, causal=True)
    O = torch.full_like(O_ref, 7.0)
    lse = torch.full_like(lse_ref, 7.0)
    chunk = 512 if d == 128 else 256
    done = [0] * len(lengths)
    while any(dn < S for dn, S in zip(done, lengths)):
        ranges, Kc, Vc = [], K.clone(), V.clone()
        for b, S in enumerate(lengths):
            r0, r1 = (done[b], min(S, done[b] + chunk)) if done[b] < S else (0, 0)
            ranges.append((r0, r1))
            t0 = w.cu_seqlens[b]
            Kc[t0 + r1: t0 + S] = float("nan")               # keys that have not arrived yet
            Vc[t0 + r1: t0 + S] = float("nan")
            done[b] = max(done[b], r1)
        scratch = B.dam_sparse_attention_rows(Q, Kc, Vc, blob, shape, ranges, O, lse)
        assert B.dam_poll_status(scratch) == 0
    _check(w, O, lse, masks, _all_rows)                      # the chunked output itself against the oracle
    assert torch.equal(O, O_ref)
    assert torch.equal(lse, lse_ref)


@pytest.mark.parametrize("lengths,Hq,ranges", [
    ([600] * 16, 4, [(256, 600)] * 16),                          # the last batch whose ranges travel with the launch
    ([600, 0, 256] * 5 + [700, 40], 4, [(0, 512), (0, 0), (0, 256)] * 5 + [(512, 700), (0, 40)]),      # one sequence more
    ([32700], 128, [(20480, 20992)]),                            # 16384 items, as many as a CTA marks
    ([33000], 128, [(20480, 20992)]),                            # 16512: claimed one after the other
])
def test_row_ranges_of_long_lists_and_many_sequences(lengths, Hq, ranges):
    """Rows of the single call, bit for bit, and no others."""
    _rows_as_in_the_single_call(lengths, Hq, 64, ranges)


@pytest.mark.parametrize("S,Hq", [(30720, 32), (30976, 32), (32700, 128), (33000, 128)])      # 3840, 3872, 16384, 16512 items
def test_row_ranges_of_long_lists_at_head_dim_128(S, Hq):
    """The lengths of work lists at which the marks of the wanted items, and with them the slots for K and V, change."""
    _rows_as_in_the_single_call([S], Hq, 128, [(20480, 20992)])


def _rows_as_in_the_single_call(lengths, Hq, d, ranges):
    torch.manual_seed(23)
    cu = np.concatenate([[0], np.cumsum(lengths)]).tolist()
    Q = torch.randn(cu[-1], Hq, d, dtype=torch.bfloat16, device=DEV)
    K, V = (torch.randn(cu[-1], 2, d, dtype=torch.bfloat16, device=DEV) for _ in range(2))
    shape = B.make_shape(cu, Hq, 2, d, torch.bfloat16, DEV)
    blob, _ = B.dam_build_masks(Q, K, shape, B.make_rule(64, 0.1, 0.5, gather_columns=True))
    O_ref, lse_ref, _ = B.dam_sparse_attention(Q, K, V, blob, shape, causal=True)
    O, lse = torch.full_like(O_ref, 7.0), torch.full_like(lse_ref, 7.0)
    scratch = B.dam_sparse_attention_rows(Q, K, V, blob, shape, ranges, O, lse)
    assert B.dam_poll_status(scratch) == 0
    inside = torch.zeros(cu[-1], dtype=torch.bool, device=DEV)
    for t0, (r0, r1) in zip(cu, ranges):
        inside[t0 + r0: t0 + r1] = True
    assert torch.equal(O[inside], O_ref[inside]) and torch.equal(lse[:, inside], lse_ref[:, inside])
    assert (O[~inside] == 7.0).all() and (lse[:, ~inside] == 7.0).all()


def test_row_ranges_under_stream_capture():
    """Ranges that travel with the launch are captured with it; a batch whose ranges would be copied from host memory at
    every replay is refused, and the capture around the refused call stays valid."""
    def case(n):
        torch.manual_seed(31)
        Q = torch.randn(300 * n, 2, 64, dtype=torch.bfloat16, device=DEV)
        K, V = (torch.randn(300 * n, 1, 64, dtype=torch.bfloat16, device=DEV) for _ in range(2))
        shape = B.make_shape([300 * b for b in range(n + 1)], 2, 1, 64, torch.bfloat16, DEV)
        rule = B.make_rule(64, 0.1, 0.5, gather_columns=True)
        blob, _ = B.dam_build_masks(Q, K, shape, rule)
        scratch = torch.zeros(B.dam_mask_sizes(shape, rule)[2], dtype=torch.uint8, device=DEV)
        return Q, K, V, blob, shape, [(256, 300)] * n, torch.zeros_like(Q), torch.zeros(2, 300 * n, device=DEV), scratch

    few, many = case(16), case(17)
    B.dam_sparse_attention_rows(*many[:8], scratch=many[8])                   # (a first call outside of the capture)
    B.dam_sparse_attention_rows(*few[:8], scratch=few[8])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.dam_sparse_attention_rows(*few[:8], scratch=few[8])
        with pytest.raises(RuntimeError):
            B.dam_sparse_attention_rows(*many[:8], scratch=many[8])
    few[0].neg_()
    want = few[6].clone()
    B.dam_sparse_attention_rows(*few[:6], want, few[7], scratch=few[8])
    few[6].zero_()
    graph.replay()
    torch.cuda.synchronize()
    inside = (torch.arange(300 * 16, device=DEV) % 300) >= 256
    assert torch.equal(few[6][inside], want[inside]) and not few[6][~inside].any() and want[inside].any()


def test_row_ranges_leave_other_rows_alone_and_reject_odd_bounds():
    w = synth.small_case(0, 4, 2, 128, 128, seed=22, dtype=torch.bfloat16, lengths=[768, 512])
    shape = _shape(w)
    rule = B.make_rule(w.pcl_max, w.tau, w.mu, w.lam, w.eps)
    Q, K, V = w.Q.to(DEV), w.K.to(DEV), w.V.to(DEV)
    blob, _ = B.dam_build_masks(Q, K, shape, rule)
    O_ref, lse_ref, _ = B.dam_sparse_attention(Q, K, V, blob, shape, causal=True)
    O = torch.full_like(O_ref, 7.0)
    lse = torch.full_like(lse_ref, 7.0)
    B.dam_sparse_attention_rows(Q, K, V, blob, shape, [(256, 512), (0, 0)], O, lse)
    assert torch.equal(O[256:512], O_ref[256:512]) and torch.equal(lse[:, 256:512], lse_ref[:, 256:512])
    keep = torch.ones(O.shape[0], dtype=torch.bool, device=DEV)
    keep[256:512] = False
    assert (O[keep] == 7.0).all() and (lse[:, keep] == 7.0).all()
    for bad in ([(128, 512), (0, 0)], [(0, 300), (0, 0)], [(0, 1024), (0, 0)], [(512, 256), (0, 0)]):
        with pytest.raises(B.DamError):
            B.dam_sparse_attention_rows(Q, K, V, blob, shape, bad, O, lse)


@pytest.mark.parametrize("gather", [False, True])
def test_inactive_keys_with_huge_logits(gather):
    """Keys outside every pattern whose logits dwarf the active ones (K rows below the window scaled up): the
    row maximum over all entries of a tile then lies far above the masked one, which is the case the softmax
    must detect (the reference may only follow the masked maximum) and must survive without overflow."""
    w = synth.small_case(0, 4, 2, 128, 128, seed=31, dtype=torch.bfloat16, lengths=[1280, 520])
    rng = np.random.default_rng(5)
    K = w.K.clone()
    for b, S in enumerate([1280, 520]):
        t0 = w.cu_seqlens[b]
        rows = rng.choice(np.arange(128, S), size=(S - 128) // 3, replace=False)
        K[t0 + torch.as_tensor(rows)] *= 12.0                # logits up to a few hundred in either direction
    w.K = K
    if hasattr(w, "_host_qkv"):
        del w._host_qkv
    _, _, _, _, _, worst = _masked_case(w, _sample_rows(128), gather=gather)
    assert all(np.isfinite(worst))
