"""GPU parity of the verification attention against the fp64 oracle, through the C ABI.

Tolerance: max-abs 2e-2 on bf16 outputs of O(1) magnitude (fp32 accumulation, probabilities and
outputs rounded to bf16: relative 2^-8 each); lse within 2e-3."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2509_15235_b200 import synth

pytestmark = pytest.mark.gpu
TOL = 2e-2
LSE_TOL = 2e-3


@pytest.fixture(scope="module")
def gu():
    import gpu_util
    return gpu_util


def _check(gu, q, k, v, kv_len, mask, scale, split_form=0):
    out, lse, status = gu.run_attn(q, k, v, kv_len, mask, scale, split_form=split_form)
    want, want_lse = oracle.tree_attn(q, k, v, kv_len, mask, scale)
    assert status == 0
    assert not np.isnan(out).any()
    err = np.abs(out - want).max()
    assert err <= TOL, f"max abs err {err}"
    finite = np.isfinite(want_lse)
    assert np.array_equal(np.isfinite(lse), finite)
    if finite.any():
        assert np.abs(lse[finite] - want_lse[finite]).max() <= LSE_TOL
    return err


def _case(cfg, layer=0, S_max=None):
    t = synth.make_tree_inputs(cfg)
    x = synth.make_layer_tensors(cfg, layer, S_max=S_max)
    mask, _, _ = oracle.tree_mask(t["parents"])
    return x["q"], x["k_cache"], x["v_cache"], t["kv_len"], mask


def test_tiny_config_full_parity(gu):
    cfg = synth.get_config("tiny")
    _check(gu, *_case(cfg), 1 / math.sqrt(cfg.D))


@pytest.mark.parametrize("Hq,Hkv,D,N,S,S_max", [
    (4, 4, 64, 8, 256, 320),      # tiny-like
    (4, 4, 128, 60, 707, 832),    # MHA, ragged tail, several tiles
    (14, 2, 128, 60, 533, 640),   # GQA ratio 7 (Qwen2.5-VL-7B-like)
    (16, 2, 128, 16, 300, 384),   # GQA ratio 8, small tree
    (8, 1, 128, 128, 200, 384),   # GQA ratio 8, largest tree: 1024 query rows per kv head
    (2, 2, 64, 1, 77, 128),       # a single node (plain decode step)
    (4, 2, 128, 31, 1000, 1088),  # the paper's 30-token tree plus root
    (3, 3, 128, 65, 130, 256),    # two mask words
])
@pytest.mark.parametrize("split_form", [0, 1, 2, 3])
def test_shapes_span_tiles_tails_and_group_sizes(gu, Hq, Hkv, D, N, S, S_max, split_form):
    rng = np.random.Generator(np.random.Philox(Hq * 1000 + N))
    B = 2
    q = synth.normal_bf16((B, N, Hq, D), 1 + N)
    k = synth.normal_bf16((B, Hkv, S_max, D), 2 + N)
    v = synth.normal_bf16((B, Hkv, S_max, D), 3 + N)
    kv_len = np.array([S, max(0, S - 61)], dtype=np.int32)
    parents = np.stack([synth.draw_tree(N, 6, 4, rng) for _ in range(B)])
    mask, _, _ = oracle.tree_mask(parents)
    _check(gu, q, k, v, kv_len, mask, 1 / math.sqrt(D), split_form=split_form)


# Head size 64 on the tensor-core kernel: one node on an empty cache, a full and a just overfull 64-row block, a row block
# of 128 with a ragged rest, more steps than the rings have stages (6), a tree that straddles two steps.
@pytest.mark.parametrize("Hq,Hkv,N,S,S_max", [
    (4, 4, 1, 0, 64), (4, 4, 64, 127, 256), (5, 1, 13, 640, 700), (16, 4, 127, 2049, 2304), (8, 2, 33, 1000, 1152),
    (2, 2, 128, 64, 192),
])
@pytest.mark.parametrize("split_form", [0, 1, 2, 3])
def test_head_size_64_edges(gu, Hq, Hkv, N, S, S_max, split_form):
    rng = np.random.Generator(np.random.Philox(Hq * 1000 + N + 64))
    B, D = 3, 64
    q = synth.normal_bf16((B, N, Hq, D), 5 + N)
    k = synth.normal_bf16((B, Hkv, S_max, D), 6 + N)
    v = synth.normal_bf16((B, Hkv, S_max, D), 7 + N)
    kv_len = np.array([S, S // 3, max(0, S - 1)], dtype=np.int32)
    parents = np.stack([synth.draw_tree(N, 6, 4, rng) for _ in range(B)])
    mask, _, _ = oracle.tree_mask(parents)
    _check(gu, q, k, v, kv_len, mask, 1 / math.sqrt(D), split_form=split_form)


# Units of 256 query rows in two tiles, which the host chooses by the capacity (40000 slots: mostly NaN here): an empty cache
# and several steps; a second block whose second tile has 36 rows; a third block with 4 rows in its second tile; 136 rows,
# 8 of them in the second tile; head size 64; clusters of three CTAs and of one; more kv heads than groups of CTAs (several segments per CTA).
@pytest.mark.parametrize("Hq,Hkv,D,N,kv_len,S_max,split_form", [
    (16, 2, 128, 128, [0, 700], 40000, 0), (28, 4, 128, 60, [1, 1000], 40000, 0), (16, 2, 128, 128, [700, 0, 64, 333, 5], 20000, 2),
    (28, 4, 128, 92, [515, 127], 40000, 0), (8, 1, 128, 17, [250, 40], 40000, 0), (16, 4, 64, 100, [3000, 64], 40000, 0),
    (16, 4, 64, 128, [172, 1, 100, 172, 30, 128, 77, 0, 172, 129], 300, 2), (28, 4, 128, 128, [172, 1, 100, 172, 30, 128, 77, 0, 172, 129], 300, 0),
])
def test_two_tile_units(gu, Hq, Hkv, D, N, kv_len, S_max, split_form):
    B, used = len(kv_len), max(kv_len) + N
    rng = np.random.Generator(np.random.Philox(Hq * 1000 + N + D))
    q = synth.normal_bf16((B, N, Hq, D), 15 + N)
    k = np.full((B, Hkv, S_max, D), 0x7FC0, dtype=np.uint16)
    v = np.full((B, Hkv, S_max, D), 0x7FC0, dtype=np.uint16)
    k[:, :, :used] = synth.normal_bf16((B, Hkv, used, D), 16 + N)
    v[:, :, :used] = synth.normal_bf16((B, Hkv, used, D), 17 + N)
    for b in range(B):
        k[b, :, kv_len[b] + N:] = 0x7FC0
        v[b, :, kv_len[b] + N:] = 0x7FC0
    parents = np.stack([synth.draw_tree(N, 6, 4, rng) for _ in range(B)])
    mask, _, _ = oracle.tree_mask(parents)
    _, kernels = gu.kernels_of(lambda: _check(gu, q, k, v, np.array(kv_len, dtype=np.int32), mask, 1 / math.sqrt(D), split_form=split_form))
    assert any("attn_tc5_wide_kernel" in n for n in kernels), kernels      # the estimates choose it: a change there must not go unseen


# The merge of a cluster's partials at head size 64 over every cluster size that 4 to 96 units lead to (15 units or fewer: eight
# CTAs each, 16 to 22: six, ... 34 to 45: three), with units of 128 and of 256 rows: the share of a rank is then often no whole
# number of warps (43 rows x 16 column quads in rounds of 512 or 256).
@pytest.mark.parametrize("N", [31, 128])
@pytest.mark.parametrize("B", [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 12])
def test_head_size_64_cluster_merge_shares(gu, B, N):
    rng = np.random.Generator(np.random.Philox(6400 + B))
    Hq, Hkv, D, S_max = 16, 4, 64, 640
    q = synth.normal_bf16((B, N, Hq, D), 25 + B)
    k = synth.normal_bf16((B, Hkv, S_max, D), 26 + B)
    v = synth.normal_bf16((B, Hkv, S_max, D), 27 + B)
    kv_len = rng.integers(0, S_max - N + 1, size=B).astype(np.int32)
    parents = np.stack([synth.draw_tree(N, 6, 4, rng) for _ in range(B)])
    mask, _, _ = oracle.tree_mask(parents)
    _check(gu, q, k, v, kv_len, mask, 1 / math.sqrt(D), split_form=2)


@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("N,kv_len,S_max", [
    (16, [3, 40, 240], 256),                  # one and two steps: most ranks of a cluster have none
    (16, [1400, 900, 2100], 2176),            # one to three steps per rank
    (17, [4400, 3300, 2900], 4480),           # three to five; two row blocks, the last of 8 rows
])
def test_units_of_128_rows_in_clusters(gu, D, N, kv_len, S_max):
    """The cluster form whose two groups of softmax warps take alternate steps: none, one, odd and even numbers of them."""
    B, Hq, Hkv = len(kv_len), 16, 2
    rng = np.random.Generator(np.random.Philox(4100 + N))
    q = synth.normal_bf16((B, N, Hq, D), 4101)
    k = synth.normal_bf16((B, Hkv, S_max, D), 4102)
    v = synth.normal_bf16((B, Hkv, S_max, D), 4103)
    parents = np.stack([synth.draw_tree(N, 6, 4, rng) for _ in range(B)])
    mask, _, _ = oracle.tree_mask(parents)
    _check(gu, q, k, v, np.asarray(kv_len, dtype=np.int32), mask, 1 / math.sqrt(D), split_form=2)


@pytest.mark.parametrize("split_form", [1, 3])
@pytest.mark.parametrize("Hkv,D,N,kv_len,S_max", [
    (48, 128, 60, [0, 5, 70, 900], 1024),     # units of 1, 1, 2 and 8 steps: ranges that begin or end where a unit has no work
    (80, 128, 3, [1300, 125], 1408),          # units of 11 and 1 steps, three rows each
    (52, 64, 33, [700, 300, 1], 768),
])
def test_more_units_than_ctas(gu, Hkv, D, N, kv_len, S_max, split_form):
    """The even split with several segments per CTA: their starts count as steps when the line is cut, and the q rows of later
    segments come through the K ring."""
    B = len(kv_len)
    rng = np.random.Generator(np.random.Philox(4000 + N))
    q = synth.normal_bf16((B, N, Hkv, D), 4001)
    k = synth.normal_bf16((B, Hkv, S_max, D), 4002)
    v = synth.normal_bf16((B, Hkv, S_max, D), 4003)
    parents = np.stack([synth.draw_tree(N, 6, 4, rng) for _ in range(B)])
    mask, _, _ = oracle.tree_mask(parents)
    _check(gu, q, k, v, np.asarray(kv_len, dtype=np.int32), mask, 1 / math.sqrt(D), split_form=split_form)


# Nodes that see one key (their own slot; kv_len 0) or two (the one committed key and their own): a row's sum is then one or
# two exponentials, and every column of a step has a node whose weight is formed there.  Small integers in q and k make the
# scores exact, so lse carries the roundings of the scaling, of two exponentials (2 ulp each) and of one logarithm: below
# 2^-22 * (2 + |score|) each, 2e-6 in all for scores up to 4.
@pytest.mark.parametrize("static", [False, True])
@pytest.mark.parametrize("Hq,Hkv,D,N,S_max", [(4, 4, 64, 60, 256), (4, 1, 64, 100, 256), (4, 4, 128, 60, 256), (4, 1, 128, 100, 256),
                                              (16, 2, 64, 128, 40000), (16, 2, 128, 128, 40000)])
def test_lse_of_rows_with_one_or_two_keys(gu, Hq, Hkv, D, N, S_max, static):
    _one_or_two_keys(gu, Hq, Hkv, D, N, S_max, static)


def _one_or_two_keys(gu, Hq, Hkv, D, N, S_max, static=False, split_form=0):
    from paper_2509_15235_b200 import binding
    rng = np.random.Generator(np.random.Philox(Hq * 1000 + N + D))
    B, scale = 2, 1 / 16
    small = lambda *shape: synth.f32_to_bf16_bits(rng.integers(-2, 3, size=shape).astype(np.float32))
    q, k = small(B, N, Hq, D), np.zeros((B, Hkv, S_max, D), dtype=np.uint16)
    k[:, :, :N + 1] = small(B, Hkv, N + 1, D)
    v = np.zeros_like(k)
    v[:, :, :N + 1] = synth.normal_bf16((B, Hkv, N + 1, D), 5 + N)
    kv_len = np.array([0, 1], dtype=np.int32)
    mask = np.zeros((B, N, (N + 63) // 64), dtype=np.uint64)
    for i in range(N):
        mask[:, i, i // 64] = np.uint64(1 << (i % 64))
    if static:
        out = torch.zeros((B, N, Hq, D), dtype=torch.bfloat16, device="cuda")
        lse = torch.zeros((B, Hq, N), dtype=torch.float32, device="cuda")
        binding.tree_verify_attn_static(gu.bf16_dev(q), gu.bf16_dev(k), gu.bf16_dev(v), gu.i32_dev(kv_len), gu.u64_dev(mask), scale, out, lse)
        out, lse = out.float().cpu().numpy(), lse.cpu().numpy()
    else:
        out, lse, status = gu.run_attn(q, k, v, kv_len, mask, scale, split_form=split_form)
        assert status == 0
    want, want_lse = oracle.tree_attn(q, k[:, :, :N + 1], v[:, :, :N + 1], kv_len, mask, scale)
    assert np.abs(out - want).max() <= TOL
    assert np.abs(lse - want_lse).max() <= 2e-6


# ---- units of 128 rows in clusters, whose two groups of softmax warps take alternate steps ----
def _ran_alternate_steps(kernels):
    """The one-tile kernel in its cluster form with units of 128 rows: template arguments false, true, ..."""
    return any("attn_tc5_kernel<false, true" in n or "attn_tc5_kernelILb0ELb1E" in n for n in kernels)


def _alternate_case(D, seed, B=24):
    """24 sequences x 2 kv heads of 128 rows: clusters of three CTAs, four steps to each, so that both groups of a CTA have a second
    step; lengths end in every part of the last step, and what lies past them is NaN."""
    N, Hq, Hkv, S_max = 16, 16, 2, 1536
    rng = np.random.Generator(np.random.Philox(seed))
    q = synth.normal_bf16((B, N, Hq, D), seed + 1)
    k = synth.normal_bf16((B, Hkv, S_max, D), seed + 2)
    v = synth.normal_bf16((B, Hkv, S_max, D), seed + 3)
    kv_len = np.array([S_max - N - 1 - 5 * b for b in range(B)], dtype=np.int32)
    parents = np.stack([synth.draw_tree(N, 6, 4, rng) for _ in range(B)])
    mask, _, _ = oracle.tree_mask(parents)
    return q, k, v, kv_len, mask


def _nan_past_the_end(kv_len, N, *caches):
    for c in caches:
        for b, S in enumerate(kv_len):
            c[b, :, S + N:] = 0x7FC0


@pytest.mark.parametrize("D", [128, 64])
def test_alternate_steps_move_the_reference_maximum(gu, D):
    """Scores that climb by 6 c (8.7 c in log2 units) per step, c by row from -2 to 2, so that rows of one warp move their reference in
    other steps, and values that shrink by e^6 per step: with c = 1 every step has the same part in a row's output, whatever has become
    of the reference since.  A row's output is measured against its largest element."""
    q, k, v, kv_len, mask = _alternate_case(D, 7100)
    B, N, Hq, _ = q.shape
    step = np.arange(k.shape[2]) // 128
    qf, kf, vf = (synth.bf16_bits_to_f32(x) for x in (q, k, v))
    c = np.array([1, 2, 0.5, -1, 1, -2, 0, 1], dtype=np.float32)
    qf[..., 0] = c[(np.arange(N)[:, None] + np.arange(Hq)) % 8]
    kf[..., 0] = 6 * 16 * step                                       # (exact in bf16; the scale is 1/16)
    vf *= np.exp(6.0 * (11 - step))[:, None].astype(np.float32)
    q, k, v = (synth.f32_to_bf16_bits(x) for x in (qf, kf, vf))
    clean = (k.copy(), v.copy())
    _nan_past_the_end(kv_len, N, k, v)
    (out, lse, status), kernels = gu.kernels_of(lambda: gu.run_attn(q, k, v, kv_len, mask, 1 / 16, split_form=2))
    assert status == 0 and _ran_alternate_steps(kernels), kernels
    want, want_lse = oracle.tree_attn(q, *clean, kv_len, mask, 1 / 16)
    assert np.isfinite(out).all()
    assert (np.abs(out - want) / np.abs(want).max(axis=-1, keepdims=True)).max() <= TOL
    assert np.abs(lse - want_lse).max() <= LSE_TOL


@pytest.mark.parametrize("D", [128, 64])
@pytest.mark.parametrize("special", [0x7FC0, 0x7F80])
def test_alternate_steps_nan_and_infinite_scores(gu, D, special):
    """One such key per sequence, in even and odd steps of every rank, in either half and every column modulo 16 of a step; the last
    sequence has none."""
    q, k, v, kv_len, mask = _alternate_case(D, 7200)
    B, N, Hq, _ = q.shape
    _nan_past_the_end(kv_len, N, k, v)
    for b in range(B - 1):
        k[b, :, (b % 11) * 128 + (64 if b >= 11 else 0) + (7 * b) % 64, 3] = special
    (out, _, status), kernels = gu.kernels_of(lambda: gu.run_attn(q, k, v, kv_len, mask, 0.1, split_form=2))
    assert status == 0 and _ran_alternate_steps(kernels), kernels
    want = np.ones((B, N, Hq), dtype=bool) if special == 0x7FC0 else synth.bf16_bits_to_f32(q)[..., 3] > 0
    want[B - 1] = False
    assert np.isnan(out[want]).all() and np.isfinite(out[~want]).all()


@pytest.mark.parametrize("Hq,Hkv,D,N,S_max", [(4, 1, 64, 100, 256), (4, 1, 128, 100, 256), (16, 2, 128, 128, 512)])
def test_alternate_steps_lse_of_rows_with_one_or_two_keys(gu, Hq, Hkv, D, N, S_max):
    _, kernels = gu.kernels_of(lambda: _one_or_two_keys(gu, Hq, Hkv, D, N, S_max, split_form=2))
    assert _ran_alternate_steps(kernels), kernels

@pytest.mark.parametrize("B,N,S,clusters", [(8, 16, 12000, True), (8, 16, 24000, False), (6, 13, 20000, True), (6, 13, 28000, False)])
def test_long_calls_of_one_row_block_leave_the_clusters(gu, B, N, S, clusters):
    """16 and 2 heads, 104 and 128 rows per kv head: from where clusters of six and eight are the slower form, the even split and its merge
    kernel serve the call.  Few tokens in use: the form follows the capacity."""
    q = synth.normal_bf16((B, N, 16, 128), 8100)
    kv_len = np.array([300 + 17 * b for b in range(B)], dtype=np.int32)
    used = int(kv_len.max()) + N
    k, v = (np.zeros((B, 2, S + 128, 128), dtype=np.uint16) for _ in range(2))
    k[:, :, :used] = synth.normal_bf16((B, 2, used, 128), 8101)
    v[:, :, :used] = synth.normal_bf16((B, 2, used, 128), 8102)
    rng = np.random.Generator(np.random.Philox(8103))
    mask, _, _ = oracle.tree_mask(np.stack([synth.draw_tree(N, 6, 4, rng) for _ in range(B)]))
    (out, lse, status), kernels = gu.kernels_of(lambda: gu.run_attn(q, k, v, kv_len, mask, 0.09))
    assert status == 0 and _ran_alternate_steps(kernels) == clusters and any("attn_tc5_merge_kernel" in n for n in kernels) != clusters
    want, want_lse = oracle.tree_attn(q, k[:, :, :used], v[:, :, :used], kv_len, mask, 0.09)
    assert np.abs(out - want).max() <= TOL and np.abs(lse - want_lse).max() <= LSE_TOL


# P of a step lies in the tensor memory that the scores two steps on overwrite, and the order of the products alone keeps the two
# apart: every repetition gives the same bits.  One-tile clusters and the two-tile kernel.
@pytest.mark.parametrize("Hq,Hkv,D,B,N,S,S_max,split_form,kernel", [
    (16, 2, 128, 4, 60, 4000, 4224, 2, "attn_tc5_kernel"), (16, 4, 64, 4, 60, 4000, 4224, 2, "attn_tc5_kernel"),
    (16, 2, 128, 4, 128, 4000, 40000, 0, "attn_tc5_wide_kernel"),
])
def test_products_in_shared_tensor_memory_repeat_bit_for_bit(gu, Hq, Hkv, D, B, N, S, S_max, split_form, kernel):
    from paper_2509_15235_b200 import binding
    rng = np.random.Generator(np.random.Philox(73))
    gen = torch.Generator("cuda").manual_seed(74)
    rand = lambda *shape: torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)
    q, k, v = rand(B, N, Hq, D), rand(B, Hkv, S_max, D), rand(B, Hkv, S_max, D)
    mask, _, _ = oracle.tree_mask(np.stack([synth.draw_tree(N, 6, 4, rng) for _ in range(B)]))
    mask, kv_len = gu.u64_dev(mask), gu.i32_dev([S - 37 * b for b in range(B)])
    ctx = binding.VerifyContext(B, N, Hq, Hkv, D, S_max, 1)
    ctx.ctx_set_option(binding.OPT_SPLIT_FORM, split_form)
    ctx.cache_register(0, k, v)
    outs = [torch.zeros_like(q) for _ in range(8)]
    _, kernels = gu.kernels_of(lambda: ctx.tree_verify_attn(0, q, kv_len, mask, 0.09, outs[0]))
    assert any(kernel in n for n in kernels) and (kernel != "attn_tc5_kernel" or _ran_alternate_steps(kernels)), kernels
    first = outs[0].clone()
    for rep in range(40):                                            # eight calls back to back, then the comparison
        for o in outs:
            ctx.tree_verify_attn(0, q, kv_len, mask, 0.09, o)
        for o in outs:
            assert torch.equal(o, first)
    assert ctx.status_poll() == 0
    ctx.close()


# A NaN in a key (or an infinite score) makes every row that sees it NaN, whatever column of a step the key falls on.  One
# sequence per step column modulo 16, one whose second 64 tokens are all such keys (the duplicated-row layout keeps a state of
# its own for those), one without any.
@pytest.mark.parametrize("static", [False, True])
@pytest.mark.parametrize("Hq,Hkv,D,N,S_max", [(2, 2, 64, 20, 256), (8, 1, 64, 20, 256), (2, 2, 128, 20, 256), (8, 1, 128, 20, 256),
                                              (32, 2, 64, 20, 40000), (32, 2, 128, 20, 40000)])
def test_nan_and_infinite_scores_reach_the_rows_that_see_them(gu, Hq, Hkv, D, N, S_max, static):
    from paper_2509_15235_b200 import binding
    B, S, used = 18, 192, 256
    q = synth.normal_bf16((B, N, Hq, D), 91)
    k = np.zeros((B, Hkv, S_max, D), dtype=np.uint16)
    v = np.zeros_like(k)
    k[:, :, :used] = synth.normal_bf16((B, Hkv, used, D), 92)
    v[:, :, :used] = synth.normal_bf16((B, Hkv, used, D), 93)
    mask, _, _ = oracle.tree_mask(np.tile(np.array([-1, 0, 0] + [1] * (N - 3), dtype=np.int32), (B, 1)))
    kv_len = np.full(B, S, dtype=np.int32)
    for special in (0x7FC0, 0x7F80):                                 # NaN, +inf in one element of the key
        for b in range(16):
            k[b, :, 2 + 16 * (b % 8) + b, 3] = special
        k[16, :, 64:128, 3] = special
        if static:
            out = torch.zeros((B, N, Hq, D), dtype=torch.bfloat16, device="cuda")
            binding.tree_verify_attn_static(gu.bf16_dev(q), gu.bf16_dev(k), gu.bf16_dev(v), gu.i32_dev(kv_len), gu.u64_dev(mask), 0.1, out)
            out = out.float().cpu().numpy()
        else:
            out, _, status = gu.run_attn(q, k, v, kv_len, mask, 0.1)
            assert status == 0
        # an infinite element of the key: the score is +inf where q > 0 there, else -inf and the key has no weight
        want = np.ones((B, N, Hq), dtype=bool) if special == 0x7FC0 else synth.bf16_bits_to_f32(q)[..., 3] > 0
        want[17] = False
        assert np.isnan(out[want]).all()
        assert np.isfinite(out[~want]).all()


# Hidden tree rows have weight exactly 0 in every column of a step: rows that see nothing are zeros (also where one CTA has the
# whole unit and writes the output itself), and the largest finite v in rows that nobody sees changes nothing.
@pytest.mark.parametrize("Hq,Hkv,D,N,S_max", [(2, 2, 64, 40, 64), (8, 1, 64, 40, 64), (2, 2, 128, 40, 64), (8, 1, 128, 40, 64),
                                              (16, 2, 64, 40, 40000), (16, 2, 128, 40, 40000)])
@pytest.mark.parametrize("split_form", [0, 1, 2, 3])
def test_hidden_rows_have_no_weight_in_any_column(gu, Hq, Hkv, D, N, S_max, split_form):
    B = 2
    q = synth.normal_bf16((B, N, Hq, D), 61)
    k = np.zeros((B, Hkv, S_max, D), dtype=np.uint16)
    v = np.zeros_like(k)
    k[:, :, :64] = synth.normal_bf16((B, Hkv, 64, D), 62)
    v[:, :, :64] = synth.normal_bf16((B, Hkv, 64, D), 63)
    v[:, :, 8:40] = 0x7F7F                                           # 3.4e38, seen by nobody
    mask = np.zeros((B, N, 1), dtype=np.uint64)
    mask[:, 1::2] = np.uint64(0b10100010)                            # every other node sees slots 1, 5 and 7, the rest nothing
    kv_len = np.zeros(B, dtype=np.int32)
    out, lse, status = gu.run_attn(q, k, v, kv_len, mask, 0.1, split_form=split_form)
    want, want_lse = oracle.tree_attn(q, k[:, :, :64], v[:, :, :64], kv_len, mask, 0.1)
    assert status == 0
    assert (out[:, 0::2] == 0).all() and np.isneginf(lse[:, :, 0::2]).all()
    assert np.abs(out - want).max() <= TOL
    assert np.abs(lse[:, :, 1::2] - want_lse[:, :, 1::2]).max() <= LSE_TOL


def test_arbitrary_mask_bits_all_ones_and_zero_rows(gu):
    B, N, Hq, Hkv, D, S_max = 2, 20, 4, 2, 128, 256
    q = synth.normal_bf16((B, N, Hq, D), 21); k = synth.normal_bf16((B, Hkv, S_max, D), 22)
    v = synth.normal_bf16((B, Hkv, S_max, D), 23)
    rng = np.random.default_rng(9)
    mask = rng.integers(0, 1 << 20, size=(B, N, 1), dtype=np.int64).astype(np.uint64)
    mask[0, 3, 0] = (1 << 20) - 1          # all ones
    mask[1, 5, 0] = 0                      # no tree key at all
    _check(gu, q, k, v, np.array([100, 0], dtype=np.int32), mask, 0.11)


def test_empty_allowed_set_gives_zero_and_minus_inf(gu):
    B, N, Hq, Hkv, D, S_max = 1, 4, 2, 2, 64, 64
    q = synth.normal_bf16((B, N, Hq, D), 31); k = synth.normal_bf16((B, Hkv, S_max, D), 32)
    v = synth.normal_bf16((B, Hkv, S_max, D), 33)
    mask = np.array([[[0], [2], [0], [8]]], dtype=np.uint64)
    out, lse, status = gu.run_attn(q, k, v, np.array([0], dtype=np.int32), mask, 0.5)
    want, want_lse = oracle.tree_attn(q, k, v, [0], mask, 0.5)
    assert status == 0 and (out[0, 0] == 0).all() and (out[0, 2] == 0).all()
    assert np.isneginf(lse[0, :, 0]).all() and np.isneginf(lse[0, :, 2]).all()
    assert np.abs(out - want).max() <= TOL


def test_slots_past_the_tree_may_hold_nan_patterns(gu):
    cfg = synth.get_config("tiny")
    q, k, v, kv_len, mask = _case(cfg, S_max=384)
    k = k.copy(); v = v.copy()
    end = int(kv_len[0]) + cfg.N
    k[:, :, end:] = 0x7FC0; v[:, :, end:] = 0x7FC0
    k[:, :, end + 3] = 0x7F80; v[:, :, end + 3] = 0xFF80      # +inf / -inf
    _check(gu, q, k, v, kv_len, mask, 0.125)


def test_non_ancestor_rows_do_not_influence_a_node(gu):
    """Hidden tree rows get weight exactly 0, so replacing them by other finite rows leaves a node's
    output bit-identical (a NaN there would not: 0 * NaN; hidden rows hold finite data by contract)."""
    B, N, Hq, Hkv, D, S_max = 1, 12, 2, 1, 128, 128
    rng = np.random.Generator(np.random.Philox(77))
    q = synth.normal_bf16((B, N, Hq, D), 41); k = synth.normal_bf16((B, Hkv, S_max, D), 42)
    v = synth.normal_bf16((B, Hkv, S_max, D), 43)
    parents = synth.draw_tree(N, 3, 3, rng)[None]
    mask, _, _ = oracle.tree_mask(parents)
    S = 50
    base, _, _ = gu.run_attn(q, k, v, [S], mask, 0.1)
    i = N - 1
    k2, v2 = k.copy(), v.copy()
    for t in range(N):
        if not (int(mask[0, i, 0]) >> t) & 1:
            k2[0, :, S + t] = k[0, :, (t * 7) % S]; v2[0, :, S + t] = 0x42C8   # other finite rows (v = 100)
    out2, _, _ = gu.run_attn(q, k2, v2, [S], mask, 0.1)
    assert np.array_equal(out2[0, i], base[0, i])


def test_large_scores_stay_finite(gu):
    """Scores of magnitude ~1e3: the running-max rescale must keep everything finite."""
    B, N, Hq, Hkv, D, S_max = 1, 8, 2, 2, 64, 192
    q = synth.f32_to_bf16_bits(synth.bf16_bits_to_f32(synth.normal_bf16((B, N, Hq, D), 51)) * 30)
    k = synth.f32_to_bf16_bits(synth.bf16_bits_to_f32(synth.normal_bf16((B, Hkv, S_max, D), 52)) * 30)
    v = synth.normal_bf16((B, Hkv, S_max, D), 53)
    mask, _, _ = oracle.tree_mask(np.arange(-1, N - 1, dtype=np.int32)[None])
    out, lse, _ = gu.run_attn(q, k, v, [150], mask, 0.125)
    want, want_lse = oracle.tree_attn(q, k, v, [150], mask, 0.125)
    assert np.isfinite(out).all() and np.abs(out - want).max() <= TOL
    assert np.abs(lse - want_lse).max() <= 2e-3 * np.abs(want_lse).max()


def test_overlong_sequence_is_zeroed_with_status(gu):
    B, N, Hq, Hkv, D, S_max = 2, 8, 2, 2, 64, 128
    q = synth.normal_bf16((B, N, Hq, D), 61); k = synth.normal_bf16((B, Hkv, S_max, D), 62)
    v = synth.normal_bf16((B, Hkv, S_max, D), 63)
    mask, _, _ = oracle.tree_mask(np.tile(np.arange(-1, N - 1, dtype=np.int32), (B, 1)))
    out, lse, status = gu.run_attn(q, k, v, [125, 100], mask, 0.125)
    assert status == -4 and (out[0] == 0).all()
    want, _ = oracle.tree_attn(q[1:], k[1:], v[1:], [100], mask[1:], 0.125)
    assert np.abs(out[1] - want[0]).max() <= TOL


def test_host_side_argument_errors(gu):
    from paper_2509_15235_b200 import binding
    ctx = binding.VerifyContext(1, 8, 2, 2, 64, 128, 2)
    q = torch.zeros((1, 8, 2, 64), dtype=torch.bfloat16, device="cuda")
    kv_len = torch.zeros(1, dtype=torch.int32, device="cuda")
    mask = torch.zeros((1, 8, 1), dtype=torch.int64, device="cuda")
    with pytest.raises(binding.VispecError) as e:
        ctx.tree_verify_attn(0, q, kv_len, mask, 1.0, q.clone())
    assert e.value.code == -9                                    # nothing registered
    cache = torch.zeros((1, 2, 128, 64), dtype=torch.bfloat16, device="cuda")
    ctx.cache_register(0, cache, cache.clone())
    with pytest.raises(binding.VispecError) as e:
        ctx.tree_verify_attn(2, q, kv_len, mask, 1.0, q.clone())
    assert e.value.code == -4                                    # layer out of range
    with pytest.raises(binding.VispecError) as e:
        ctx.tree_verify_attn(0, q, kv_len, mask, 1.0, q.clone(), k_cache=cache.clone())
    assert e.value.code == -9                                    # not the registered pointer
    big = torch.zeros((1, 9, 2, 64), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(binding.VispecError) as e:
        ctx.tree_verify_attn(0, big, kv_len, mask, 1.0, big.clone())
    assert e.value.code == -3                                    # N > N_max
    ctx.tree_verify_attn(0, q, kv_len, mask, 1.0, q.clone(), k_cache=cache)
    torch.cuda.synchronize()


@pytest.mark.parametrize("split_form", [0, 1, 2])
@pytest.mark.parametrize("name", ["llava7b", "qwen7b"])
def test_full_size_layer_parity(gu, name, split_form):
    """One whole layer at benchmark size, every output element against the oracle, for both ways of
    combining the pieces of a head (partials + merge kernel; clusters) and for the library's own choice (the
    launch configuration bench.py times; on qwen7b that is the layout with 64-row blocks, which the forced forms
    do not take)."""
    cfg = synth.get_config(name)
    _check(gu, *_case(cfg, layer=1), 1 / math.sqrt(cfg.D), split_form=split_form)


def test_full_size_batched_variable_length_parity(gu):
    cfg = synth.get_config("llava13b_b4")
    q, k, v, kv_len, mask = _case(cfg, layer=0)
    # the oracle on 4 x 40 heads x ~4000 keys takes a while: check 8 heads of every sequence
    heads = [0, 5, 13, 21, 27, 33, 38, 39]
    out, lse, status = gu.run_attn(q, k, v, kv_len, mask, 1 / math.sqrt(cfg.D))
    assert status == 0 and not np.isnan(out).any()
    want, want_lse = oracle.tree_attn(q[:, :, heads], k[:, heads], v[:, heads], kv_len, mask, 1 / math.sqrt(cfg.D))
    assert np.abs(out[:, :, heads] - want).max() <= TOL
    assert np.abs(lse[:, heads] - want_lse).max() <= LSE_TOL
    # and every one of the 40 heads of the longest sequence
    b = int(np.argmax(kv_len))
    want, want_lse = oracle.tree_attn(q[b:b + 1], k[b:b + 1], v[b:b + 1], kv_len[b:b + 1], mask[b:b + 1], 1 / math.sqrt(cfg.D))
    assert np.abs(out[b:b + 1] - want).max() <= TOL
    assert np.abs(lse[b:b + 1] - want_lse).max() <= LSE_TOL


@pytest.mark.parametrize("name", ["qwen3b_S2048_N16_B1", "qwen3b_S8192_N60_B4", "qwen3b_S32768_N128_B1",
                                  "qwen3b_S16384_N16_B8"])
def test_long_response_sweep_cells(gu, name):
    """Sweep cells at full size: the whole GPU result is produced, and the oracle recomputes every
    output of one kv head's group (heads are independent, so this samples the result exactly)."""
    cfg = synth.get_config(name)
    q, k, v, kv_len, mask = _case(cfg)
    scale = 1 / math.sqrt(cfg.D)
    out, lse, status = gu.run_attn(q, k, v, kv_len, mask, scale)
    assert status == 0 and not np.isnan(out).any()
    kvh = cfg.Hkv - 1
    hs = slice(kvh * cfg.G, (kvh + 1) * cfg.G)
    want, want_lse = oracle.tree_attn(q[:, :, hs], k[:, kvh:kvh + 1], v[:, kvh:kvh + 1], kv_len, mask, scale)
    assert np.abs(out[:, :, hs] - want).max() <= TOL
    assert np.abs(lse[:, hs] - want_lse).max() <= LSE_TOL


def test_options_and_fallbacks_give_the_same_attention(gu):
    """Early prefix prefetch off, more sequences than the tensor-core kernel takes per call (generic kernel),
    and a non-positive scale (generic kernel: the maximum no longer commutes with the scale)."""
    from paper_2509_15235_b200 import binding
    rng = np.random.Generator(np.random.Philox(2024))
    Hq, Hkv, D, N, S_max = 4, 2, 128, 12, 384
    for B, scale, early in ((2, 0.09, 0), (33, 0.09, None), (2, 0.0, None), (2, -0.05, None)):
        q = synth.normal_bf16((B, N, Hq, D), 71 + B); k = synth.normal_bf16((B, Hkv, S_max, D), 72 + B)
        v = synth.normal_bf16((B, Hkv, S_max, D), 73 + B)
        kv_len = rng.integers(0, S_max - N, size=B).astype(np.int32)
        parents = np.stack([synth.draw_tree(N, 4, 3, rng) for _ in range(B)])
        mask, _, _ = oracle.tree_mask(parents)
        out, lse, status = gu.run_attn(q, k, v, kv_len, mask, scale, early_prefetch=early)
        want, want_lse = oracle.tree_attn(q, k, v, kv_len, mask, scale)
        assert status == 0
        assert np.abs(out - want).max() <= TOL
        assert np.abs(lse - want_lse).max() <= LSE_TOL
    ctx = binding.VerifyContext(1, 8, 2, 2, 64, 128, 1)
    with pytest.raises(binding.VispecError) as e:
        ctx.ctx_set_option(99, 1)
    assert e.value.code == -5
    with pytest.raises(binding.VispecError) as e:
        ctx.ctx_set_option(binding.OPT_SPLIT_FORM, 7)
    assert e.value.code == -4


def test_redundant_image_keys_stress_the_softmax(gu):
    """Sec. 4.1 of the paper: image tokens are highly redundant, identical tokens get identical scores (Eq. 2)
    and their softmax mass is spread evenly (Eq. 3-4).  1296 identical 'image' keys followed by ordinary text
    keys: a huge, flat block of probability mass, against the oracle; and with every key identical the output
    must be the mean of the visible V rows (Eq. 4), checked directly."""
    B, N, Hq, Hkv, D, S, S_max = 1, 16, 4, 2, 128, 1500, 1664
    rng = np.random.Generator(np.random.Philox(404))
    q = synth.normal_bf16((B, N, Hq, D), 81); k = synth.normal_bf16((B, Hkv, S_max, D), 82)
    v = synth.normal_bf16((B, Hkv, S_max, D), 83)
    k[:, :, :1296] = k[:, :, :1]                       # the image span repeats one key per head
    parents = synth.draw_tree(N, 4, 3, rng)[None]
    mask, _, _ = oracle.tree_mask(parents)
    _check(gu, q, k, v, np.array([S], dtype=np.int32), mask, 1 / math.sqrt(D))
    k[:, :, :] = k[:, :, :1]                           # every key identical: weights are uniform over the visible set
    out, lse, status = gu.run_attn(q, k, v, [S], mask, 1 / math.sqrt(D))
    assert status == 0
    vf = synth.bf16_bits_to_f32(v).astype(np.float64)
    for i in range(N):
        vis = list(range(S)) + [S + t for t in range(N) if (int(mask[0, i, 0]) >> t) & 1]
        for h in range(Hq):
            assert np.abs(out[0, i, h] - vf[0, h // (Hq // Hkv), vis].mean(axis=0)).max() <= TOL


def test_stream_probe_runs_and_validates_its_arguments(gu):
    """The measurement aid: it only reads, so the check is that it runs clean on ragged lengths (including a
    rejected sequence, which it skips) and that the host-side validation answers."""
    from paper_2509_15235_b200 import binding
    ctx = binding.VerifyContext(3, 60, 4, 2, 128, 1024, 2)
    k = torch.zeros((3, 2, 1024, 128), dtype=torch.bfloat16, device="cuda")
    ctx.cache_register(0, k, k.clone())
    ctx.stream_probe(0, gu.i32_dev([900, 0, 1000]), 60)        # 1000 + 60 > 1024: skipped
    torch.cuda.synchronize()
    assert ctx.status_poll() == 0
    with pytest.raises(binding.VispecError) as e:
        ctx.stream_probe(1, gu.i32_dev([1, 2, 3]), 60)
    assert e.value.code == -9                                   # layer 1 has no registered cache
    ctx64 = binding.VerifyContext(1, 8, 2, 2, 64, 128, 1)
    c = torch.zeros((1, 2, 128, 64), dtype=torch.bfloat16, device="cuda")
    ctx64.cache_register(0, c, c.clone())
    with pytest.raises(binding.VispecError) as e:
        ctx64.stream_probe(0, gu.i32_dev([10]), 8)
    assert e.value.code == -5                                   # D = 64: no TMA maps


def test_stream_probe_with_nothing_to_read_keeps_the_stream_order(gu):
    """A kernel that starts early (the commit) waits for the kernel before it, here a probe whose sequences are all out of range;
    the probe must not end ahead of the rotary placement before it, whose rows the commit moves."""
    from paper_2509_15235_b200 import binding
    B, N, Hq, Hkv, D, S_max = 8, 128, 32, 32, 128, 512
    ctx = binding.VerifyContext(B, N, Hq, Hkv, D, S_max, 1)
    rows = lambda seed: torch.randn((B, N, Hkv, D), generator=torch.Generator("cuda").manual_seed(seed), device="cuda", dtype=torch.bfloat16)
    kv_len, none = gu.i32_dev([100] * B), gu.i32_dev([S_max] * B)
    path = gu.i32_dev([[0, 127] + [-1] * (N - 2)] * B)                # the last row of the tree moves to slot 101
    alen, pos = gu.i32_dev([2] * B), gu.i32_dev(np.zeros((B, N)))
    k, v = (torch.zeros((B, Hkv, S_max, D), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    ctx.cache_register(0, k, v)
    for rep in range(10):
        kn, vn, q = rows(2 * rep), rows(2 * rep + 1), rows(99)
        ctx.rope_tree_rows(0, q, kn, vn, pos, kv_len, 10000.0)
        ctx.stream_probe(0, none, N)
        ctx.kv_compact(0, 1, path, alen, kv_len)
        torch.cuda.synchronize()
        assert torch.equal(k[:, :, 101], kn[:, 127]) and torch.equal(v[:, :, 101], vn[:, 127])   # (position 0: no rotation)
    assert ctx.status_poll() == 0
    ctx.close()


def test_seeded_random_shapes_against_the_oracle(gu):
    """Sixty seeded draws of (batch, heads, group size, tree size, lengths, split form): every output element
    against the oracle.  Lengths straddle tile boundaries; some sequences are empty."""
    rng = np.random.Generator(np.random.Philox(2024))
    for case in range(60):
        B = int(rng.integers(1, 6))
        Hkv = int(rng.choice([1, 2, 3, 4, 8]))
        G = int(rng.choice([1, 2, 4, 7, 8]))
        N = int(rng.choice([1, 2, 7, 16, 31, 60, 64, 65, 100, 128]))
        S_hi = int(rng.choice([0, 5, 127, 128, 129, 400, 1000, 1400]))
        kv_len = rng.integers(0, S_hi + 1, size=B).astype(np.int32)
        S_max = (int(kv_len.max()) + N + 127) // 128 * 128 + int(rng.choice([0, 128]))
        split_form = int(rng.integers(0, 4))
        q = synth.normal_bf16((B, N, Hkv * G, 128), 9000 + 3 * case)
        k = synth.normal_bf16((B, Hkv, S_max, 128), 9001 + 3 * case)
        v = synth.normal_bf16((B, Hkv, S_max, 128), 9002 + 3 * case)
        parents = np.stack([synth.draw_tree(N, 8, 0, rng) for _ in range(B)])
        mask, _, _ = oracle.tree_mask(parents)
        _check(gu, q, k, v, kv_len, mask, 1 / math.sqrt(128), split_form=split_form)
