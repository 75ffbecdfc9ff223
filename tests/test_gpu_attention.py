"""GPU parity of bp_block_attention against the fp64 oracle (bf16 tensor-core path and fp32 path).

Tolerance: max |O - O_ref| / max |O_ref| <= 2e-2 per (sequence, query head) slice (bf16 inputs,
fp32 accumulation); log-sum-exp within 2e-3.  Small ragged cases are compared in full, on both
splits of the keys (the flat split and the cluster split, each forced, the cluster split also in
clusters of 3: contexts this short stay in one CTA per unit when the library chooses; those clusters
merge through distributed shared memory, or through the workspace where a unit has at most 34 rows --
test_cluster_merges takes both merges at other sizes); the full-size workloads run
exactly as the benchmark launches them (the library's own choice of split) and are compared on
sampled sequences (and KV heads for the 32K-context case).
"""
import numpy as np
import pytest
import torch

import paper_2606_31315_gb300 as bp
from paper_2606_31315_gb300 import workloads as wl

from _gpu import ATTN_TOL, LSE_TOL, attention_errors, run_attention, to_dev

pytestmark = pytest.mark.gpu

CAUSAL, BIDIR = bp.MASK_CAUSAL, bp.MASK_BIDIR


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    bp.build()
    bp.load()


def _check(a, mask, seqs=None, kv_head=None, split="auto"):
    o, lse = run_attention(a, mask, split)
    seqs = range(len(a["cu_q"]) - 1) if seqs is None else seqs
    err, lerr = attention_errors(o, lse, a, mask, seqs, kv_head)
    assert err <= ATTN_TOL, err
    assert lerr <= LSE_TOL, lerr
    return o, lse


@pytest.mark.parametrize("mask", [CAUSAL, BIDIR])
@pytest.mark.parametrize("ctx,block", [
    ((0, 1, 127, 300, 1000), (1, 8, 16, 24, 13)),   # ragged, tile-crossing contexts, B=1 decode
    ((129, 0, 5), (64, 2, 33)),                     # B=64: two 128-row query tiles; L=0
    ((2048,), (16,)),                                # Qwen3-4B verify shape, one sequence
    ((4000, 10, 255, 256, 257), (16, 16, 16, 16, 16)),
])
@pytest.mark.parametrize("split", ["flat", "cluster", "cluster3"])
def test_ragged_small(ctx, block, mask, split):
    w = wl.custom(seed=sum(ctx) + len(block), ctx=ctx, block=block, num_q_heads=32, num_kv_heads=8)
    _check(wl.attention_inputs(w), mask, split=split)


@pytest.mark.parametrize("hq,hkv", [(8, 8), (64, 8), (16, 2), (4, 1), (24, 8)])
@pytest.mark.parametrize("split", ["flat", "cluster", "cluster3"])
def test_group_sizes(hq, hkv, split):
    # (24, 8): a group of 3 does not divide the 128-row tile, so Q is gathered without TMA (cluster split)
    w = wl.custom(seed=hq * 10 + hkv, ctx=(300, 77), block=(12, 31), num_q_heads=hq, num_kv_heads=hkv)
    for mask in (CAUSAL, BIDIR):
        _check(wl.attention_inputs(w), mask, split=split)


@pytest.mark.parametrize("ctx,block", [
    ((3, 1, 0, 300), (1, 1, 2, 1)),                  # fewer key tiles than CTAs: CTAs without work
    ((40000,), (16,)),                                # one unit per KV head cut over ~19 CTAs each
    ((9000, 120, 130, 2500, 31), (16, 9, 64, 1, 24)),  # cuts mid-unit, B=64 (two query tiles), B=1
])
def test_flat_split_cuts(ctx, block):
    """The flat split's ranges start and end anywhere inside a unit; partial stretches are merged by
    the second kernel in CTA order."""
    w = wl.custom(seed=len(ctx) * 7 + block[0], ctx=ctx, block=block, num_q_heads=32, num_kv_heads=8)
    a = wl.attention_inputs(w)
    for mask in (CAUSAL, BIDIR):
        _check(a, mask, split="flat")


@pytest.mark.parametrize("n", [256, 257])
def test_many_sequences(n):
    """Up to 256 sequences take the flat split (their offsets fit the CTA's table); 257 the cluster split."""
    rng = np.random.default_rng(n)
    w = wl.custom(seed=n, ctx=tuple(int(x) for x in rng.integers(0, 300, n)),
                  block=tuple(int(x) for x in rng.integers(1, 17, n)), num_q_heads=32, num_kv_heads=8)
    a = wl.attention_inputs(w)
    _check(a, CAUSAL, seqs=[0, 1, n // 2, n - 1], split="flat")


def _attn_kernels(a, split):
    from torch.profiler import ProfilerActivity, profile

    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        run_attention(a, CAUSAL, split)
        torch.cuda.synchronize()
    return {e.name for e in prof.events() if "attn_" in e.name}


def test_split_choice():
    """Left to the library, a batch-1 verify (2K keys) takes the cluster split (one kernel) and 64 short
    sequences, which would need four waves of the cluster split, the flat split (two kernels); each can
    be forced."""
    _attn_kernels(wl.attention_inputs(wl.custom(seed=1, ctx=(100,), block=(4,), num_q_heads=32, num_kv_heads=8)),
                  "auto")  # the profiler's first session may miss kernels while it starts
    small = wl.attention_inputs(wl.get("qwen3_4b"))
    names = _attn_kernels(small, "auto")
    assert not any("attn_combine_kernel" in x for x in names) and any("attn_bf16_tc_kernel" in x for x in names)
    assert any("attn_combine_kernel" in x for x in _attn_kernels(small, "flat"))
    many = wl.attention_inputs(wl.custom(seed=9, ctx=(512,) * 64, block=(16,) * 64, num_q_heads=32,
                                         num_kv_heads=8))
    assert any("attn_combine_kernel" in x for x in _attn_kernels(many, "auto"))
    assert not any("attn_combine_kernel" in x for x in _attn_kernels(many, "cluster"))
    err, lerr = attention_errors(*run_attention(many, CAUSAL), many, CAUSAL, [0, 17, 63])
    assert err <= ATTN_TOL and lerr <= LSE_TOL


@pytest.mark.parametrize("n, ctx, block, flat", [
    (1, 70000, 16, True), (10, 9000, 16, True), (8, 12000, 16, False), (9, 5000, 16, False),
    (20, 4000, 16, True), (32, 1500, 16, False), (10, 4096, 40, True), (16, 1200, 40, False)])
def test_split_by_estimate(n, ctx, block, flat):
    """Clusters against the flat split, by the library's estimates.  One wave: wide clusters or few SMs on long
    runs go flat, nearly full grids stay in clusters (128 CTAs: K's ring ahead; 144: not).  Two waves: flat where the
    second is nearly empty.  Blocks of 40 have two query tiles, whose clusters share K and V."""
    a = wl.attention_inputs(wl.custom(seed=n, ctx=(ctx,) * n, block=(block,) * n, num_q_heads=32, num_kv_heads=8))
    _attn_kernels(a, "auto")
    assert any("attn_combine_kernel" in x for x in _attn_kernels(a, "auto")) == flat
    err, lerr = attention_errors(*run_attention(a, CAUSAL), a, CAUSAL, [n // 2])
    assert err <= ATTN_TOL and lerr <= LSE_TOL


def test_qwen3_4b_full():
    a = wl.attention_inputs(wl.get("qwen3_4b"))
    _check(a, CAUSAL)
    _check(a, BIDIR)


def test_ragged_batch_full_size_sampled():
    w = wl.get("ragged")
    a = wl.attention_inputs(w)
    lens = np.diff(a["cu_kv"])
    seqs = sorted({0, 5, 31, int(np.argmax(lens)), int(np.argmin(lens))})
    _check(a, CAUSAL, seqs=seqs)


def test_drafter_bidir_full_size_sampled():
    a = wl.attention_inputs(wl.get("drafter_bidir"))
    _check(a, BIDIR, seqs=[0, 9, 15])


def test_long_context_full_size_sampled():
    a = wl.attention_inputs(wl.get("long_context"))
    o, lse = run_attention(a, CAUSAL)
    for s, kvh in ((0, 0), (7, 5), (3, 7)):
        err, lerr = attention_errors(o, lse, a, CAUSAL, [s], kv_head=kvh)
        assert err <= ATTN_TOL and lerr <= LSE_TOL, (s, kvh, err, lerr)


def test_tiny_fp32():
    a = wl.attention_inputs(wl.get("tiny"))
    for mask in (CAUSAL, BIDIR):
        o, lse = run_attention(a, mask)
        err, lerr = attention_errors(o, lse, a, mask, [0])
        assert err <= 1e-5 and lerr <= 1e-5, (err, lerr)


def test_causal_last_row_equals_bidir_last_row():
    a = wl.attention_inputs(wl.custom(seed=5, ctx=(700, 90), block=(16, 9), num_q_heads=32, num_kv_heads=8))
    oc, _ = run_attention(a, CAUSAL)
    ob, _ = run_attention(a, BIDIR)
    last = a["cu_q"][1:] - 1
    np.testing.assert_allclose(oc[last], ob[last], rtol=0, atol=1e-2)


def test_empty_blocks_and_empty_batch():
    a = wl.attention_inputs(wl.custom(seed=6, ctx=(10, 0, 40), block=(0, 0, 8), num_q_heads=32, num_kv_heads=8))
    _check(a, CAUSAL)
    q = torch.zeros((0, 32, 128), dtype=torch.bfloat16, device="cuda")
    k = torch.zeros((0, 8, 128), dtype=torch.bfloat16, device="cuda")
    cu = torch.zeros(1, dtype=torch.int32, device="cuda")
    o, _ = bp.block_attention(q, k, k, cu, cu, 0, 0)
    assert o.shape == q.shape


def test_invalid_arguments_are_rejected_on_the_host():
    a = wl.attention_inputs(wl.custom(seed=1, ctx=(10,), block=(4,), num_q_heads=6, num_kv_heads=4))
    q, k, v = to_dev(a["q"], "bf16"), to_dev(a["k"], "bf16"), to_dev(a["v"], "bf16")
    cu_q, cu_kv = to_dev(a["cu_q"]), to_dev(a["cu_kv"])
    with pytest.raises(bp.BlockPilotError) as e:
        bp.block_attention(q, k, v, cu_q, cu_kv, 4, 14)  # 6 % 4 != 0
    assert e.value.status == 1
    w64 = wl.custom(seed=2, ctx=(10,), block=(4,), num_q_heads=4, num_kv_heads=2, head_dim=64)
    a64 = wl.attention_inputs(w64)
    with pytest.raises(bp.BlockPilotError) as e:
        bp.block_attention(to_dev(a64["q"], "bf16"), to_dev(a64["k"], "bf16"), to_dev(a64["v"], "bf16"),
                           to_dev(a64["cu_q"]), to_dev(a64["cu_kv"]), 4, 14)
    assert e.value.status == 2


@pytest.mark.parametrize("ctx,block,hq,hkv,d", [
    ((0, 1, 63, 64, 65), (1, 8, 16, 2, 33), 4, 2, 64),     # chunk edges; 66 rows: three row tiles, the last of 2
    ((1000, 7, 0), (8, 0, 24), 8, 1, 128),                 # a wide group (192 rows), an empty block, no context
    ((2047,), (64,), 4, 4, 128),                           # one long unit per head: the widest cluster split
    ((500, 129), (9, 16), 6, 2, 80),                       # D padded to the 128-column tile
    ((300, 40), (5, 12), 3, 1, 33),                        # D not a multiple of 4: scalar loads and stores
    ((40,) * 90, (4,) * 90, 4, 2, 64),                     # more units than SMs: no clusters
])
def test_fp32_shapes(ctx, block, hq, hkv, d):
    """fp32 sums of at most 2111 keys and 128 columns: the error of a dot and of a weighted sum is a few
    sqrt(length) roundings of 2^-24, well inside 1e-5 of the slice's largest value."""
    w = wl.custom(seed=d + len(ctx), ctx=ctx, block=block, num_q_heads=hq, num_kv_heads=hkv, head_dim=d, dtype="f32")
    a = wl.attention_inputs(w)
    for mask in (CAUSAL, BIDIR):
        o, lse = run_attention(a, mask)
        err, lerr = attention_errors(o, lse, a, mask, range(len(ctx)))
        assert err <= 1e-5 and lerr <= 1e-5, (err, lerr)


@pytest.mark.parametrize("hq,hkv,d", [(8, 8, 32), (8, 2, 128), (6, 2, 33), (4, 1, 64)])
@pytest.mark.parametrize("ctx,block", [
    ((4,), (1,)), ((0,), (8,)), ((31,), (1,)), ((55,), (9,)),                 # one sequence, up to a chunk of keys
    ((4, 0, 2, 16, 9) * 40, (1, 8, 0, 2, 3) * 40),                            # hundreds of short ones, some empty
    ((40, 30, 0, 50) * 60, (1, 2, 8, 13) * 60),                               # on either side of the line by head_dim
])
def test_fp32_short_contexts(ctx, block, hq, hkv, d):
    """Contexts of at most one 64-key chunk, by the row kernel or the tiled one.  Bars as test_fp32_shapes."""
    w = wl.custom(seed=d + len(ctx), ctx=ctx, block=block, num_q_heads=hq, num_kv_heads=hkv, head_dim=d, dtype="f32")
    a = wl.attention_inputs(w)
    for mask in (CAUSAL, BIDIR):
        o, lse = run_attention(a, mask)
        err, lerr = attention_errors(o, lse, a, mask, range(0, len(ctx), max(1, len(ctx) // 8)))
        assert err <= 1e-5 and lerr <= 1e-5, (err, lerr)


def test_fp32_unaligned_bases():
    """Tensors that start off a 16-byte boundary give the same values as aligned ones (same order of sums)."""
    a = wl.attention_inputs(wl.custom(seed=3, ctx=(200, 30), block=(8, 5), num_q_heads=4, num_kv_heads=2, head_dim=64,
                                      dtype="f32"))
    cu_q, cu_kv = to_dev(a["cu_q"]), to_dev(a["cu_kv"])

    def shifted(x):
        flat = torch.zeros(x.numel() + 1, device="cuda")
        flat[1:] = x.reshape(-1)
        return flat[1:].view(x.shape)

    q, k, v = to_dev(a["q"]), to_dev(a["k"]), to_dev(a["v"])
    o, _ = bp.block_attention(q, k, v, cu_q, cu_kv, a["max_q_len"], a["max_kv_len"])
    o1, _ = bp.block_attention(shifted(q), shifted(k), shifted(v), cu_q, cu_kv, a["max_q_len"], a["max_kv_len"],
                               out=shifted(torch.zeros_like(q)))
    assert torch.equal(o, o1)


@pytest.mark.parametrize("block", [(16, 1, 9, 16, 8, 12, 16, 3, 16, 5), (24, 1, 17, 20, 8, 32, 24, 3, 31, 5)])
def test_k_ring_ahead_of_v(block):
    """80 units of one CTA each, up to 33 key tiles: fewer CTAs than SMs and long runs, so K's ring
    refills ahead of V's; runs of 1 to 33 tiles wrap the rings at every phase, in both row layouts."""
    ctx = (2049, 4100, 2303, 31, 0, 900, 2176, 1, 3000, 128)
    a = wl.attention_inputs(wl.custom(seed=len(block) + block[0], ctx=ctx, block=block, num_q_heads=32, num_kv_heads=8))
    for mask in (CAUSAL, BIDIR):
        _check(a, mask, split="cluster")


def test_uneven_batch_takes_the_flat_split():
    """One 9000-key sequence among short ones: the flat split when the library chooses (the longest unit alone
    would take longer than every tile spread over all SMs); a batch of equal lengths keeps whole units."""
    ctx = (9000,) + tuple(range(300, 2100, 100)) + (31, 0)
    uneven = wl.attention_inputs(wl.custom(seed=8, ctx=ctx, block=(16, 9, 24) * 7, num_q_heads=32, num_kv_heads=8))
    _attn_kernels(uneven, "auto")
    assert any("attn_combine_kernel" in x for x in _attn_kernels(uneven, "auto"))
    err, lerr = attention_errors(*run_attention(uneven, BIDIR), uneven, BIDIR, [0, 1, 10, 19, 20])
    assert err <= ATTN_TOL and lerr <= LSE_TOL
    even = wl.attention_inputs(wl.custom(seed=8, ctx=(1500,) * 32, block=(16,) * 32, num_q_heads=32, num_kv_heads=8))
    assert not any("attn_combine_kernel" in x for x in _attn_kernels(even, "auto"))


def _run(a, mask, split="auto", ws_bytes=None, max_kv=None, page=0):
    """run_attention with a workspace of ws_bytes, another max_kv_len or a paged cache."""
    from _gpu import attention_ws, forced_split

    q, cu_q, cu_kv = to_dev(a["q"], "bf16"), to_dev(a["cu_q"]), to_dev(a["cu_kv"])
    lse = torch.empty(q.shape[0], q.shape[1], device="cuda")
    ws = attention_ws(a) if ws_bytes is None else bp.workspace(ws_bytes, "cuda")
    max_kv = max_kv or a["max_kv_len"]
    with forced_split(split):
        if page:
            pk = wl.paged_kv(a["k"], a["v"], a["cu_kv"], page, seed=page)
            bt = np.zeros((len(a["cu_q"]) - 1, max(pk["block_table"].shape[1], -(-max_kv // page))), dtype=np.int32)
            bt[:, :pk["block_table"].shape[1]] = pk["block_table"]
            o, _ = bp.block_attention_paged(q, to_dev(pk["k_cache"], "bf16"), to_dev(pk["v_cache"], "bf16"), cu_q, cu_kv,
                                            to_dev(bt), page, int(a["cu_kv"][-1]), a["max_q_len"], max_kv, mask=mask,
                                            lse=lse, ws=ws)
        else:
            o, _ = bp.block_attention(q, to_dev(a["k"], "bf16"), to_dev(a["v"], "bf16"), cu_q, cu_kv, a["max_q_len"],
                                      max_kv, mask=mask, lse=lse, ws=ws)
    assert bp.get_status(ws) == 0
    return o.float().cpu().numpy(), lse.cpu().numpy()


@pytest.mark.parametrize("n", [4, 5, 8, 11, 16])
@pytest.mark.parametrize("ctx,block,page", [
    ((2100,), (1,), 0), ((2100,), (9,), 64), ((3000,), (12,), 0), ((2050,), (16,), 16), ((2500,), (24,), 0),
    ((2080,), (32,), 128), ((2600, 200), (16, 3), 0), ((300, 2300), (24, 32), 64),
])
def test_cluster_merges(n, ctx, block, page):
    """Clusters of n on both row layouts, merged through the workspace (where a CTA owns few rows) and, without the
    workspace, through distributed shared memory: one sequence, or two of which one has fewer tiles than CTAs; owners
    with fewer rows than others or none; 2 KV heads, so that clusters of 16 are resident.  Both merges add the same
    partials in fp32, in another order: they differ by bf16 roundings of the output, 2^-8 of its size at most."""
    a = wl.attention_inputs(wl.custom(seed=n + ctx[0], ctx=ctx, block=block, num_q_heads=8, num_kv_heads=2))
    for mask in (CAUSAL, BIDIR):
        full = _run(a, mask, f"cluster:{n}", page=page)
        chip = _run(a, mask, f"cluster:{n}", ws_bytes=256, page=page)
        for o, lse in (full, chip):
            err, lerr = attention_errors(o, lse, a, mask, range(len(ctx)))
            assert err <= ATTN_TOL and lerr <= LSE_TOL
        assert np.abs(full[0] - chip[0]).max() <= 2 ** -8 * max(1.0, np.abs(full[0]).max())
        np.testing.assert_allclose(full[1], chip[1], rtol=0, atol=1e-5)


@pytest.mark.parametrize("ctx,block,hq,hkv", [
    ((2000,) * 2, (16, 12), 32, 8),                                           # equal parts, 9 groups of CTAs a unit
    ((1500, 1400, 90, 0, 3), (16, 9, 1, 0, 24), 32, 8),                       # parts; few tiles, none, an empty block
    ((700,) * 12, (16, 3) * 6, 32, 8),                                        # a group a unit, K's ring ahead
    ((300, 290, 310, 20) * 10, (9, 16, 1, 24) * 10, 32, 8),                   # rounds there and back over the groups
    ((130,) * 64, (4,) * 64, 16, 16),                                         # as many sequences as are dealt; 9 groups
    ((5000,) + (200,) * 11, (8,) * 12, 32, 8),                                # one long among short: cut evenly
    ((900,) * 5, (16,) * 5, 8, 1),                                            # one KV head: dozens of parts
    ((260, 250, 240), (32, 31, 30), 32, 32),                                  # four groups for three sequences
])
@pytest.mark.parametrize("page", [0, 16, 64])
def test_units_dealt_out(ctx, block, hq, hkv, page):
    """The flat split whose kernel may deal the units out, whole or in equal parts, by the lengths it finds."""
    a = wl.attention_inputs(wl.custom(seed=len(ctx) + hkv, ctx=ctx, block=block, num_q_heads=hq, num_kv_heads=hkv))
    seqs = range(0, len(ctx), max(1, len(ctx) // 6))
    for mask in (CAUSAL, BIDIR):
        o, lse = _run(a, mask, "dealt", page=page)
        err, lerr = attention_errors(o, lse, a, mask, seqs)
        assert err <= ATTN_TOL and lerr <= LSE_TOL, (err, lerr)


def _merges(a, **kw):
    from torch.profiler import ProfilerActivity, profile

    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        _run(a, CAUSAL, **kw)
        torch.cuda.synchronize()
    return any("attn_combine_kernel" in e.name for e in prof.events())


@pytest.mark.parametrize("n, ctx, bound, flat", [
    (2, 500, 8192, False), (4, 2000, 32768, False), (8, 1000, 8192, False), (12, 500, 8192, False),
    (16, 2000, 8192, False), (16, 4000, 16384, True), (24, 2000, 8192, True)])
@pytest.mark.parametrize("page", [0, 64])
def test_loose_bound_on_the_lengths(n, ctx, bound, flat, page):
    """max_kv_len as a capacity far above the lengths: the values of the exact bound (to the rounding of another
    split), and where equal lengths take less than about 25 us the clusters an exact bound gets."""
    a = wl.attention_inputs(wl.custom(seed=n, ctx=(ctx,) * n, block=(16,) * n, num_q_heads=32, num_kv_heads=8))
    _merges(a)
    assert _merges(a, max_kv=bound, page=page) == flat
    o, lse = _run(a, CAUSAL, max_kv=bound, page=page)
    err, lerr = attention_errors(o, lse, a, CAUSAL, [0, n - 1])
    assert err <= ATTN_TOL and lerr <= LSE_TOL


@pytest.mark.parametrize("n, ctx, hq, hkv, flat", [
    (1, 16000, 16, 2, False), (1, 16000, 32, 4, False), (24, 16000, 32, 1, True), (4, 4000, 32, 1, False),
    (24, 16000, 16, 2, True), (10, 4000, 32, 16, True), (4, 4000, 32, 16, False), (10, 4000, 32, 32, True)])
def test_split_by_estimate_other_head_counts(n, ctx, hq, hkv, flat):
    """The faster split as timed, for 1 to 32 KV heads."""
    a = wl.attention_inputs(wl.custom(seed=n + hkv, ctx=(ctx,) * n, block=(16,) * n, num_q_heads=hq, num_kv_heads=hkv))
    _merges(a)
    assert _merges(a) == flat
    o, lse = _run(a, CAUSAL)
    err, lerr = attention_errors(o, lse, a, CAUSAL, [n - 1], 0)
    assert err <= ATTN_TOL and lerr <= LSE_TOL
