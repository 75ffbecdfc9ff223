"""GPU parity of bp_policy_select against the fp64 oracle.

Bars: logits within 1e-3 relative to max |o| (fp32 accumulation of bf16/fp32 products); the
selected block size exact unless the oracle's top-2 margin is below 1e-4 * max |o|.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2606_31315_gb300 as bp
from paper_2606_31315_gb300 import workloads as wl

from _gpu import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    bp.build()
    bp.load()


def _run(pin):
    dt = "bf16" if pin["wdtype"] == "bf16" else None
    f = lambda k: to_dev(pin[k], dt if k in ("feats", "w1", "w2") else None)  # noqa: E731
    ri = to_dev(pin["row_index"]) if pin.get("row_index") is not None else None
    bs, lo = bp.policy_select(f("feats"), f("w1"), f("b1"), f("w2"), f("b2"), f("candidates"), row_index=ri)
    return bs.cpu().numpy(), lo.cpu().numpy()


def _oracle(pin):
    d = pin["wdtype"]
    return oracle.policy_select(wl.as_f64(pin["feats"], d), wl.as_f64(pin["w1"], d), pin["b1"],
                                wl.as_f64(pin["w2"], d), pin["b2"], pin["candidates"], row_index=pin.get("row_index"))


def _compare(pin):
    bs, lo = _run(pin)
    ref = _oracle(pin)
    scale = np.abs(ref["logits"]).max()
    assert np.abs(lo - ref["logits"]).max() <= 1e-3 * scale
    ok = ref["top2_margin"] >= 1e-4 * scale
    np.testing.assert_array_equal(bs[ok], ref["block_size"][ok])


def test_tiny_fp32():
    _compare(wl.policy_inputs(wl.get("tiny")))


def test_ragged_bf16_32_requests():
    _compare(wl.policy_inputs(wl.get("ragged")))


def test_more_requests_than_one_group():
    w = wl.custom(seed=5, policy=dict(num_reqs=70, d_in=512, hidden=300, wdtype="bf16", feat_std=1.0))
    _compare(wl.policy_inputs(w))


def test_ties_choose_lowest_index():
    pin = wl.policy_inputs(wl.get("tiny"))
    pin["w2"] = np.zeros_like(pin["w2"])
    pin["b2"] = np.array([0, 1, 3, 2, 3, 3, 0, 1, 3], dtype=np.float32)
    bs, _ = _run(pin)
    assert np.all(bs == pin["candidates"][2])


def test_paper_input_width_streams_w1():
    # Section 3.1 feeds the predictor the last-token logit vector, so d_in = V = 151936: far more
    # 64-column W1 atoms per CTA than fit in shared memory at once, so they stream through a ring.
    w = wl.custom(seed=6, policy=dict(num_reqs=4, d_in=151936, hidden=256, wdtype="bf16", feat_std=3.0))
    _compare(wl.policy_inputs(w))


@pytest.mark.parametrize("d_in", [4104, 5160])
def test_d_in_tail_and_two_request_groups(d_in):
    # d_in is not a multiple of 64 (the last atom is zero-filled), 70 requests span two groups of 64
    # (the second only partly filled) and hidden = 300 leaves the last W1 tile partial.  Split over
    # 9 CTAs per tile, d_in = 4104 (65 atoms, 8 per CTA) is loaded at once; d_in = 5160 (81 atoms, 9
    # per CTA) streams through the ring and wraps around it.
    w = wl.custom(seed=7, policy=dict(num_reqs=70, d_in=d_in, hidden=300, wdtype="bf16", feat_std=1.0))
    _compare(wl.policy_inputs(w))


@pytest.mark.parametrize("n,d_in,hidden", [
    (4, 41992, 256),     # 2 tiles of 657 atoms (the last of 8 columns): dozens of runs per tile
    (33, 40000, 900),    # a partial tile of 4 rows, 48 padded requests
    (64, 82000, 300),    # a full group
    (130, 41000, 300),   # three request groups, the last of two
    (1, 40000, 128),     # one tile cut over every CTA, runs of 4 or 5 atoms
    (33, 120000, 900),   # 48 padded requests on runs long enough for the flat split
    (130, 130000, 300),  # so are these three groups
    (17, 5912, 600),     # short runs: clusters in either workspace
])
@pytest.mark.parametrize("gather", [True, False])
def test_streamed_splits(n, d_in, hidden, gather):
    """Wide inputs on both splits of the stream: flat over the SMs in a workspace of the size the library asks
    for, clusters in one without the flat split's region; feature rows in place or gathered.  Against the oracle,
    and with each other to the rounding of fp32 sums in another order (bound: sqrt(d_in) 2^-24 of |w||x|, a few
    1e-6 of the largest logit; 1e-4 is far inside the bar)."""
    w = wl.custom(seed=n + hidden, policy=dict(num_reqs=n, d_in=d_in, hidden=hidden, wdtype="bf16", feat_std=1.0))
    pin = wl.policy_inputs(w)
    if not gather:
        pin["feats"], pin["row_index"] = np.ascontiguousarray(pin["feats"][pin["row_index"]]), None
    ref = _oracle(pin)
    scale = np.abs(ref["logits"]).max()
    f = lambda k: to_dev(pin[k], "bf16" if k in ("feats", "w1", "w2") else None)  # noqa: E731
    ri = to_dev(pin["row_index"]) if gather else None
    args = [f(k) for k in ("feats", "w1", "b1", "w2", "b2", "candidates")]
    c = len(pin["candidates"])
    up = lambda x: -(-x // 256) * 256  # noqa: E731
    groups, tiles = -(-n // 64), -(-hidden // 128)
    least = 256 + up(4 * n * hidden) + up(4 * groups * tiles * 64 * c) + up(4 * groups) + up(groups * 64 * d_in * 2)
    full = bp.policy_select_workspace_size(n, d_in, hidden, c)
    assert least < full
    for size in (full, least):
        ws = bp.workspace(size, "cuda")
        for _ in range(2):  # the tickets are back at zero after a call
            bs, lo = bp.policy_select(*args, row_index=ri, ws=ws)
        assert bp.get_status(ws) == 0
        assert np.abs(lo.cpu().numpy() - ref["logits"]).max() <= 1e-4 * scale
        ok = ref["top2_margin"] >= 1e-4 * scale
        np.testing.assert_array_equal(bs.cpu().numpy()[ok], ref["block_size"][ok])
    with pytest.raises(bp.BlockPilotError) as e:
        bp.policy_select(*args, row_index=ri, ws=bp.workspace(least, "cuda")[:-1])
    assert e.value.status == 4


@pytest.mark.parametrize("n,d_in,hidden", [
    (1, 4, 1),          # one copy, one row
    (33, 36, 65),       # a request and a row past a tile, a chunk of 4 columns
    (32, 1000, 64),     # exactly one tile
    (70, 4100, 300),    # three request tiles, d_in split over a cluster
    (5, 40960, 130),    # the widest input the fp32 path takes
])
def test_fp32_tiles(n, d_in, hidden):
    """fp32 sums of d_in and hidden terms: errors of a few sqrt(length) 2^-24 of the terms, 1e-6 of the logits."""
    w = wl.custom(seed=n + hidden, policy=dict(num_reqs=n, d_in=d_in, hidden=hidden, wdtype="f32", feat_std=1.0))
    pin = wl.policy_inputs(w)
    bs, lo = _run(pin)
    ref = _oracle(pin)
    scale = np.abs(ref["logits"]).max()
    assert np.abs(lo - ref["logits"]).max() <= 1e-5 * scale
    ok = ref["top2_margin"] >= 1e-4 * scale
    np.testing.assert_array_equal(bs[ok], ref["block_size"][ok])


def test_one_wide_request_of_any_row_stride():
    """The stride of a single row is not used: one wider than a tensor map can hold is taken too."""
    w = wl.custom(seed=3, policy=dict(num_reqs=1, d_in=98304, hidden=64, wdtype="bf16", feat_std=1.0))
    pin = wl.policy_inputs(w)
    f = lambda k: to_dev(pin[k], "bf16" if k in ("feats", "w1", "w2") else None)  # noqa: E731
    rest = [f(k) for k in ("w1", "b1", "w2", "b2", "candidates")]
    feats = f("feats")[:1]
    bs, lo = bp.policy_select(feats, *rest)
    bs1, lo1 = bp.policy_select(feats.as_strided((1, 98304), (1 << 40, 1)), *rest)
    assert torch.equal(bs, bs1) and torch.equal(lo, lo1)


@pytest.mark.parametrize("hidden", [1, 255, 1025, 3262])
@pytest.mark.parametrize("cand", [1, 16, 17, 64])
@pytest.mark.parametrize("dtype, tol", [(torch.float32, 1e-5), (torch.bfloat16, 1e-5)])
def test_output_layer_rounds(dtype, tol, hidden, cand):
    """Candidates in rounds of 16, hidden units past a thread's loads in flight.  fp32 sums of 72 and hidden terms:
    a few sqrt(length) 2^-24 of the terms.  (72 bf16 columns: h stays fp32 and W2 is exact in fp32.)"""
    gen = torch.Generator().manual_seed(hidden + cand)
    rnd = lambda *s: torch.randn(*s, generator=gen)  # noqa: E731
    x, w1, b1, w2, b2 = rnd(3, 72), rnd(hidden, 72) / 8, rnd(hidden), rnd(cand, hidden) / hidden ** 0.5, rnd(cand)
    x, w1, w2 = (t.to(dtype) for t in (x, w1, w2))
    sizes = torch.arange(cand, dtype=torch.int32) + 2
    bs, lo = bp.policy_select(*(t.cuda() for t in (x, w1, b1, w2, b2, sizes)))
    h = (x.double() @ w1.double().T + b1.double()).clamp_min(0)
    ref = h @ w2.double().T + b2.double()
    assert (lo.cpu().double() - ref).abs().max() <= tol * ref.abs().max() + 1e-6
    top = ref.topk(min(2, cand)).values
    clear = (top[:, 0] - top[:, -1] > 1e-4) if cand > 1 else torch.ones(3, dtype=torch.bool)
    assert torch.equal(bs.cpu()[clear], sizes[ref.argmax(1)][clear])
