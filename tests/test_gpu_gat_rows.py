"""The batched GAT reduce at the shapes where it can go wrong: every number of heads it takes, every row width, rows at the
edges of its rounds (8 edges) and chunks (32 edges), rows of one block, split hubs, and rows without edges."""
import pytest
import torch

from gpu_util import check_against_oracle, make_gat_layer, make_sage_layer, run_device, small_workload, to_numpy
from paper_2307_00228_b200 import binding as B
from paper_2307_00228_b200 import host

pytestmark = pytest.mark.gpu

EDGES = (2100, 1025, 257, 256, 65, 64, 63, 40, 33, 32, 31, 25, 24, 17, 16, 9, 8, 7, 1)


@pytest.mark.parametrize("dtype,heads,hd", [("f32", 1, 32), ("f32", 2, 16), ("f32", 8, 4), ("f32", 4, 16), ("f32", 8, 8), ("f32", 1, 128),
                                            ("f32", 4, 32), ("bf16", 1, 64), ("bf16", 2, 32), ("bf16", 8, 8), ("bf16", 4, 32), ("bf16", 8, 16),
                                            ("bf16", 2, 128), ("bf16", 8, 32)])
@pytest.mark.parametrize("threshold", [0, 128])
def test_heads_widths_and_row_lengths(dtype, heads, hd, threshold):
    layer = make_gat_layer(11, "elu", 32, heads, hd, dtype)
    w = small_workload(12, 700, 14, dtype, [layer], hubs=EDGES, threshold=threshold, p_zero=0.4)
    got, _ = run_device(w)
    check_against_oracle(w, got, label=(dtype, heads, hd, threshold))


@pytest.mark.parametrize("n", [700, (1 << 17) + 77])   # one kernel per layer, and kernels by row length
@pytest.mark.parametrize("slope", [-0.3, 0.0])
@pytest.mark.parametrize("dtype,heads,hd", [("f32", 4, 4), ("f32", 2, 16), ("bf16", 4, 32), ("bf16", 8, 8)])
def test_any_leaky_slope(dtype, heads, hd, slope, n):
    """A slope that is zero or negative: places of a round without an edge must stay out of the softmax (rows of 1 to 33 edges
    leave every number of such places)."""
    layer = make_gat_layer(17, "none", 32, heads, hd, dtype)
    layer.leaky_slope = slope
    w = small_workload(18, n, 9, dtype, [layer], hubs=tuple(range(1, 34)) + (300, 65), p_zero=0.3)
    got, _ = run_device(w)
    check_against_oracle(w, got, label=(dtype, heads, hd, slope, n), exact=False)


def test_bias_need_not_be_aligned():
    layer = make_gat_layer(13, "none", 32, 4, 16, "f32")
    w = small_workload(14, 300, 12, "f32", [layer], hubs=(300, 40))
    d = host.upload(w)
    want = d.infer().clone()
    wide = torch.empty(65, device="cuda")
    wide[1:] = d.layers[0].bias
    d.layers[0].bias = wide[1:]
    assert d.layers[0].bias.data_ptr() % 16 != 0
    assert torch.equal(d.infer(), want)


@pytest.mark.parametrize("dtype,dims", [("f32", (64, 16)), ("f32", (100, 20)), ("bf16", (8, 128)), ("bf16", (264, 64))])
@pytest.mark.parametrize("op,raw", [("max", False), ("min", True), ("max", True), ("mean", True), ("gcn", False)])
def test_rows_without_edges(dtype, dims, op, raw):
    """Nearly all rows empty (more than one block's worth): zeros, the identity of a raw partial reduce, or act(bias)."""
    layer = make_sage_layer(15, "sum" if op == "gcn" else op, "elu", *dims, dtype, allow_reorder=not raw)
    if op == "gcn":
        layer.op, layer.W = "gcn", layer.W[: dims[0]]
    w = small_workload(16, 5003, 5, dtype, [layer], p_zero=0.97)
    if not raw:
        got, _ = run_device(w)
        check_against_oracle(w, got, label=(dtype, dims, op))
        return
    d = host.upload(w)
    out = torch.full((w.n, dims[0]), float("nan"), device="cuda")
    B.it_layer_gather(d.graph, d.layers[0], d.x, None, 0, True, out, d.workspace)
    empty = torch.from_numpy((w.indptr[1:] == w.indptr[:-1])).cuda()
    identity = {"max": float("-inf"), "min": float("inf"), "mean": 0.0}[op]
    assert bool((out[empty] == identity).all())
    assert bool(torch.isfinite(out[~empty]).all()) and to_numpy(out[~empty]).size > 0
