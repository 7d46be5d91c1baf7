"""Graphs beyond the line of the one-kernel path: the kernels by row length (very short, short, one warp per row, pieces of long
vertices, rows without edges) on more than 2^17 vertices, against the oracle; and both sides of that line against each other."""
import numpy as np
import pytest
import torch

from gpu_util import check_against_oracle, make_gat_layer, make_msg_layer, make_plain_layer, make_sage_layer, run_device, small_workload
from paper_2307_00228_b200 import binding as B
from paper_2307_00228_b200 import host

pytestmark = pytest.mark.gpu

N = (1 << 17) + 77
HUBS = (20000, 4097, 2100, 1025, 1024, 700, 257, 256, 65, 64, 63, 33, 32, 31, 9, 8)


@pytest.mark.parametrize("dtype,fi", [("f32", 4), ("f32", 16), ("f32", 32), ("f32", 60), ("f32", 64), ("f32", 100), ("f32", 132), ("bf16", 8), ("bf16", 32),
                                      ("bf16", 64), ("bf16", 120), ("bf16", 128), ("bf16", 264)])
@pytest.mark.parametrize("op,max_deg", [("mean", 5), ("max", 14)])   # rows of at most four edges on average, and longer ones
def test_pooling(dtype, fi, op, max_deg):
    layer = make_sage_layer(21, op, "relu", fi, 16, dtype, weights=op == "max", allow_reorder=False)
    w = small_workload(22, N, max_deg, dtype, [layer], hubs=HUBS, weights=op == "max", threshold=4096)
    got, _ = run_device(w)
    check_against_oracle(w, got, label=(dtype, fi, op), exact=False)


@pytest.mark.parametrize("dtype,fi", [("bf16", 64), ("f32", 20), ("f32", 32), ("bf16", 128), ("f32", 100)])
@pytest.mark.parametrize("op,weights,max_deg", [("max", False, 9), ("sum", True, 9), ("mean", False, 60), ("min", True, 60)])
def test_no_vertex_in_pieces(dtype, fi, op, weights, max_deg):
    """Rows of at most 1024 edges only: few long ones (walked one at a time), and tens of thousands (chunks of one row after the other)."""
    layer = make_sage_layer(30, op, "relu", fi, 16, dtype, weights=weights, allow_reorder=False)
    w = small_workload(31, N, max_deg, dtype, [layer], hubs=HUBS[4:], weights=weights)
    got, _ = run_device(w)
    check_against_oracle(w, got, label=(dtype, fi, op, max_deg), exact=False)


@pytest.mark.parametrize("dtype,heads,hd", [("f32", 4, 4), ("f32", 4, 16), ("f32", 2, 64), ("bf16", 2, 16), ("bf16", 8, 8), ("bf16", 4, 32), ("f32", 1, 8)])
def test_gat(dtype, heads, hd):
    layer = make_gat_layer(23, "elu", 32, heads, hd, dtype)
    w = small_workload(24, N, 9, dtype, [layer], hubs=HUBS, threshold=4096, p_zero=0.4)
    got, _ = run_device(w)
    check_against_oracle(w, got, label=(dtype, heads, hd), exact=False)


@pytest.mark.parametrize("dtype,heads,hd", [("f32", 4, 8), ("bf16", 4, 16), ("f32", 8, 4), ("bf16", 8, 8)])
@pytest.mark.parametrize("hubs", [HUBS, HUBS[4:]])   # with and without pieces
def test_gat_of_128_byte_rows_with_many_heads(dtype, heads, hd, hubs):
    """More than eight edges per vertex on average: the per-edge softmax, or the batched one where it wins."""
    layer = make_gat_layer(32, "elu", 32, heads, hd, dtype)
    w = small_workload(33, N, 24, dtype, [layer], hubs=hubs, p_zero=0.1)
    assert w.e > 8 * w.n
    got, _ = run_device(w)
    check_against_oracle(w, got, label=(dtype, heads, hd), exact=False)


@pytest.mark.parametrize("kind,dtype,fi", [("mean", "f32", 4), ("max", "f32", 8), ("min", "bf16", 32), ("sum", "f32", 64), ("mean", "bf16", 128), ("max", "f32", 128),
                                           ("max", "bf16", 600), ("min", "f32", 384), ("max", "f32", 12),
                                           ("gat", "f32", (4, 4)), ("gat", "bf16", (4, 16)), ("gat", "bf16", (8, 8)), ("gat", "f32", (2, 32)), ("gat", "f32", (8, 16)),
                                           ("gat", "bf16", (1, 256))])
@pytest.mark.parametrize("p_zero", [0.0, 0.4, 0.97])
def test_small_graph_rows_without_edges_beside_the_short_ones(kind, dtype, fi, p_zero):
    """One kernel per layer: rows of every width, of one column chunk and of several, on graphs with no, some and mostly vertices without
    edges (shares of a warp with a remainder); rows and pieces of 64 and 65 edges (graphs of few edges) next to them."""
    hubs = (500, 193, 129, 128, 66, 65, 64, 63, 33, 32, 31, 17, 16, 9, 8, 7)
    if kind == "gat":
        layer = make_gat_layer(35, "elu", 32, *fi, dtype)
    else:
        layer = make_sage_layer(35, kind, "relu", fi, 16, dtype, weights=kind == "sum", allow_reorder=False)
    w = small_workload(36, 5001, 24, dtype, [layer], hubs=hubs, weights=kind == "sum", p_zero=p_zero)
    got, _ = run_device(w)
    check_against_oracle(w, got, label=(kind, dtype, fi, p_zero))


@pytest.mark.parametrize("n,deg", [(1000, 1100), (3700, 245), (3700, 270), (3000, 400)])
@pytest.mark.parametrize("kind", ["sum", "max", "gat"])
def test_few_vertices_of_many_edges(n, deg, kind):
    """Both sides of the line between one kernel and kernels by list: about 245 and 270 edges per vertex, fewer vertices, and far beyond it."""
    layer = make_gat_layer(34, "elu", 32, 4, 16, "f32") if kind == "gat" else make_sage_layer(34, kind, "relu", 132, 16, "f32", allow_reorder=False)
    w = small_workload(35, n, 2 * deg, "f32", [layer], hubs=(5000, 129, 128, 127), p_zero=0.0)
    got, _ = run_device(w)
    check_against_oracle(w, got, label=(n, deg, kind), exact=False)


@pytest.mark.parametrize("n", [900, N])
@pytest.mark.parametrize("kind", ["sum", "gat"])
def test_the_threshold_changes_no_bit(n, kind):
    """What is gathered in pieces does not depend on the shadow rows: thresholds far below, between and above the bounds of the lists."""
    layer = make_gat_layer(36, "elu", 32, 4, 8, "f32") if kind == "gat" else make_sage_layer(36, "sum", "relu", 32, 16, "f32", weights=True, allow_reorder=False)
    w = small_workload(37, n, 40, "f32", [layer], hubs=HUBS, weights=True)
    base, d = run_device(w, threshold=0)
    check_against_oracle(w, base, label=(n, kind), exact=False)
    deg = np.diff(w.indptr)
    for T in (1, 7, 8, 9, 32, 33, 300, 1024, 1025, 4096, 20000):
        rows, split = B.it_split_hubs(d.graph, T)
        assert rows == int(np.maximum(1, -(-deg // T)).sum()) and split == int((deg > T).sum())
        assert np.array_equal(d.infer().double().cpu().numpy(), base), T


@pytest.mark.parametrize("dtype,fi", [("bf16", 64), ("bf16", 40), ("bf16", 264), ("f32", 32), ("f32", 132)])
@pytest.mark.parametrize("op,weights", [("max", False), ("min", False), ("min", True), ("sum", True)])
def test_every_reduce(dtype, fi, op, weights):
    """Plain maxima and minima (packed pairs in bf16), weighted ones and weighted sums, rows that fill their lane group and rows that do
    not, rows of more than one column chunk; very short, short and long rows, and pieces."""
    layer = make_sage_layer(40, op, "none", fi, 16, dtype, weights=weights, allow_reorder=False)
    w = small_workload(41, N, 7, dtype, [layer], hubs=HUBS, weights=weights, threshold=300)
    got, _ = run_device(w)
    check_against_oracle(w, got, label=(dtype, fi, op, weights), exact=False)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("kind", ["edge_features", "messages", "gat_edge_logits", "wide"])
def test_rows_in_edge_order_and_column_chunks(dtype, kind):
    """Edge features next to the source rows, learned messages, attention logits with an edge term, rows of more than 512 bytes."""
    if kind == "edge_features":
        layer = make_sage_layer(42, "mean", "relu", 32, 16, dtype, edge_dim=16)
    elif kind == "messages":
        layer = make_msg_layer(43, "max", "relu", 32, 32, 16, dtype, edge_dim=8)
    elif kind == "gat_edge_logits":
        layer = make_gat_layer(44, "elu", 32, 4, 16, dtype, edge_dim=8)
    else:
        layer = make_sage_layer(45, "mean", "relu", 320, 16, dtype, allow_reorder=False)
    w = small_workload(46, N, 6, dtype, [layer], hubs=HUBS, threshold=64, edge_dim=layer.edge_dim)
    got, _ = run_device(w)
    check_against_oracle(w, got, label=(dtype, kind), exact=False)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("op", ["sum", "mean", "max", "min"])
def test_raw_partial_results(dtype, op):
    """What a part hands to the others, by value: whole numbers, so that fp32 sums are exact in any order."""
    layer = make_sage_layer(47, op, "none", 32, 16, dtype, allow_reorder=False)
    w = small_workload(48, N, 6, "f32", [layer], hubs=HUBS, p_zero=0.5)
    w.x, w.dtype = np.round(w.x * 2).astype(np.float32), "f32"
    d = host.upload(w)
    x = d.x.to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    lay = host.layer_to_device(layer, dtype)
    out = torch.full((w.n, 32), float("nan"), device="cuda")
    ws = torch.empty(B.it_workspace_bytes(d.graph, [lay]), dtype=torch.uint8, device="cuda")
    B.it_layer_gather(d.graph, lay, x, None, 0, True, out, ws)
    rows = torch.from_numpy(np.repeat(np.arange(w.n), np.diff(w.indptr))).cuda()
    src = d.x[torch.from_numpy(w.indices.astype(np.int64)).cuda()]
    start = {"max": float("-inf"), "min": float("inf")}.get(op, 0.0)
    want = torch.full((w.n, 32), start, device="cuda")
    if op in ("max", "min"):
        want.scatter_reduce_(0, rows[:, None].expand(-1, 32), src, "amax" if op == "max" else "amin")
    else:
        want = want.double().index_add_(0, rows, src.double()).float()
    assert torch.equal(out, want)


@pytest.mark.parametrize("kind", ["mean", "gat"])
def test_a_vertex_of_more_pieces_than_one_block_should_fold(kind):
    """5M edges on one vertex: pieces longer than 512 edges, and a remainder."""
    layer = make_gat_layer(38, "none", 8, 1, 16, "f32") if kind == "gat" else make_sage_layer(38, kind, "none", 8, 16, "f32", allow_reorder=False)
    w = small_workload(39, N, 4, "f32", [layer], hubs=(5_000_011, 8192 * 512, 8192 * 512 + 1, 5000))
    got, _ = run_device(w)
    check_against_oracle(w, got, label=kind, exact=False)


def test_self_term_and_bias_of_rows_without_edges():
    for layer in (make_sage_layer(25, "mean", "elu", 64, 32, "bf16"), make_plain_layer(26, "gcn", "elu", 64, 32, "bf16")):
        w = small_workload(27, N, 4, "bf16", [layer], hubs=HUBS[:6], p_zero=0.9)
        got, _ = run_device(w)
        check_against_oracle(w, got, label=layer.op, exact=False)


@pytest.mark.parametrize("dtype,dims,kind", [("f32", (64, 64), "mean"), ("bf16", (128, 128), "gat"), ("f32", (16, 48), "max")])
def test_both_sides_of_the_small_graph_line(dtype, dims, kind):
    """The same rows in a graph of 2^17 vertices (one kernel per layer) and in one of more (kernels by list): sums may differ by
    the order of at most a few hundred additions, 2^-24 each, or one rounding of a stored bf16 result (2^-8)."""
    layer = make_gat_layer(28, "none", dims[0], 4, dims[1] // 4, dtype) if kind == "gat" else make_sage_layer(28, kind, "none", *dims, dtype)
    w = small_workload(29, 1 << 17, 6, dtype, [layer], hubs=HUBS[1:])
    d = host.upload(w)
    small = d.infer().float()
    extra = np.concatenate([w.indptr, np.full(500, w.indptr[-1])])   # 500 more vertices without edges
    g = B.it_graph_create(torch.from_numpy(extra).cuda(), torch.from_numpy(w.indices).cuda())
    x = torch.cat([d.x, torch.zeros((500, dims[0]), dtype=d.x.dtype, device="cuda")])
    out = torch.empty((x.shape[0], dims[1]), dtype=x.dtype, device="cuda")
    ws = torch.empty(B.it_workspace_bytes(g, d.layers), dtype=torch.uint8, device="cuda")
    big = B.it_infer(g, d.layers, x, out, ws)[: w.n].float()
    scale = small.abs().mean()
    assert float((big - small).abs().max()) <= (2.0 ** -24 * 4096 if dtype == "f32" else 2.0 ** -6) * float(torch.maximum(small.abs().max(), scale))
