"""Layers with learned messages (the general apply_edge: m = w_e act_edge([h_u | e_vu] W_edge + b_edge), Eq. (1))
against the CPU oracle, through the C ABI: every reduce and GCN, both storage types, with and without edge
features and edge weights, on split and unsplit graphs, stacked, and the argument checks."""
import numpy as np
import pytest
import torch

from gpu_util import check_against_oracle, make_gat_layer, make_msg_layer, make_sage_layer, run_device, small_workload
from paper_2307_00228_b200 import binding as B
from paper_2307_00228_b200 import host
from workloads import Workload
from workloads import rng as wrng

pytestmark = pytest.mark.gpu

HUBS = (257, 300, 1000, 2500, 33, 32, 9, 8, 1)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("op", ["sum", "mean", "max", "min", "gcn"])
@pytest.mark.parametrize("edge_dim", [0, 8])
@pytest.mark.parametrize("threshold", [0, 64])
def test_message_layer_parity(dtype, op, edge_dim, threshold):
    layer = make_msg_layer(1, op, "relu", 32, 32, 64, dtype, act_edge="elu", weights=(op in ("sum", "max")), edge_dim=edge_dim)
    w = small_workload(2, 1500, 30, dtype, [layer], hubs=HUBS, weights=True, threshold=threshold, edge_dim=edge_dim)
    got, d = run_device(w)
    if threshold:
        assert d.n_split_owners > 0
    check_against_oracle(w, got, label=(dtype, op, edge_dim, threshold))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("dims", [(16, 8, 16, 24), (64, 16, 128, 32), (24, 40, 48, 16), (128, 32, 64, 128)])
def test_message_shapes(dtype, dims):
    """(in_dim, edge_dim, msg_dim, out_dim): message rows of several widths, K that is not a whole number of k-blocks."""
    fi, de, fm, fo = dims
    layer = make_msg_layer(3, "sum", "none", fi, fm, fo, dtype, act_edge="relu", edge_dim=de)
    w = small_workload(4, 700, 14, dtype, [layer], hubs=(300, 40), threshold=128, edge_dim=de)
    got, _ = run_device(w)
    check_against_oracle(w, got, label=(dtype, dims))


@pytest.mark.parametrize("act", ["none", "relu", "elu"])
@pytest.mark.parametrize("fm", [8, 24, 72, 120, 128])
def test_messages_finished_in_the_product(fm, act):
    """bf16 messages leave the per-edge product finished: widths that are no multiple of 16 columns or of a 128-byte panel, every
    activation, a last tile with few rows (oracle and metric of the other layers: one more rounding to bf16 is in both)."""
    layer = make_msg_layer(9, "sum", "none", 32, fm, 32, "bf16", act_edge=act, edge_dim=16)
    w = small_workload(10, 701, 13, "bf16", [layer], hubs=(300, 41), threshold=128, edge_dim=16)
    got, _ = run_device(w)
    check_against_oracle(w, got, label=(fm, act))


# in-degrees whose sums put the ends of vertices at, before and after the 128-edge tiles of the per-edge product, vertices of several
# tiles and of so many that a block folds their parts, runs of vertices without edges longer than a tile
TILE_DEGREES = {
    "one edge": [0, 1, 0],
    "one tile": [0, 100, 28],
    "a tile and an edge": [64, 64, 1],
    "aligned": [128, 256, 0, 128, 16, 112],
    "crossing": [127, 2, 127, 1, 300, 83] + [0] * 300 + [15, 17, 16, 0, 1, 31] * 9,
    "long": [5, 6500, 3, 0, 129, 40] + [3] * 50,
}


def tile_workload(deg, layer, seed):
    deg = np.asarray(deg)
    base = small_workload(seed, len(deg), 0, "bf16", [layer])
    rng = np.random.default_rng(seed)
    e = int(deg.sum())
    ef = wrng.f32_to_bf16_bits(rng.standard_normal((e, layer.edge_dim)).astype(np.float32))
    return Workload("tiles", len(deg), e, np.concatenate(([0], np.cumsum(deg))), rng.integers(0, len(deg), e).astype(np.int32),
                    rng.random(e, dtype=np.float32), "bf16", base.x, [layer], 0, ef)


@pytest.mark.parametrize("degrees", TILE_DEGREES)
@pytest.mark.parametrize("fm,weights", [(40, False), (128, True)])
def test_messages_written_by_their_product(degrees, fm, weights):
    """Few edges: tiles of finished messages are written, the last one in part (oracle and tolerance of the other message tests)."""
    layer = make_msg_layer(13, "sum", "none", 16, fm, 24, "bf16", act_edge="relu", weights=weights, edge_dim=8)
    w = tile_workload(TILE_DEGREES[degrees], layer, 14)
    got, _ = run_device(w)
    check_against_oracle(w, got, label=(degrees, fm))


@pytest.mark.parametrize("op,weights,fm,tail", [("sum", False, 64, 0), ("sum", True, 24, 1), ("mean", False, 24, 127), ("mean", True, 120, 64), ("max", False, 64, 1),
                                                ("min", True, 64, 0), ("max", False, 120, 5), ("gcn", True, 120, 127), ("min", False, 24, 0), ("max", True, 24, 3)])
def test_messages_reduced_by_their_product(op, weights, fm, tail):
    """Many edges: written by the product with the caller's workspace, reduced tile by tile where they are made without one (their rows
    then do not fit); every pattern of ends of vertices, a last tile of `tail` edges (0: a whole one).  Oracle and tolerance of the other
    message tests: a sum in another order differs in fp32 only."""
    layer = make_msg_layer(15, op, "none", 16, fm, 24, "bf16", act_edge="elu" if op == "sum" else "relu", weights=weights, edge_dim=8)
    bulk = np.random.default_rng(16).integers(0, 48, 58_000) if fm < 120 else np.random.default_rng(16).integers(0, 96, 29_000)
    deg = [d for p in TILE_DEGREES.values() for d in p] + bulk.tolist()
    deg.append((tail - sum(deg)) % 128)
    assert sum(deg) % 128 == tail and sum(deg) > 5 << 18
    w = tile_workload(deg, layer, 17)
    got, d = run_device(w)
    check_against_oracle(w, got, label=(op, weights, fm, tail))
    again, _ = run_device(w, int32_indptr=True)
    assert np.array_equal(got, again)
    assert w.e * fm * 2 > 32 << 20   # the message rows alone exceed the built-in scratch
    reduced = static_forward(d)
    assert_same_reduce(op, d.out.float(), reduced.float())
    assert torch.equal(reduced, static_forward(d))


def static_forward(d):
    out = torch.full_like(d.out, float("nan"))
    B.it_layer_forward_static(d.graph, d.layers[0], d.x, out)
    B.it_graph_check(d.graph)
    return out


def assert_same_reduce(op, a, b):
    """Two orders of the same reduce: max and min the same bits; sums differ by a rounding (2^-8) of the bf16 aggregate and one of the output,
    of products of the order of the largest."""
    if op in ("max", "min"):
        assert torch.equal(a.nan_to_num(nan=12345.0), b.nan_to_num(nan=12345.0))
        return
    ok = torch.isfinite(a)
    assert torch.equal(ok, torch.isfinite(b))
    assert (a[ok] - b[ok]).abs().max() <= 2.0 ** -7 * a[ok].abs().max()


@pytest.mark.parametrize("op,fm,deg_max", [("max", 64, 90), ("mean", 128, 60), ("mean", 72, 80)])
def test_messages_reduced_by_their_product_with_a_workspace(op, fm, deg_max):
    """As many edges as make the reduce in the product the faster form: the scratch then holds no message rows (oracle and tolerance of
    the other message tests)."""
    e = (320 << 20) // fm + 1000
    deg = np.random.default_rng(21).integers(0, deg_max, 2 * e // (deg_max - 1) + 1000)
    layer = make_msg_layer(22, op, "none", 16, fm, 24, "bf16", act_edge="relu", edge_dim=8)
    w = tile_workload(deg, layer, 23)
    assert w.e >= e and w.e >= 14 * w.n
    got, d = run_device(w)
    assert B.it_workspace_bytes(d.graph, d.layers) < w.e * fm * 2
    check_against_oracle(w, got, label=(op, fm))


@pytest.mark.parametrize("op,fm", [("max", 64), ("min", 24), ("sum", 40), ("mean", 120), ("max", 8), ("sum", 16)])
def test_infinite_and_undefined_messages_reduce_the_same_in_their_product(op, fm):
    """Messages of +-inf and NaN, and the narrowest rows: the reduce in the product gives what the gather gives of the written rows (max and
    min: the same bits; sums: to the rounding of bf16 outputs, infinities and NaN where they are)."""
    layer = make_msg_layer(31, op, "none", 16, fm, 24, "bf16", act_edge="none", edge_dim=8)
    deg = [d for p in TILE_DEGREES.values() for d in p] + np.random.default_rng(32).integers(0, 60, (32 << 20) // (2 * fm) // 25).tolist()
    w = tile_workload(deg, layer, 33)
    rng = np.random.default_rng(34)
    bits = w.edge_feat.view(np.uint16)
    bits[rng.random(w.e) < 0.01, 0] = 0x7f80    # inf times weights of both signs
    bits[rng.random(w.e) < 0.002, 1] = 0x7fc0
    got, d = run_device(w)
    assert w.e * fm * 2 > 32 << 20
    assert not torch.isfinite(d.out).all() and torch.isfinite(d.out).any()
    assert_same_reduce(op, d.out.float(), static_forward(d).float())


def test_message_layers_stack_with_plain_layers():
    layers = [make_msg_layer(5, "mean", "relu", 32, 64, 32, "f32", act_edge="relu", edge_dim=8),
              make_sage_layer(6, "sum", "relu", 32, 32, "f32", edge_dim=8),
              make_msg_layer(7, "max", "none", 32, 16, 16, "f32", act_edge="elu", edge_dim=8)]
    w = small_workload(8, 900, 10, "f32", layers, hubs=(200,), threshold=64, edge_dim=8)
    got, d = run_device(w)
    check_against_oracle(w, got)
    # it_infer is the sequence of it_layer_forward calls
    h = d.x
    for lay, src in zip(d.layers, w.layers):
        o = torch.empty((w.n, src.out_dim), device="cuda")
        B.it_layer_forward(d.graph, lay, h, o, d.workspace)
        h = o
    torch.cuda.synchronize()
    assert torch.equal(h, d.out)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("threshold", [0, 100])
@pytest.mark.parametrize("heads,hd,de", [(2, 16, 8), (4, 32, 16), (1, 8, 8)])
def test_gat_with_edge_features_in_the_logits(dtype, threshold, heads, hd, de):
    """e = LeakyReLU(a_src . z_u + a_dst . z_v + a_edge . e_vu): split and unsplit, all row kernels (hubs up to 2500 edges)."""
    layer = make_gat_layer(21, "elu", 32, heads, hd, dtype, edge_dim=de)
    w = small_workload(22, 1300, 25, dtype, [layer], hubs=HUBS, threshold=threshold, edge_dim=de)
    got, d = run_device(w)
    if threshold:
        assert d.n_split_owners > 0
    check_against_oracle(w, got, label=(dtype, threshold, heads, hd, de))


def test_gat_edge_logits_change_the_result_and_stack():
    layers = [make_gat_layer(23, "elu", 32, 2, 16, "f32", edge_dim=8), make_gat_layer(24, "none", 32, 2, 8, "f32", edge_dim=8)]
    w = small_workload(25, 800, 12, "f32", layers, hubs=(300,), threshold=64, edge_dim=8)
    got, _ = run_device(w)
    check_against_oracle(w, got)
    plain = [make_gat_layer(23, "elu", 32, 2, 16, "f32"), make_gat_layer(24, "none", 32, 2, 8, "f32")]
    for a, b in zip(plain, layers):   # the same parameters without the edge term
        a.W, a.bias, a.att_src, a.att_dst = b.W, b.bias, b.att_src, b.att_dst
    w2 = small_workload(25, 800, 12, "f32", plain, hubs=(300,), threshold=64)
    base, _ = run_device(w2)
    assert np.abs(got - base).max() > 1e-3


def test_message_argument_checks():
    layer = make_msg_layer(9, "sum", "none", 16, 16, 16, "f32", edge_dim=8)
    w = small_workload(10, 100, 5, "f32", [layer], edge_dim=8)
    d = host.upload(w)
    out = torch.empty((w.n, 16), device="cuda")

    def status_of(fn):
        with pytest.raises(B.ItError) as ei:
            fn()
        return ei.value.status_name

    bad = host.layer_to_device(make_msg_layer(11, "sum", "none", 16, 6, 16, "f32", edge_dim=8), "f32")   # 24-byte message rows
    assert status_of(lambda: B.it_workspace_bytes(d.graph, [bad])) == "IT_ERR_INVALID_ARG"
    no_w = host.layer_to_device(layer, "f32")
    no_w.W_edge = None
    assert status_of(lambda: B.it_layer_forward(d.graph, no_w, d.x, out, d.workspace)) == "IT_ERR_INVALID_ARG"
    gat = host.layer_to_device(layer, "f32")
    gat.op = "gat"
    gat.edge_dim = 0
    assert status_of(lambda: B.it_workspace_bytes(d.graph, [gat])) == "IT_ERR_UNSUPPORTED"   # learned messages are not for GAT
    g2 = host.layer_to_device(make_gat_layer(12, "none", 16, 2, 8, "f32", edge_dim=8), "f32")
    g2.att_edge = None
    ws = torch.empty(B.it_workspace_bytes(d.graph, [g2]), dtype=torch.uint8, device="cuda")
    assert status_of(lambda: B.it_layer_forward(d.graph, g2, d.x, out, ws)) == "IT_ERR_INVALID_ARG"
    assert torch.ones(3, device="cuda").sum().item() == 3
