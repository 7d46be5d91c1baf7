"""Rows of 80 bytes and more that are no power of two fill a lane group up to its last lanes: the narrowest and widest
row of every group, with rows of every length in one kernel (graphs of 900 vertices; the kernels by row length:
test_gpu_lists.py), against the oracle."""
import pytest

from gpu_util import check_against_oracle, make_sage_layer, run_device, small_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,fi", [("f32", 20), ("f32", 28), ("f32", 36), ("f32", 60), ("f32", 68), ("f32", 100), ("f32", 124),
                                      ("bf16", 40), ("bf16", 56), ("bf16", 72), ("bf16", 120), ("bf16", 136), ("bf16", 248)])
@pytest.mark.parametrize("max_deg", [3, 60])   # rows of at most four edges on average, and longer ones
def test_padded_rows_in_every_bucket(dtype, fi, max_deg):
    for op, weights in (("mean", False), ("max", True)):
        layer = make_sage_layer(7, op, "none", fi, 16, dtype, weights=weights, allow_reorder=False)
        w = small_workload(8, 900, max_deg, dtype, [layer], hubs=(2100, 700, 300, 90), weights=weights)
        got, _ = run_device(w)
        check_against_oracle(w, got, label=(dtype, fi, op, max_deg))


@pytest.mark.parametrize("dtype,dims", [("bf16", (64, 8)), ("bf16", (64, 24)), ("bf16", (96, 40)), ("bf16", (64, 104)), ("bf16", (40, 200)), ("bf16", (600, 40)),
                                        ("bf16", (128, 264)), ("bf16", (64, 48)), ("bf16", (64, 96)), ("f32", (64, 48)), ("f32", (128, 112)), ("f32", (128, 80)),
                                        ("f32", (64, 100)), ("f32", (20, 12)), ("f32", (32, 176))])
def test_output_widths_of_the_dense_products(dtype, dims):
    """Outputs that are no whole 128-byte panel, no multiple of 16 columns, or split over several column ranges; one output, and
    two side by side (transform-first layers), with rows that end inside a 128-row tile."""
    fi, fo = dims
    for op, reorder, n in (("mean", False, 300), ("sum", True, 1285)):
        layer = make_sage_layer(9, op, "relu", fi, fo, dtype, allow_reorder=reorder)
        w = small_workload(10, n, 9, dtype, [layer], hubs=(200,))
        got, _ = run_device(w)
        check_against_oracle(w, got, label=(dtype, dims, op))
