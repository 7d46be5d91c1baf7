"""Rows of 80 bytes and more that are no power of two fill a lane group up to its last lanes: the narrowest and widest
row of every group, in buckets of every length class (very short, short, one warp, one block), against the oracle."""
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
