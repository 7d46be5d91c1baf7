"""A launch that the runtime refuses is reported by the call that made it, and by no later one.  The refusal is made on the host:
the stream's capture has been invalidated (by a query of the capturing stream), after which nothing may be launched into it."""
import ctypes

import pytest
import torch

from gpu_util import make_gat_layer, make_sage_layer, small_workload
from paper_2307_00228_b200 import binding as B
from paper_2307_00228_b200 import host

pytestmark = pytest.mark.gpu
RELAXED = 2


class _InvalidCapture:
    """A stream whose capture has been invalidated; the capture is ended on exit."""

    def __enter__(self):
        self.rt = ctypes.CDLL("libcudart.so.12")
        self.stream = torch.cuda.Stream()
        self.s = ctypes.c_void_p(self.stream.cuda_stream)
        assert self.rt.cudaStreamBeginCapture(self.s, RELAXED) == 0
        assert self.rt.cudaStreamQuery(self.s) != 0
        self.rt.cudaGetLastError()
        return self.stream

    def __exit__(self, *exc):
        graph = ctypes.c_void_p()
        assert self.rt.cudaStreamEndCapture(self.s, ctypes.byref(graph)) != 0
        self.rt.cudaGetLastError()


@pytest.mark.parametrize("kind", ["gat", "mean", "split_mean"])
def test_a_refused_launch_is_reported_once(kind):
    layer = make_gat_layer(1, "none", 32, 2, 16, "f32") if kind == "gat" else make_sage_layer(1, "mean", "none", 32, 32, "f32", allow_reorder=False)
    w = small_workload(2, 300, 9, "f32", [layer], hubs=(100,) if kind != "split_mean" else (2000,))   # (100 edges: in one piece)
    d = host.upload(w)
    out = torch.zeros((w.n, 32), device="cuda")
    scores = torch.zeros((w.n, 4), device="cuda") if kind == "gat" else None
    gather = lambda stream=None: B.it_layer_gather(d.graph, d.layers[0], d.x, scores, 0, False, out, d.workspace, stream=stream)  # noqa: E731
    gather()
    torch.cuda.synchronize()
    with _InvalidCapture() as stream:
        with pytest.raises(B.ItError) as ei:
            gather(stream)
        assert ei.value.status_name == "IT_ERR_CUDA"
    B.it_aggregate_finish(torch.ones((w.n, 32), device="cuda"), torch.ones(w.n, device="cuda"), out)
    gather()
    torch.cuda.synchronize()
    assert bool(torch.isfinite(out).all())


def test_a_refused_creation_leaves_nothing_behind():
    """The validation cannot be queued or waited for: the creation is refused, the next graphs are not, and start without a timeout."""
    w = small_workload(3, 300, 9, "f32", [make_sage_layer(1, "mean", "none", 32, 32, "f32")])
    ip, ix = torch.from_numpy(w.indptr).cuda(), torch.from_numpy(w.indices).cuda()
    torch.cuda.synchronize()
    with _InvalidCapture() as stream:
        for _ in range(3):
            with pytest.raises(B.ItError) as ei:
                B.it_graph_create(ip, ix, stream=stream)
            assert ei.value.status_name == "IT_ERR_CUDA"
    bad = ix.clone()
    bad[0] = w.n
    for _ in range(3):
        with pytest.raises(B.ItError) as ei:
            B.it_graph_create(ip, bad)
        assert ei.value.status_name == "IT_ERR_BAD_GRAPH"
        g = B.it_graph_create(ip, ix)
        B.it_graph_check(g)
        B.it_graph_destroy(g)
