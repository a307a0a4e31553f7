"""The first call for node gradients allocates the accumulator that every later
call finds zero.  Made inside a stream capture it must be zero all the same for
calls that run before the graph's first launch, and when the graph is dropped.

The memory that the accumulator is given is filled beforehand: blocks of its
size (256 KiB, which CUDA cuts from a larger piece and hands out as they are),
written by other volumes and freed.  So a fill that was only recorded shows."""
import numpy as np
import pytest

import synth
from synth import Grid

from gpu_helpers import load_pf, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

GRID = Grid(32, 32, 32, 0.1, 0.3, (0.0, 0.0, 0.0))
JUNK = Grid(64, 32, 32, 0.1, 0.3, (0.0, 0.0, 0.0))  # its node values and its weights: 256 KiB each


@pytest.mark.parametrize("launch_graph", [False, True])
def test_first_node_gradients_inside_a_capture(launch_graph):
    torch = torch_cuda()
    pf = load_pf()
    scene = synth.room_scene(0)
    field = synth.analytic_tsdf(scene, GRID)
    P = synth.room_view(scene, 0)
    pts = to_dev(synth.render_points(scene, synth.ROOM64_INTR, P, 3))[None].contiguous()
    poses = to_dev(P @ synth.perturbation(3, 0, 1.0, 2.0))[None].contiguous()

    def call(vol, out):
        pf.pf_align_loss(vol.handle, pts, None, pts.shape[1], 1, poses, None, None, *out)

    def outputs():
        f64 = dict(dtype=torch.float64, device="cuda")
        return [torch.empty(1, **f64), torch.empty(1, dtype=torch.int32, device="cuda"), torch.empty(1, 6, **f64),
                torch.full((GRID.n_nodes,), 7.0, device="cuda")]

    vols = [pf.Volume.from_grid(GRID) for _ in range(2)]
    for v in vols:
        v.upload(*field)
    want, got, graphed = outputs(), outputs(), outputs()
    call(vols[0], want)
    assert int(want[1]) > 1000 and float(want[3].abs().max()) > 0
    junk = [pf.Volume.from_grid(JUNK, cell_view=-1) for _ in range(16)]
    for v in junk:
        v.upload(np.full(JUNK.n_nodes, 0.5, dtype=np.float32), np.ones(JUNK.n_nodes, dtype=np.float32))
    for v in junk:
        v.close()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="relaxed"):
        call(vols[1], graphed)
    call(vols[1], got)
    assert all(torch.equal(p, q) for p, q in zip(want, got))
    if launch_graph:
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(p, q) for p, q in zip(want, graphed))
    del graph
    got = outputs()
    call(vols[1], got)
    assert all(torch.equal(p, q) for p, q in zip(want, got))
    for v in vols:
        v.close()
