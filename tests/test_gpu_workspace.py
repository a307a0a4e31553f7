"""The search's workspace: reservations add up, whatever order they came in."""
import numpy as np
import pytest

import synth

from gpu_helpers import load_pf, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

INTR = synth.ROOM64_INTR
N_PIX = INTR.width * INTR.height


def room(pf):
    vol = pf.Volume.from_grid(synth.ROOM64_GRID)
    vol.upload(*synth.analytic_tsdf(synth.room_scene(0), synth.ROOM64_GRID))
    return vol


def frame(view=1):
    scene = synth.room_scene(0)
    P = synth.room_view(scene, view)
    depth = synth.render_depth(scene, INTR, P).astype(np.float32)
    return to_dev(depth), P @ synth.perturbation(5, view, 2.0, 3.0)


def params(pf, k, **kw):
    return pf.track_params(to_dev(synth.templates(k).astype(np.float32)), k_sched=(k,) * 3, decim_sched=(1,) * 3,
                           n_iters=4, **kw)


def test_a_frame_within_separate_reservations_is_taken():
    torch_cuda()
    pf = load_pf()
    depth, P0 = frame()
    prm = params(pf, 4096)
    whole, parts = room(pf), room(pf)
    want = whole.track_frame(depth, INTR, prm, P0)
    parts.reserve(64, 4096)     # particles
    parts.reserve(N_PIX, 32)    # pixels
    got = parts.track_frame(depth, INTR, prm, P0)
    assert want[0] == got[0] == pf.PF_OK and np.array_equal(want[1], got[1])
    whole.close()
    parts.close()


def outgrow(pf, torch, vol):
    """Calls that need more of every scratch buffer of the volume."""
    pts = torch.zeros((3000, 4), device="cuda")
    vol.fitness(pts, torch.zeros((30000, 12), device="cuda"))
    vol.reserve(4 * N_PIX, 20000)
    vol.align_loss(pts.expand(300, 3000, 4).contiguous(), torch.eye(4, dtype=torch.float64, device="cuda").expand(300, 4, 4).contiguous())
    # what was freed, if anything, is written over
    junk = [torch.full((n,), float("nan"), device="cuda") for n in (1 << 16, 1 << 18, 1 << 20, 1 << 22) for _ in range(4)]
    torch.cuda.synchronize()
    del junk


@pytest.mark.parametrize("use_graph", [True, False])
def test_a_batch_outlives_the_growth_of_its_members(use_graph):
    torch = torch_cuda()
    pf = load_pf()
    frames = [frame(v) for v in (1, 2)]
    prm = params(pf, 500)
    got = []
    for grow in (False, True):
        vols = [room(pf) for _ in frames]
        batch = pf.Batch(vols, [INTR] * 2, [prm] * 2, use_graph=use_graph)
        for i, (depth, P0) in enumerate(frames):
            batch.depth[i].copy_(depth)
            batch.pose[i].copy_(to_dev(P0))
            batch.rel[i].copy_(torch.eye(4, dtype=torch.float64))
        batch.step()
        if grow:
            outgrow(pf, torch, vols[1])
        batch.step()
        if grow:
            outgrow(pf, torch, vols[0])
            batch.set_points_per_block(4096)  # new tables, on the new buffers
        batch.step()
        torch.cuda.synchronize()
        got.append([batch.pose[0].cpu().numpy(), batch.pose[1].cpu().numpy(), batch.stats[0].cpu().numpy(),
                    batch.stats[1].cpu().numpy(), *vols[0].download(), *vols[1].download()])
        batch.close()
        for v in vols:
            v.close()
    assert all(np.array_equal(a, b) for a, b in zip(*got))


def test_captured_calls_outlive_the_growth_of_the_workspace():
    torch = torch_cuda()
    pf = load_pf()
    depth, P0 = frame()
    prm = params(pf, 500)
    vol = room(pf)
    pts = to_dev(synth.render_points(synth.room_scene(0), INTR, synth.room_view(synth.room_scene(0), 1), 3))[None].contiguous()
    init = to_dev(P0).reshape(16).contiguous()
    out = torch.empty(16, dtype=torch.float64, device="cuda")
    loss = [torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty(1, dtype=torch.int32, device="cuda"),
            torch.empty(1, 6, dtype=torch.float64, device="cuda"), torch.empty(synth.ROOM64_GRID.n_nodes, device="cuda")]

    def calls():
        vol.track_frame_async(depth, INTR, prm, init, out)
        pf.pf_align_loss(vol.handle, pts, None, pts.shape[1], 1, init.view(1, 4, 4), None, None, *loss)

    calls()
    torch.cuda.synchronize()
    want = [out.clone(), *(q.clone() for q in loss)]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    outgrow(pf, torch, vol)
    for q in (out, *loss):
        q.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, [out, *loss]))
    calls()  # on the new buffers
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(want, [out, *loss]))
    del graph
    vol.close()
