"""The alignment loss and the polish read the cell view's float records where
a volume has them and the node array where it has not; both must give the same
bits, on every storage type.  The node-gradient accumulator returns to zero
after each call, for node counts off the vector width and for an output that
is not 16-byte aligned."""
import pytest

import synth
from synth import Grid

from gpu_helpers import load_pf, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

GRID = Grid(61, 47, 53, 0.06, 0.18, (0.0, 0.1, 0.0))  # 151 951 nodes: one off a multiple of four


def volume(pf, dtype, cell_view, **kw):
    vol = pf.Volume.from_grid(GRID, tsdf_dtype=getattr(pf, dtype), cell_view=cell_view, **kw)
    vol.upload(*synth.analytic_tsdf(synth.room_scene(0), GRID, hole_bricks=0.02))
    return vol


def frames(torch, n):
    scene = synth.room_scene(0)
    pts = [to_dev(synth.render_points(scene, synth.ROOM64_INTR, synth.room_view(scene, f), 3)) for f in range(n)]
    counts = torch.tensor([len(p) - 7 * f for f, p in enumerate(pts)], dtype=torch.int32, device="cuda")
    pad = torch.full((n, max(len(p) for p in pts), 4), 1.0e9, device="cuda")
    for f, p in enumerate(pts):
        pad[f, :len(p)] = p
    poses = torch.stack([to_dev(synth.room_view(scene, f) @ synth.perturbation(3, f, 1.0, 2.0)) for f in range(n)])
    xi = to_dev(0.02 * (synth.uniform01(8, 6 * n).reshape(n, 6) - 0.5))
    return pad, counts, poses, xi


@pytest.mark.parametrize("dtype", ["PF_F32", "PF_F16", "PF_BF16", "PF_FP8E4M3"])
def test_records_and_nodes_give_the_same_bits(dtype):
    torch = torch_cuda()
    pf = load_pf()
    pts, counts, poses, xi = frames(torch, 3)
    dloss = torch.tensor([1.0, -0.5, 3.0], dtype=torch.float64, device="cuda")
    out = []
    views = [dict(cell_view=-1), dict(cell_view=1), dict(cell_view=2)]
    if dtype == "PF_F32":
        views.append(dict(cell_view=1, search_dtype=pf.PF_F16))  # a rounded view must not be read
    for kw in views:
        vol = volume(pf, dtype, **kw)
        a = vol.align_loss(pts, poses, counts=counts, xi=xi, dloss=dloss, grad_xi=True, grad_tsdf=True)
        buf = torch.full((GRID.n_nodes + 1,), 7.0, device="cuda")
        b = [torch.empty_like(q) for q in a[:3]]
        pf.pf_align_loss(vol.handle, pts, counts, pts.shape[1], 3, poses, xi, dloss, b[0], b[1], b[2], buf[1:])
        assert torch.equal(a[3], buf[1:]) and float(buf[0]) == 7.0  # a second call, unaligned output
        assert all(torch.equal(p, q) for p, q in zip(a[:3], b))
        pose = poses[1].clone().contiguous()
        trace, acc = vol.polish(pts[1], pose, steps=6, n_dev=counts[1:2])
        out.append([*a, pose, trace, acc])
        vol.close()
    assert int(out[0][1].sum()) > 1000 and float(out[0][3].abs().max()) > 0 and int(out[0][6]) >= 2
    for other in out[1:]:
        assert all(torch.equal(p, q) for p, q in zip(out[0], other))


def test_polish_without_a_solvable_system_keeps_the_pose():
    """No point in the grid: no objective, no candidate, every step a no-op."""
    torch = torch_cuda()
    pf = load_pf()
    vol = volume(pf, "PF_F32", 1)
    pts = torch.full((50, 4), 100.0, device="cuda")
    start = to_dev(synth.room_view(synth.room_scene(0), 0))
    pose = start.clone()
    trace, acc = vol.polish(pts, pose, steps=3)
    assert torch.equal(pose, start) and int(acc) == 0 and bool(torch.isinf(trace).all())
    again = start.clone()  # the state starts afresh on the next call
    trace, acc = vol.polish(to_dev(synth.render_points(synth.room_scene(0), synth.ROOM64_INTR, start.cpu().numpy())), again, steps=2)
    assert bool(torch.isfinite(trace).all())
    vol.close()
