"""Fusion where its culls and short cuts can go wrong, against the oracle, and
the cell view's row-wise refresh against the node array.

A near obstacle covers half of the image (the tiles behind it are dropped by
the depth cull), the rest is far or missing; later views see the same free
space again (only weights change), a surface where free space was, and free
space where the surface was.  Ragged grids put the last tile, row and plane of
each axis in play; images smaller and larger than the cull's 64 x 64 blocks;
weights saturate.  After every fusion the fitness on the cell view must equal
the fitness on the node array bit for bit: every record whose corners changed
was rewritten."""
import numpy as np
import pytest

import oracle
import synth
from synth import Grid, Intrinsics

from gpu_helpers import abi, load_pf, perturbed_poses, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

GRIDS = [Grid(33, 17, 9, 0.06, 0.18, (-0.9, -0.5, 0.4)), Grid(64, 40, 41, 0.04, 0.12, (-1.2, -0.8, 0.3)),
         Grid(100, 71, 8, 0.03, 0.1, (-1.5, -1.0, 0.9))]
CAMS = [Intrinsics(48, 37, 40.0, 41.0, 23.3, 18.1), Intrinsics(173, 97, 120.0, 118.0, 86.0, 48.0)]


def views(intr, n):
    """n (depth, pose): an obstacle that moves across a far wall, with holes."""
    out = []
    for s in range(n):
        d = np.full((intr.height, intr.width), 2.1, dtype=np.float32)
        x = intr.width * (s % 3) // 4
        d[:, x:x + intr.width // 2] = 0.9 + 0.05 * s
        d[synth.uniform01(50 + s, d.size).reshape(d.shape) < 0.1] = 0.0
        d[: intr.height // 8] = 0.0
        out.append((synth.add_depth_noise(d, 70 + s, 0.004), synth.perturbation(90, s, 4.0 * (s > 0), 6.0 * (s > 0))))
    return out


@pytest.mark.parametrize("grid", GRIDS, ids=lambda g: f"{g.nx}x{g.ny}x{g.nz}")
@pytest.mark.parametrize("intr", CAMS, ids=lambda c: f"{c.width}x{c.height}")
@pytest.mark.parametrize("dtype,u8", [("PF_F32", 0), ("PF_F16", 1), ("PF_FP8E4M3", 1)])
def test_fusion_and_view_after_every_frame(grid, intr, dtype, u8):
    torch_cuda()
    pf = load_pf()
    vol = pf.Volume.from_grid(grid, max_weight=3, tsdf_dtype=getattr(pf, dtype), weight_u8=u8, cell_view=1)
    ovol = oracle.Volume(abi(grid), max_weight=3)
    clear = np.ones(grid.n_nodes, dtype=bool)
    pts = to_dev(np.concatenate([synth.uniform01(7, 3 * 3000).reshape(-1, 3) * [g * grid.voxel_size for g in
                 (grid.nx, grid.ny, grid.nz)] + grid.origin, np.zeros((3000, 1))], 1).astype(np.float32))
    poses = to_dev(perturbed_poses(np.eye(4), 64, 3.0, 5.0, seed=1))
    for depth, P in views(intr, 5):
        vol.integrate(to_dev(depth), intr, P)
        clear &= ~oracle.integrate(ovol, depth, abi(intr), P, ambiguity=True).astype(bool)
        t, w = vol.download()
        assert np.array_equal(w[clear], ovol.weight[clear].astype(np.float32))
        seen = clear & (w > 0)
        assert np.count_nonzero(seen) > 500
        if dtype == "PF_F32":
            assert np.max(np.abs(t[seen] - ovol.tsdf[seen])) <= 1e-5
        got = []
        for layout in (2, 3):
            vol.set_fitness_variant(layout + 4)
            E, C = vol.fitness(pts, poses)
            got.append((E.cpu().numpy(), C.cpu().numpy()))
        assert np.array_equal(got[0][1], got[1][1])
        # (e4m3 narrow records are scaled once more: equal within the float tolerance)
        if dtype == "PF_FP8E4M3":
            fin = np.isfinite(got[0][0])
            assert np.allclose(got[0][0][fin], got[1][0][fin], rtol=1e-5, atol=0)
        else:
            assert np.array_equal(got[0][0], got[1][0])
    vol.close()
