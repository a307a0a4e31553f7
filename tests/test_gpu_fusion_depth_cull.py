"""Grids of more than 100 000 fusion tiles (32 x 8 x 8 nodes) drop tiles that lie
behind every depth of the pixels they cover, smaller ones do not look: plates
two nodes thick on either side of that count, where each node counts as much as
in a full grid, against the oracle.

A near obstacle hides half of the far plate, with holes in the image; images
below and above the cull's 64 x 64 blocks; at the origin and kilometres from it,
where a tile's place in the camera frame is a difference of large numbers."""
import numpy as np
import pytest

import oracle
import synth
from synth import Grid, Intrinsics

from gpu_helpers import abi, load_pf, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

CAMS = [Intrinsics(48, 37, 24.0, 24.0, 23.3, 18.1), Intrinsics(173, 97, 84.0, 82.0, 86.0, 48.0)]


@pytest.mark.parametrize("ny", [2512, 2544])  # 314 and 318 x 315 tiles
@pytest.mark.parametrize("intr", CAMS, ids=lambda c: f"{c.width}x{c.height}")
@pytest.mark.parametrize("far", [0.0, 1.0])
def test_fusion_on_either_side_of_the_tile_count(ny, intr, far):
    torch_cuda()
    pf = load_pf()
    nz, vs = 2520, 1.0 / 512.0
    shift = far * np.array([1024.0, -2048.0, 512.0])
    grid = Grid(2, ny, nz, vs, 0.03, tuple(shift + (-0.5 * vs, -0.5 * ny * vs, 0.3)))
    vol = pf.Volume.from_grid(grid, max_weight=3, cell_view=-1)
    ovol = oracle.Volume(abi(grid), max_weight=3)
    clear = np.ones(grid.n_nodes, dtype=bool)
    for s in range(2):
        d = np.full((intr.height, intr.width), 4.5, dtype=np.float32)
        d[intr.height * s // 4:intr.height * (2 + s) // 4] = 1.1 + 0.4 * s
        d[synth.uniform01(50 + s, d.size).reshape(d.shape) < 0.1] = 0.0
        P = synth.perturbation(90, s, 2.0 * s, 0.05 * s)
        P[:3, 3] += shift
        vol.integrate(to_dev(d), intr, P)
        clear &= ~oracle.integrate(ovol, d, abi(intr), P, ambiguity=True).astype(bool)
    t, w = vol.download()
    assert np.array_equal(w[clear], ovol.weight[clear].astype(np.float32))
    seen = clear & (w > 0)
    assert np.count_nonzero(seen) > 500000 and np.count_nonzero(clear & (w == 0)) > 500000
    # float offsets from a double-precision tile base: 1e-7 m of a truncation of 0.03 m
    assert np.max(np.abs(t[seen] - ovol.tsdf[seen])) <= 1e-5
    vol.close()
