"""The ray cast's jumps in a grid a kilometre from the origin, where a sample's
place on the grid is a difference of large floats, against the plain march in
float64 of the same volumes as in test_gpu_raycast_march.

There a sample's place is off by up to ~1e-4 voxel and 1 pixel in 1000 may
differ, depths of the others by 1e-4 m.  Here it is off by half a unit of the
last place of 1024 m, 6.1e-5 m or 1.2e-3 voxel of 0.05 m on each axis: twelve
times that, so twelve times the share and the depth."""
import numpy as np
import pytest

from synth import Grid, Intrinsics

from gpu_helpers import abi, load_pf, torch_cuda
from test_gpu_raycast_march import VIEWS, blob_grid, plain_march

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(64, 64, 64), (33, 40, 65), (97, 66, 8)])
def test_jumps_agree_with_the_plain_march_far_from_the_origin(dims):
    torch = torch_cuda()
    pf = load_pf()
    grid = abi(Grid(*dims, 0.05, 0.15, (1024.0, -1500.0, 1100.0)))
    intr = abi(Intrinsics(96, 72, 70.0, 70.0, 47.5, 35.5))
    t, w = blob_grid(*dims, seed=sum(dims))
    vol = pf.Volume.from_grid(grid)
    vol.upload(t, w)
    hits = 0
    for view in sorted(VIEWS):
        P = VIEWS[view]([0.05 * (n - 1) for n in dims])
        P[:3, 3] = (P[:3, 3] + grid.origin).astype(np.float32)
        d = vol.raycast(intr, P, normals=False)[0].cpu().numpy().astype(np.float64)
        ref = plain_march(torch, t, w, grid, intr, P)
        hits += np.count_nonzero(ref > 0)
        differ = ((d > 0) != (ref > 0)) | (np.abs(d - ref) > 1.2e-3)
        assert np.count_nonzero(differ) <= 1.2e-2 * d.size, (view, np.count_nonzero(differ))
    assert hits > 500  # (few rays of some views meet a surface)
    vol.close()
