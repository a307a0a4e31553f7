"""The ray cast's jumps over bricks without surface, against a plain march in
float64 that evaluates every sample (torch, on the same uploaded values).

The volumes are free space with isolated solid nodes at the edges of bricks
(8 nodes) and of the surface map's words (32 nodes) and at the grid's own
edges, a wall, and unobserved nodes; ragged sizes; rays along the axes (an
infinite slope on two axes), oblique ones, and a camera outside the grid.
Fusion's own marking is covered by casting after fusing onto the upload.

A float march and a float64 one may take another side only where a value or a
cell face lies within rounding of a sample: positions are off by at most
~1e-4 voxel of samples 1.5 voxels apart, eight faces or zero crossings each,
so under 1 pixel in 1000 may differ; depths of the others within 1e-4 m."""
import numpy as np
import pytest

import synth
from synth import Grid, Intrinsics

from gpu_helpers import abi, load_pf, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def plain_march(torch, t, w, grid, intr, P):
    """Depth image of the march over every sample, float64."""
    dev = "cuda"
    v = torch.as_tensor(np.where(w > 0, t, np.nan), dtype=torch.float64, device=dev)
    vv, uu = torch.meshgrid(torch.arange(intr.height, dtype=torch.float64, device=dev),
                            torch.arange(intr.width, dtype=torch.float64, device=dev), indexing="ij")
    R, o = (torch.as_tensor(q, dtype=torch.float64, device=dev) for q in (P[:3, :3], P[:3, 3]))
    d = torch.stack([(uu - intr.cx) / intr.fx, (vv - intr.cy) / intr.fy, torch.ones_like(uu)], -1) @ R.T
    org = torch.as_tensor(grid.origin, dtype=torch.float64, device=dev)
    top = torch.tensor([grid.nx - 1, grid.ny - 1, grid.nz - 1], dtype=torch.float64, device=dev)
    step = float(np.float32(0.5) * np.float32(grid.trunc))
    hit, prev = torch.zeros_like(uu), torch.full_like(uu, np.nan)
    nx, nxy = grid.nx, grid.nx * grid.ny
    for i in range(int((intr.depth_max - intr.depth_min) / step) + 1):
        z = intr.depth_min + i * step
        g = (o + z * d - org) / grid.voxel_size
        c = g.floor()
        ok = ((g >= 0) & (g < top)).all(-1)
        f = g - c
        c = torch.where(ok[..., None], c, torch.zeros_like(c)).long()
        b = c[..., 0] + nx * c[..., 1] + nxy * c[..., 2]
        x = [v[b + s] + f[..., 0] * (v[b + s + 1] - v[b + s]) for s in (0, nx, nxy, nxy + nx)]
        y = [x[0] + f[..., 1] * (x[1] - x[0]), x[2] + f[..., 1] * (x[3] - x[2])]
        s = torch.where(ok, y[0] + f[..., 2] * (y[1] - y[0]), torch.full_like(prev, np.nan))
        new = (hit == 0) & (prev > 0) & (s <= 0)
        hit = torch.where(new, z - step + step * prev / (prev - s), hit)
        prev = s
    return hit.cpu().numpy()


def blob_grid(nx, ny, nz, seed):
    """Free space, solid nodes at brick and word edges, a wall, unobserved nodes."""
    t = np.ones((nz, ny, nx), dtype=np.float32)
    w = np.ones_like(t)
    u = synth.uniform01(seed, 3 * 40).reshape(40, 3)
    at = [0, 1, 7, 8, 9, 15, 16, 31, 32, 33, 63, 64]
    for a, b, c in u:
        i, j, k = (min(n - 1, at[int(q * len(at))]) for q, n in ((a, nx), (b, ny), (c, nz)))
        t[k, j, i] = -1.0 if a < 0.5 else -0.25
    t[:, ny - 3:, :] = -0.5                         # a wall
    t[:, ny - 5:ny - 3, :] = 0.25
    hole = synth.uniform01(seed + 1, t.size).reshape(t.shape) < 0.002
    w[hole] = 0.0
    t[hole] = 1.0
    return t.reshape(-1), w.reshape(-1)


VIEWS = {
    "along_y": lambda s: np.array([[1.0, 0, 0, 0.5 * s[0]], [0, 0, 1, 0.02 * s[1]], [0, -1, 0, 0.5 * s[2]], [0, 0, 0, 1]]),
    "along_minus_x": lambda s: np.array([[0.0, 0, -1, 0.97 * s[0]], [1, 0, 0, 0.4 * s[1]], [0, -1, 0, 0.6 * s[2]], [0, 0, 0, 1]]),
    "oblique": lambda s: synth.look_at((0.1 * s[0], 0.15 * s[1], 0.2 * s[2]), (0.9 * s[0], 0.8 * s[1], 0.7 * s[2])),
    "from_outside": lambda s: synth.look_at((-0.3 * s[0], -0.2 * s[1], 1.2 * s[2]), (0.5 * s[0], 0.5 * s[1], 0.5 * s[2])),
}


@pytest.mark.parametrize("dims", [(64, 64, 64), (33, 40, 65), (9, 70, 31), (97, 66, 8)])
@pytest.mark.parametrize("view", sorted(VIEWS))
def test_jumps_agree_with_the_plain_march(dims, view):
    torch = torch_cuda()
    pf = load_pf()
    grid = Grid(*dims, 0.05, 0.15, (0.1, -0.2, 0.3))
    intr = Intrinsics(96, 72, 70.0, 70.0, 47.5, 35.5)
    t, w = blob_grid(*dims, seed=sum(dims))
    P = VIEWS[view]([0.05 * (n - 1) for n in dims])
    P[:3, 3] += grid.origin
    vol = pf.Volume.from_grid(grid)
    vol.upload(t, w)
    g, c = abi(grid), abi(intr)
    for fused in (False, True):
        if fused:  # a bowl in front of the camera: solid nodes that fusion writes
            u, v = np.meshgrid(np.arange(96.0), np.arange(72.0))
            depth = (0.8 + 0.004 * np.hypot(u - 40.0, v - 30.0)).astype(np.float32)
            vol.integrate(to_dev(depth), intr, P)
            t, w = vol.download()
        d = vol.raycast(intr, P, normals=False)[0].cpu().numpy().astype(np.float64)
        ref = plain_march(torch, t, w, g, c, P)
        differ = ((d > 0) != (ref > 0)) | (np.abs(d - ref) > 1e-4)
        assert np.count_nonzero(differ) <= 1e-3 * d.size, (fused, np.count_nonzero(differ))
    vol.close()
