"""Fitness of points at the grid's faces: from four cells inside to two outside
each of the six, in order of that distance, so that warps lie on either side of
the bound within which a chunk's samples skip the range test, and some straddle
it.  Every node is observed and in the band, so a point counts exactly when its
cell is in the grid.  Against the oracle, and to the bit between the kernel's
forms: with few and with many thread blocks (and so registers) an SM."""
import numpy as np
import pytest

import oracle
import synth
from synth import Grid

from gpu_helpers import abi, compare_fitness, load_pf, perturbed_poses, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

GRID = Grid(48, 40, 33, 0.05, 0.15, (-0.3, 0.2, 0.1))
N_POINTS = 8 * 1024 - 5  # eight tiles, the last ragged


def field():
    k, j, i = np.meshgrid(*(np.arange(n, dtype=np.float64) for n in (GRID.nz, GRID.ny, GRID.nx)), indexing="ij")
    t = 0.45 * np.sin(0.7 * i + 0.3 * j) + 0.45 * np.cos(0.5 * k - 0.4 * j)
    return t.astype(np.float32).reshape(-1), np.ones(t.size, dtype=np.float32)


def face_points(P):
    """Camera-frame points (N, 4) near the faces, deepest inside first."""
    u = synth.uniform01(21, 4 * N_POINTS).reshape(N_POINTS, 4)
    n = np.array([GRID.nx, GRID.ny, GRID.nz], dtype=np.float64)
    g = (0.12 + 0.76 * u[:, :3]) * (n - 1)  # away from the other faces
    depth = np.sort(6.0 * u[:, 3] - 2.0)[::-1]
    face = np.arange(N_POINTS) // 4 % 6  # groups of four: every warp has all six
    axis, high = face % 3, face >= 3
    rows = np.arange(N_POINTS)
    g[rows, axis] = np.where(high, n[axis] - 1 - depth, depth)
    w = g * GRID.voxel_size + np.asarray(GRID.origin)
    x = (w - P[:3, 3]) @ P[:3, :3]
    return np.concatenate([x, np.zeros((N_POINTS, 1))], 1).astype(np.float32)


@pytest.mark.parametrize("dtype,search", [("PF_F32", "PF_F32"), ("PF_F32", "PF_F16"), ("PF_FP8E4M3", "PF_F32")])
@pytest.mark.parametrize("spread", [0.05, 4.0])  # degrees and centimetres: particles on lanes, points on lanes
def test_samples_at_the_faces(dtype, search, spread):
    torch = torch_cuda()
    pf = load_pf()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    t, w = field()
    vol = pf.Volume.from_grid(GRID, tsdf_dtype=getattr(pf, dtype), search_dtype=getattr(pf, search))
    vol.upload(t, w)
    P = synth.look_at((0.8, 1.1, 0.9), (1.2, 0.7, 1.0))
    pts = face_points(P)
    edge = 32 * (sms // 8)  # the last pose count that takes the form with more registers
    poses = perturbed_poses(P, 2 * edge, spread, spread, seed=4)
    dp = to_dev(pts)
    for variant in (2, 3, 6, 7, 10, 11):
        vol.set_fitness_variant(variant)
        ref = None
        for k in (32, edge, edge + 1, 2 * edge):
            E, C = vol.fitness(dp, to_dev(poses[:k]))
            got = E[:32].cpu().numpy(), C[:32].cpu().numpy()
            ref = ref or got
            assert np.array_equal(ref[0], got[0]) and np.array_equal(ref[1], got[1]), (variant, k)
        # about a third of the points lies outside
        assert np.all(ref[1] > N_POINTS // 2) and np.all(ref[1] < N_POINTS * 3 // 4 + 200)
        if dtype == "PF_F32" and (search == "PF_F32" or variant & 3 == 2):
            orc = oracle.fitness(oracle.Volume(abi(GRID), t, w), pts, poses[:32], ambiguity=True, cap=64)
            assert np.all(orc.amb <= 64)
            compare_fitness(*ref, orc)
    vol.close()
