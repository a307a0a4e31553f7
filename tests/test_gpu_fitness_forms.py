"""A fitness launch with no more thread blocks than SMs takes a form of the
kernel with more registers a thread: the same operations in the same order, so
a pose's fitness must not depend, to the bit, on how many other chunks of poses
share the launch (the points are tiled alike in all of these)."""
import numpy as np
import pytest

import synth

from gpu_helpers import load_pf, perturbed_poses, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,search", [("PF_F32", "PF_F32"), ("PF_F32", "PF_F16"), ("PF_BF16", "PF_F32"),
                                          ("PF_FP8E4M3", "PF_F32")])
@pytest.mark.parametrize("spread", [0.05, 4.0])  # particles on lanes, points on lanes
def test_fitness_is_the_same_in_either_form(dtype, search, spread):
    torch = torch_cuda()
    pf = load_pf()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    scene = synth.room_scene(0)
    vol = pf.Volume.from_grid(synth.ROOM64_GRID, tsdf_dtype=getattr(pf, dtype), search_dtype=getattr(pf, search))
    vol.upload(*synth.analytic_tsdf(scene, synth.ROOM64_GRID, hole_bricks=0.02))
    P = synth.room_view(scene, 1)
    pts = to_dev(synth.render_points(scene, synth.ROOM64_INTR, P)[:8 * 1024 - 5])  # eight tiles, the last ragged
    edge = 32 * (sms // 8)  # the last pose count that takes the form with more registers
    poses = to_dev(perturbed_poses(P, 2 * edge, spread, spread, seed=4))
    for layout in (2, 3):
        vol.set_fitness_variant(layout)
        ref = None
        for k in (32, edge, edge + 1, 2 * edge):
            E, C = vol.fitness(pts, poses[:k].contiguous())
            got = E[:32].cpu().numpy(), C[:32].cpu().numpy()
            assert np.count_nonzero(got[1]) > 16
            ref = ref or got
            assert np.array_equal(ref[0], got[0]) and np.array_equal(ref[1], got[1]), k
    vol.close()
