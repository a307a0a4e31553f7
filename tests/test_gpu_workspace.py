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
