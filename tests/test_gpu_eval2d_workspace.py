"""The workspace fsmi_eval_2d takes by default follows the library's rules: none where every beam has a warp and
no gains are computed, the queue counter where the thread's schedule leaves beams to balance, the gains where
the batch visits more cells than the map holds."""
import ctypes

import numpy as np
import pytest
import torch

from paper_1905_02238_gb300 import fsmi, synth

pytestmark = pytest.mark.gpu


def _scene(P):
    grid = np.full((2048, 2048), 0.3, np.float32)
    poses = np.stack([synth.pose_2d(900.0 + 3 * k, 1000.0, 0.1 * k) for k in range(P)])
    return tuple(torch.from_numpy(a).cuda() for a in (grid, poses, synth.beam_dirs_2d(360)))


@pytest.mark.parametrize("sched,P,R,want", [
    (None, 2, 64.0, 0),                                                        # a warp for every beam
    (fsmi.Schedule(warps_per_block=1, blocks_per_sm=1, queue_chunk=1), 2, 64.0, 256),   # 152 warps for 720 beams
    (fsmi.Schedule(warps_per_block=1, blocks_per_sm=1, queue_chunk=-1), 2, 64.0, 0),    # the caller asks for none
    (None, 40, 64.0, 256),                                                     # 14,400 beams, few cells
    (None, 80, 1024.0, 256 + 16 * 2048 * 2048),                                # more visits than cells
])
def test_default_workspace(monkeypatch, sched, P, R, want):
    g, p, d = _scene(P)
    prm = fsmi.Params(sigma=1.5, delta_occ=1.5, delta_emp=0.67, max_range=R)
    taken = []
    default_ws = fsmi._default_ws
    monkeypatch.setattr(fsmi, "_default_ws", lambda n, dev: taken.append(n) or default_ws(n, dev))
    fsmi.set_schedule(fsmi.KIND_2D, sched)
    try:
        got = fsmi.eval_2d(g, p, d, prm)
    finally:
        fsmi.set_schedule(fsmi.KIND_2D, None)
    assert taken == ([want] if want else [])
    assert torch.equal(got, fsmi.eval_2d(g, p, d, prm, ws=torch.empty(0, dtype=torch.uint8, device="cuda")))


def test_refused_arguments():
    lib, nb = fsmi.load(), ctypes.c_size_t(7)
    cp = fsmi.Params(max_range=64.0).c()
    assert lib.fsmi_eval_2d_workspace_size(0, 16, 1, 1, ctypes.byref(cp), ctypes.byref(nb)) == 1
    assert lib.fsmi_eval_2d_workspace_size(16, 16, 1, 1, None, ctypes.byref(nb)) == 1
    assert lib.fsmi_eval_2d_workspace_size(16, 16, 1, 1, ctypes.byref(cp), None) == 1
    assert lib.fsmi_eval_2d_workspace_size(16, 16, 0, 9, ctypes.byref(cp), ctypes.byref(nb)) == 0 and nb.value == 0
    g, p, d = _scene(1)
    with pytest.raises(fsmi.FsmiError, match="fsmi_eval_2d: "):
        fsmi.eval_2d(g, p, d, fsmi.Params(max_range=1025.0))
