"""The 3D cell form in blocks of 128 virtual cells (csrc/evalrle.cuh): rays whose cell counts lie around the
lanes' groups of 4, the blocks and the passes of the banded convolution (1 .. 5, 31 .. 33, 127 .. 130, 255 .. 258,
383 .. 385), with the compiled-in radii and others, worlds of short and of long runs, several split lengths.
Against the FP64 oracle, and the fused call against the encoder and the run-input call bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_1905_02238_gb300 import fsmi, synth
from tests.parity import assert_mi_close

pytestmark = pytest.mark.gpu

CASES = [
    dict(variant=fsmi.EXACT, sigma=2.0),
    dict(variant=fsmi.EXACT, sigma=1.0),
    dict(variant=fsmi.APPROX, approx_reading=1, trunc_delta=6, sigma=2.0),
    dict(variant=fsmi.APPROX, approx_reading=0, trunc_delta=6, sigma=2.0),
    dict(variant=fsmi.APPROX, approx_reading=0, trunc_delta=3, sigma=1.3),
    dict(variant=fsmi.UNIFORM, uniform_h=4),
    dict(variant=fsmi.UNIFORM, uniform_h=0),
]


def _world(noise):
    vox = synth.voxel_world(400, 9, 7, n_boxes=6, seed=21, noise_seed=22, noise_frac=noise)
    # along +x from x = 400 - n: n cells to the volume's end; and a few slanted rays
    poses = np.stack([synth.pose_3d(400 - n + 0.1, 4.5, 3.5, 0.0, 0.0)
                      for n in (1, 2, 3, 4, 5, 31, 32, 33, 127, 128, 129, 130, 255, 256, 257, 258, 383, 384, 385)])
    a = np.radians([0.0, 0.4, -0.7])
    dirs = synth.q30(np.stack([np.cos(a), np.sin(a), np.zeros(3)], axis=1))
    return vox, poses, dirs


@pytest.mark.parametrize("noise", [0.0, 0.3])
@pytest.mark.parametrize("cap", [7, 64, 255])
@pytest.mark.parametrize("deltas", [(1.5, 0.67), (3.0, 0.4), (40.0, 0.02)])
def test_block_edges(noise, cap, deltas):
    vox, poses, dirs = _world(noise)
    v, p, d = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (vox, poses, dirs))
    for kw in CASES:
        prm = dict(delta_occ=deltas[0], delta_emp=deltas[1], max_range=384.0, run_cap=cap, **kw)
        got, nr = fsmi.eval_3d(v, p, d, fsmi.Params(**prm), with_runs=True)
        ref, nr_ref = oracle.eval_3d(vox, poses, dirs, oracle.Params(**prm))
        np.testing.assert_array_equal(nr.cpu().numpy(), nr_ref)
        assert_mi_close(got.cpu().numpy(), ref, f"{kw}")
        assert torch.equal(got, fsmi.eval_3d(v, p, d, fsmi.Params(**prm)))
        off, ro, rl = fsmi.rle_encode_3d(v, p, d, fsmi.Params(**prm), capacity=int(nr_ref.sum()))
        assert torch.equal(got.view(-1), fsmi.eval_rle(off, ro, rl, fsmi.Params(**prm)))
    assert fsmi.device_status() == 0
