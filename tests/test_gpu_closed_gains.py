"""Deltas far from 1, whose per-cell gains have no polynomial (csrc/evalrle.cuh closed_gains): the closed forms are
evaluated once per span of equal values of a block of cells. Worlds of long spans, of short ones and of different
values in every cell; ray lengths around the blocks; every evaluation path in the fused, the run-input and
the mixed call, against the FP64 oracle and bit for bit against one another."""
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
    dict(variant=fsmi.APPROX, approx_reading=0, trunc_delta=6, sigma=2.0),
    dict(variant=fsmi.APPROX, approx_reading=1, trunc_delta=3, sigma=2.0),
    dict(variant=fsmi.UNIFORM, uniform_h=4),
]


@pytest.mark.parametrize("world", [0.0, 0.3, 1.0])
@pytest.mark.parametrize("R", [1, 3, 33, 64, 65, 127, 130, 200, 260])
def test_closed_form_gains(world, R):
    if world < 1.0:
        vox = synth.voxel_world(280, 9, 7, n_boxes=5, seed=41, noise_seed=42, noise_frac=world)
    else:
        vox = np.random.default_rng(43).uniform(0.02, 0.9, (7, 9, 280)).astype(np.float32)
    poses = np.stack([synth.pose_3d(280 - n + 0.1, 4.5, 3.5, 0.0, 0.0) for n in (1, 2, 5, 31, 64, 65, 127, 129, 256, 270)])
    a = np.radians([0.0, 0.4, -0.7])
    dirs = synth.q30(np.stack([np.cos(a), np.sin(a), np.zeros(3)], axis=1))
    v, p, d = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (vox, poses, dirs))
    sets, n = fsmi.make_sets([(fsmi.SET_3D, 0, len(poses), 0, 3, float(R), 0)], "cuda")
    vols = fsmi.make_volumes([v], "cuda")
    for deltas in ((40.0, 0.02), (1.5, 0.02)):
        for kw in CASES:
            prm = dict(delta_occ=deltas[0], delta_emp=deltas[1], max_range=float(R), run_cap=7, **kw)
            got, nr = fsmi.eval_3d(v, p, d, fsmi.Params(**prm), with_runs=True)
            ref, nr_ref = oracle.eval_3d(vox, poses, dirs, oracle.Params(**prm))
            np.testing.assert_array_equal(nr.cpu().numpy(), nr_ref)
            assert_mi_close(got.cpu().numpy(), ref, f"{deltas} {kw}")
            off, ro, rl = fsmi.rle_encode_3d(v, p, d, fsmi.Params(**prm), capacity=int(nr_ref.sum()))
            assert torch.equal(got.view(-1), fsmi.eval_rle(off, ro, rl, fsmi.Params(**prm)))
            for bound in (float(R), 300.0):
                mixed = fsmi.eval_mixed(sets, n, volumes=vols, poses3=p, dirs3=d, prm3=fsmi.Params(**{**prm, "max_range": bound}))
                assert torch.equal(mixed, got.view(-1)), (deltas, kw, bound)
    assert fsmi.device_status() == 0
