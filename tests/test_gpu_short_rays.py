"""3D rays of at most 64 samples, which go in blocks of 64 cells, two per lane (csrc/evalrle.cuh kShortRay), and the
lengths around that line: every evaluation path, in the fused call, the run-input call and the mixed call's
range classes, against the FP64 oracle; fused, run-input and mixed results bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_1905_02238_gb300 import fsmi, synth
from tests.parity import assert_mi_close

pytestmark = pytest.mark.gpu

CASES = [
    dict(variant=fsmi.EXACT, sigma=2.0),                                         # compiled-in radius 15
    dict(variant=fsmi.EXACT, sigma=1.0),                                         # any radius
    dict(variant=fsmi.APPROX, approx_reading=1, trunc_delta=6, sigma=2.0),       # 6
    dict(variant=fsmi.APPROX, approx_reading=0, trunc_delta=6, sigma=2.0),       # Theorem 5, radius 15
    dict(variant=fsmi.APPROX, approx_reading=0, trunc_delta=3, sigma=1.3),
    dict(variant=fsmi.UNIFORM, uniform_h=4),                                     # 4
    dict(variant=fsmi.UNIFORM, uniform_h=9),
]


@pytest.mark.parametrize("R", [1, 2, 3, 4, 31, 32, 33, 62, 63, 64, 65, 66])
@pytest.mark.parametrize("noise", [0.0, 0.3])
def test_ranges(R, noise):
    vox = synth.voxel_world(120, 9, 7, n_boxes=4, seed=31, noise_seed=32, noise_frac=noise)
    # along +x from x = 120 - n: n cells to the volume's end, cut at R; and slanted rays
    poses = np.stack([synth.pose_3d(120 - n + 0.1, 4.5, 3.5, 0.0, 0.0) for n in (1, 2, 3, 5, 30, 31, 33, 62, 63, 64, 65, 66, 90)])
    a = np.radians([0.0, 0.4, -0.7])
    dirs = synth.q30(np.stack([np.cos(a), np.sin(a), np.zeros(3)], axis=1))
    v, p, d = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (vox, poses, dirs))
    sets, n = fsmi.make_sets([(fsmi.SET_3D, 0, len(poses), 0, 3, float(R), 0)], "cuda")
    vols = fsmi.make_volumes([v], "cuda")
    for cap in (7, 64):
        for kw in CASES:
            prm = dict(delta_occ=1.5, delta_emp=0.67, max_range=float(R), run_cap=cap, **kw)
            got, nr = fsmi.eval_3d(v, p, d, fsmi.Params(**prm), with_runs=True)
            ref, nr_ref = oracle.eval_3d(vox, poses, dirs, oracle.Params(**prm))
            np.testing.assert_array_equal(nr.cpu().numpy(), nr_ref)
            assert_mi_close(got.cpu().numpy(), ref, f"R={R} cap={cap} {kw}")
            off, ro, rl = fsmi.rle_encode_3d(v, p, d, fsmi.Params(**prm), capacity=int(nr_ref.sum()))
            assert torch.equal(got.view(-1), fsmi.eval_rle(off, ro, rl, fsmi.Params(**prm)))
            # the class of the set's range under the call's bound and under a longer one
            for bound in (float(R), 100.0):
                mixed = fsmi.eval_mixed(sets, n, volumes=vols, poses3=p, dirs3=d, prm3=fsmi.Params(**{**prm, "max_range": bound}))
                assert torch.equal(mixed, got.view(-1)), (R, cap, kw, bound)
    assert fsmi.device_status() == 0
