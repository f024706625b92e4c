"""Exact 2D FSMI along direction vectors shorter than a unit (the traversal takes any; a cell is then up to
sqrt 2 / |d| wide in units of the beam's distance): the mass form covers widths up to its table's limit, wider
beams take the boundary form, in every kernel that sums grid cells. Against the FP64 oracle, with the full
window bit-identical to the full sweep."""
import numpy as np
import pytest
import torch

import oracle
from paper_1905_02238_gb300 import fsmi, synth
from tests.parity import assert_mi_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 0.999, 0.93, 0.6, 0.3, 0.1])
@pytest.mark.parametrize("sigma", [1.0, 1.5, 2.0, 5.0])
def test_short_directions(scale, sigma):
    rng = np.random.default_rng(17)
    grid = rng.uniform(0.02, 0.98, size=(90, 120)).astype(np.float32)
    poses = np.stack([synth.pose_2d(*rng.uniform(25, 60, 2), rng.uniform(0, 6.28)) for _ in range(4)])
    dirs = np.rint(synth.beam_dirs_2d(31) * scale).astype(np.int32)
    g, p, d = (torch.from_numpy(a).cuda() for a in (grid, poses, dirs))
    off = torch.tensor([0, 4], dtype=torch.int32, device="cuda")
    sets, n = fsmi.make_sets([(fsmi.SET_2D, 0, 4, 0, 31, 50.0)], "cuda")
    for e0 in (0, 1):
        kw = dict(sigma=sigma, delta_occ=1.5, delta_emp=0.67, max_range=50.0, e0_mode=e0)
        ref = oracle.eval_2d(grid, poses, dirs, oracle.Params(**kw))
        prm = fsmi.Params(**kw)
        got = fsmi.eval_2d(g, p, d, prm)
        assert_mi_close(got.cpu().numpy(), ref, f"eval_2d e0={e0}")
        mixed = fsmi.eval_mixed(sets, n, grid=g, poses2=p, dirs2=d, prm2=prm)
        assert torch.equal(mixed.view(4, 31), got)
        beam = fsmi.eval_trajectories_2d(g, p[:1], off[:1].new_tensor([0, 1]), d, prm)[0]
        assert_mi_close(beam.cpu().numpy().reshape(-1), ref[0], f"trajectory e0={e0}")
        full = [fsmi.eval_2d(g, p, d, fsmi.Params(flags=f, **kw)) for f in (fsmi.FLAG_FULL_WINDOW, fsmi.FLAG_FULL_SWEEP)]
        assert torch.equal(full[0], full[1])
    assert fsmi.device_status() == 0
