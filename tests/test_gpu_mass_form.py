"""The exact 2D sum in mass form (csrc/cell_mass.cuh, eval2d.cuh) against the FP64 oracle at the edges
of its rounds (beams of 1 .. 66 cells and the lengths around), at both degrees and on either side of
their limits in sigma, with and without the no-return event; and its table against the Gaussian mass
in FP64."""
import math
import os
import re

import numpy as np
import pytest
import torch

import oracle
from paper_1905_02238_gb300 import fsmi, synth
from tests.parity import assert_mi_close

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("D,sigma,bound", [(3, 1.5, 6e-8), (3, 2.0, 6e-9), (4, 1.0, 3e-8)])
def test_table(D, sigma, bound):
    # widest cell of a grid; the bound is fit_cell_mass.py's printed error rounded up, relative to the
    # mass at the centre
    src = open(os.path.join(ROOT, "paper_1905_02238_gb300", "csrc", "cell_mass.cuh")).read()
    body = re.search(r"T%d\[%d\]\[kMassOrder \+ 1\] = \{(.*?)\}\};" % (D, D + 1), src, re.S)[1]
    T = np.array([float(v) for v in re.findall(r"[-0-9.]+e[-+]\d+", body)]).reshape(D + 1, -1)
    z = np.linspace(0.0, 7.0, 1401)
    for t in np.linspace(0.05, 1.0, 12) * math.sqrt(0.5) / sigma:
        exact = np.array([0.5 * (math.erfc((a - t) / math.sqrt(2)) - math.erfc((a + t) / math.sqrt(2))) for a in z])
        s = z * z / (2 * math.log(2))
        q = sum((T[i] * t ** (2 * np.arange(T.shape[1]))).sum() * s ** i for i in range(D + 1))
        got = 2 * t * np.exp(-0.5 * z * z) / math.sqrt(2 * math.pi) * q
        assert np.abs(got - exact).max() <= bound * exact[0]


@pytest.mark.gpu
@pytest.mark.parametrize("sigma", [0.99, 1.0, 1.49, 1.5, 2.0, 12.0])
@pytest.mark.parametrize("e0", [0, 1])
def test_round_edges(sigma, e0):
    rng = np.random.default_rng(8)
    grid = rng.uniform(0.02, 0.98, size=(97, 141)).astype(np.float32)
    poses = np.stack([synth.pose_2d(*rng.uniform(30, 60, 2), rng.uniform(0, 6.28)) for _ in range(3)])
    dirs = synth.beam_dirs_2d(29)
    g, p, d = (torch.from_numpy(a).cuda() for a in (grid, poses, dirs))
    for R in (0.4, 1.0, 8.0, 24.0, 31.0, 32.5, 46.0, 52.0, 64.0, 90.0):
        kw = dict(sigma=sigma, delta_occ=1.5, delta_emp=0.67, max_range=R, e0_mode=e0)
        got = fsmi.eval_2d(g, p, d, fsmi.Params(**kw))
        assert_mi_close(got.cpu().numpy(), oracle.eval_2d(grid, poses, dirs, oracle.Params(**kw)), f"R={R}")
        full = [fsmi.eval_2d(g, p, d, fsmi.Params(flags=f, **kw)) for f in (fsmi.FLAG_FULL_WINDOW, fsmi.FLAG_FULL_SWEEP)]
        assert torch.equal(full[0], full[1])
    assert fsmi.device_status() == 0
