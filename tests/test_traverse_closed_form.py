"""The closed form of the 2D traversal (csrc/dda2d.cuh, Fixed): i_k = floor(V_0 + k am / aM) in fixed
point with 32 fractional bits. Restated here in integers and compared with the oracle's exact traversal:
whenever no V_k lies within the slack of an integer the cells are the same, whatever the error of the
slope estimate (the kernel's is 1.5 units at most); a diagonal step is always caught; and few beams
other than lattice directions are."""
import os
import re

import numpy as np
import pytest

import oracle
from paper_1905_02238_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SLACK = int(re.search(r"kSlack = (\d+)", open(os.path.join(ROOT, "paper_1905_02238_gb300", "csrc", "dda2d.cuh")).read())[1])


def closed_form(W, H, ox, oy, dx, dy, R, err):
    """Cell ids of the beam, or None where the kernel walks it. err: error of the slope, in its last bit."""
    rfix = int(round(R * 65536))
    cx, cy = ox >> 16, oy >> 16
    cx -= dx < 0 and ox & 0xFFFF == 0
    cy -= dy < 0 and oy & 0xFFFF == 0
    if (dx | dy) == 0 or not (0 <= cx < W and 0 <= cy < H):
        return []
    xmaj = abs(dx) >= abs(dy)
    (aM, am), (dM, dm) = ((abs(dx), abs(dy)), (dx, dy)) if xmaj else ((abs(dy), abs(dx)), (dy, dx))
    if am == aM:
        return None
    sM, sm = (1 if dM > 0 else -1), (1 if dm > 0 else -1)
    (cM, cm), (dimM, dimm), (oM, om) = (((cx, cy), (W, H), (ox, oy)) if xmaj else ((cy, cx), (H, W), (oy, ox)))
    nM0 = ((cM + 1) << 16) - oM if sM > 0 else oM - (cM << 16)
    nm0 = 0 if am == 0 else ((cm + 1) << 16) - om if sm > 0 else om - (cm << 16)
    LM, Lm = ((rfix * aM - 1) >> 30) + 1, ((rfix * am - 1) >> 30) + 1 if am else 0
    K = min(-(-(LM - nM0) // 65536) if LM > nM0 else 0, dimM - 1 - cM if sM > 0 else cM)
    if am == 0:
        slope, V0, I = 0, 1 << 31, 1 << 20
    else:
        slope = (am << 32) // aM + err
        V0 = (1 << 32) + (nM0 * slope >> 16) - (nm0 << 16)
        I = min(-(-(Lm - nm0) // 65536) if Lm > nm0 else 0, dimm - 1 - cm if sm > 0 else cm)
    assert 0 <= V0 and 1.5 * (K + 2) + 2 < SLACK
    cells = []
    for k1 in range(K + 1):
        V = V0 + k1 * slope
        if (V & 0xFFFFFFFF) + SLACK & 0xFFFFFFFF < 2 * SLACK:
            return None
        i, inn = (0 if k1 == 0 else V - slope >> 32), V >> 32
        if i > I:
            break
        assert len(cells) == k1 + i  # the list index in closed form
        a, b = cM + sM * k1, cm + sm * i
        cells.append(b * W + a if xmaj else a * W + b)
        if inn > i and i < I:
            b += sm
            cells.append(b * W + a if xmaj else a * W + b)
    return cells


@pytest.mark.parametrize("err", [-2, 0, 1])
def test_random_beams(err):
    rng = np.random.default_rng(3)
    walked = 0
    for t in range(1500):
        W, H = (int(v) for v in rng.integers(1, 400, 2))
        R = float(np.exp(rng.uniform(np.log(0.3), np.log(1024.0))))
        pose = synth.pose_2d(rng.uniform(0, W), rng.uniform(0, H), rng.uniform(0, 2 * np.pi))
        if t % 5 == 0:
            pose[:2] &= ~0xFFFF  # on grid lines
        u = synth.q30([np.cos(t * 0.1), np.sin(t * 0.1)])
        d = oracle.beam_dir_2d(pose, u)
        got = closed_form(W, H, int(pose[0]), int(pose[1]), int(d[0]), int(d[1]), R, err)
        ref, _ = oracle.trace_2d(W, H, int(pose[0]), int(pose[1]), int(d[0]), int(d[1]), R, 4096)
        if got is None:
            walked += 1
        else:
            np.testing.assert_array_equal(got, ref)
    assert walked < 1500 * 0.01


def test_axes_and_lattice_directions():
    q = 1 << 30
    dirs = [(q, 0), (-q, 0), (0, q), (0, -q), (q, 1), (q, -1), (1, q), (-1, -q)]
    for a, b in ((1, 1), (-1, 1), (2, 1), (1, -2), (3, 2), (-4, 1), (7, 5)):
        c = int(round(q / np.hypot(a, b)))
        dirs += [(a * c, b * c), (a * c + 1, b * c), (a * c, b * c - 1)]
    for W, H in ((64, 48), (1, 1), (33, 65), (32, 31)):
        for ox, oy in ((W * 32768, H * 32768), (W // 2 << 16, H // 2 << 16), (65535, 1), (32768, H * 65536 - 32768)):
            for dx, dy in dirs:
                for R in (0.5, 1.0, 31.0, 32.0, 33.5, 64.0, 300.0):
                    got = closed_form(W, H, ox, oy, dx, dy, R, 0)
                    if got is not None:
                        ref, _ = oracle.trace_2d(W, H, ox, oy, dx, dy, R, 4096)
                        np.testing.assert_array_equal(got, ref)
