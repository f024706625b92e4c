"""Rounding of the 3D prefix products (csrc/evalrle.cuh scan_block) on long spans of equal probability: a lane
multiplies its four cells' factors one after the other; as ((1-o)(1-o))((1-o)(1-o)) the two halves round alike and
the product drifts (rms 1.04e-6 against 7.6e-7 at 700 cells, 6.9e-7 with the lanes' blocks of n / 32 cells).

With delta_emp = 1 (f_emp = 0) and Uniform-FSMI of H = 0 a ray's MI is f(delta_occ, o) sum_j P(e_j), so the ratio to
the one-cell ray is sum_j P(e_j) / o: compared with a replay of the products in FP32. Tolerance 5e-7: the
sum's own rounding, at most 32 additions per lane and 5 over the lanes at 2^-24 each, with random signs below 2e-7,
and four more roundings. Runs are split every 16 cells, so that the cell form is taken."""
import numpy as np
import pytest
import torch

from paper_1905_02238_gb300 import fsmi, synth

pytestmark = pytest.mark.gpu
F = np.float32
PROBS = (0.1, 0.05, 0.02, 0.03, 0.07, 0.15, 0.01, 0.005, 0.2, 0.12, 0.08, 0.06, 0.0137, 0.0411, 0.25, 0.0073)
X = 1024


def _replay(o, n):
    """sum_j P(e_j) of n cells of probability o: blocks of 128 cells, 4 per lane, a warp scan per block."""
    x, total, start = F(1) - F(o), 0.0, F(1)
    for base in range(0, n, 128):
        cells = np.clip(n - base - 4 * np.arange(32), 0, 4)
        prod = np.ones(32, F)
        for l in range(32):
            for _ in range(cells[l]):
                prod[l] = F(prod[l] * x)
        k = 1
        while k < 32:
            prod[k:] = (prod[k:] * prod[:-k]).astype(F)
            k *= 2
        for l in range(32):
            E = F(start * prod[l - 1]) if l else start
            for _ in range(cells[l]):
                total += float(F(E * F(o)))
                E = F(E * x)
        start = F(start * prod[31])
    return total


@pytest.mark.parametrize("n", [65, 127, 129, 384, 700, 1000])
def test_equal_cells(n):
    vox = np.ascontiguousarray(np.broadcast_to(np.array(PROBS, F)[None, :, None], (1, len(PROBS), X)))
    poses = np.stack([synth.pose_3d(X - m + 0.1, y + 0.5, 0.5, 0.0, 0.0) for y in range(len(PROBS)) for m in (n, 1)])
    dirs = synth.q30(np.array([[1.0, 0.0, 0.0]]))
    prm = fsmi.Params(variant=fsmi.UNIFORM, uniform_h=0, delta_occ=1.5, delta_emp=1.0, max_range=float(X), run_cap=16)
    v, p, d = (torch.from_numpy(a).cuda() for a in (vox, poses, dirs))
    out = fsmi.eval_3d(v, p, d, prm)
    off, ro, rl = fsmi.rle_encode_3d(v, p, d, prm, capacity=len(poses) * X)
    assert torch.equal(out.view(-1), fsmi.eval_rle(off, ro, rl, prm))
    mi = out.view(-1).cpu().numpy().astype(np.float64)
    for i, o in enumerate(PROBS):
        got, want = mi[2 * i] / mi[2 * i + 1] * float(F(o)), _replay(o, n)
        assert abs(got / want - 1.0) < 5e-7, (n, o, got / want - 1.0)
    assert fsmi.device_status() == 0
