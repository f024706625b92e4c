"""Rounding of the 2D prefix products (csrc/fsmi_device.cuh cell_prefixes) on long spans of equal probability,
as free and unknown space are: a lane multiplies its cells' factors one after the other, so that their
roundings differ from cell to cell; grouped as ((1-o)(1-o))((1-o)(1-o)) every group rounds alike and the
product drifts (at 700 to 1400 cells a bias of up to 2.1e-6 against 1.1e-6).

With delta_emp = 1 (f_emp = 0) and a Gaussian narrower than a cell, Approx-FSMI with Delta = 0 is
f(delta_occ, o) sum_j P(e_j), so the ratio to the one-cell beam is sum_j P(e_j) / o: compared with a replay of the
products in FP32. Tolerance 5e-7: the sum's own rounding, at most 44 additions per lane and 5 over the lanes
at 2^-24 each, with random signs below 2e-7, and four more roundings."""
import numpy as np
import pytest
import torch

from paper_1905_02238_gb300 import fsmi

pytestmark = pytest.mark.gpu
F = np.float32
PROBS = (0.1, 0.05, 0.02, 0.03, 0.07, 0.15, 0.01, 0.005)


def _replay(o, n):
    """sum_j P(e_j) of n cells of probability o: lanes' blocks of 4 ceil(n / 128) cells, then a warp scan."""
    K, x = 4 * ((n + 127) // 128), F(1) - F(o)
    cells = np.clip(n - K * np.arange(32), 0, K)
    prod = np.ones(32, F)
    for l in range(32):
        for _ in range(cells[l]):
            prod[l] = F(prod[l] * x)
    k = 1
    while k < 32:
        prod[k:] = (prod[k:] * prod[:-k]).astype(F)
        k *= 2
    total = 0.0
    for l in range(32):
        E = prod[l - 1] if l else F(1)
        for _ in range(cells[l]):
            total += float(F(E * F(o)))
            E = F(E * x)
    return total


@pytest.mark.parametrize("n", [3, 64, 129, 360, 700, 1400])
def test_equal_cells(n):
    off = np.concatenate([[0], np.cumsum([n, 1] * len(PROBS))]).astype(np.int32)
    o = np.concatenate([np.full(n + 1, p, F) for p in PROBS])
    l = np.concatenate([np.concatenate([np.arange(n), [0]]) for _ in PROBS]).astype(F)
    lend = np.array([n, 1] * len(PROBS), F)
    prm = fsmi.Params(variant=fsmi.APPROX, trunc_delta=0, sigma=0.05, delta_occ=1.5, delta_emp=1.0, max_range=64.0)
    mi = fsmi.eval_beams(*(torch.from_numpy(a).cuda() for a in (off, o, l, lend)), prm).cpu().numpy().astype(np.float64)
    for i, p in enumerate(PROBS):
        got, want = mi[2 * i] / mi[2 * i + 1] * float(F(p)), _replay(p, n)
        assert abs(got / want - 1.0) < 5e-7, (n, p, got / want - 1.0)
    assert fsmi.device_status() == 0
