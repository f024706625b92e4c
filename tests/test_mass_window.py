"""The window of the exact 2D sum in mass form (csrc/eval2d.cuh exact_mass_sum), replayed on the CPU: rounds of
64 source cells, two adjacent ones per lane, while more than 32 remain, then one per lane; coverage trials
from the previous round's counts; comparisons in FP32 as in the kernel, sums in FP64. The trials end
at the fewest pairs that cover the round, every target within the cuts of a source lies in the pairs the source
visits, every pair read stays in the array, and what is left out of the sum stays within the stated bounds:
for a first-hit cell the cells after it below 2^-31, those before it below 2^-27 of the largest C_k among them
(the Gaussian mass beyond the cut on that side), and the MI of a beam on the maps in use changed by less than
2^-25 of itself (half an FP32 rounding) for sigma from 1 to 20 cells."""
import math
import os
import re

import numpy as np
import pytest
from scipy.special import erfc

import oracle
from paper_1905_02238_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SQ = math.sqrt(math.log2(math.e))
F = np.float32


def _cuts():
    """The cuts for the targets below a source and above it."""
    src = open(os.path.join(ROOT, "paper_1905_02238_gb300", "csrc", "eval2d.cuh")).read()
    return [float(re.search(r"constexpr float %s = ([0-9.]+)f[;,]" % n, src).group(1)) for n in ("kMassCut", "kTailCutDefault")]


def _step():
    return F(F(_cuts()[0]) - F(_cuts()[1]))


def _trials(g, ok, n):
    steps = 0
    if ok(g):
        while g > 0 and ok(g - 1):
            g -= 1
    else:
        while not ok(g):
            g += 1
            steps += 1
            assert steps <= n + 2, "trials do not end"
    assert g == 0 or not ok(g - 1)  # the fewest pairs that cover the round
    return g


def visited(x, cut, e0, mu0):
    """First and last + 1 target of every source of a beam with scaled cell centres x (FP32)."""
    n, step = len(x), _step()
    at = lambda m: np.where(m < 0, mu0, x[np.clip(m, 0, n - 1)]).astype(F)  # noqa: E731
    mlo, plast = -1 if e0 else 0, (n - 1) >> 1
    span = x[n - 1] - x[0]
    per = F(n) / span if span > F(0) else F(0)
    GN = GP = int(min(cut * per, F(n + 1))) >> 1
    lo, hi = np.zeros(n, int), np.zeros(n, int)
    for kb in range(0, n, 64):
        two = n - kb > 32
        k = kb + (2 if two else 1) * np.arange(32)
        a = k[k < n]
        b = np.where(two & (a + 1 < n), a + 1, a)
        pa, below, above = a >> 1, (x[a] - cut).astype(F), (x[b] + F(cut - step)).astype(F)

        def neg_ok(G):
            m = 2 * (pa - G) - 1
            return bool(np.all((m < mlo) | (at(m) < below)))

        def pos_ok(G):
            m = 2 * (pa + G) + 2
            return bool(np.all((m >= n) | (at(m) >= above)))

        GN, GP = _trials(GN, neg_ok, n), _trials(GP, pos_ok, n)
        p, end = np.maximum(pa - GN, -1), np.minimum(pa + GP, plast)
        assert p.min() >= -1 and end.max() <= n >> 1  # the pairs that were built
        for s in (a, b):
            lo[s], hi[s] = 2 * p, np.minimum(2 * end + 2, n)
    return lo, hi


def _beams(world, count):
    if world == "office":
        grid, poses, dirs = synth.office_scene(n_poses=8, size=1024)
        R = 200.0
    else:
        grid, poses, dirs = synth.random_grid_200()
        R = 64.0
    H, W = grid.shape
    for b in range(count):
        p = poses[b % len(poses)]
        d = oracle.beam_dir_2d(p, dirs[(b * 7) % len(dirs)])
        cells, l = oracle.trace_2d(W, H, p[0], p[1], d[0], d[1], R)
        if len(cells) > 1:
            yield grid.reshape(-1)[cells].astype(np.float64), l.astype(np.float64)


def test_mass_beyond_the_cuts():
    cut, cut_before = _cuts()
    assert 0.5 * erfc(cut / SQ) < 2.0 ** -31
    assert 0.5 * erfc(cut_before / SQ) < 2.0 ** -27


@pytest.mark.parametrize("world", ["office", "random"])
@pytest.mark.parametrize("sigma", [1.0, 1.5, 2.0, 3.0, 5.0, 10.0, 20.0])
def test_left_out(world, sigma):
    cs = SQ / (sigma * math.sqrt(2.0))
    cut, cut_before = (F(F(0.70710678) * F(cs) + F(c)) for c in _cuts())
    worst = 0.0
    for i, (o, l) in enumerate(_beams(world, 40)):
        n = len(o)
        P = o * np.concatenate([[1.0], np.cumprod(1.0 - o)[:-1]])
        C = oracle.c_k(o, 1.5, 0.67)
        mu = 0.5 * (l[1:] + l[:-1])
        z = (l[None, :] - mu[:, None]) / (sigma * math.sqrt(2.0))
        up, dn = 0.5 * erfc(z), 0.5 * erfc(-z)
        G = np.where(z[:, 1:] <= 0, dn[:, 1:] - dn[:, :-1], up[:, :-1] - up[:, 1:])  # [first hit j][source k]
        ls = l.astype(F) * F(cs)
        x = (F(0.5) * (ls[:-1] + ls[1:])).astype(F)
        mu0 = F(ls[0] - F(0.5) * F(cs))
        lo, hi = visited(x, cut, i % 2, mu0)
        j, k = np.arange(n)[:, None], np.arange(n)[None, :]
        out = (j < lo[k]) | (j >= hi[k])
        assert not (out & (x[:, None] >= (x - cut)[None, :]) & (x[:, None] < (x + cut_before)[None, :])).any()
        for side, share in ((out & (k > j), 2.0 ** -31), (out & (k < j), 2.0 ** -27)):
            left, C_max = np.where(side, C[None, :] * G, 0.0).sum(1), np.where(side, C[None, :], 0.0).max(1)
            assert (left <= share * C_max).all()
        W = P[:, None] * C[None, :] * G
        worst = max(worst, W[out].sum() / W.sum())
    assert worst < 2.0 ** -25, worst


@pytest.mark.parametrize("e0", [0, 1])
def test_indices_on_any_lengths(e0):
    # 1 .. 70 cells and a long beam, cells of any width down to zero, windows from a cell to the whole beam
    rng = np.random.default_rng(5)
    for n in list(range(1, 71)) + [127, 128, 129, 400]:
        w = rng.uniform(0.0, 1.4142, n) * (rng.random(n) > 0.1)
        l = np.concatenate([[0.0], np.cumsum(w)]).astype(F)
        for sigma in (1.0, 3.0, 20.0):
            cs = F(SQ / (sigma * math.sqrt(2.0)))
            x = (F(0.5) * (l[:-1] * cs + l[1:] * cs)).astype(F)
            for cuts in ([F(F(0.70710678) * cs + F(c)) for c in _cuts()], [F(11.3)] * 2):
                lo, hi = visited(x, F(cuts[1] + _step()), e0, F(l[0] * cs - F(0.5) * cs))
                for s in range(n):
                    inside = np.nonzero((x >= x[s] - cuts[0]) & (x < x[s] + cuts[1]))[0]
                    if len(inside):
                        assert lo[s] <= inside[0] and inside[-1] < hi[s]
