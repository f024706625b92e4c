"""The per-cell gain of the 3D kernels (csrc/fsmi_api.cu fit_gains): the 8-term polynomial may stand in for the
14-term one only where it is as accurate. A ray of one cell under Uniform-FSMI with H = 0 has the MI
o f(delta_occ, o); its error against 64 bits over 16,384 probabilities is compared with that of the 14-term
polynomial, replayed in FP32. Tolerance 1.2 in the root mean square: the two share two roundings outside the
polynomial, and at equal truncation their polynomials' rounding differs by up to 1.2 (1.5 and nearer to 1);
where truncation reaches FP32 rounding the 8-term form is 1.4 off or more."""
import numpy as np
import pytest
import torch

from paper_1905_02238_gb300 import fsmi, synth

pytestmark = pytest.mark.gpu
F = np.float32


def _gain(d, o):
    o = o.astype(np.longdouble)
    a, omo = (d - 1) * o, 1 - o
    return d * o / (1 + a) * np.log1p((d - 1) * omo / (1 + a)) - omo / (1 + a) * np.log1p(a)


def _long(d, o, terms=14):
    j = np.arange(terms)
    at = (np.cos(np.pi * (j + 0.5) / terms) + 1) / 2
    h = (_gain(d, at) / (at * (1 - at))).astype(np.float64)
    c = [(h * np.cos(np.pi * k * (j + 0.5) / terms)).sum() * (2 if k else 1) / terms for k in range(terms)]
    p = np.polynomial.chebyshev.cheb2poly(c).astype(F)
    x = (2.0 * o.astype(np.float64) - 1.0).astype(F)
    h = np.full_like(x, p[-1])
    for k in range(terms - 2, -1, -1):
        h = (h.astype(np.float64) * x + float(p[k])).astype(F)  # one rounding, as fma (the product is exact)
    return (o * (F(1) - o)).astype(F) * h


@pytest.mark.parametrize("docc,demp", [(1.5, 0.67), (1.4, 0.7), (1.56, 0.67), (1.56, 1.5), (1.575, 0.66), (1.6, 0.62),
                                       (2.0, 0.5)])
def test_error_of_the_gain(docc, demp):
    o = np.linspace(0.01, 0.99, 16384).astype(F)
    vox = o.reshape(128, 128, 1)  # [Z][Y][X]
    poses = np.stack([synth.pose_3d(0.0, y + 0.5, z + 0.5, 0.0, 0.0) for z in range(128) for y in range(128)])
    dirs = synth.q30(np.array([[1.0, 0.0, 0.0]]))
    prm = fsmi.Params(variant=fsmi.UNIFORM, uniform_h=0, delta_occ=docc, delta_emp=demp, max_range=1.0)
    got = fsmi.eval_3d(*(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (vox, poses, dirs)), prm)
    d = np.longdouble(F(docc))
    want = o.astype(np.longdouble) * _gain(d, o)
    rms = lambda v: float(np.sqrt((((v.astype(np.longdouble) - want) / want) ** 2).mean()))  # noqa: E731
    assert rms(got.cpu().numpy().reshape(-1)) <= 1.2 * rms(o * _long(d, o))
    assert fsmi.device_status() == 0
