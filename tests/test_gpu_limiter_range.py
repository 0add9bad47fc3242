"""The FP32 limiter over the range of f.

The limiter's ratio is the same for f and any multiple of f.  A caller whose
units make f small or large, and the tails of any f, must get the limited
gradient and not the plain one, also where the squares of f are subnormal in
FP32.  One step without collisions (a collision time of about 1e15, so that the
equilibria weigh nothing) on an f that varies by 30 % from cell to cell and node to node
shows every node's foot values; errors relative to each node's largest value.

Bounds.  The suite's 1e-5 for a mixed step while the squares are normal.  Below,
each of the about six roundings in numerator and denominator is off by up to
2^-150, so the limiter by at most 6 2^-149 / den with den >= (lim_K dx)^3 phi^2,
and den >= 2 d2^2 for the projection d2 it multiplies: the foot value is off by
at most 6 2^-149 / (sqrt(2 (lim_K dx)^3) phi), of which a step takes less than
its Courant number, 0.2 times the case's.
"""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2212_05645_gb300 import workloads as wl

from gpu_common import need_gpu, pair, pair_rykov

pytestmark = pytest.mark.gpu

SIZES = [((5, 4), (15, 13)), ((4, 3, 3), (9, 9, 7))]


def case(cells, base, model, s):
    w = dataclasses.replace(wl.sweep_box(cells, base=base, max_refine=0, precision="mixed"), Kn=1e15 * s)
    w.model = model
    return w


def start(r, s):
    """f and its W in the oracle run r; returns f."""
    u = np.random.default_rng(2).uniform(-0.3, 0.3, r.f.shape)
    f = (s * (1.0 + u)).astype(np.float32).astype(np.float64)
    r.f, r.Wc = f.copy(), r._moments(f)
    return f


@pytest.mark.parametrize("model", ["shakhov", "rykov"])
@pytest.mark.parametrize("cells,base", SIZES)
@pytest.mark.parametrize("s", [1e12, 1.0, 1e-12, 1e-18, 5e-20])
def test_limited_foot_values(cells, base, s, model):
    avs = need_gpu()
    w = case(cells, base, model, s)
    r, g = (pair_rykov if model == "rykov" else pair)(w, avs, precision="mixed", amp=0.0)
    f = start(r, s)
    g.set_f(f)
    g.set_W(r.Wc)
    dt = 0.2 * r.dt()
    r.step(dt)
    g.step(1, dt=dt)
    e = (np.abs(g.get_f() - r.f) / f.max(axis=0, keepdims=True)).max()
    g.close()
    eps2 = (0.3 * w.mesh.vol.min() ** (1.0 / w.D)) ** 3
    sub = 6 * 2.0 ** -149 / (np.sqrt(2 * eps2) * f.min()) / f.min() * 0.2 if f.min() ** 2 < 2.0 ** -126 / eps2 else 0.0
    print(f"\n{cells} {model} s={s:g}: {e:.2e}, bound {1e-5 + sub:.2e}")
    assert e < 1e-5 + sub


@pytest.mark.parametrize("cells,base", SIZES)
def test_the_limiter_acts_here(cells, base):
    """The same step without the limiter differs by far more than the bounds."""
    out = []
    for limiter in (1, 2):
        r = O.Run(case(cells, base, "shakhov", 1.0), limiter=limiter)
        r.init_field()
        f = start(r, 1.0)
        r.step(0.2 * r.dt())
        out.append(r.f)
    assert (np.abs(out[0] - out[1]) / f.max(axis=0, keepdims=True)).max() > 5e-3
