"""FP32 face groups whose two faces see different gases.

Two interior faces that follow each other in the face order share a group.  They
may belong to different cells (an unstructured numbering, the end of a row of a
structured one) or to one cell at a shock, so that their mean velocities lie far
apart; each face's interface state must come out as it would alone.  A cold
stream at 24 sqrt(R T) fills half of a periodic box, along its sides gas at rest;
cells and faces are numbered at random, so that most groups mix the two.  The
cells of the gas at rest that one step does not join to the stream (it reaches
two cells) are compared with the FP64 oracle; collisions dominate (Kn = 1e-3), so
that f and W follow the interface states.

Bounds: 1e-5 for f and its moments, as the suite's other mixed steps.  The carried
W is FP64 but for its face fluxes, sums of FP32 terms of size rho (R T)^(3/2) in a
gas at rest, of which a step takes dt sqrt(R T) / h on each of 2 D faces: with 16
roundings of 2^-24 in a flux, 2 D 16 2^-24 dt sqrt(R T) / h, about 1e-7.
"""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2212_05645_gb300 import workloads as wl

from gpu_common import field_err, need_gpu, pair, pair_rykov, rel_err

pytestmark = pytest.mark.gpu

SPEED = 24.0


def shuffled(cells, base, model, seed=11):
    w = wl.sweep_box(cells, Kn=1e-3, base=base, max_refine=0, precision="mixed")
    m, D = w.mesh, w.D
    rng = np.random.default_rng(seed)
    new = rng.permutation(m.Nc)                     # old cell -> new cell
    old = np.argsort(new)
    face = rng.permutation(m.Nf)
    mesh = wl.Mesh(D, new[m.faceL][face].astype(np.int32), new[m.faceR][face].astype(np.int32), m.An[face], m.rL[face],
                   m.rR[face], m.vol[old], m.xc[old], m.bc, name="shuffled").contiguous()
    W = wl.sweep_W(mesh)
    stream = mesh.xc[:, 0] < 0.5
    c = wl.sqrt_RT(1.0)
    W[stream, 2] += SPEED * c
    lo, hi = np.full(D, -5.0 * c), np.full(D, 5.0 * c)
    hi[1] += SPEED * c
    w = dataclasses.replace(w, mesh=mesh, W_init=W, vlo=tuple(lo), vhi=tuple(hi))
    w.model = model
    return w


@pytest.mark.parametrize("model", ["shakhov", "rykov"])
@pytest.mark.parametrize("cells,base", [
    ((36, 35), (10, 34)),            # one warp per group
    ((20, 18), (15, 51)),            # 64 threads
    ((21, 17), (41, 160)),           # 128 threads, rows over 48 KB
    ((16, 8, 7), (7, 17, 4)),        # 3D, one warp
    ((16, 5, 5), (8, 40, 9)),        # 3D, 64 threads
])
def test_stream_beside_gas_at_rest(cells, base, model):
    avs = need_gpu()
    w = shuffled(cells, base, model)
    r, g = (pair_rykov if model == "rykov" else pair)(w, avs, precision="mixed", amp=1e-3)
    dt = r.dt()
    r.step(dt)
    g.step(1, dt=dt)
    x, h = w.mesh.xc[:, 0], 1.0 / cells[0]
    rest = (x > 0.5 + 2.5 * h) & (x < 1.0 - 2.5 * h)
    assert rest.sum() >= 2 * w.mesh.Nc // cells[0]
    W, q = g.moments()
    e = field_err(W[rest], r.Wc[rest], w.D)
    if model == "rykov":
        Wo, qt, qr = O.moments_rykov(w.D, r.xi, r.w, r.f)
        qo = qt + qr
    else:
        Wo, qo = O.moments(w.D, r.xi, r.w, r.f)
    ef = field_err(g.f_moments()[rest], Wo[rest], w.D, q[rest], qo[rest])
    df = rel_err(g.get_f()[rest], r.f[rest])
    print(f"\n{cells} {base} {model} Nf={w.mesh.Nf} Nv={g.Nv}: W {e}, f moments {ef}, f {df:.2e}")
    g.close()
    tol = 2 * w.D * 16 * 2.0 ** -24 * dt * wl.sqrt_RT(1.0) * max(cells)
    assert max(e.values()) < tol, (e, tol)
    assert max(ef.values()) < 1e-5, ef
    assert df < 1e-5, df
