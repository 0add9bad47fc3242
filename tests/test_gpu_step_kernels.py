"""The step's kernels at the sizes where their launch rules change, against the
FP64 oracle.

FP32 form, either gas: one warp or 128 threads per face group (rows of at most
512 nodes, or 1024 with many faces), one or two faces per group (a last group
that repeats its face where the number is odd), three or four ring slots (rows
beyond 48 KB, 3D), one warp or 128 threads per cell (256 nodes, 2432 cells),
64 or 128 threads and one or more quads per thread in the foot and sweep kernels,
rows that end within a quad.  FP64 form: tables of the axes from the size where
a row has twice their entries, and the kernels without them below.

Bounds, set before the first run: 1e-12 in the FP64 form, 1e-5 in the mixed form
(f after implicit steps 1e-4), as the suite's other comparisons of these forms.
"""
import dataclasses

import numpy as np
import pytest

import oracle as O
from paper_2212_05645_gb300 import workloads as wl

from gpu_common import field_err, need_gpu, pair, pair_rykov, rel_err

pytestmark = pytest.mark.gpu


def box(cells, base, precision="mixed", model="shakhov"):
    w = wl.sweep_box(cells, base=base, max_refine=0, precision=precision)
    w.model = model
    return w


def sphere(n, base, precision="mixed", model="shakhov"):
    w = wl.sphere(n_r=n[0], n_theta=n[1], n_phi=n[2], C1=1.0, max_refine=0, precision=precision, learned=False)
    w = dataclasses.replace(w, base=base)
    w.model = model
    return w


def walled(cells, base, precision="mixed", model="shakhov"):
    wall, hot, lid = (wl._bc_row(wl.BC_WALL, U=(u, 0.0, 0.0), T=T) for u, T in ((0.0, 1.0), (0.0, 1.3), (0.3, 1.0)))
    mesh = wl.cartesian_mesh(cells, (1.0, 1.0), bcs=[(wall, hot), (wall, lid)])
    w = box(cells, base, precision=precision, model=model)
    return dataclasses.replace(w, name="walled-" + w.name, mesh=mesh, W_init=wl.sweep_W(mesh))


def run(w, implicit=None, steps=2, tol=1e-5, ftol=1e-5):
    avs = need_gpu()
    ryk = w.model == "rykov"
    r, g = (pair_rykov if ryk else pair)(w, avs, precision=w.precision, amp=1e-2)
    assert g.Nv == int(np.prod(w.base))
    if implicit is None:
        dt = r.dt()
        for _ in range(steps):
            r.step(dt)
        g.step(steps, dt=dt)
    else:
        dt = r.dt(2.0)
        for _ in range(steps):
            r.step_implicit(dt, **implicit)
        g.step_implicit(steps, dt=dt, **implicit)
    W, q = g.moments()
    e = field_err(W, r.Wc, w.D)
    if ryk:
        Wo, qt, qr = O.moments_rykov(w.D, r.xi, r.w, r.f)
        qo = qt + qr
        e["Erot"] = float(np.abs(W[:, -1] / r.Wc[:, -1] - 1.0).max())
    else:
        Wo, qo = O.moments(w.D, r.xi, r.w, r.f)
    ef = field_err(g.f_moments(), Wo, w.D, q, qo)
    df = rel_err(g.get_f(), r.f)
    print(f"\n{w.name} {w.model} {w.precision} Nc={w.mesh.Nc} Nf={len(w.mesh.faceL)} Nv={g.Nv}: W {e}, f moments {ef}, f {df:.2e}")
    assert max(e.values()) < tol, e
    assert max(ef.values()) < tol, ef
    assert df < ftol, df
    g.close()


BOXES = {
    "tiny": ((3, 2), (2, 3)),
    "warp-odd": ((5, 4), (5, 7)),
    "64-threads-last": ((5, 4), (16, 16)),
    "past-256": ((5, 4), (43, 6)),
    "warp-last": ((5, 4), (32, 16)),
    "past-512-few-faces": ((5, 4), (27, 19)),
    "past-512-two-faces": ((20, 18), (27, 19)),
    "two-faces-warp": ((36, 35), (5, 7)),
    "past-512-many-faces": ((50, 49), (27, 19)),
    "two-quads": ((50, 49), (47, 47)),
    "long-rows": ((20, 18), (79, 79)),
}


@pytest.mark.parametrize("model", ["shakhov", "rykov"])
@pytest.mark.parametrize("case", sorted(BOXES))
def test_mixed_step_2d(case, model):
    cells, base = BOXES[case]
    run(box(cells, base, model=model), steps=1 if cells[0] == 50 else 2)


@pytest.mark.parametrize("model", ["shakhov", "rykov"])
@pytest.mark.parametrize("cells,base", [((2, 1), (4, 5)), ((5, 4), (5, 7)), ((5, 4), (16, 16)), ((20, 18), (27, 19))])
def test_mixed_step_walls(cells, base, model):
    """Boundary faces, several to a block where a group is one warp."""
    run(walled(cells, base, model=model))


@pytest.mark.parametrize("model", ["shakhov", "rykov"])
@pytest.mark.parametrize("n,base", [((3, 4, 4), (5, 6, 7)), ((3, 4, 4), (8, 8, 8)), ((3, 4, 4), (9, 9, 7)),
                                    ((6, 6, 8), (9, 9, 7))])
def test_mixed_step_3d(n, base, model):
    run(sphere(n, base, model=model))


@pytest.mark.parametrize("model", ["shakhov", "rykov"])
@pytest.mark.parametrize("kw", [dict(k_macro=3, k_micro=1), dict(k_macro=8, k_micro=3), dict(k_macro=2, k_micro=0)])
@pytest.mark.parametrize("cells,base", [((5, 4), (5, 7)), ((1, 1), (4, 5)), ((20, 18), (27, 19))])
def test_mixed_implicit_step(cells, base, kw, model):
    """Sweeps that clear nothing and add nothing at the end: one symmetric
    iteration, several, none; one cell between walls; rows of one warp and more."""
    run((walled if cells == (1, 1) else box)(cells, base, model=model), implicit=kw, ftol=1e-4)


@pytest.mark.parametrize("model", ["shakhov", "rykov"])
def test_mixed_implicit_step_3d(model):
    run(sphere((3, 4, 4), (9, 9, 7), model=model), implicit=dict(k_macro=8, k_micro=2), ftol=1e-4)


@pytest.mark.parametrize("base", [(4, 3), (4, 4), (5, 3), (32, 31)])
def test_fp64_axis_tables_rule(base):
    """A row of twice the tables' entries takes them, a shorter one does not."""
    run(box((5, 4), base, precision="fp64"), tol=1e-12, ftol=1e-12)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("base", [(5, 7), (27, 19)])
def test_f_widened_exactly(precision, base):
    """get_f returns the stored value itself: signed zeros, subnormals of the
    element type, its smallest and largest numbers."""
    avs = need_gpu()
    w = box((5, 4), base, precision=precision)
    g = avs.AVS(w, precision=precision)
    rng = np.random.default_rng(3)
    T = np.float32 if precision == "mixed" else np.float64
    t = np.finfo(T)
    f = rng.standard_normal(g.get_f().shape).astype(T)
    special = np.array([0.0, -0.0, t.smallest_subnormal, -t.smallest_subnormal, t.tiny, -t.tiny, t.tiny / 2, t.max, t.min,
                        7 * t.smallest_subnormal], dtype=T)
    f.reshape(-1)[:: 3][: 4 * len(special)] = np.tile(special, 4)
    f.reshape(-1)[-len(special):] = special
    f = f.astype(np.float64)
    g.set_f(f)
    out = g.get_f()
    assert np.array_equal(out.view(np.uint64), f.view(np.uint64))
    cells = np.array([7, 0, 19], dtype=np.int32)
    assert np.array_equal(np.asarray(g.get_f_cells(cells)).view(np.uint64), f[cells].view(np.uint64))
    g.close()
