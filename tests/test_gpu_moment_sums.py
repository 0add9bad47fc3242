"""Sums over the velocity nodes of long rows in the FP32 cell kernels.

Carried raw moments, summed while f is written, feed the lagged heat flux of the
next step, a small difference of large sums.  Their FP32 chains must not grow with
the row (a cell of many cells is one warp), and the kernel that forms the moments
again after f was changed must give the same bits in every form the launch rules
choose: one warp or 128 threads per cell, rows of several runs, either gas, and in
the FP64 form with tables of the axes and without.
"""
import numpy as np
import pytest

import oracle as O
from paper_2212_05645_gb300 import workloads as wl

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def box(cells, base, model="shakhov", precision="mixed", Kn=0.05):
    w = wl.sweep_box(cells, Kn=Kn, base=base, max_refine=0, precision=precision)
    w.model = model
    return w


def uneven(xi, w):
    """One distribution: the first and last 128 nodes large and symmetric, the
    others far below the rounding of a lane's sum of |c_x| c^2 f once it holds the
    first ones, and at negative c_x only, so that they are the heat flux."""
    m = np.abs(xi[:, 0]) * (xi * xi).sum(1) * w
    f = np.zeros(len(w))
    f[:128] = f[-128:] = 1.0005
    f[128:-128] = np.where(xi[128:-128, 0] < 0, 0.8 * 2.0 ** -23, 0.0)
    return (f / m).astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("model", ["shakhov", "rykov"])
def test_lagged_heat_flux_of_a_long_row(model):
    """A uniform gas with collisions that outweigh everything else takes the
    equilibrium of W and its lagged heat flux in one step.  With W at rest the part
    of the new f that is odd in c is proportional to that heat flux: compared with
    the oracle's by projection.  2548 cells x 64000 nodes, the oracle on 27 cells of
    the same gas.

    Bound: a run is 16 terms, one sum of lanes and five over the warp, the state ten
    more roundings: 32 2^-24 of half the sum of |c_x| c^2 f, relative to
    rho (R T)^(3/2)."""
    avs = need_gpu()
    import torch
    base = (40, 40, 40)
    r = O.Run(box((3, 3, 3), base, model, Kn=1e-9))
    f1 = uneven(r.xi, r.w)
    m = np.abs(r.xi[:, 0]) * (r.xi * r.xi).sum(1)
    rho, RT = (r.w * f1).sum(), float((r.w * f1 * (r.xi * r.xi).sum(1)).sum() / (r.w * f1).sum() / 3.0)
    rows = np.stack([f1, 0.8 * RT * f1]) if model == "rykov" else f1[None]
    r.f = np.ascontiguousarray(np.broadcast_to(rows, (27,) + rows.shape))
    r.Wc = r._moments(r.f)
    r.Wc[:, 1:4] = 0.0
    W = np.ascontiguousarray(np.broadcast_to(r.Wc[0], (2548, r.Wc.shape[1])))
    g = avs.AVS(box((14, 14, 13), base, model, Kn=1e-9), precision="mixed")
    assert g.Nc == 2548 >= 16 * torch.cuda.get_device_properties(0).multi_processor_count
    g.set_f(torch.from_numpy(rows).cuda().expand(g.Nc, -1, -1).contiguous())
    g.set_W(W)
    q0 = np.abs(sum(O.moments_rykov(3, r.xi, r.w, r.f)[1:]) if model == "rykov" else O.moments(3, r.xi, r.w, r.f)[1]).max()
    dt = r.dt()
    g.step(1, dt=dt)
    r.step(dt)
    f = g.get_f_cells(np.array([0, 1274, 2547], dtype=np.int32))
    g.close()
    odd = r.f[0] - r.f[0][:, ::-1]                      # the nodes are symmetric in their order
    got = np.einsum("iak,ak->i", np.asarray(f) - np.asarray(f)[:, :, ::-1], odd) / (odd * odd).sum()
    e = np.abs(got - 1.0).max() * q0 / (rho * RT ** 1.5)
    bound = 32 * 2.0 ** -24 * 0.5 * float((r.w * f1 * m).sum()) / (rho * RT ** 1.5)
    print(f"\n{model}: heat flux {q0 / (rho * RT ** 1.5):.2e} of rho (RT)^1.5, taken {got}, error {e:.2e}, bound {bound:.2e}")
    assert e < bound


@pytest.mark.parametrize("cells,base,model,precision", [
    ((50, 49), (47, 47), "shakhov", "mixed"),            # one warp per cell, three runs
    ((50, 49), (47, 47), "rykov", "mixed"),
    ((14, 14, 13), (13, 13, 13), "shakhov", "mixed"),
    ((14, 14, 13), (13, 13, 13), "rykov", "mixed"),
    ((6, 5), (80, 64), "shakhov", "mixed"),              # 128 threads, two runs
    ((6, 5), (80, 64), "rykov", "mixed"),
    ((6, 5), (32, 31), "shakhov", "fp64"),               # tables of the axes
    ((6, 5), (4, 3), "shakhov", "fp64"),                 # rows too short for them
])
def test_carried_moments_equal_recomputed(cells, base, model, precision):
    """Three steps with the carried moments against three that drop them after
    every step, bit for bit."""
    avs = need_gpu()
    out = []
    for drop in (False, True):
        g = avs.AVS(box(cells, base, model, precision), precision=precision)
        g.init_field(amp=1e-3, seed=5)
        dt = g.dt()
        for _ in range(3):
            g.step(1, dt=dt)
            if drop:
                g.set_W(g.moments()[0])
        out.append((g.get_f(), g.moments()[0]))
        g.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1], out[1][1])
