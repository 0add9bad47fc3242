"""Rows beyond 48 KB and meshes of one warp per cell in the FP32 form, against the
FP64 oracle.

Face rows over 48 KB take groups of two faces in 128 threads where the mesh has
enough faces (608 on 152 SMs): here with walls and far-field faces beside them and
an odd number of interior faces, so that the last group repeats its face, in 2D and
3D and for both gases (the diatomic gas in 3D sums its 34 moments face by face).
3D cells take one warp from 2432 cells on.  Bound as the suite's other mixed steps,
1e-5.
"""
import numpy as np
import pytest

from gpu_common import need_gpu
from test_gpu_step_kernels import run, sphere, walled

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,cells,base,model", [
    (walled, (21, 18), (79, 79), "shakhov"),
    (walled, (21, 18), (65, 64), "rykov"),
    (sphere, (5, 7, 9), (24, 24, 22), "shakhov"),
    (sphere, (5, 7, 9), (19, 18, 18), "rykov"),
])
def test_groups_of_long_rows(make, cells, base, model):
    need_gpu()
    import torch
    w = make(cells, base, model=model)
    NA = (2 if w.D == 2 else 1) + (model == "rykov")
    inner = int((w.mesh.faceR >= 0).sum())
    assert inner % 2 == 1 and inner < w.mesh.Nf
    assert w.mesh.Nf >= 4 * torch.cuda.get_device_properties(0).multi_processor_count
    assert NA * 4 * int(np.prod(base)) > 49152
    run(w, steps=2)


@pytest.mark.parametrize("model", ["shakhov", "rykov"])
@pytest.mark.parametrize("base", [(9, 9, 7), (13, 13, 13)])
def test_one_warp_per_cell_3d(base, model):
    need_gpu()
    import torch
    w = sphere((10, 16, 16), base, model=model)
    assert w.mesh.Nc >= 16 * torch.cuda.get_device_properties(0).multi_processor_count
    run(w, steps=2)
