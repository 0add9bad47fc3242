"""The first step of a small context allocates no device memory.

Mapping memory takes as long as a whole step of the smallest cases, so the step's
face buffer is there when the context is.  Many contexts are kept alive, so that
the driver's blocks fill up and the next ones map memory; none of them may do so
in its first step.
"""
import pytest

from paper_2212_05645_gb300 import workloads as wl

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,precision", [("shakhov", "mixed"), ("rykov", "mixed"), ("shakhov", "fp64")])
@pytest.mark.parametrize("implicit", [False, True])
def test_first_step_maps_no_memory(model, precision, implicit):
    avs = need_gpu()
    import torch
    w = wl.triangle_box(120, precision=precision)
    w.model = model
    keep = []
    for n in range(25):
        g = avs.AVS(w)
        g.init_field()
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        if implicit:
            g.step_implicit(1)
        else:
            g.step(1)
        torch.cuda.synchronize()
        taken = before - torch.cuda.mem_get_info()[0]
        keep.append(g)
        # the first context also loads the kernels
        assert n == 0 or taken == 0, f"context {n}: {taken} bytes"
    for g in keep:
        g.close()
