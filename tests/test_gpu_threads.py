"""Contexts in several threads, each on its own stream.

A context belongs to one thread at a time; contexts of different threads share
nothing that a launch depends on.  The shared memory that a step's kernels take
differs with the mesh (faces per cell) and, in the FP64 form, with the velocity
space (entries of the axes' tables), while the limit that the runtime checks a
launch against is one per kernel: it has to be the same whoever sets it.
"""
import threading

import numpy as np
import pytest

from paper_2212_05645_gb300 import workloads as wl

from gpu_common import need_gpu

pytestmark = pytest.mark.gpu


def tables(base):
    return wl.sweep_box((3, 2), base=base, max_refine=0, precision="fp64")


PAIRS = {
    # three and four faces per cell: 66 and 78 KB for a cell
    "faces": lambda: (wl.triangle_box(300, base=(20, 20), max_refine=0, precision="mixed"),
                      wl.sweep_box((10, 10), base=(20, 20), max_refine=0, precision="mixed")),
    # 1286 and 2916 table entries: 41 and 93 KB
    "tables": lambda: (tables((1270, 16)), tables((2900, 16))),
}


@pytest.mark.parametrize("pair", sorted(PAIRS))
def test_two_threads_step_their_contexts(pair):
    avs = need_gpu()
    import torch
    ws = PAIRS[pair]()
    out, errors = [None, None], []
    both = threading.Barrier(2, timeout=60)

    def work(j, alone):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                g = avs.AVS(ws[j])
                g.init_field(amp=1e-3, seed=5)
                dt = g.dt()
                if not alone:
                    both.wait()
                for _ in range(25):
                    g.step(50, dt=dt)
                W = g.moments()[0]
                g.close()
            if alone:
                out[j] = W
            else:
                assert np.array_equal(W, out[j])
        except Exception as e:                      # reported by the test's own thread
            errors.append((j, repr(e)))

    for alone in (True, False):
        threads = [threading.Thread(target=work, args=(j, alone)) for j in (0, 1)]
        for t in threads:
            t.start()
            if alone:
                t.join()
        for t in threads:
            t.join()
        assert not errors, errors
