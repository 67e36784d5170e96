"""Reading back the FP64 gradient (icon_dycore_debug_field "grad4") works on the
dycore's own stream and keeps no host copy of the field: it returns while
another stream still runs, and the process grows by much less than the field."""
import os
import subprocess
import sys

import pytest

from c_harness import ROOT
from parity import gpu_params, setup, to_torch

pytestmark = pytest.mark.gpu


def test_waits_for_no_other_stream(built_lib, cuda):
    import torch
    import paper_2608_21150_gb300 as P
    grid, z, op, od, st = setup(1, 7, 1800.0)
    own = torch.cuda.Stream()
    d = P.Dycore(P.Grid(grid, radius=op.radius), z, gpu_params(op, autotune=0, stream=own.cuda_stream))
    t = to_torch(st, cuda)
    f = torch.empty((4, grid.n_cells, 7), dtype=torch.float64, device=cuda)
    torch.cuda.synchronize()
    d.nh_solve(t)
    d.debug_field("grad4", f)  # first use of what the read-back needs
    busy = torch.cuda.Event()
    torch.cuda._sleep(1_000_000_000)  # about half a second on the default stream
    busy.record()
    d.debug_field("grad4", f)
    assert not busy.query()
    torch.cuda.synchronize()


CHILD = r"""
import resource
import numpy as np
import torch
import paper_2608_21150_gb300 as P
from icon_inputs import make_grid, make_vct
grid, z = make_grid(4), make_vct(200)
d = P.Dycore(P.Grid(grid), z, dict(dtime=60.0, ndyn_substeps=5, autotune=0))
f = torch.empty((4, grid.n_cells, 200), dtype=torch.float64, device="cuda")
small = torch.empty((grid.n_cells, 200), dtype=torch.float64, device="cuda")
d.debug_field("divd", small)
before = resource.getrusage(resource.RUSAGE_SELF).ru_maxrss
d.debug_field("grad4", f)
print(resource.getrusage(resource.RUSAGE_SELF).ru_maxrss - before, f.numel() * 8 // 1024)
"""


def test_keeps_no_host_copy(built_lib, cuda):
    p = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT),
                       capture_output=True, text=True)
    assert p.returncode == 0, p.stderr
    grown, field = (int(x) for x in p.stdout.split()[-2:])  # KiB
    assert grown < field // 8, (grown, field)
