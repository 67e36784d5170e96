"""The FP64 stencils' folded forms at the ends of their inputs: the gradient in
a cell's own basis read back in its frame, against the mixed mode's gradient;
diffusion with a zero and a negative Smagorinsky factor and from rest (square
roots of zero), with and without the enhanced temperature diffusion's factor,
against the oracle at the FP64 stage tolerance."""
import dataclasses

import numpy as np
import pytest

from oracle import Dycore as OracleDycore
from parity import gpu_params, rel_err, setup, to_numpy, to_torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fac", [0.0, -0.001])
@pytest.mark.parametrize("rest", [False, True], ids=["wind", "rest"])
def test_diffusion_factor_and_rest(built_lib, cuda, fac, rest):
    import paper_2608_21150_gb300 as P
    grid, z, op, _, st = setup(2, 30, 1800.0)
    op = dataclasses.replace(op, hdiff_smag_fac=fac)
    od = OracleDycore(grid, z, op)
    st = od.substep(st)
    if rest:
        st["vn"] = np.zeros_like(st["vn"])
    d = P.Dycore(P.Grid(grid, radius=op.radius), z, gpu_params(op))
    t = to_torch(st, cuda)
    d.nh_diff(t)
    err = rel_err(to_numpy(t), od.diffusion(dict(st)), od)
    assert max(err.values()) < 1e-12, err


def test_gradient_read_back_in_the_cell_frame(built_lib, cuda):
    import torch
    import paper_2608_21150_gb300 as P
    grid, z, op, od, st = setup(2, 29, 1800.0)
    g = P.Grid(grid, radius=op.radius)
    out = {}
    for prec, dt in ((P.ICON_PREC_FP64, torch.float64), (P.ICON_PREC_MIXED, torch.float32)):
        d = P.Dycore(g, z, gpu_params(op, precision=prec, autotune=0))
        t = to_torch(st, cuda)
        d.nh_solve(t)
        f = torch.empty((4, st["rho"].shape[0], 29), dtype=dt, device=cuda)
        d.debug_field("grad4", f)
        out[prec] = f.cpu().numpy().astype(np.float64)
    # FP32 differences of perturbations: a few 2^-24 of the perturbations over the cell distance
    for a, b in zip(out[P.ICON_PREC_FP64], out[P.ICON_PREC_MIXED]):
        assert np.max(np.abs(a - b)) < 1e-4 * np.max(np.abs(a))
