"""The mixed mode's FP32 stencils take four consecutive levels per thread on
rows padded to a multiple of four, and read the caller's FP64 rows in aligned
pairs where they can.  Level counts of every remainder by four against the
FP64 oracle (the mixed mode's 2e-5 after one step), over flat ground and over
the mountain; very few levels, and state arrays that start on an odd 8 bytes,
bit for bit against the one-launch velocity advection (which stages single
levels) and against aligned arrays."""
import numpy as np
import pytest

from icon_inputs import make_grid, make_vct, jw_type_state, mountain_height, terrain_following_z
from oracle import DycoreParams
from oracle import Dycore as OracleDycore
from oracle.terrain import TerrainDycore
from parity import gpu_params, rel_err, to_numpy, to_torch

pytestmark = pytest.mark.gpu


def _setup(bis, nlev, dt, terrain):
    grid, z = make_grid(bis), make_vct(nlev)
    if terrain:
        z = terrain_following_z(z, mountain_height(grid.cell_xyz))
    op = DycoreParams(dtime=dt, ndyn_substeps=5, rayleigh_coeff=0.05)
    od = (TerrainDycore if terrain else OracleDycore)(grid, z, op)
    st = jw_type_state(grid, z, seed=5)
    st["exner_pr"] = od.initial_exner_pr(st["exner"])
    return grid, z, op, od, st


@pytest.mark.parametrize("terrain", [False, True], ids=["flat", "terrain"])
@pytest.mark.parametrize("nlev", [29, 31, 32])
def test_every_remainder_matches_the_oracle(built_lib, cuda, nlev, terrain):
    import paper_2608_21150_gb300 as P
    grid, z, op, od, st = _setup(2, nlev, 1800.0, terrain)
    d = P.Dycore(P.Grid(grid, radius=op.radius), z, gpu_params(op, precision=P.ICON_PREC_MIXED, autotune=0))
    t = to_torch(st, cuda)
    d.step(t)
    d.synchronize()
    errs = rel_err(to_numpy(t), od.step(st), od)
    assert all(e < 2e-5 for e in errs.values()), errs


@pytest.mark.parametrize("terrain", [False, True], ids=["flat", "terrain"])
@pytest.mark.parametrize("nlev", [2, 3, 4, 5, 8, 10])
def test_few_levels_and_odd_addresses_bitwise(built_lib, cuda, nlev, terrain):
    import torch
    import paper_2608_21150_gb300 as P
    grid, z, op, od, st = _setup(1, nlev, 900.0, terrain)
    g = P.Grid(grid, radius=op.radius)
    out = {}
    for name, over, odd in (("aligned", {}, 0), ("odd", {}, 1), ("fused", dict(fused_advection=1), 0)):
        d = P.Dycore(g, z, gpu_params(op, precision=P.ICON_PREC_MIXED, autotune=0, **over))
        t = {}
        for k, v in st.items():
            buf = torch.empty(v.size + 1, dtype=torch.float64, device=cuda)
            t[k] = buf[odd:odd + v.size].view(*v.shape)
            t[k].copy_(torch.from_numpy(np.ascontiguousarray(v)))
            assert t[k].data_ptr() % 16 == 8 * odd
        for _ in range(2):
            d.step(t)
        d.synchronize()
        out[name] = to_numpy(t)
        d.close()
    for name in ("odd", "fused"):
        for k in out[name]:
            assert np.array_equal(out[name][k].view(np.uint64), out["aligned"][k].view(np.uint64)), (name, k)
