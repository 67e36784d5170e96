"""A step's kernels are placed while their predecessors drain and wait for them
on the device; a profiled step waits between launches instead.  Both give the
same bits, over several steps without a synchronisation between them, as one
graph and as separate launches on the caller's stream, from grids whose kernels
fit the GPU several times over to grids of several waves; a training step's
kernels likewise."""
import numpy as np
import pytest

from icon_inputs import make_grid, make_vct, jw_type_state, mountain_height, terrain_following_z
from oracle import DycoreParams
from oracle import Dycore as OracleDycore
from oracle.terrain import TerrainDycore
from parity import gpu_params, to_numpy, to_torch
from test_gpu_mlp import init_params

pytestmark = pytest.mark.gpu

STEPS = 3


@pytest.mark.parametrize("prec", ["FP64", "MIXED", "MIXED_F64COL"])
@pytest.mark.parametrize("bis,nlev,terrain", [(0, 2, False), (1, 7, True), (2, 30, False), (4, 65, False),
                                              (4, 31, True)])
def test_a_chained_step_is_the_step_with_waits(built_lib, cuda, bis, nlev, terrain, prec):
    import paper_2608_21150_gb300 as P
    grid, z = make_grid(bis), make_vct(nlev)
    if terrain:
        z = terrain_following_z(z, mountain_height(grid.cell_xyz))
    op = DycoreParams(dtime=450.0, ndyn_substeps=5, rayleigh_coeff=0.05)
    st = jw_type_state(grid, z, seed=8)
    st["exner_pr"] = (TerrainDycore if terrain else OracleDycore)(grid, z, op).initial_exner_pr(st["exner"])
    g = P.Grid(grid, radius=op.radius)
    out = {}
    for name, more in (("waits", {}), ("graph", {}), ("launches", dict(use_graph=0)),
                       ("one launch of A1-A4", dict(use_graph=0, fused_advection=1))):
        if "A1" in name and (terrain or prec == "FP64"):
            continue
        d = P.Dycore(g, z, gpu_params(op, precision=getattr(P, "ICON_PREC_" + prec), autotune=0, synchronous=0,
                                      **more))
        t = to_torch(st, cuda)
        if name == "waits":
            d.profile(t, STEPS)
        else:
            for _ in range(STEPS):
                d.step(t)
        d.synchronize()
        out[name] = to_numpy(t)
        d.close()
    for name in out:
        for k, v in out["waits"].items():
            assert np.array_equal(out[name][k].view(np.uint64), v.view(np.uint64)), (name, k)


@pytest.mark.parametrize("dims", [(33, 31, 70, 192), (450, 512, 269, 1024)])
def test_a_chained_training_step_is_the_one_with_waits(built_lib, cuda, dims):
    import torch
    import paper_2608_21150_gb300 as P
    I, H, O, B = dims
    rng = np.random.default_rng(B)
    p = init_params(rng, I, H, O)
    x = torch.from_numpy(rng.standard_normal((STEPS, B, I)).astype(np.float32)).to(cuda)
    t = torch.from_numpy(rng.standard_normal((STEPS, B, O)).astype(np.float32)).to(cuda)

    def train():
        net = P.MLP(I, H, O, max_batch=B)
        net.set_params(p)
        loss = [net.train_step(x[i], t[i], 1e-3) for i in range(STEPS)]
        return loss, net.params(), net.grads()

    chained = train()
    with P.Profile():
        waits = train()
    assert chained[0] == waits[0]
    assert np.array_equal(chained[1], waits[1]) and np.array_equal(chained[2], waits[2])
