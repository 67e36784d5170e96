"""The column solve runs small grids with 16 columns per CTA and larger ones
with 32, and in chunks of 4, 6 or 8 levels.  A column's result does not depend
on the form that solved it, nor on its neighbours: every form evaluates the
same operations in the same order, so the results agree bit for bit.  Sizes
around the groups of columns and the chunks of levels, both arithmetics."""
import numpy as np
import pytest

from icon_inputs import make_grid, make_vct, jw_type_state, mountain_height, terrain_following_z
from oracle import DycoreParams
from oracle import Dycore as OracleDycore
from oracle.terrain import TerrainDycore
from parity import gpu_params, to_torch, to_numpy

pytestmark = pytest.mark.gpu

WIDE = 19457  # columns from which the wide form is used (19 456), and one more: a ragged last group


def _columns(nlev, n, cuda):
    """n columns of the balanced jet with noise in every input."""
    import torch
    z = make_vct(nlev)
    st = jw_type_state(make_grid(1), z, seed=6)
    rng = np.random.default_rng(nlev)
    pick = rng.integers(0, st["rho"].shape[0], n)
    f = {k: st[k][pick] * (1.0 + 1e-5 * rng.standard_normal((n, nlev))) for k in ("rho", "exner", "theta_v")}
    half = {k: s * rng.standard_normal((n, nlev + 1)) for k, s in (("w", 0.05), ("ddt_w0", 1e-4), ("ddt_w1", 1e-4))}
    for a in half.values():
        a[:, 0] = 0.0
        a[:, -1] = 0.0
    f.update(half)
    f["div_m"] = 1e-6 * rng.standard_normal((n, nlev))
    f["div_t"] = f["div_m"] * f["theta_v"]
    f["rho_pred"] = f["rho"] * (1.0 + 1e-5 * rng.standard_normal((n, nlev)))
    f["theta_pred"] = f["theta_v"] * (1.0 + 1e-5 * rng.standard_normal((n, nlev)))
    return z, {k: torch.from_numpy(np.ascontiguousarray(a)).to(cuda) for k, a in f.items()}


@pytest.mark.parametrize("nlev", [2, 3, 7, 8, 9, 17, 52])
@pytest.mark.parametrize("corrector", [False, True], ids=["predictor", "corrector"])
def test_a_columns_result_does_not_depend_on_the_form(built_lib, cuda, nlev, corrector):
    import torch
    import paper_2608_21150_gb300 as P
    z, f = _columns(nlev, WIDE, cuda)
    names = ["w", "rho", "exner", "theta_v", "ddt_w0", "div_m", "div_t"]
    names += ["rho_pred", "theta_pred", "ddt_w1"] if corrector else []
    for prec in (P.ICON_PREC_FP64, P.ICON_PREC_MIXED):
        params = dict(dtime=360.0, ndyn_substeps=5, rayleigh_coeff=0.05, precision=prec)

        def solve(n):
            a = {k: f[k][:n].clone() for k in names}
            out = {k + "_new": torch.full_like(a[v], np.nan)
                   for k, v in (("w", "w"), ("rho", "rho"), ("exner", "exner"), ("theta", "theta_v"))}
            P.column_solve_noalloc(z, params, **a, **out)
            return {k: v.view(torch.int64) for k, v in out.items()}

        big = solve(WIDE)
        assert all(bool(torch.isfinite(v.view(torch.float64)).all()) for v in big.values())
        for n in (1, 15, 16, 17, 33, WIDE - 2):
            got = solve(n)
            for k in got:
                assert torch.equal(got[k], big[k][:n]), (prec, n, k)


@pytest.mark.parametrize("terrain", [False, True], ids=["flat", "terrain"])
@pytest.mark.parametrize("precision", ["fp64", "mixed", "mixed_f64col"])
@pytest.mark.parametrize("nlev", [7, 17])
def test_the_steps_forms_agree_bitwise(built_lib, cuda, terrain, precision, nlev):
    """R2B0 and R2B1 (80 and 320 cells: ragged groups of 32), the narrow form
    against the wide ones in every chunk length."""
    import paper_2608_21150_gb300 as P
    prec = {"fp64": P.ICON_PREC_FP64, "mixed": P.ICON_PREC_MIXED, "mixed_f64col": P.ICON_PREC_MIXED_F64COL}[precision]
    for bis in (0, 1):
        grid, z = make_grid(bis), make_vct(nlev)
        if terrain:
            z = terrain_following_z(z, mountain_height(grid.cell_xyz))
        op = DycoreParams(dtime=900.0, ndyn_substeps=5, rayleigh_coeff=0.05)
        od = (TerrainDycore if terrain else OracleDycore)(grid, z, op)
        st = jw_type_state(grid, z, seed=4)
        st["exner_pr"] = od.initial_exner_pr(st["exner"])
        g = P.Grid(grid, radius=op.radius)
        ref = None
        for kc in (0, 4, 6, 8):
            d = P.Dycore(g, z, gpu_params(op, precision=prec, autotune=0, column_chunk=kc))
            t = to_torch(st, cuda)
            for _ in range(2):
                d.step(t)
            d.synchronize()
            got = to_numpy(t)
            d.close()
            if ref is None:
                ref = got
                assert all(np.all(np.isfinite(v)) for v in ref.values())
            for k in ref:
                assert np.array_equal(got[k].view(np.uint64), ref[k].view(np.uint64)), (bis, kc, k)
