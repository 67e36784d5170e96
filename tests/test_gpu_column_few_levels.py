"""Column solves of a few levels take shorter chunks: the allocation-free entry
point chunks of 2 at up to four levels, the step chunks of 4 for its predictor.
On both sides of that line the results are those of the 16-column form, whose
chunks of 8 hold all the levels, bit for bit."""
import pytest

from parity import gpu_params, setup
from test_gpu_column_forms import WIDE, _columns

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nlev", [2, 3, 4, 5])
@pytest.mark.parametrize("corrector", [False, True], ids=["predictor", "corrector"])
@pytest.mark.parametrize("prec", ["FP64", "MIXED"])
def test_few_levels_of_many_columns(built_lib, cuda, nlev, corrector, prec):
    import torch
    import paper_2608_21150_gb300 as P
    z, f = _columns(nlev, WIDE, cuda)
    names = ["w", "rho", "exner", "theta_v", "ddt_w0", "div_m", "div_t"]
    names += ["rho_pred", "theta_pred", "ddt_w1"] if corrector else []
    params = dict(dtime=360.0, ndyn_substeps=5, rayleigh_coeff=0.05, precision=getattr(P, "ICON_PREC_" + prec))

    def solve(part):
        a = {k: f[k][part].contiguous() for k in names}
        out = {k + "_new": torch.full_like(a[v], float("nan"))
               for k, v in (("w", "w"), ("rho", "rho"), ("exner", "exner"), ("theta", "theta_v"))}
        P.column_solve_noalloc(z, params, **a, **out)
        return out

    whole = solve(slice(0, WIDE))
    for part in (slice(0, WIDE // 2), slice(WIDE // 2, WIDE)):
        for k, v in solve(part).items():
            assert bool(torch.isfinite(v).all())
            assert torch.equal(v.view(torch.int64), whole[k][part].view(torch.int64)), k


@pytest.mark.parametrize("nlev,chunk", [(2, 4), (4, 4), (5, 8)])
def test_default_chunk_of_few_levels(built_lib, cuda, nlev, chunk):
    import paper_2608_21150_gb300 as P
    grid, z, op, od, st = setup(4, nlev, 450.0)
    d = P.Dycore(P.Grid(grid, radius=op.radius), z, gpu_params(op, autotune=0))
    assert d.launch_config().endswith(";column_chunk=%d" % chunk)
