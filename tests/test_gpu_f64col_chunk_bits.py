"""The mixed mode with the FP64 column solve gives the same bits in every chunk
length too: the solve spells its multiply-adds out, so that no instantiation
leaves one to the compiler.  45 levels, which no chunk divides."""
import numpy as np
import pytest

from parity import gpu_params, setup, to_numpy, to_torch

pytestmark = pytest.mark.gpu


def test_f64col_chunk_lengths_agree_bitwise(built_lib, cuda):
    import paper_2608_21150_gb300 as P
    grid, z, op, od, st = setup(3, 45, 900.0, rayleigh=0.05, seed=4)
    g = P.Grid(grid, radius=op.radius)
    outs = []
    for kc in (0, 4, 6, 8):
        d = P.Dycore(g, z, gpu_params(op, precision=P.ICON_PREC_MIXED_F64COL, autotune=0, column_chunk=kc))
        t = to_torch(st, cuda)
        for _ in range(2):
            d.step(t)
        d.synchronize()
        outs.append(to_numpy(t))
        d.close()
    for got in outs[1:]:
        for k, v in outs[0].items():
            assert np.array_equal(got[k].view(np.uint64), v.view(np.uint64)), k
