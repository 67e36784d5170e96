"""The text of icon_dycore_launch_config keeps the form its callers parse:
"name=threads,...;column_chunk=K", the list ending in the column solve's threads
and K one number, also where the predictor and the corrector differ; what was
added stands between the two as further ";key=value" entries."""
import re

import pytest

from parity import gpu_params, setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bis,chunk,tuned", [(1, 0, 0), (1, 6, 0), (4, 0, 0), (4, 4, 0), (4, 6, 0), (4, 8, 0),
                                             (4, 0, 1)])
def test_form_of_the_launch_config(built_lib, cuda, bis, chunk, tuned):
    import paper_2608_21150_gb300 as P
    grid, z, op, od, st = setup(bis, 5, 450.0)
    d = P.Dycore(P.Grid(grid, radius=op.radius), z, gpu_params(op, autotune=tuned, column_chunk=chunk))
    text = d.launch_config()
    m = re.fullmatch(r"((?:\w+=\d+[tw]?,)*\w+=\d+)((?:;\w+=\w+)*);column_chunk=([468])", text)
    assert m, text
    names = dict(x.split("=") for x in m.group(1).split(","))
    more = dict(x.split("=") for x in m.group(2).split(";") if x)
    assert list(names)[-1] == "column_threads"
    assert all(int(v.rstrip("tw")) % 32 == 0 for v in names.values())
    assert set(more) == {"column_columns", "column_corrector_threads", "column_corrector_chunk"}
    wide = chunk or bis == 4
    assert int(more["column_columns"]) == (32 if wide else 16)
    if not tuned:
        want = (chunk, chunk) if chunk else (8, 4) if wide else (8, 8)
        assert (int(m.group(3)), int(more["column_corrector_chunk"])) == want
    # a worker thread per level (or two levels) of a chunk and one warp more
    for threads, k in ((names["column_threads"], m.group(3)),
                       (more["column_corrector_threads"], more["column_corrector_chunk"])):
        levels = 1 if not wide or int(k) == 4 else 2
        assert int(threads) == int(more["column_columns"]) * int(k) // levels + 32
