"""The matrix-vector pass of a rank-one box at the sizes where its blocks, its
rows in flight and its column groups end: every sketch against the oracle.
Tolerances as for the other passes (binary64 1e-12; binary32 accumulation of
at most 2e4 terms 1e-5)."""
import numpy as np
import pytest

import workloads as W
from oracle import ttnn as O
from oracle.tree import Tree

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2412_06111_gb300 import api  # noqa: E402

from _lib_util import Run, rel  # noqa: E402

FORMS = {"f64": (api.F64, torch.float64, 1e-12), "f32": (api.F32, torch.float32, 1e-5),
         "bf16": (api.BF16, torch.bfloat16, 1e-5)}


# rows = the box's extents on the first two modes; r, p set the column groups (of 8)
@pytest.mark.parametrize("rows,r,p", [((1, 2), 3, 2), ((7, 73), 4, 2), ((16, 32), 5, 3), ((19, 27), 8, 4),
                                      ((127, 149), 9, 8)])
@pytest.mark.parametrize("fmt", list(FORMS))
def test_rows_of_a_rank_one_box(rows, r, p, fmt):
    dtype, tdt, tol = FORMS[fmt]
    tr = W.balanced_binary(3)
    dims = [130, 150, 24]
    n = len(tr[0])
    off, ext = [3, 1, 17], [rows[0], rows[1], 1]
    off[0], off[1] = min(3, dims[0] - rows[0]), min(1, dims[1] - rows[1])
    data = torch.from_numpy(W.gaussian(ext, 5)).to(tdt)
    run = Run(tr, dims, [r] * n, [p] * n, 71, dtype=dtype)
    try:
        api.ttnn_update_dense(run.state, data.cuda(), off, ext, lam=0.5)
        om, ps, pr = run.sketches()
    finally:
        run.close()
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    T = 0.5 * W.embed_box(dims, off, ext, data.double().numpy())
    wom, wps, wpr = O.sketch_ttnn(T, t, O.Drm(t, 71, fmt, "ttnn"))
    assert rel(pr, wpr) <= tol
    for v in t.sketched():
        assert rel(om[v], wom[v]) <= tol and rel(ps[v], wps[v]) <= tol, v
