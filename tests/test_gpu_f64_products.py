"""The binary64 first-level products on the tensor cores (digits of eight bits,
exact sums): tile, k and column-group edges, scales that grow along the
reduction, rows of very different magnitude, zeros and subnormals, entries that
are not finite.  Every sketch against the oracle at the binary64 tolerance of
the other passes (1e-12), and no further from it than twice the FP64 units."""
import numpy as np
import pytest

import workloads as W
from oracle import ttnn as O
from oracle.tree import Tree

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2412_06111_gb300 import api  # noqa: E402

from _lib_util import Run, rel  # noqa: E402

TOL = 1e-12
# dims of a 3-mode tree ((0, 1), 2): rows nL = n0 n1, columns nR = n2; r, p
SHAPES = {
    "rows_128": ([16, 8, 64], 4, 3),         # one row tile, one B tile
    "rows_129_k_65": ([3, 43, 65], 2, 1),    # one row and one k over
    "rows_127_k_63": ([127, 1, 63], 5, 4),
    "k_31": ([40, 33, 31], 8, 8),            # below one tile of k
    "odd_long": ([37, 35, 129], 7, 6),
    "columns_33": ([30, 40, 70], 16, 17),    # two column groups, 33 columns
    "columns_96": ([50, 52, 90], 40, 16),    # three column groups
    "many_tiles": ([190, 110, 200], 6, 5),
}


def _both(dims, r, p, data, off=None, ext=None):
    tr = W.balanced_binary(3)
    n = len(tr[0])
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    out = []
    for flags in (0, api.FLAG_SIMT_PASS):
        run = Run(tr, dims, [r] * n, [p] * n, 31, dtype=api.F64, flags=flags)
        try:
            api.ttnn_update_dense(run.state, torch.from_numpy(data).cuda(), off, ext)
            assert api.ttnn_plan_pass_counts(run.plan) == ((0, 1) if flags else (1, 0))
            out.append(run.sketches())
        finally:
            run.close()
    T = data if off is None else W.embed_box(dims, off, ext, data)
    return t, out, O.sketch_ttnn(T, t, O.Drm(t, 31, "f64", "ttnn"))


def _check(t, out, want):
    errs = [[rel(o[2], want[2])] + [rel(o[k][v], want[k][v]) for v in t.sketched() for k in (0, 1)] for o in out]
    assert max(errs[0]) <= TOL, max(errs[0])
    assert max(errs[0]) <= max(2 * max(errs[1]), 1e-15 * 8), (max(errs[0]), max(errs[1]))


@pytest.mark.parametrize("shape", list(SHAPES))
def test_products_match_oracle(shape):
    dims, r, p = SHAPES[shape]
    _check(*_both(dims, r, p, W.gaussian(dims, 4)))


@pytest.mark.parametrize("axes", [(2,), (0, 1), (0, 1, 2)])
@pytest.mark.parametrize("span", [6, 40])
def test_scales_that_grow_along_the_reduction(axes, span):
    # every row tile meets larger and larger entries: its sums move down
    dims = [20, 24, 300]
    data = W.gaussian(dims, 5)
    for a in axes:
        sh = [1, 1, 1]
        sh[a] = dims[a]
        data = data * (10.0 ** np.linspace(-span, span, dims[a])).reshape(sh)
    _check(*_both(dims, 6, 4, data))


def test_zero_rows_subnormals_and_boxes():
    dims = [20, 24, 90]
    data = W.gaussian(dims, 6)
    data[3] = 0.0
    data[:, 5, :] *= 1e-310
    data[:, :, 7] = 0.0
    _check(*_both(dims, 6, 4, data))
    off, ext = [3, 0, 11], [13, 24, 71]
    _check(*_both(dims, 6, 4, np.ascontiguousarray(W.gaussian(ext, 8)), off, ext))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_entries_that_are_not_finite_reach_the_same_sketches(bad):
    dims = [20, 24, 90]
    data = W.gaussian(dims, 7)
    data[2, 3, 4] = bad
    with np.errstate(invalid="ignore"):
        t, out, want = _both(dims, 6, 4, data)
    for v in t.sketched():
        for k in (0, 1):
            assert np.array_equal(np.isfinite(out[0][k][v]), np.isfinite(want[k][v])), (v, k)
    assert np.array_equal(np.isfinite(out[0][2]), np.isfinite(want[2]))
