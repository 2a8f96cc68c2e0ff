"""Plan flags reach the tensor-core GEMMs of a walk (Khatri-Rao prefixes, large
cores of TTN-format input) as they reach its other ops and the first-level
products."""
import re

import numpy as np
import pytest

import workloads as W
from oracle import rounding as OR
from oracle import ttnn as O
from oracle.tree import Tree

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2412_06111_gb300 import api  # noqa: E402

from _lib_util import Run, rel  # noqa: E402

# a tree, dims, r, p whose whole update has a prefix product, and a network
# with one large core (three products) and one just below the size
PREFIX = (W.from_nested((((0, 1), 2), [3, 4])), [27, 19, 64, 9, 5], 9, 8)
LARGE = (W.balanced_binary(4), [40, 30, 35, 33], 20, 8)
RANKS = [1, 64, 128, 128, 64, 128, 127]
LINE = re.compile(r"us  \[ttnn\] L(\d+) tensor-core gemm (.*)")


def _cores(tr, dims):
    return W.ttn_cores(tr, dims, RANKS, np.random.default_rng(21))


def _open(case, dtype, flags):
    tr, dims, r, p = case
    n = len(tr[0])
    return Run(tr, dims, [r] * n, [p] * n, 42, dtype=dtype, flags=flags)


def _update(run, case):
    """One update; returns the sketches' distance from the oracle as a call."""
    tr, dims, r, p = case
    n = len(tr[0])
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    if case is LARGE:
        cores = _cores(tr, dims)
        api.ttnn_update_ttn(run.state, [torch.from_numpy(np.ascontiguousarray(cores[v])).cuda() for v in range(n)],
                            RANKS)
        want = lambda: OR.sketch_ttn_input(cores, t, O.Drm(t, 42, "f32", "round"))
    else:
        data = torch.from_numpy(W.gaussian(dims, 9)).float()
        api.ttnn_update_dense(run.state, data.cuda())
        want = lambda: O.sketch_ttnn(data.double().numpy(), t, O.Drm(t, 42, "f32", "ttnn"))

    def distance():
        (om, ps, pr), (Om, Ps, Pr) = run.sketches(), want()
        return max([rel(pr, Pr)] + [e for v in t.sketched() for e in (rel(om[v], Om[v]), rel(ps[v], Ps[v]))])

    return distance


@pytest.mark.parametrize("case,products", [(PREFIX, 1), (LARGE, 3)], ids=["prefix", "large_cores"])
def test_dump_shows_every_product(case, products, capfd):
    run = _open(case, api.F32, api.FLAG_DUMP_PROGRAM)
    try:
        distance = _update(run, case)
        lines = LINE.findall(capfd.readouterr().err)
        assert len(lines) == products, lines
        assert distance() <= 1e-5
    finally:
        run.close()
