"""Entries and operands near the ends of their number format, on the
tensor-core GEMMs: results that binary32 (binary64) can hold are reached, with
the accuracy of the FP32 (FP64) units.  Tolerance: the updates' own (binary32
accumulation 1e-5)."""
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

# factors of the cores of nodes 0 (root), 1 and 4 (transfer) and their first
# children 2 and 5: the environment of a transfer node times its first child's
# sketch, the operand of one product, leaves binary32 in both directions
NETWORKS = {
    "large_operand": {0: 1e30, 2: 1e20, 5: 1e20, 1: 1e-30, 4: 1e-30},
    "larger_sketch": {0: 1e20, 2: 1e31, 5: 1e31, 1: 1e-30, 4: 1e-30},
    "small_operand": {0: 1e-30, 2: 1e-25, 5: 1e-25, 1: 1e30, 4: 1e30},
    "smaller_environment": {0: 1e-36, 2: 1e-20, 5: 1e-20, 1: 1e25, 4: 1e25},
}


@pytest.mark.parametrize("network", list(NETWORKS))
def test_environments_and_sketches_of_any_size(network):
    tr, dims, r, p = W.balanced_binary(4), [40, 30, 35, 33], 20, 9
    R, n = [1, 64, 128, 128, 64, 128, 127], 7
    cores = W.ttn_cores(tr, dims, R, np.random.default_rng(21))
    for v, f in NETWORKS[network].items():
        cores[v] = cores[v] * f
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    Om, Ps, Pr = OR.sketch_ttn_input(cores, t, O.Drm(t, 42, "f32", "round"))
    assert all(1e-30 < np.abs(x).max() < 1e35 for x in [Pr, *Om.values(), *Ps.values()])
    run = Run(tr, dims, [r] * n, [p] * n, 42, dtype=api.F32)
    try:
        api.ttnn_update_ttn(run.state, [torch.from_numpy(np.ascontiguousarray(cores[v])).cuda() for v in range(n)], R)
        om, ps, pr = run.sketches()
    finally:
        run.close()
    assert rel(pr, Pr) <= 1e-5
    for v in t.sketched():
        assert rel(om[v], Om[v]) <= 1e-5 and rel(ps[v], Ps[v]) <= 1e-5, v
