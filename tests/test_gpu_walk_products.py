"""Walk contractions on their wide forms, at the sizes where those begin and
end: large cores of TTN-format input and Khatri-Rao prefixes as tensor-core
GEMMs, and contractions with an output axis across the lanes.  Tolerances: the
updates' own (binary32 accumulation 1e-5, binary64 1e-12)."""
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

FMT = {api.F64: "f64", api.F32: "f32", api.BF16: "bf16"}
TOL = {api.F64: 1e-12, api.F32: 1e-5, api.BF16: 1e-5}
B4, B8 = W.balanced_binary(4), W.balanced_binary(8)
ID4 = (B4[0], B4[1], [m == [0] for m in B4[1]])   # the first child of its parent is an identity leaf
PAIR = W.from_nested(([0, 1], (2, 3)))            # a leaf of two modes

# name: tree, dims, r, p, rank of each node (one: of all)
CORES = {
    "at_threshold": (B4, [40, 30, 35, 33], 20, 8, {0: 1, 1: 64, 2: 128, 3: 128, 4: 64, 5: 128, 6: 127}),
    "odd": (B4, [40, 30, 35, 33], 20, 11, {0: 1, 1: 17, 2: 257, 3: 255, 4: 31, 5: 129, 6: 263}),
    "one_row": (B4, [40, 30, 35, 33], 20, 9, {0: 1, 1: 1, 2: 1031, 3: 1033, 4: 2, 5: 1024, 6: 513}),
    "one_inner": (B4, [40, 30, 35, 33], 20, 10, {0: 1, 1: 1027, 2: 1025, 3: 1, 4: 1024, 5: 1, 6: 1024}),
    "wide": (B4, [64, 50, 55, 49], 32, 16, {0: 1, 1: 128, 2: 96, 3: 88, 4: 127, 5: 97, 6: 89}),
    "deep": (B8, [20, 19, 18, 17, 20, 19, 18, 17], 8, 4, 139),
    "toy": (W.toy_tree(), [30, 25, 20, 24, 28, 26], 7, 5, 141),
    "identity_first": (ID4, [9, 30, 35, 33], 6, 3, 151),
    "identity_second": (W.tensor_train(4), [30, 25, 20, 24], 7, 5, 104),   # general path
}


def check_ttn(tr, dims, r, p, ranks, dtype, scale=1.0):
    n = len(tr[0])
    R = [ranks] * n if isinstance(ranks, int) else [ranks[v] for v in range(n)]
    cores = W.ttn_cores(tr, dims, R, np.random.default_rng(21), scale)
    run = Run(tr, dims, [r] * n, [p] * n, 42, dtype=dtype)
    try:
        dev = [torch.from_numpy(np.ascontiguousarray(cores[v])).cuda() for v in range(n)]
        for _ in range(2):   # into a fresh state, and onto one
            api.ttnn_update_ttn(run.state, dev, R, lam=-0.625)
        t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
        Om, Ps, Pr = OR.sketch_ttn_input(cores, t, O.Drm(t, 42, FMT[dtype], "round"))
        om, ps, pr = run.sketches()
    finally:
        run.close()
    assert rel(pr, -1.25 * Pr) <= TOL[dtype]
    for v in t.sketched():
        assert rel(om[v], -1.25 * Om[v]) <= TOL[dtype], v
        assert rel(ps[v], -1.25 * Ps[v]) <= TOL[dtype], v


@pytest.mark.parametrize("dtype", [api.F32, api.BF16])
@pytest.mark.parametrize("case", list(CORES))
def test_large_cores_match_oracle(case, dtype):
    check_ttn(*CORES[case], dtype)


# widths of the lane axis (8, 16 and 32 lanes, cut beyond) and reductions long
# enough to be split over blocks, with and without weights per column
@pytest.mark.parametrize("dtype", [api.F64, api.F32])
@pytest.mark.parametrize("r,p", [(3, 1), (4, 3), (8, 0), (9, 7), (16, 16), (33, 0), (24, 41)])
@pytest.mark.parametrize("tr,dims,ranks", [(B4, [70, 71, 72, 69], 37), (B4, [2500, 80, 2049, 70], 17),
                                           (PAIR, [2100, 3, 70, 80], 40)], ids=["short", "split", "pair"])
def test_lane_contractions_match_oracle(tr, dims, ranks, r, p, dtype):
    check_ttn(tr, dims, r, p, ranks, dtype)


# Khatri-Rao prefix of D1 on the tensor cores: just beyond its threshold at 17
# and 32 columns; smaller where the split-K form has few blocks or holds too
# few columns; odd extents
@pytest.mark.parametrize("dtype", [api.F32, api.BF16])
@pytest.mark.parametrize("dims,r,p", [([101, 67, 41, 17, 3], 20, 12), ([127, 103, 41, 1, 17], 11, 6),
                                      ([33, 35, 34, 17, 5], 18, 15), ([27, 19, 64, 9, 5], 9, 8),
                                      ([61, 50, 49, 3, 17], 32, 16)])
def test_prefix_products_match_oracle(dims, r, p, dtype):
    tr = W.from_nested((((0, 1), 2), [3, 4]))
    n = len(tr[0])
    tdt = {api.F32: torch.float32, api.BF16: torch.bfloat16}[dtype]
    data = torch.from_numpy(W.gaussian(dims, 9)).to(tdt)
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    Om, Ps, Pr = O.sketch_ttnn(data.double().numpy(), t, O.Drm(t, 83, FMT[dtype], "ttnn"))
    run = Run(tr, dims, [r] * n, [p] * n, 83, dtype=dtype)
    try:
        api.ttnn_update_dense(run.state, data.cuda())
        om, ps, pr = run.sketches()
    finally:
        run.close()
    assert rel(pr, Pr) <= 1e-5
    for v in t.sketched():
        assert rel(om[v], Om[v]) <= 1e-5 and rel(ps[v], Ps[v]) <= 1e-5, v
