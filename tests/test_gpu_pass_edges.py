"""First-level tensor-core passes at the edges of their tiles and chunks: row
blocks and column chunks that end inside a tile, one, two and more than four
chunks (their partial sums of D1 folded in chunk order), every width of 16
columns from 16 to 80, each storage format, against the oracle.  Tolerance: the
passes' own (binary32 accumulation, 1e-5; 1e-4 for binary32 DRM blocks split in
two)."""
import numpy as np
import pytest

import workloads as W
from oracle import quant as Q
from oracle import ttnn as O
from oracle.tree import Tree

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2412_06111_gb300 import api  # noqa: E402

from _lib_util import Run, rel  # noqa: E402

TREE = W.from_nested(([0, 1], [2, 3]))   # nL = dims[0] dims[1], nR = dims[2] dims[3]
FORMS = {"bf16": (api.BF16, 1e-5), "f32": (api.F32, 1e-4), "bf16x2": (api.BF16X2, 1e-5), "e4m3": (api.E4M3, 1e-5)}


@pytest.mark.parametrize("fmt", sorted(FORMS))
@pytest.mark.parametrize("dims,r,p", [([8, 16, 8, 16], 4, 2),      # one tile
                                      ([8, 1000, 8, 6], 4, 2),     # nR inside a tile
                                      ([8, 13, 16, 97], 20, 10),   # nL inside a tile, 2 chunks
                                      ([8, 33, 16, 97], 11, 5),
                                      ([8, 1201, 16, 97], 32, 16),
                                      ([8, 50, 80, 78], 20, 10)])  # 5 chunks
def test_pass_edges_match_oracle(dims, r, p, fmt):
    dtype, tol = FORMS[fmt]
    n = len(TREE[0])
    t = Tree(TREE[0], TREE[1], dims, [r] * n, [p] * n, TREE[2])
    T = W.gaussian(dims, 5).astype(np.float32).astype(np.float64)
    run = Run(TREE, dims, [r] * n, [p] * n, 31, dtype=dtype)
    try:
        if fmt == "bf16":
            data = torch.from_numpy(T).to(torch.bfloat16)
            T = data.double().numpy()
        elif fmt == "e4m3":
            q, s = Q.fp8_tile_quantize(T.reshape(dims[0] * dims[1], -1))
            data, T = torch.from_numpy(Q.e4m3_encode(q).reshape(-1)), Q.fp8_dequantize_bf16(q, s).reshape(dims)
        else:
            data = torch.from_numpy(T.astype(np.float32))
            if fmt == "bf16x2":
                hi, lo = Q.split_bf16x2(T)
                T = hi + lo
        scale = torch.from_numpy(s.astype(np.float32).reshape(-1)).cuda() if fmt == "e4m3" else None
        api.ttnn_update_dense(run.state, data.cuda(), tile_scale=scale)
        assert api.ttnn_plan_pass_counts(run.plan) == (1, 0)
        om, ps, pr = run.sketches()
    finally:
        run.close()
    drm = O.Drm(t, 31, {"bf16x2": "bf16"}.get(fmt, fmt))
    wom, wps, wpr = O.sketch_ttnn(T, t, drm)
    assert rel(pr, wpr) <= tol
    for v in t.sketched():
        assert rel(om[v], wom[v]) <= tol and rel(ps[v], wps[v]) <= tol, v
