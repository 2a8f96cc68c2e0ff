"""First-level products of tensors and boxes that TMA cannot stage (odd row
strides, bases off 16 bytes, binary32 boxes) on the tensor-core GEMM, at the
sizes where its tiles, its split and its column groups end: every sketch
against the oracle, and no further from it than the SIMT pass.  Tolerance: the
passes' own (binary32 accumulation, 1e-5)."""
import numpy as np
import pytest

import workloads as W
from oracle import sttnn as OS
from oracle import ttnn as O
from oracle.tree import Tree

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2412_06111_gb300 import api  # noqa: E402

from _lib_util import Run, rel  # noqa: E402

FORMS = {"f32": (api.F32, torch.float32), "bf16": (api.BF16, torch.bfloat16)}
# name: tree, dims, r, p, variant, box extents of mode 0 (None: whole), first element's place
CASES = {
    "tile_plus_one": (W.balanced_binary(3), [43, 48, 1033], 9, 7, 0, None, 0),   # nL = 16*128+16, nR = 8*128+9
    "tile_minus_one": (W.balanced_binary(3), [31, 65, 1151], 20, 12, 0, None, 0),  # nL = 15*128+95, nR = 9*128-1
    "one_column": (W.balanced_binary(3), [1031, 1019, 3], 3, 0, 0, None, 0),     # nR below one k tile
    "one_row_tile": (W.balanced_binary(3), [5, 7, 60013], 4, 3, 0, None, 0),     # nL below one row tile
    "wide": (W.balanced_binary(4), [37, 41, 39, 36], 32, 16, 0, None, 0),        # 80 columns
    "sttnn": (W.balanced_binary(4), [37, 41, 39, 37], 11, 6, 1, None, 0),
    "tt": (W.tensor_train(4), [41, 37, 39, 37], 10, 5, 0, None, 0),              # identity leaf, no left block
    "slab": (W.balanced_binary(4), [64, 32, 40, 48], 12, 6, 0, 40, 0),
    "odd_slab": (W.balanced_binary(4), [50, 33, 41, 47], 12, 6, 0, 37, 0),
    "odd_base": (W.balanced_binary(4), [37, 41, 39, 37], 11, 6, 0, None, 1),
}


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("fmt", list(FORMS))
def test_odd_products_match_oracle(case, fmt):
    tr, dims, r, p, variant, slab, first = CASES[case]
    dtype, tdt = FORMS[fmt]
    n = len(tr[0])
    off = [0] * len(dims)
    ext = list(dims)
    if slab is not None:
        off[0], ext[0] = dims[0] - slab - 3, slab
    assert int(np.prod(ext)) >= 1 << 21      # the size from which the GEMM takes over
    data = torch.from_numpy(W.gaussian(ext, 9)).to(tdt)
    dev = torch.empty(data.numel() + first, dtype=tdt, device="cuda")
    dev[first:].copy_(data.reshape(-1))
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    T = W.embed_box(dims, off, ext, data.double().numpy())
    drm = O.Drm(t, 83, fmt, "sttnn" if variant else "ttnn")
    wom, wps, wpr = (OS.sketch_sttnn if variant else O.sketch_ttnn)(T, t, drm)
    args = (None, None) if slab is None else (off, ext)
    for flags in (0, api.FLAG_SIMT_PASS):
        run = Run(tr, dims, [r] * n, [p] * n, 83, dtype=dtype, variant=variant, flags=flags)
        try:
            api.ttnn_update_dense(run.state, dev[first:], *args)
            if not flags and not (fmt == "bf16" and case == "slab"):
                assert api.ttnn_plan_pass_counts(run.plan) == (1, 0)
            om, ps, pr = run.sketches()
        finally:
            run.close()
        assert rel(pr, wpr) <= 1e-5
        for v in t.sketched():
            assert rel(om[v], wom[v]) <= 1e-5 and rel(ps[v], wps[v]) <= 1e-5, v


def test_static_scratch_keeps_the_smaller_form():
    # 53^4 binary32 at r = 16, p = 8 fits the fixed 32 MiB with the SIMT
    # products and not with the tensor-core GEMM's pieces: it still runs there
    tr, dims = W.balanced_binary(4), [53, 53, 53, 53]
    n = len(tr[0])
    data = torch.from_numpy(W.gaussian(dims, 3)).float().cuda()
    run = Run(tr, dims, [16] * n, [8] * n, 5, dtype=api.F32)
    other = api.ttnn_state_create(run.plan)
    try:
        api.ttnn_update_dense_static(run.state, data)
        api.ttnn_update_dense(other, data)
        torch.cuda.synchronize()
        buf = np.zeros(run.sizes[0], dtype=np.float32)
        api.ttnn_state_save(other, buf)
        assert rel(run.state_host(), buf) <= 1e-5
    finally:
        api.ttnn_state_destroy(other)
        run.close()
