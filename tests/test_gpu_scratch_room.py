"""Forms that trade scratch for speed: taken where the scratch is there, the
general forms elsewhere, and the results the same."""
import numpy as np
import pytest

import workloads as W
from oracle import ttnn as O
from oracle.tree import Tree

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2412_06111_gb300 import api  # noqa: E402

from _lib_util import Run, rel  # noqa: E402


def _distance(run, tr, dims, r, p, fmt, dense, seed):
    n = len(tr[0])
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    Om, Ps, Pr = O.sketch_ttnn(dense, t, O.Drm(t, seed, fmt, "ttnn"))
    om, ps, pr = run.sketches()
    return max([rel(pr, Pr)] + [e for v in t.sketched() for e in (rel(om[v], Om[v]), rel(ps[v], Ps[v]))])


@pytest.mark.parametrize("dims", [[64, 32, 40, 48], [16, 16, 128, 128]])
def test_grown_workspace_is_used(dims):
    # a plan sized for TMA passes may lack the room for the tensor-core GEMM of
    # an odd box; once a TTN-format update has grown the workspace it is there
    tr, r, p = W.balanced_binary(4), 12, 6
    n = len(tr[0])
    off, ext = [0, 0, 1, 0], [m - 1 for m in dims]
    data = torch.from_numpy(W.gaussian(ext, 3)).to(torch.bfloat16)
    run = Run(tr, dims, [r] * n, [p] * n, 5, dtype=api.BF16)
    try:
        api.ttnn_update_dense(run.state, data.cuda(), off, ext)
        before = api.ttnn_plan_pass_counts(run.plan)
        cores = W.ttn_cores(tr, dims, [150] * n, np.random.default_rng(1))
        api.ttnn_update_ttn(run.state, [torch.from_numpy(np.ascontiguousarray(cores[v])).cuda() for v in range(n)],
                            [150] * n)
        api.ttnn_state_zero(run.state)
        api.ttnn_update_dense(run.state, data.cuda(), off, ext)
        assert api.ttnn_plan_pass_counts(run.plan) == (before[0] + 1, before[1])
        dense = W.embed_box(dims, off, ext, data.double().numpy())
        assert _distance(run, tr, dims, r, p, "bf16", dense, 5) <= 1e-5
    finally:
        run.close()


@pytest.mark.parametrize("dtype,fmt,tol", [(api.F64, "f64", 1e-12), (api.F32, "f32", 1e-5)])
def test_plan_creation_goes_without_optional_memory(dtype, fmt, tol):
    # each device allocation of a plan fails in turn: where the block only
    # makes updates faster the plan is made without it, and its updates agree
    tr, dims, r, p = W.balanced_binary(3), [45, 47, 1009], 6, 4
    n = len(tr[0])
    data = W.gaussian(dims, 8)
    tdt = torch.float64 if dtype == api.F64 else torch.float32
    dev = torch.from_numpy(data).to(tdt).cuda()
    dense = dev.double().cpu().numpy()
    make = lambda: Run(tr, dims, [r] * n, [p] * n, 3, dtype=dtype)
    whole = make()
    full = api.ttnn_plan_device_bytes(whole.plan)[0]
    whole.close()
    less = 0
    try:
        for k in range(1, 64):
            api.ttnn_debug_fail_alloc(k)
            try:
                run = make()
            except api.TtnnError as e:
                assert e.status == 2
                continue
            api.ttnn_debug_fail_alloc(0)
            size = api.ttnn_plan_device_bytes(run.plan)[0]
            try:
                api.ttnn_update_dense(run.state, dev)
                assert _distance(run, tr, dims, r, p, fmt, dense, 3) <= tol
            finally:
                run.close()
            assert size <= full
            less += size < full
            if size == full:
                break
    finally:
        api.ttnn_debug_fail_alloc(0)
    assert less >= 2      # the prepared operands; the larger workspace
