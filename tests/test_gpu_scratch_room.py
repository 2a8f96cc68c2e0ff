"""Forms that trade scratch for speed: taken where the scratch is there, the
general forms elsewhere, and the results the same."""
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


def test_ttn_updates_run_where_the_workspace_cannot_grow():
    # large cores take more scratch on the tensor cores than in the general
    # form: without memory for it, and in a capture, the general form runs
    tr, dims, r, p = W.balanced_binary(4), [64] * 4, 25, 12
    n, R = len(tr[0]), [96] * len(tr[0])
    cores = W.ttn_cores(tr, dims, R, np.random.default_rng(2))
    dev = [torch.from_numpy(np.ascontiguousarray(cores[v])).cuda() for v in range(n)]
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    Om, Ps, Pr = OR.sketch_ttn_input(cores, t, O.Drm(t, 6, "f32", "round"))

    def distance(run, scale):
        om, ps, pr = run.sketches()
        return max([rel(pr, scale * Pr)] + [e for v in t.sketched() for e in
                                            (rel(om[v], scale * Om[v]), rel(ps[v], scale * Ps[v]))])

    make = lambda: Run(tr, dims, [r] * n, [p] * n, 6, dtype=api.F32, flags=api.FLAG_STRUCTURED_ONLY)
    run, room = make(), make()
    try:
        api.ttnn_update_ttn(room.state, dev, R)
        assert distance(room, 1) <= 1e-5
        api.ttnn_debug_fail_alloc(1)
        api.ttnn_update_ttn(run.state, dev, R)
        api.ttnn_debug_fail_alloc(0)
        assert distance(run, 1) <= 1e-5
        small = api.ttnn_plan_device_bytes(run.plan)[1]
        assert small < api.ttnn_plan_device_bytes(room.plan)[1]
        graph = torch.cuda.CUDAGraph()
        stream = torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=stream):
            api.ttnn_update_ttn(run.state, dev, R, stream=stream.cuda_stream)
        graph.replay()
        assert distance(run, 2) <= 1e-5
        assert api.ttnn_plan_device_bytes(run.plan)[1] == small
    finally:
        api.ttnn_debug_fail_alloc(0)
        run.close()
        room.close()


def _served(srv, dims, r, p, k):
    tr = W.balanced_binary(3)
    n = len(tr[0])
    return api.ttnn_server_open(srv, tr, dims, [r] * n, [p] * n, k, sketch_dtype=api.F64)


def test_admission_gives_up_memory_that_only_makes_updates_faster():
    tr, dims, r, p = W.balanced_binary(3), [45, 47, 1009], 6, 4
    n = len(tr[0])
    static = 32 << 20     # the library's scratch block counts against the budget
    probe = api.ttnn_server_create(8 << 30)
    try:
        _served(probe, dims, r, p, 1)
        full = api.ttnn_server_stats(probe)["device_bytes"]
    finally:
        api.ttnn_server_destroy(probe)
    tight = api.ttnn_server_create(full - 1 + static)
    try:
        _served(tight, dims, r, p, 1)
        least = api.ttnn_server_stats(tight)["device_bytes"]
        assert least < full
    finally:
        api.ttnn_server_destroy(tight)
    # room for a few streams of the least size: the first is opened in full
    count = max(3, -(-full // least))
    data = [W.gaussian(dims, 20 + k) for k in range(3)]
    srv = api.ttnn_server_create(count * least + static)
    try:
        ids = [_served(srv, dims, r, p, 1)]
        assert api.ttnn_server_stats(srv)["device_bytes"] == full
        dev = [torch.from_numpy(x).cuda() for x in data]
        assert api.ttnn_server_wait(srv, api.ttnn_server_submit(srv, ids[0], dev[0]), 5_000_000) == 0
        ids += [_served(srv, dims, r, p, 1) for _ in range(count - 1)]
        with pytest.raises(api.TtnnError) as ei:
            _served(srv, dims, r, p, 1)
        assert ei.value.status == 6                        # EBUSY
        for s, d in zip(ids[1:], dev[1:]):
            assert api.ttnn_server_wait(srv, api.ttnn_server_submit(srv, s, d), 5_000_000) == 0
        # the trimmed stream goes on
        assert api.ttnn_server_wait(srv, api.ttnn_server_submit(srv, ids[0], dev[1]), 5_000_000) == 0
        t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
        for s, dense in zip(ids, (data[0] + data[1], data[1], data[2])):
            state = api.ttnn_server_stream_state(srv, s)
            plan_nodes = Run(tr, dims, [r] * n, [p] * n, 1, dtype=api.F64)
            try:
                buf = np.zeros(plan_nodes.sizes[0])
                api.ttnn_state_save(state, buf)
                api.ttnn_state_load(plan_nodes.state, buf)
                assert _distance(plan_nodes, tr, dims, r, p, "f64", dense, 1) <= 1e-12
            finally:
                plan_nodes.close()
    finally:
        api.ttnn_server_destroy(srv)
