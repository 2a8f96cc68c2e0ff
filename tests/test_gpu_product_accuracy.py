"""The tensor-core GEMMs are as accurate as the FP32 units they stand in for
(dropping a third piece or a product of order two of binary32 operands leaves a
few 1e-6), and are what ran; merged over the streams of a server they give the
same bits as alone."""
import numpy as np
import pytest

import test_gpu_walk_products as P
import workloads as W
from oracle import rounding as OR
from oracle import ttnn as O
from oracle.tree import Tree

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2412_06111_gb300 import api  # noqa: E402

from _lib_util import Run, rel  # noqa: E402

TDT = {api.F64: torch.float64, api.F32: torch.float32, api.BF16: torch.bfloat16}


def _worst(t, got, want):
    return max([rel(got[2], want[2])] + [rel(got[k][v], want[k][v]) for k in (0, 1) for v in t.sketched()])


# odd tensors: long and short reductions, 80 columns, one row tile; the FP32
# units err by 1e-7 to 1e-6 (more the longer the sums)
@pytest.mark.parametrize("dtype", [api.F32, api.BF16])
@pytest.mark.parametrize("tr,dims,r,p", [(W.balanced_binary(3), [43, 48, 1033], 9, 7),
                                         (W.balanced_binary(3), [1031, 1019, 3], 3, 0),
                                         (W.balanced_binary(3), [5, 7, 60013], 4, 3),
                                         (W.balanced_binary(4), [37, 41, 39, 36], 32, 16)])
def test_first_level_products_are_as_accurate_as_the_fp32_units(tr, dims, r, p, dtype):
    n = len(tr[0])
    data = torch.from_numpy(W.gaussian(dims, 9)).to(TDT[dtype])
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    want = O.sketch_ttnn(data.double().numpy(), t, O.Drm(t, 83, P.FMT[dtype], "ttnn"))
    err = []
    for flags in (0, api.FLAG_SIMT_PASS):
        run = Run(tr, dims, [r] * n, [p] * n, 83, dtype=dtype, flags=flags)
        try:
            api.ttnn_update_dense(run.state, data.cuda())
            assert api.ttnn_plan_pass_counts(run.plan) == ((0, 1) if flags else (1, 0))
            err.append(_worst(t, run.sketches(), want))
        finally:
            run.close()
    assert err[0] <= max(2 * err[1], 1e-6), err


@pytest.mark.parametrize("case", [c for c in P.CORES if c != "identity_second"])
def test_large_cores_are_as_accurate_as_fp32(case, capfd):
    tr, dims, r, p, ranks = P.CORES[case]
    n = len(tr[0])
    R = [ranks] * n if isinstance(ranks, int) else [ranks[v] for v in range(n)]
    cores = W.ttn_cores(tr, dims, R, np.random.default_rng(23))
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    want = OR.sketch_ttn_input(cores, t, O.Drm(t, 44, "f32", "round"))
    run = Run(tr, dims, [r] * n, [p] * n, 44, dtype=api.F32, flags=api.FLAG_DUMP_PROGRAM)
    try:
        api.ttnn_update_ttn(run.state, [torch.from_numpy(np.ascontiguousarray(cores[v])).cuda() for v in range(n)], R)
        assert "tensor-core gemm" in capfd.readouterr().err
        assert _worst(t, run.sketches(), want) <= 1.5e-6
    finally:
        run.close()


@pytest.mark.parametrize("dtype", [api.F32, api.BF16])
@pytest.mark.parametrize("dims,r,p", [([101, 67, 41, 17, 3], 20, 12), ([27, 19, 64, 9, 5], 9, 8),
                                      ([61, 50, 49, 3, 17], 32, 16)])
def test_prefixes_are_as_accurate_as_fp32(dims, r, p, dtype, capfd):
    tr = W.from_nested((((0, 1), 2), [3, 4]))
    n = len(tr[0])
    data = torch.from_numpy(W.gaussian(dims, 10)).to(TDT[dtype])
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    want = O.sketch_ttnn(data.double().numpy(), t, O.Drm(t, 83, P.FMT[dtype], "ttnn"))
    run = Run(tr, dims, [r] * n, [p] * n, 83, dtype=dtype, flags=api.FLAG_DUMP_PROGRAM)
    try:
        api.ttnn_update_dense(run.state, data.cuda())
        assert "tensor-core gemm" in capfd.readouterr().err
        assert _worst(t, run.sketches(), want) <= 1.5e-6
    finally:
        run.close()


def test_served_products_equal_alone_bitwise():
    # walks with prefix products of two plans, and first-level products on both
    # GEMMs, batched by one worker
    pre = W.from_nested((((0, 1), 2), [3, 4]))
    streams = [(pre, [27, 19, 64, 9, 5], 9, 8, api.F32), (pre, [29, 18, 64, 9, 5], 9, 8, api.BF16),
               (W.balanced_binary(4), [37, 41, 39, 37], 11, 6, api.F32), (W.balanced_binary(3), [30, 41, 43], 5, 4, api.F64)]
    srv = api.ttnn_server_create(64 << 30, max_batch=8, workers=1)
    alone = []
    try:
        ids, tickets, keep = [], [], []
        for j, (tr, dims, r, p, dt) in enumerate(streams):
            n = len(tr[0])
            ids.append(api.ttnn_server_open(srv, tr, dims, [r] * n, [p] * n, 100 + j, sketch_dtype=dt))
            alone.append(Run(tr, dims, [r] * n, [p] * n, 100 + j, dtype=dt))
        for k in range(12):
            for j, (tr, dims, r, p, dt) in enumerate(streams):
                x = torch.from_numpy(W.gaussian(dims, 50 * j + k)).to(TDT[dt]).cuda()
                keep.append((j, x))
        torch.cuda.synchronize()
        for j, x in keep:
            tickets.append(api.ttnn_server_submit(srv, ids[j], x))
        for ticket in tickets:
            assert api.ttnn_server_wait(srv, ticket, 10_000_000) == 0
        rep = api.ttnn_server_stats(srv)
        assert rep["batches"] < len(keep)          # requests were merged
        for j, x in keep:
            api.ttnn_update_dense(alone[j].state, x)
        for j, run in enumerate(alone):
            state = api.ttnn_server_stream_state(srv, ids[j])
            n, eb = run.sizes[0], run.sizes[1]
            buf = np.zeros(n, dtype=np.float64 if eb == 8 else np.float32)
            api.ttnn_state_save(state, buf)
            assert np.array_equal(buf.astype(np.float64), run.state_host()), j
    finally:
        api.ttnn_server_destroy(srv)
        for run in alone:
            run.close()
