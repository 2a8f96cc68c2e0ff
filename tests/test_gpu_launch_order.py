"""Kernels of an update placed before the kernel they follow has ended read
what it wrote: updates and recoveries queued back to back equal the same with
the device idle between any two, and a captured graph of them, bit for bit."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
from paper_2412_06111_gb300 import api  # noqa: E402

from _lib_util import Run  # noqa: E402

CASES = {   # tree, dims, r, p, update boxes (offset, extent); the last has one row
    "tt": (W.tensor_train(4), [16, 12, 10, 14], 4, 3,
           [(None, None), ([0, 2, 1, 3], [16, 1, 9, 7]), ([3, 0, 0, 0], [1, 12, 10, 14])]),
    "binary": (W.balanced_binary(5), [9, 8, 10, 9, 8], 4, 2,
               [(None, None), ([1, 0, 2, 1, 0], [8, 7, 6, 5, 4]), ([3, 4, 0, 0, 0], [1, 1, 10, 9, 8])]),
}


@pytest.mark.parametrize("dtype", [api.F64, api.F32, api.BF16])
@pytest.mark.parametrize("case", sorted(CASES))
def test_queued_calls_equal_idle_ones(case, dtype):
    tr, dims, r, p, boxes = CASES[case]
    n = len(tr[0])
    tdt = {api.F64: torch.float64, api.F32: torch.float32, api.BF16: torch.bfloat16}[dtype]
    data = [torch.from_numpy(W.gaussian(dims if e is None else e, 3 + k)).to(tdt).cuda()
            for k, (_, e) in enumerate(boxes)]
    run = Run(tr, dims, [r] * n, [p] * n, 7, dtype=dtype)
    cores = torch.zeros(run.sizes[2], dtype=torch.float64, device="cuda")
    stream = torch.cuda.Stream()

    def updates(between):
        api.ttnn_state_zero(run.state, stream=stream.cuda_stream)
        for _ in range(4):
            for d, (off, ext) in zip(data, boxes):
                between()
                api.ttnn_update_dense(run.state, d, off, ext, stream=stream.cuda_stream)
        between()

    try:
        torch.cuda.synchronize()
        updates(torch.cuda.synchronize)
        want = run.state_host()
        api.ttnn_recover(run.state, cores, stream=stream.cuda_stream)
        torch.cuda.synchronize()
        wcores = cores.clone()
        for _ in range(20):
            updates(lambda: None)
            api.ttnn_recover(run.state, cores, stream=stream.cuda_stream)
            torch.cuda.synchronize()
            assert (run.state_host() == want).all() and bool((cores == wcores).all())
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            updates(lambda: None)
        api.ttnn_state_zero(run.state)
        torch.cuda.synchronize()
        graph.replay()
        assert (run.state_host() == want).all()
    finally:
        run.close()
