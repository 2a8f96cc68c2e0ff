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


ETIMEOUT = 5


def _expect_timeout(run, update):
    update(run)
    core = torch.zeros(run.sizes[2], dtype=torch.float64, device="cuda")
    with pytest.raises(api.TtnnError) as ei:
        api.ttnn_recover(run.state, core)
    assert ei.value.status == ETIMEOUT
    api.ttnn_plan_sync(run.plan)   # reported once


# products of a walk alone: the large cores; a prefix behind a first-level
# product small enough for the FP32 units (which have no waits)
@pytest.mark.parametrize("case", [LARGE, PREFIX], ids=["large_cores", "prefix"])
def test_walk_waits_running_out_report_timeout(case):
    bad, good = (_open(case, api.F32, f) for f in (api.FLAG_WAIT_TEST, 0))
    try:
        _expect_timeout(bad, lambda run: _update(run, case))
        assert _update(good, case)() <= 1e-5   # the context is intact
    finally:
        bad.close()
        good.close()


# first-level products on the two GEMMs: odd rows, K- and MN-major operands of
# every type, one CTA and many
@pytest.mark.parametrize("dtype,dims", [(api.F32, [43, 41, 39, 37]), (api.BF16, [43, 41, 39, 37]),
                                        (api.F64, [43, 41, 39, 37]), (api.F64, [8, 4, 6, 8])])
def test_first_level_waits_running_out_report_timeout(dtype, dims):
    case = (W.balanced_binary(4), dims, 6, 3)
    tdt = {api.F64: torch.float64, api.F32: torch.float32, api.BF16: torch.bfloat16}[dtype]
    data = torch.from_numpy(W.gaussian(dims, 9)).to(tdt).cuda()
    bad, good = (_open(case, dtype, f) for f in (api.FLAG_WAIT_TEST, 0))
    try:
        _expect_timeout(bad, lambda run: api.ttnn_update_dense(run.state, data))
        assert api.ttnn_plan_pass_counts(bad.plan) == (1, 0)
        api.ttnn_update_dense(good.state, data)
        good.recover()
        assert np.isfinite(good.state_host()).all()
    finally:
        bad.close()
        good.close()


@pytest.mark.parametrize("case", [PREFIX, LARGE], ids=["prefix", "large_cores"])
def test_products_leave_the_reserved_sms(case, capfd):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for flags, used in ((0, sms), (api.FLAG_RESERVE_SMS, sms - 8)):   # (at most eight sketched nodes)
        run = _open(case, api.F32, api.FLAG_DUMP_PROGRAM | flags)
        try:
            distance = _update(run, case)
            lines = LINE.findall(capfd.readouterr().err)
            assert lines and all(line.endswith(" SMs %d" % used) for _, line in lines), lines
            assert distance() <= 1e-5
        finally:
            run.close()


@pytest.mark.parametrize("case", [PREFIX, LARGE], ids=["prefix", "large_cores"])
def test_simt_pass_keeps_products_off_the_tensor_cores(case, capfd):
    run = _open(case, api.F32, api.FLAG_DUMP_PROGRAM | api.FLAG_SIMT_PASS)
    try:
        distance = _update(run, case)
        assert not LINE.findall(capfd.readouterr().err)
        assert distance() <= 1e-5
    finally:
        run.close()
