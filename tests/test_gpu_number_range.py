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


def _sketch_errors(tr, dims, r, p, data, dtype, seed, flags):
    n = len(tr[0])
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    want = O.sketch_ttnn(data.astype(np.float64), t, O.Drm(t, seed, {api.F32: "f32", api.F64: "f64"}[dtype], "ttnn"))
    run = Run(tr, dims, [r] * n, [p] * n, seed, dtype=dtype, flags=flags)
    try:
        api.ttnn_update_dense(run.state, torch.from_numpy(data).cuda())
        assert api.ttnn_plan_pass_counts(run.plan) == ((0, 1) if flags else (1, 0))
        got = run.sketches()
    finally:
        run.close()
    return max([rel(got[2], want[2])] + [rel(got[k][v], want[k][v]) for k in (0, 1) for v in t.sketched()])


# binary32 entries whose low bits a bfloat16 piece could not hold (its numbers
# end at 2^-133) and ones near the largest; no further off than twice the FP32
# units, whose own error is about 2e-7 (floor 5e-7)
@pytest.mark.parametrize("scale", [1e-36, 1e-34, 1e-30, 1.0, 1e30, 1e33])
def test_binary32_tensors_of_any_size(scale):
    dims = [43, 41, 39, 37]
    data = W.gaussian(dims, 9).astype(np.float32) * np.float32(scale)
    tc, simt = (_sketch_errors(W.balanced_binary(4), dims, 11, 6, data, api.F32, 83, f) for f in (0, api.FLAG_SIMT_PASS))
    assert tc <= max(2 * simt, 5e-7), (tc, simt)


def test_small_core_keeps_its_bits():
    # a large core of 1e-36 below a root of 1e30; binary32 FMAs err by 4e-7
    tr, dims, r, p = W.balanced_binary(4), [40, 30, 35, 33], 20, 9
    R, n = [1, 64, 128, 128, 64, 128, 127], 7
    cores = W.ttn_cores(tr, dims, R, np.random.default_rng(22))
    cores[0], cores[1] = cores[0] * 1e30, cores[1] * 1e-36
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    Om, Ps, Pr = OR.sketch_ttn_input(cores, t, O.Drm(t, 43, "f32", "round"))
    run = Run(tr, dims, [r] * n, [p] * n, 43, dtype=api.F32)
    try:
        api.ttnn_update_ttn(run.state, [torch.from_numpy(np.ascontiguousarray(cores[v])).cuda() for v in range(n)], R)
        om, ps, pr = run.sketches()
    finally:
        run.close()
    assert max([rel(pr, Pr)] + [e for v in t.sketched() for e in (rel(om[v], Om[v]), rel(ps[v], Ps[v]))]) <= 1e-6


def _same_values_that_are_not_finite(got, want):
    got, want = np.asarray(got, np.float64).ravel(), np.asarray(want, np.float64).ravel()
    return np.array_equal(np.nan_to_num(got, nan=2.0, posinf=3.0, neginf=-3.0)[~np.isfinite(want)],
                          np.nan_to_num(want, nan=2.0, posinf=3.0, neginf=-3.0)[~np.isfinite(want)]) and \
        np.array_equal(np.isfinite(got), np.isfinite(want))


def _check_not_finite(dims, r, p, dtype, data, flags=0):
    """Every sketch has NaN, +Inf and -Inf where the definition has them."""
    tr = W.balanced_binary(len(dims))
    n = len(tr[0])
    t = Tree(tr[0], tr[1], dims, [r] * n, [p] * n, tr[2])
    with np.errstate(invalid="ignore", over="ignore"):
        want = O.sketch_ttnn(data.astype(np.float64), t, O.Drm(t, 31, {api.F32: "f32", api.F64: "f64"}[dtype], "ttnn"))
    run = Run(tr, dims, [r] * n, [p] * n, 31, dtype=dtype, flags=flags)
    try:
        api.ttnn_update_dense(run.state, torch.from_numpy(data).cuda())
        assert api.ttnn_plan_pass_counts(run.plan) == ((0, 1) if flags else (1, 0))
        got = run.sketches()
    finally:
        run.close()
    assert _same_values_that_are_not_finite(got[2], want[2])
    for k in (0, 1):
        for v in t.sketched():
            assert _same_values_that_are_not_finite(got[k][v], want[k][v]), (k, v)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_binary32_entries_that_are_not_finite(bad):
    dims = [43, 41, 39, 37]
    data = W.gaussian(dims, 9).astype(np.float32)
    data[7, 8, 9, 10] = bad
    _check_not_finite(dims, 11, 6, api.F32, data)


def test_binary32_nan_with_all_its_bits_low():
    dims = [43, 41, 39, 37]
    data = W.gaussian(dims, 9).astype(np.float32)
    data.reshape(-1).view(np.uint32)[123457] = 0x7F800001
    _check_not_finite(dims, 11, 6, api.F32, data)


# a row tile of one CTA and tiles cut over many; an entry early and one late
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("dims,at", [([12, 10, 12], 5), ([20, 24, 90], 777), ([37, 35, 129], 160000),
                                     ([190, 110, 200], 3000000)])
def test_binary64_entries_that_are_not_finite(dims, at, bad):
    data = W.gaussian(dims, 9)
    data.reshape(-1)[at] = bad
    _check_not_finite(dims, 6, 4, api.F64, data)


def test_binary64_infinities_of_both_signs_in_one_row():
    dims = [20, 24, 90]
    data = W.gaussian(dims, 9)
    data[3, 4, 7], data[3, 4, 60], data[3, 5, 7] = np.inf, -np.inf, np.inf
    _check_not_finite(dims, 6, 4, api.F64, data)


# the second and third group of 32 columns take their own part of the operand
@pytest.mark.parametrize("dims,r,p", [([30, 40, 70], 16, 17), ([50, 52, 90], 40, 16)])
def test_binary64_infinity_in_later_column_groups(dims, r, p):
    data = W.gaussian(dims, 9)
    data[11, 13, 17] = np.inf
    _check_not_finite(dims, r, p, api.F64, data)
