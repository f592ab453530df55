"""The fp32 passes over column groups (rows wider than 4096 or with a radix above 8) and the fp32 column passes of the
two-sided product, against the oracle: every tile layout and phase form, row counts around the 32- and 64-row tiles."""
import numpy as np
import pytest
import torch

import paper_2605_29843_b200 as harp
from oracle import harp_oracle as orc
from paper_2605_29843_b200 import workloads as wl
from harp_testlib import TOL, gpu_apply, host_rows, promote, to_device, to_host_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radices,perm", [
    ((16, 16, 8), "identity"),            # contiguous and strided sixteen-wide blocks, an upper pass
    ((16, 16, 8), "random"),              # permutation and signs in a kernel of their own
    ((2, 16, 9, 4), "identity"),          # strides 1 and 2 that no 16-byte access fits
    ((4, 4, 4, 43), "identity"),          # radix above 16 in the upper pass
    ((8, 8, 8, 8, 2), "identity"),
    ((8, 8, 5, 3, 11), "identity"),
    ((4, 4, 4, 4, 4, 4, 2), "identity"),  # pairs of radix-4 stages
    ((32, 16), "identity"),               # a first pass these kernels do not take
])
@pytest.mark.parametrize("n_rows", [1, 33, 64, 127])
def test_rows_match_the_oracle(radices, perm, n_rows):
    spec = wl.tiny_plan(61, radices, kind="qr", perm=perm, signs=True)
    plan, oplan = harp.plan_from_spec(spec), orc.OraclePlan.from_spec(spec)
    xh = host_rows(np.random.default_rng(62).standard_normal((n_rows, spec.d)), "f32")
    for tr, fn in ((False, orc.forward), (True, orc.transpose)):
        got, guards = gpu_apply(plan, xh, "f32", tr)
        assert guards
        assert orc.rel_err_rows(got, fn(oplan, promote(xh, "f32"))) <= TOL["f32"]
    assert harp.harp_plan_error_word(plan) == 0


@pytest.mark.parametrize("radices,perm", [((16, 16, 8), "identity"), ((16, 16, 8), "random"), ((2, 16, 9, 4), "identity"), ((16, 16), "identity"),
                                          ((4, 4, 4, 43), "identity"), ((8, 8, 8, 8, 2), "identity"), ((8, 8, 5, 3, 11), "identity"),
                                          ((4, 4, 4, 4, 4, 4, 2), "identity")])
@pytest.mark.parametrize("n_rows", [1, 33, 64, 127])
def test_passes_match_the_oracle(monkeypatch, radices, perm, n_rows):
    """The same batches with the passes for all of them: by themselves the smaller ones take the whole-row kernels."""
    monkeypatch.setenv("HARP_F32_PASSES", "1")
    test_rows_match_the_oracle(radices, perm, n_rows)


@pytest.mark.parametrize("radices,few,many", [((16, 16, 4), 64, 1024), ((8, 8, 8, 8, 2), 500, 128)])
def test_small_batches_take_one_launch(radices, few, many):
    """`few` rows are one wave of the whole-row kernels, `many` are faster in two passes."""
    plan = harp.plan_from_spec(wl.tiny_plan(71, radices, kind="qr", perm="identity", signs=True))
    for n_rows, launches in ((few, 1), (many, 2)):
        x = torch.zeros((n_rows, plan.d), device="cuda")
        before = harp.harp_launch_count()
        harp.apply_(plan, x)
        torch.cuda.synchronize()
        assert harp.harp_launch_count() - before == launches


@pytest.mark.parametrize("r_out,r_in", [((8, 8, 8), (4, 3, 5)), ((16, 16, 2), (7, 4)), ((2, 2, 2, 2, 3), (4, 4, 4, 4, 4)),
                                        ((43, 4), (4, 17)), ((64,), (2, 2)), ((8, 8, 8, 8), (8, 9))])
def test_two_sided_fp32(r_out, r_in):
    p_out = wl.tiny_plan(63, r_out, kind="qr", perm="identity", signs=True)
    p_in = wl.tiny_plan(64, r_in, kind="qr", perm="identity", signs=True)
    wh = host_rows(np.random.default_rng(65).standard_normal((p_out.d, p_in.d)), "f32")
    wd = to_device(wh, "f32")
    plan_out, plan_in = harp.plan_from_spec(p_out), harp.plan_from_spec(p_in)
    harp.two_sided_(wd, plan_out, plan_in)
    torch.cuda.synchronize()
    want = orc.two_sided(orc.OraclePlan.from_spec(p_out), orc.OraclePlan.from_spec(p_in), promote(wh, "f32"))
    # two sides, each within the one-sided tolerance of the row (column) norm
    err = np.abs(to_host_f64(wd) - want)
    scale = np.minimum(np.linalg.norm(want, axis=1, keepdims=True), np.linalg.norm(want, axis=0, keepdims=True))
    assert np.max(err / scale) <= 2 * TOL["f32"]
    assert harp.harp_plan_error_word(plan_out) == 0


@pytest.mark.parametrize("r_out,r_in", [((2, 2, 2, 2, 3), (4, 3, 5)), ((43, 4), (4, 17)), ((41, 3, 3), (4, 4)), ((64,), (2, 2)), ((8, 8, 8), (8, 9))])
def test_two_sided_fp32_in_place(monkeypatch, r_out, r_in):
    """Column passes for small matrices too, which by themselves go through the transposed copy."""
    monkeypatch.setenv("HARP_F32_PASSES", "1")
    test_two_sided_fp32(r_out, r_in)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_a_driver_without_tensor_maps(monkeypatch, dtype):
    """Plans whose passes cannot be fed by bulk copies keep the kernels that need none: rows, permuted rows and both sides of a matrix."""
    monkeypatch.setenv("HARP_NO_TENSOR_MAPS", "1")
    for radices, perm in (((16, 16, 8), "random"), ((8, 8, 8, 8, 2), "identity"), ((16, 16, 43), "identity")):
        spec = wl.tiny_plan(66, radices, kind="qr", perm=perm, signs=True)
        plan, oplan = harp.plan_from_spec(spec), orc.OraclePlan.from_spec(spec)
        xh = host_rows(np.random.default_rng(67).standard_normal((70, spec.d)), dtype)
        for tr, fn in ((False, orc.forward), (True, orc.transpose)):
            got, guards = gpu_apply(plan, xh, dtype, tr)
            assert guards and orc.rel_err_rows(got, fn(oplan, promote(xh, dtype))) <= TOL[dtype]
    p_out = wl.tiny_plan(68, (8, 8, 8), kind="qr", perm="identity", signs=True)
    p_in = wl.tiny_plan(69, (8, 8), kind="qr", perm="identity", signs=True)
    wh = host_rows(np.random.default_rng(70).standard_normal((p_out.d, p_in.d)), dtype)
    wd = to_device(wh, dtype)
    harp.two_sided_(wd, harp.plan_from_spec(p_out), harp.plan_from_spec(p_in))
    torch.cuda.synchronize()
    want = orc.two_sided(orc.OraclePlan.from_spec(p_out), orc.OraclePlan.from_spec(p_in), promote(wh, dtype))
    scale = np.minimum(np.linalg.norm(want, axis=1, keepdims=True), np.linalg.norm(want, axis=0, keepdims=True))
    assert np.max(np.abs(to_host_f64(wd) - want) / scale) <= 2 * TOL[dtype]


def _launches(call):
    before = harp.harp_launch_count()
    call()
    torch.cuda.synchronize()
    return harp.harp_launch_count() - before


def test_covers_with_and_without_register_passes():
    """A third pass in place of a wide tile of one row a lane, where no pass with its block kernels in registers takes part: rows of
    radices (8, 8, 15, 10) 31 and 38 us, columns of (2, 2, 2, 2, 48, 2, 2, 2)."""
    plan = harp.plan_from_spec(wl.tiny_plan(72, (8, 8, 15, 10), kind="qr", perm="identity", signs=True))
    x = torch.zeros((48, plan.d), device="cuda")
    assert _launches(lambda: harp.apply_(plan, x)) == 3
    p_out = harp.plan_from_spec(wl.tiny_plan(73, (2, 2, 2, 2, 48, 2, 2, 2), kind="qr", perm="identity", signs=True))
    p_in = harp.plan_from_spec(wl.tiny_plan(74, (12, 11, 14, 2), kind="qr", perm="identity", signs=True))
    w, rows = torch.zeros((p_out.d, p_in.d), device="cuda"), torch.zeros((p_out.d, p_in.d), device="cuda")
    assert _launches(lambda: harp.two_sided_(w, p_out, p_in)) - _launches(lambda: harp.apply_(p_in, rows)) == 3


def test_permuted_rows_of_a_large_radix_take_the_faster_route():
    """256 rows of radices (4, 4, 15, 4) behind a random permutation: the whole-row kernel (20.7 us) and not a permutation and two passes (27.8)."""
    plan = harp.plan_from_spec(wl.tiny_plan(75, (4, 4, 15, 4), kind="qr", perm="random", signs=True))
    x = torch.zeros((256, plan.d), device="cuda")
    assert _launches(lambda: harp.apply_(plan, x)) == 1


@pytest.mark.parametrize("radices,n_rows", [((8, 8, 2, 8, 8), 300), ((4, 3, 4, 2, 4, 4, 7), 300), ((8, 5, 4, 8, 8), 400), ((2,) * 10 + (8,), 400)])
def test_batches_that_are_faster_in_passes_take_them(radices, n_rows):
    """Half a wave to a wave of the whole-row kernel: 42, 55, 49 and 38 us there, 27, 39, 35 and 15 in two passes."""
    plan = harp.plan_from_spec(wl.tiny_plan(76, radices, kind="qr", perm="identity", signs=True))
    x = torch.zeros((n_rows, plan.d), device="cuda")
    assert _launches(lambda: harp.apply_(plan, x)) == 2
