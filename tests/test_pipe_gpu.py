"""The two-pass path's kernels that are fed by bulk tensor copies, against the oracle at the edges of the batches they take (9 and 17
rows) and of their tiles (16, 32 and 64 rows): slabs of one, three, seven and eight 64-blocks, one and two upper phases of
every width, dense upper blocks of up to 32 and 48, and batches of several tiles per team of warps."""
import numpy as np
import pytest
import torch

import paper_2605_29843_b200 as harp
from oracle import c_oracle, harp_oracle as orc
from paper_2605_29843_b200 import workloads as wl
from harp_testlib import TOL, gpu_apply, host_rows, promote, to_device, to_host_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radices", [(8, 8, 16), (8, 8, 8, 8), (8, 8, 3, 16), (8, 8, 7, 5, 3), (8, 8, 8, 8, 2), (8, 8, 8, 8, 7), (16, 16, 7, 5),
                                     (16, 16, 43), (16, 16, 47), (8, 8, 8, 19)])
@pytest.mark.parametrize("n_rows", [8, 9, 16, 17, 31, 33, 65, 131, 2049, 6001])
def test_matches_the_oracle(radices, n_rows):
    check_rows(radices, n_rows)


@pytest.mark.parametrize("radices", [(8, 8, 8, 9, 2), (8, 8, 8, 10, 3), (8, 8, 8, 13, 2), (16, 16, 9, 2)])
@pytest.mark.parametrize("n_rows", [16, 17, 700])
def test_two_upper_phases_with_a_block_wider_than_eight(radices, n_rows):
    """Tiles of 32 positions read the fragments of two neighbouring groups of sixteen, which lie phase by phase within each group."""
    check_rows(radices, n_rows)


@pytest.mark.parametrize("radices,n_rows", [((8, 8, 8, 8, 8), 83), ((8, 8, 8, 8, 8), 84), ((8, 8, 6, 8, 8), 111), ((8, 8, 6, 8, 8), 112), ((8, 8, 4, 8, 8), 168)])
def test_slab_pass_in_front_of_an_upper_pass_of_even_radices(radices, n_rows):
    check_rows(radices, n_rows)


def check_rows(radices, n_rows):
    spec = wl.make_plan(81, int(np.prod(radices)), radices, "qr", perm="identity", signs=True)
    plan, oplan = harp.plan_from_spec(spec), orc.OraclePlan.from_spec(spec)
    xh = host_rows(np.random.default_rng(82).standard_normal((n_rows, spec.d)), "bf16")
    edges = [e for e in (0, 8, 16, 32, 64, 128, 1024, n_rows // 2, n_rows) if e <= n_rows]
    rows = np.unique(np.clip(np.concatenate([np.arange(e - 2, e + 2) for e in edges]), 0, n_rows - 1))
    for tr, fn in ((False, orc.forward), (True, orc.transpose)):
        got, guards = gpu_apply(plan, xh, "bf16", tr, harp.KERNEL_SPLIT)
        assert guards and harp.harp_plan_error_word(plan) == 0
        assert orc.rel_err_rows(got[rows], fn(oplan, promote(xh[rows], "bf16"))) <= TOL["bf16"]


@pytest.mark.parametrize("out_radices", [(16, 16, 8), (16, 8), (8, 8, 7, 16), (8, 8, 8, 5, 2), (8, 8, 5, 4)])
@pytest.mark.parametrize("in_radices", [(8,), (9, 8), (8, 8, 5), (8, 8, 8, 8, 3)])
def test_columns_match_the_oracle(out_radices, in_radices):
    """The column side: slabs of three shapes, upper passes of one phase, 8 to 12288 columns (tiles of 64, the last one ragged)."""
    p_out = wl.make_plan(83, int(np.prod(out_radices)), out_radices, "qr", perm="identity", signs=True)
    p_in = wl.make_plan(84, int(np.prod(in_radices)), in_radices, "qr", perm="identity", signs=True)
    plan = harp.plan_from_spec(p_out)
    wh = host_rows(np.random.default_rng(85).standard_normal((p_out.d, p_in.d)), "bf16")
    wd = to_device(wh, "bf16")
    harp.two_sided_(wd, plan, harp.plan_from_spec(p_in))
    torch.cuda.synchronize()
    assert harp.harp_plan_error_word(plan) == 0
    want = c_oracle.two_sided(c_oracle.CPlan(p_out), c_oracle.CPlan(p_in), promote(wh, "bf16"))
    # an entry against the smaller norm of its row and column: one bound of the rows' test per side
    scale = np.minimum(np.linalg.norm(want, axis=1, keepdims=True), np.linalg.norm(want, axis=0, keepdims=True))
    assert np.max(np.abs(to_host_f64(wd) - want) / scale) <= 2 * TOL["bf16"]


@pytest.mark.parametrize("radices", [(16, 16, 8, 7), (8, 8, 8, 8, 7), (8, 8, 8, 8, 2), (8, 8, 8, 8, 8), (16, 16, 43), (8, 8, 8, 8)])
@pytest.mark.parametrize("transpose", [False, True])
def test_a_row_has_the_same_bits_in_every_batch(radices, transpose):
    """The kernels that take over at 9, 17, 384 rows and from the wide tiles on round where the others round, and sum in their order."""
    plan = harp.plan_from_spec(wl.make_plan(86, int(np.prod(radices)), radices, "qr", perm="identity", signs=True))
    x = torch.randn((4099, plan.d), generator=torch.Generator(device="cuda").manual_seed(87), device="cuda").to(torch.bfloat16)
    want = harp.apply_(plan, x.clone(), transpose, harp.KERNEL_SPLIT)
    for n_rows in (1, 8, 9, 16, 17, 100, 383, 384, 700):
        got = harp.apply_(plan, x[:n_rows].clone(), transpose, harp.KERNEL_SPLIT)
        assert torch.equal(got.view(torch.int16), want[:n_rows].view(torch.int16)), n_rows
