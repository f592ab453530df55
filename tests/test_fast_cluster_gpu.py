"""The whole-row kernel with a cluster of two to sixteen CTAs per tile (small batches), against the oracle: every
position of the exchange between phases (before the last phase, after the first, both for a digit reversal), phases of width 8
and 16, ragged tiles, and row counts on both sides of the cluster sizes' limits."""
import numpy as np
import pytest
import torch

import paper_2605_29843_b200 as harp
from oracle import harp_oracle as orc
from paper_2605_29843_b200 import workloads as wl
from harp_testlib import TOL, gpu_apply, host_rows, promote

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radices,perm", [((4,) * 6, "digit_reversal"), ((8, 8, 8, 8), "identity"), ((16, 16, 16), "identity"),
                                          ((2, 2, 2, 2, 8, 16), "digit_reversal"), ((16, 8, 16), "identity")])
@pytest.mark.parametrize("n_rows", [1, 17, 240, 241, 528, 529, 1190])
def test_clusters_match_the_oracle(radices, perm, n_rows):
    spec = wl.make_plan(71, int(np.prod(radices)), radices, "qr", perm=perm)
    plan, oplan = harp.plan_from_spec(spec), orc.OraclePlan.from_spec(spec)
    xh = host_rows(np.random.default_rng(72).standard_normal((n_rows, spec.d)), "bf16")
    rows = np.unique(np.clip(np.r_[0:3, 14:18, n_rows // 2, n_rows - 3:n_rows], 0, n_rows - 1))
    for tr, fn in ((False, orc.forward), (True, orc.transpose)):
        got, guards = gpu_apply(plan, xh, "bf16", tr, harp.KERNEL_FAST)
        assert guards
        assert orc.rel_err_rows(got[rows], fn(oplan, promote(xh[rows], "bf16"))) <= TOL["bf16"]


def test_same_bits_as_one_cta_per_tile():
    """The same rows inside a batch too large for clusters give the same bits: only who computes what differs."""
    spec = wl.make_plan(73, 4096, (4,) * 6, "qr", perm="digit_reversal")
    plan = harp.plan_from_spec(spec)
    x = torch.randn((2400, 4096), device="cuda").to(torch.bfloat16)
    for tr in (False, True):
        big, small = x.clone(), x[:200].clone()
        harp.apply_(plan, big, transpose=tr, kernel=harp.KERNEL_FAST)
        harp.apply_(plan, small, transpose=tr, kernel=harp.KERNEL_FAST)
        assert torch.equal(big[:200], small)


@pytest.mark.parametrize("radices,perm", [((4,) * 6, "digit_reversal"), ((16, 16, 16), "identity"), ((8, 8, 8, 8), "identity"),
                                          ((2,) * 11, "identity")])
def test_same_bits_at_every_cluster_size(radices, perm):
    """One row to a few tiles (sixteen, eight, four CTAs a tile; a last tile of one row, of some, of all sixteen): the bits of one CTA per
    tile, the row behind the batch untouched, and no wait given up."""
    spec = wl.make_plan(74, int(np.prod(radices)), radices, "qr", perm=perm)
    plan = harp.plan_from_spec(spec)
    x = torch.randn((2400, spec.d), device="cuda").to(torch.bfloat16)
    for tr in (False, True):
        big = x.clone()
        harp.apply_(plan, big, transpose=tr, kernel=harp.KERNEL_FAST)
        for n in (1, 2, 8, 9, 15, 16, 17, 64, 97, 112, 113, 128, 129, 145, 250, 300):
            small = x[:n + 1].clone()
            harp.apply_(plan, small[:n], transpose=tr, kernel=harp.KERNEL_FAST)
            assert torch.equal(small[:n], big[:n]) and torch.equal(small[n], x[n]), n
    assert harp.harp_plan_error_word(plan) == 0
