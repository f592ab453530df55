"""The fp32 passes that keep their block kernels in registers, and the register-tiled stage of radix 17 to 48, against the oracle: every
shape there is a kernel for, batches around the tiles of one, two and four rows (56 and 64 for the large radices), ragged column tiles."""
import numpy as np
import pytest
import torch

import paper_2605_29843_b200 as harp
from oracle import harp_oracle as orc
from paper_2605_29843_b200 import workloads as wl
from harp_testlib import TOL, gpu_apply, host_rows, promote, to_device, to_host_f64

pytestmark = pytest.mark.gpu


def _rows_match(radices, perm, n_rows):
    spec = wl.tiny_plan(81, radices, kind="qr", perm=perm, signs=True)
    plan, oplan = harp.plan_from_spec(spec), orc.OraclePlan.from_spec(spec)
    xh = host_rows(np.random.default_rng(82).standard_normal((n_rows, spec.d)), "f32")
    for tr, fn in ((False, orc.forward), (True, orc.transpose)):
        got, guards = gpu_apply(plan, xh, "f32", tr)
        assert guards
        assert orc.rel_err_rows(got, fn(oplan, promote(xh, "f32"))) <= TOL["f32"]
    assert harp.harp_plan_error_word(plan) == 0


@pytest.mark.parametrize("n_rows", [1, 3, 300])
@pytest.mark.parametrize("radices,perm", [
    ((8, 8, 8, 8), "identity"), ((8, 8, 8, 8), "random"),      # three stages in a row, one at runs of 256
    ((8, 8, 8, 5, 2), "identity"),        # a last group of coordinates that is half a tile; units of ten
    ((8, 8, 8, 8, 2), "identity"),
    ((4, 4, 4, 4, 4, 4), "identity"),
    ((2,) * 8 + (11,), "identity"),       # a group of three quarters of a tile
    ((8, 8, 8, 8, 7), "identity"),        # 224 of 256 threads own a unit of eight
    ((8, 8, 8, 8, 8), "identity"),
    ((16, 16, 8, 7), "identity"), ((16, 16, 43), "random"),    # units of sixteen shared by four threads
])
def test_passes_in_registers(monkeypatch, radices, perm, n_rows):
    monkeypatch.setenv("HARP_F32_PASSES", "1")
    _rows_match(radices, perm, n_rows)


@pytest.mark.parametrize("radices,n_rows", [((8, 8, 8), 1), ((8, 8, 8), 5), ((8, 8, 8), 4801), ((4, 4, 4), 33), ((4, 4, 4), 9473), ((2,) * 8, 7), ((8, 8, 8, 8), 1201)])
def test_whole_rows_as_one_run_and_tiles_of_four(monkeypatch, radices, n_rows):
    """Rows shorter than a tile: several to a tile, the last one in part; batches that take two and four vectors a tile."""
    monkeypatch.setenv("HARP_F32_PASSES", "1")
    _rows_match(radices, "identity", n_rows)


@pytest.mark.parametrize("n_rows", [1, 56, 65, 400])
@pytest.mark.parametrize("radices", [(16, 16, 43), (16, 16, 17), (4, 4, 33, 2), (16, 2, 32), (16, 48), (16, 41, 3)])
def test_large_radices(monkeypatch, radices, n_rows):
    monkeypatch.setenv("HARP_F32_PASSES", "1")
    _rows_match(radices, "identity", n_rows)


@pytest.mark.parametrize("r_out", [(8, 8), (8, 8, 8), (8, 8, 8, 2), (2,) * 11, (4, 4, 4, 4, 4, 4), (8, 8, 5, 2)])
@pytest.mark.parametrize("r_in", [(4, 3), (4, 33), (4, 4, 13)])
def test_columns(monkeypatch, r_out, r_in):
    """12, 132 and 208 columns: less than a tile of 128, one and a ragged one."""
    monkeypatch.setenv("HARP_F32_PASSES", "1")
    p_out = wl.tiny_plan(83, r_out, kind="qr", perm="identity", signs=True)
    p_in = wl.tiny_plan(84, r_in, kind="qr", perm="identity", signs=True)
    wh = host_rows(np.random.default_rng(85).standard_normal((p_out.d, p_in.d)), "f32")
    wd = to_device(wh, "f32")
    plan_out = harp.plan_from_spec(p_out)
    harp.two_sided_(wd, plan_out, harp.plan_from_spec(p_in))
    torch.cuda.synchronize()
    want = orc.two_sided(orc.OraclePlan.from_spec(p_out), orc.OraclePlan.from_spec(p_in), promote(wh, "f32"))
    # two sides, each within the one-sided tolerance of the row (column) norm
    scale = np.minimum(np.linalg.norm(want, axis=1, keepdims=True), np.linalg.norm(want, axis=0, keepdims=True))
    assert np.max(np.abs(to_host_f64(wd) - want) / scale) <= 2 * TOL["f32"]
    assert harp.harp_plan_error_word(plan_out) == 0
